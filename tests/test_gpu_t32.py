"""The FP32 field of dense contexts on the tensor cores (three BF16 terms per
operand, six products, accumulators drained into FP32): edges of its tiles
and of its split and fused forms, runs cut into calls, and the values its
terms cannot hold, which the SGEMM serves.

Tolerance of the field, per element, against FP64 with the operands as given:
the products left out are below 2^-22 |q s|, a drained block is cut off by at
most an ulp per accumulated product group (2^-22 of its products), and the
additions of the blocks round n / 64 times:
(2^-21 + (n / 64 + 4) 2^-24) sum_j |q_ij s_j|."""
import numpy as np
import pytest

from paper_2501_19221_gb300 import instances as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


def _ctx(B, n, seed=0):
    J, _ = I.sk_qubo(n, seed=seed)
    return B.veloxq_create_ising_dense(J), torch.from_numpy(J).cuda().double()


def _field(B, ctx, S):
    F = torch.full_like(S, 7.0)
    B.veloxq_field_dev(ctx, S.shape[0], B.VELOXQ_PREC_FP32, S, F)
    torch.cuda.synchronize()
    return F


@pytest.mark.parametrize("n,R", [(192, 1), (193, 63), (255, 64), (257, 65), (600, 129), (1031, 128), (2049, 40),
                                 (2600, 300), (3001, 641)])
def test_field_against_fp64(B, n, R):
    ctx, Q = _ctx(B, n)
    g = torch.Generator(device="cuda").manual_seed(n)
    S = torch.rand(R, n, generator=g, device="cuda") * 2 - 1
    F = _field(B, ctx, S).double()
    ref = S.double() @ Q
    tol = (2.0 ** -21 + (n / 64 + 4) * 2.0 ** -24) * (S.double().abs() @ Q.abs())
    assert bool(((F - ref).abs() <= tol).all())
    assert float((F - ref).norm() / ref.norm()) <= 1e-6


@pytest.mark.parametrize("method", [0, 1, 2])
@pytest.mark.parametrize("n,R", [(700, 100), (2600, 520)])      # split and fused form
def test_runs_cut_into_calls(B, n, R, method):
    """Five steps in one call, one by one, and two then three: the same bits, and the oracle's update of the field
    that the call reports for its last step."""
    ctx, _ = _ctx(B, n)
    sched = B.make_schedule(c0=1.0, method=method)
    S0 = torch.rand(R, n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1)) * 0.4 - 0.2
    Y0 = torch.zeros_like(S0)
    out = []
    for cuts in ([5], [1, 1, 1, 1, 1], [2, 3]):
        S, Y, F = S0.clone(), Y0.clone(), torch.empty_like(S0)
        k = 0
        for c in cuts:
            B.veloxq_steps_dev(ctx, R, k, c, 20, sched, S, Y, F)
            k += c
        torch.cuda.synchronize()
        out.append((S, Y, F))
    for o in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], o))


@pytest.mark.parametrize("n,R", [(300, 5), (2600, 520)])
def test_integer_field_is_exact(B, n, R):
    rng = np.random.default_rng(3)
    U = np.triu(rng.integers(-1000, 1001, size=(n, n)), 1)
    Q = (U + U.T).astype(np.int32)
    ctx = B.veloxq_create_dense(Q)
    S = torch.from_numpy(rng.choice([-1.0, 1.0], size=(R, n)).astype(np.float32)).cuda()
    F = _field(B, ctx, S).cpu().numpy()
    assert np.array_equal(F, (S.cpu().numpy().astype(np.int64) @ Q.astype(np.int64)).astype(np.float32))


@pytest.mark.parametrize("value", [float("inf"), float("nan"), 3.0e38, 1.0e-36])
def test_values_outside_the_terms(B, value):
    """A state holding such a value is served by the SGEMM: the others' fields keep their accuracy, and an infinity
    gives infinities where its coupling is not zero."""
    n, R = 700, 66
    ctx, Q = _ctx(B, n)
    S = torch.rand(R, n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2)) * 2 - 1
    S[5, 11] = value
    F = _field(B, ctx, S)
    keep = torch.arange(R, device="cuda") != 5
    ref = S.double() @ Q
    tol = 1e-5 * (S.double().abs() @ Q.abs())
    assert bool(((F.double() - ref).abs() <= tol)[keep].all())
    other = torch.arange(n, device="cuda") != 11
    if np.isfinite(value):
        assert bool(((F.double() - ref).abs() <= tol)[5].all())
    elif np.isinf(value):
        assert torch.equal(F[5, other], torch.sign(Q[11, other]).float() * value)
        assert bool(torch.isnan(F[5, 11]))
    else:
        assert bool(torch.isnan(F[5]).all())
    # the same through a step, and a clean state afterwards takes the tensor cores again
    sched = B.make_schedule(c0=1.0)
    S1, Y1 = S.clone(), torch.zeros_like(S)
    B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, S1, Y1)
    S[5, 11] = 0.25
    F2 = _field(B, ctx, S)
    torch.cuda.synchronize()
    ref = S.double() @ Q
    assert float((F2.double() - ref).norm() / ref.norm()) <= 1e-6


def test_couplings_outside_the_terms(B):
    """Couplings below 2^-100: the context keeps the SGEMM."""
    n, R = 256, 8
    J, _ = I.sk_qubo(n, seed=1)
    J = J.astype(np.float64) * 2.0 ** -105
    ctx = B.veloxq_create_ising_dense(J)
    S = torch.rand(R, n, device="cuda") * 2 - 1
    F = _field(B, ctx, S)
    ref = S.double() @ torch.from_numpy(J).cuda()
    assert float((F.double() - ref).norm() / ref.norm()) <= 1e-5
