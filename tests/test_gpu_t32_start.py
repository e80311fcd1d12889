"""FP32 solves of dense instances whose start state is too large for the BF16
terms: the library's solve gives what its pieces give (the start state, and
steps that check their range)."""
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


@pytest.mark.parametrize("n,R", [(600, 12), (2600, 520)])
def test_largest_start_states(B, n, R):
    J, _ = I.sk_qubo(n, seed=0)
    ctx = B.veloxq_create_ising_dense((1e-3 * J).astype(np.float32))     # no field overflows
    sigma0 = float(np.finfo(np.float32).max)
    sched = B.make_schedule(sigma0=sigma0, c0=1.0, readout_every=0)
    got = B.veloxq_solve(ctx, R, 1, sched, seed=1)
    S, Y = torch.empty(R, n, device="cuda"), torch.empty(R, n, device="cuda")
    B.veloxq_init_state_dev(ctx, R, 1, sigma0, S, Y)
    B.veloxq_steps_dev(ctx, R, 0, 1, 1, sched, S, Y)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(S).all())
    X = (S > 0).to(torch.uint8).cpu().numpy()
    assert np.array_equal(got["E_per_replica"], B.veloxq_energy(ctx, X)["E"])


@pytest.mark.parametrize("n,R", [(700, 20), (2600, 520)])
def test_state_that_overflows_within_a_call(B, n, R):
    """Adiabatic SB has no walls: variable 11 of replica 3 starts at 1e12 and is infinite after two steps. The field of
    the third step is that of the FP32 sums of products (which a replica outside the terms' range selects): infinite
    with the coupling's sign, undefined for the variable itself, and the other replicas are not touched."""
    J, _ = I.sk_qubo(n, seed=0)
    ctx = B.veloxq_create_ising_dense(J)
    sched = B.make_schedule(c0=1.0, method=1)
    g = torch.Generator(device="cuda").manual_seed(1)
    S = torch.rand(R + 1, n, generator=g, device="cuda") * 0.2 - 0.1
    S[3, 11] = 1e12
    S[R, 5] = 1e-36
    out = []
    for r in (R, R + 1):
        s, y = S[:r].clone(), torch.zeros(r, n, device="cuda")
        f = torch.empty_like(s)
        B.veloxq_steps_dev(ctx, r, 0, 3, 20, sched, s, y, f)
        torch.cuda.synchronize()
        out.append(f[:R])
    a, b = out
    other = torch.arange(n, device="cuda") != 11
    assert bool(torch.isinf(b[3, other]).all())
    assert torch.equal(a[3, other], b[3, other]) and bool(torch.isnan(a[3, 11])) and bool(torch.isnan(b[3, 11]))
    keep = torch.arange(R, device="cuda") != 3
    assert bool(torch.isfinite(a[keep]).all())
    assert float((a[keep] - b[keep]).norm() / b[keep].norm()) <= 1e-5


def test_replays_of_a_captured_field_are_checked_one_by_one(B):
    """A replay whose state is outside the terms' range is served by the FP32 sums; the next replay with an ordinary
    state gives the tensor cores' bits again."""
    n, R = 600, 40
    J, _ = I.sk_qubo(n, seed=0)
    ctx = B.veloxq_create_ising_dense(J)
    g = torch.Generator(device="cuda").manual_seed(1)
    S0 = torch.rand(R, n, generator=g, device="cuda") * 2 - 1
    S, F = S0.clone(), torch.empty_like(S0)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        B.veloxq_field_dev(ctx, R, B.VELOXQ_PREC_FP32, S, F)
        side.synchronize()
        want = F.clone()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        B.veloxq_field_dev(ctx, R, B.VELOXQ_PREC_FP32, S, F)
        graph.capture_end()
        for value in (None, float("inf"), None):
            S.copy_(S0)
            if value is not None:
                S[2, 7] = value
            F.zero_()
            graph.replay()
            side.synchronize()
            if value is None:
                assert torch.equal(F, want)
            else:
                assert bool(torch.isinf(F[2]).any()) and bool(torch.isfinite(F[3]).all())
