"""One step of the FP32 tensor-core form against its definition: the field it
reports against FP64, and the state it leaves against the integrator in FP64
on that field, for every integrator, in the split and the fused form; and the
same through the FP32 sums of products that serve a state outside the terms'
range.

Tolerances: the field 2^-22 + (n / 64) 2^-24 of the sum of magnitudes (its
sums round n / 64 times, a few units cover the accumulators); the update
rounds at most 8 times, each by 2^-24 of the magnitudes it adds."""
import numpy as np
import pytest

from paper_2501_19221_gb300 import instances as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT, A0, C0, MOM, K, KB = 0.5, 1.0, 1.0, 0.9, 21, 4
A = A0 * KB / (K - 1)          # the default schedule rises from 0 to a0
BSB, ASB, PA = 0, 1, 2


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


def _setup(B, n, R, seed=1):
    J, _ = I.sk_qubo(n, seed=0)
    J = np.asarray(J)
    J = (np.triu(J, 1) + np.triu(J, 1).T).astype(np.float32)
    h = np.random.default_rng(2).uniform(-0.1, 0.1, n)
    ctx = B.veloxq_create_ising_dense(J, h)
    g = torch.Generator(device="cuda").manual_seed(seed)
    S = torch.rand(R, n, generator=g, device="cuda") * 2 - 1
    Y = torch.rand(R, n, generator=g, device="cuda") - 0.5
    return ctx, torch.from_numpy(J).cuda().double(), torch.from_numpy(h).cuda(), S, Y


def _step(B, ctx, S, Y, method):
    sched = B.make_schedule(dt=DT, a0=A0, c0=C0, method=method, momentum=MOM)
    s, y, f = S.clone(), Y.clone(), torch.empty_like(S)
    B.veloxq_steps_dev(ctx, S.shape[0], KB, 1, K, sched, s, y, f)
    torch.cuda.synchronize()
    return s.double(), y.double(), f.double()


def _update(method, F, b, S, Y):
    """(s, y, magnitudes of the sums) of one step in FP64; for bSB the wall's condition too."""
    s, y, phi = S.double(), Y.double(), -(F + b) / 2
    if method == PA:
        lam = (A0 - A) / A0
        m = MOM * y - DT * (lam * s - C0 * phi)
        mag = (MOM * y).abs() + DT * ((lam * s).abs() + C0 * (F.abs() + b.abs())) + s.abs()
        return (s + m).clamp(-1, 1), m, mag
    c = A0 - A + (s * s if method == ASB else 0.0)
    y1 = y + DT * (-c * s + C0 * phi)
    s1 = s + DT * A0 * y1
    mag = y.abs() + DT * ((c * s).abs() + C0 * (F.abs() + b.abs())) + s.abs()
    if method == BSB:
        out = s1.abs() > 1
        keep = (s1.abs() - 1).abs() > 1e-5          # beside the wall either side is right
        y1 = torch.where(out, torch.zeros_like(y1), y1)
        s1 = torch.where(out, torch.sign(s1), s1)
        mag = torch.where(keep, mag, torch.full_like(mag, float("inf")))
    return s1, y1, mag


def _operand(method, S):
    return torch.where(S > 0, 1.0, -1.0).double() if method == PA else S.double()


@pytest.mark.parametrize("method", [BSB, ASB, PA])
@pytest.mark.parametrize("n,R", [(700, 100), (701, 40), (2600, 520), (2603, 520)])
def test_field_and_update_of_one_step(B, n, R, method):
    ctx, Q, b, S, Y = _setup(B, n, R)
    s, y, F = _step(B, ctx, S, Y, method)
    o = _operand(method, S)
    ftol = (2.0 ** -22 + (n / 64) * 2.0 ** -24) * (o.abs() @ Q.abs())
    assert bool(((F - o @ Q).abs() <= ftol).all())
    s1, y1, mag = _update(method, F, b, S, Y)
    tol = 8 * 2.0 ** -24 * mag
    assert bool(((s - s1).abs() <= tol).all()) and bool(((y - y1).abs() <= tol).all())


@pytest.mark.parametrize("value", [1.0e-36, 3.0e38, float("inf"), float("nan")])
@pytest.mark.parametrize("n,R", [(700, 66), (2600, 520)])
def test_step_of_a_state_outside_the_terms(B, n, R, value):
    ctx, Q, b, S, Y = _setup(B, n, R, seed=3)
    S[5, 11] = value
    s, y, F = _step(B, ctx, S, Y, BSB)
    rest = torch.arange(R, device="cuda") != 5
    if value < 1.0:
        rest[:] = True
    o = S.double()[rest]
    ftol = 1e-5 * (o.abs() @ Q.abs())                # FP32 sums of products
    assert bool(((F[rest] - o @ Q).abs() <= ftol).all())
    s1, y1, mag = _update(BSB, F, b, S, Y)
    tol = 8 * 2.0 ** -24 * mag
    assert bool(((s - s1).abs() <= tol)[rest].all()) and bool(((y - y1).abs() <= tol)[rest].all())
    other = torch.arange(n, device="cuda") != 11
    if value == value:                               # the walls bring the others back, and end momenta there
        assert bool((s[5, other].abs() <= 1).all()) and bool(torch.isfinite(y[5, other]).all())
    else:
        assert bool(torch.isnan(s[5]).all())
