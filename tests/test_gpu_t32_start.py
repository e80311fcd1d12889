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
