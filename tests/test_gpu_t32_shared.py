"""FP32 runs of several steps on the tensor cores while another kernel holds
part of the GPU for longer than their waits last: the tiles go to the pairs of
SMs that are free, the run ends without an error, and its results are those of
an idle GPU, bit for bit."""
import numpy as np
import pytest

from paper_2501_19221_gb300 import instances as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RESIDENT = 1


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


@pytest.mark.parametrize("method", [0, 1, 2])
def test_solve_beside_a_long_kernel(B, method):
    # the long kernel: 64 replicas of a graph whose state stays on chip, one CTA per replica
    sp = I.chimera_ising(16, 16, 4, seed=1)
    holder = B.veloxq_create_ising_csr(sp.n, sp.rowptr, sp.col, sp.val, sp.lin)
    R, side = 64, torch.cuda.Stream()
    S, Y = torch.zeros(R, sp.n, device="cuda"), torch.zeros(R, sp.n, device="cuda")
    sched = B.make_schedule(c0=0.1, path=RESIDENT)

    def hold(steps):
        with torch.cuda.stream(side):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            B.veloxq_steps_dev(holder, R, 0, steps, steps, sched, S, Y)
            b.record()
        return a, b

    hold(1000)
    a, b = hold(20000)
    torch.cuda.synchronize()
    steps = int(20000 * 3000.0 / a.elapsed_time(b))     # about 3 s

    n, reps = 2600, 520                                 # 55 tiles: the form that runs all steps in one launch
    J, _ = I.sk_qubo(n, seed=2)
    ctx = B.veloxq_create_ising_dense(J)
    main = torch.cuda.Stream()
    B.veloxq_set_stream(ctx, main.cuda_stream)
    solve = lambda: B.veloxq_solve(ctx, reps, 40, B.make_schedule(c0=1.0, readout_every=20, method=method),
                                    seed=3)
    want = solve()
    torch.cuda.synchronize()
    _, end = hold(steps)
    got = solve()
    held = not end.query()
    torch.cuda.synchronize()
    assert np.array_equal(want["E_per_replica"], got["E_per_replica"])
    assert np.array_equal(want["x"], got["x"])
    assert held        # the solve ended beside the long kernel, not behind it
