"""The streaming path's windows (the steps between two readouts run for one
window of replicas after the other when the state lies beyond L2): the same
bits as a form fixed by VELOXQ_STREAM_FORM, which runs all replicas at once,
for odd and even numbers of steps between readouts."""
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


@pytest.mark.parametrize("method,steps,readout", [(0, 30, 7), (2, 24, 8), (1, 13, 0)])
def test_windows_equal_all_at_once(B, monkeypatch, method, steps, readout):
    sp = I.tile_planted_ising(300, seed=1).sp
    R = 256
    sched = B.make_schedule(path=2, method=method, readout_every=readout)
    ctx = B.veloxq_create_ising_csr(sp.n, sp.rowptr, sp.col, sp.val, sp.lin)
    got = B.veloxq_solve(ctx, R, steps, sched, seed=3)
    t = B.veloxq_last_timing(ctx)
    assert 32 <= t.stream_chunk < R and t.main_launches > steps
    monkeypatch.setenv("VELOXQ_STREAM_FORM", "1 0")
    ref_ctx = B.veloxq_create_ising_csr(sp.n, sp.rowptr, sp.col, sp.val, sp.lin)
    ref = B.veloxq_solve(ref_ctx, R, steps, sched, seed=3)
    assert B.veloxq_last_timing(ref_ctx).main_launches == steps
    assert np.array_equal(got["E_per_replica"], ref["E_per_replica"])
    assert np.array_equal(got["x"], ref["x"]) and got["E_int"] == ref["E_int"]
