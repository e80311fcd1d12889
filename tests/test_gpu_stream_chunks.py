"""Steps over all replicas on a context whose solves run by windows of
replicas: their chunk order is tried (a random graph of 2e5 variables keeps
its gathers in L2 by it), before and after a solve by windows, and gives the
same bits as a fixed form."""
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


@pytest.mark.parametrize("windows_first", [False, True])
def test_steps_without_windows_keep_their_chunks(B, monkeypatch, windows_first):
    h = I.xorsat_3r3x(100000, seed=1).hubo
    r = B.veloxq_hubo3_reduce(h.n, h.h, h.pairs, h.triples)
    R = 256
    make = lambda: B.veloxq_create_ising_csr(r["n"], r["rowptr"], r["col"], r["val"], r["lin"])
    often, seldom = B.make_schedule(path=2, readout_every=2), B.make_schedule(path=2, readout_every=6)
    ctx = make()
    if windows_first:
        B.veloxq_solve(ctx, R, 12, seldom, seed=3)
        t = B.veloxq_last_timing(ctx)
        assert t.main_launches > 12                    # by windows
    got = B.veloxq_solve(ctx, R, 12, often, seed=3)
    t = B.veloxq_last_timing(ctx)
    assert t.main_launches == 12 and t.stream_chunk > 0
    again = B.veloxq_solve(ctx, R, 12, seldom, seed=3)
    assert B.veloxq_last_timing(ctx).main_launches > 12
    monkeypatch.setenv("VELOXQ_STREAM_FORM", "1 0")
    ref = make()
    for res, sched in ((got, often), (again, seldom)):
        want = B.veloxq_solve(ref, R, 12, sched, seed=3)
        assert np.array_equal(res["E_per_replica"], want["E_per_replica"])
        assert np.array_equal(res["x"], want["x"])
