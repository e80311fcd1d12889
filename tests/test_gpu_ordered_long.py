"""Long solves of dense instances between the resident kernel's shared memory
and 512 variables: launched step by step instead of captured, in bounded
memory, with the resident kernel's bits; both sides of the bound on captured
launches (16384: one per step, three per readout, one at the end)."""
import os

import numpy as np
import pytest

from paper_2501_19221_gb300 import instances as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RESIDENT, DENSE = 1, 3


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


@pytest.mark.parametrize("steps,readout", [(4095, 1), (4096, 1), (16380, 0), (16381, 0), (16400, 5000)])
def test_same_bits_as_resident(B, steps, readout):
    J, _ = I.sk_qubo(300, seed=1)
    ctx = B.veloxq_create_ising_dense(J)
    out = []
    for path in (0, RESIDENT):
        out.append(B.veloxq_solve(ctx, 16, steps, B.make_schedule(readout_every=readout, path=path), seed=5))
        assert B.veloxq_last_timing(ctx).path == (path or DENSE)
    assert np.array_equal(out[0]["x"], out[1]["x"])
    assert np.array_equal(out[0]["E_per_replica"], out[1]["E_per_replica"])


def test_memory_of_a_long_run(B):
    J, _ = I.sk_qubo(300, seed=1)
    ctx = B.veloxq_create_ising_dense(J)
    sched = B.make_schedule(readout_every=1)
    B.veloxq_solve(ctx, 16, 10, sched, seed=5)

    def held():
        with open("/proc/self/statm") as f:
            return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")

    before = held()
    B.veloxq_solve(ctx, 16, 30000, sched, seed=5)       # 120001 launches: 1 GB if captured
    assert held() - before < 100 << 20
