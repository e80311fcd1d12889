"""Sparse instances that just fill the resident kernel's shared memory (the
ELL layouts with six slots and with more): they run there, in one launch, and
the vector's energy is the one reported."""
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


# 232320, 232416 and 232368 of 232448 bytes with one replica per CTA
@pytest.mark.parametrize("n,d", [(6420, 6), (6423, 6), (1017, 54)])
def test_instances_that_fill_shared_memory(B, n, d):
    rng = np.random.default_rng(n)
    i = np.repeat(np.arange(n), d // 2)
    j = (i + np.tile(np.arange(1, d // 2 + 1), n)) % n          # a ring, each row coupled to its d nearest
    w = rng.choice([-1, 1], size=i.shape[0]).astype(np.int32)
    rowptr, col, val = I._csr_from_edges(n, np.minimum(i, j), np.maximum(i, j), w)
    ctx = B.veloxq_create_ising_csr(n, rowptr, col, val.astype(np.int32))
    out = B.veloxq_solve(ctx, 8, 40, B.make_schedule(readout_every=10), seed=1)
    assert B.veloxq_last_timing(ctx).path == RESIDENT
    assert B.veloxq_energy(ctx, out["x"])["E_int"][0] == out["E_int"]
