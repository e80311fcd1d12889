"""Exact energies of sparse instances, 32 vectors per block from packed words,
at the edges of its range (vectors per block, rows per group, the largest n),
against the oracle: bit-exact for integer couplings, within the fixed-point
rounding for real ones; the no-allocation entry point gives the same."""
import numpy as np
import pytest

import oracle as O
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


@pytest.mark.parametrize("vtype", [np.int32, np.float32])
@pytest.mark.parametrize("n,batch", [(1, 64), (7, 65), (63, 63), (65, 95), (700, 97), (11264, 481), (11265, 481), (2400, 99)])
def test_packed_energies(B, n, batch, vtype):
    sp = I.random_sparse_qubo(n, min(9.0, n - 1), seed=n, vtype=np.int32, lo=-60, hi=60, empty_rows=min(3, n // 2))
    val = sp.val.astype(vtype) if vtype == np.int32 else sp.val.astype(np.float32) * np.float32(0.37)
    c = np.random.default_rng(n).integers(-9, 10, size=n).astype(np.float64)
    ctx = B.veloxq_create_csr(n, sp.rowptr, sp.col, val, c)
    integer = bool(ctx.info.is_integer)
    assert integer == (vtype == np.int32)
    p = O.problem_from_csr(n, sp.rowptr, sp.col, val.astype(np.float64), c)
    X = I.random_binary(batch, n, seed=2)
    ref = O.energy(p, X)
    Xd = torch.as_tensor(X, device="cuda")
    for fn in (B.veloxq_energy_dev, B.veloxq_energy_dev_noalloc):
        E = torch.empty(batch, dtype=torch.float64, device="cuda")
        Ei = torch.empty(batch, dtype=torch.int64, device="cuda") if integer else None
        fn(ctx, Xd, E, Ei)
        torch.cuda.synchronize()
        if integer:
            assert np.array_equal(Ei.cpu().numpy(), np.asarray(ref).astype(np.int64))
        else:
            q = O.Problem(p.n, p.er, p.ec, np.abs(p.ev), np.abs(p.c))
            tol = (p.nnz + p.n) * 2.0 ** -52 * O.energy(q, X)
            assert np.all(np.abs(E.cpu().numpy() - ref) <= tol)
