"""Exact energies of dense instances from the digit-tile kernel (64-row x
64-replica tiles, base-4096 digits) at the edges of its tiles, for every
element type, against the oracle: bit-exact int64 for integer instances, the
fixed-point rounding bound for real ones."""
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


# element type and largest magnitude: one digit, the largest values of two digits' 23 bits, three digits, and the
# real types' four to six
RANGES = [(np.int8, 127), (np.int32, 2 ** 22 - 1), (np.int32, 2 ** 30), (np.float32, 3.0), (np.float64, 3.0)]


@pytest.mark.parametrize("dtype,m", RANGES)
@pytest.mark.parametrize("n,batch", [(1, 1), (2, 65), (63, 64), (64, 63), (65, 130), (129, 1), (200, 65)])
def test_tiles(B, n, batch, dtype, m):
    rng = np.random.default_rng(n * 1000 + batch)
    if np.issubdtype(dtype, np.integer):
        Q = rng.integers(-m, m + 1, size=(n, n)).astype(dtype)
        Q[0, :] = np.array([1023, -1024, 1024, m, -m])[np.arange(n) % 5] if dtype == np.int32 else Q[0, :]
    else:
        Q = (rng.normal(size=(n, n)) * 10.0 ** rng.uniform(-4, 0, size=(n, n)) * m).astype(dtype)
    c = rng.integers(-50, 51, size=n).astype(np.float64)
    ctx = B.veloxq_create_dense(Q, c)
    X = I.random_binary(batch, n, seed=5)
    Xd = torch.as_tensor(X, device="cuda")
    integer = bool(ctx.info.is_integer)
    assert integer == np.issubdtype(dtype, np.integer)
    p = O.problem_from_dense(Q.astype(np.float64) if not integer else Q, c)
    ref = O.energy(p, X)
    for fn in (B.veloxq_energy_dev, B.veloxq_energy_dev_noalloc):
        E = torch.empty(batch, dtype=torch.float64, device="cuda")
        Ei = torch.empty(batch, dtype=torch.int64, device="cuda") if integer else None
        fn(ctx, Xd, E, Ei)
        torch.cuda.synchronize()
        if integer:
            assert np.array_equal(Ei.cpu().numpy(), ref)
        else:
            # each weight is rounded once to the fixed-point grid; the oracle's FP64 sum rounds per term
            q = O.Problem(p.n, p.er, p.ec, np.abs(p.ev), np.abs(p.c))
            tol = (p.nnz + p.n) * 2.0 ** -52 * O.energy(q, X)
            assert np.all(np.abs(E.cpu().numpy() - ref) <= tol)
