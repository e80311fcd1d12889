"""Dense instances of up to 512 variables whose couplings do not fit the
resident kernel's shared memory: the library's own choice of path sums each
field in the resident kernel's order, so that states, fields, energies and
the best vector are the resident kernel's, bit for bit. Sizes: both sides of
the variable tiles (32), of the stages (128) and of the rows' alignment (4),
replica tiles (16) with remainders."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

AUTO, RESIDENT, DENSE = 0, 1, 3


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


def _ctx(B, n, whole):
    rng = np.random.default_rng(n)
    Q = rng.integers(-100000, 100001, (n, n)) if whole else rng.standard_normal((n, n))
    Q = np.triu(Q)
    return B.veloxq_create_dense((Q + Q.T).astype(np.int32 if whole else np.float32))


@pytest.mark.parametrize("method", [0, 1, 2])
@pytest.mark.parametrize("n,R,whole", [(256, 1, True), (257, 17, True), (300, 16, False), (383, 12, True),
                                       (385, 33, False), (511, 128, True), (512, 40, False), (512, 1, True)])
def test_same_bits_as_resident(B, n, R, whole, method):
    ctx = _ctx(B, n, whole)
    out = []
    for path in (AUTO, RESIDENT):
        sched = B.make_schedule(readout_every=20, method=method, path=path)
        res = B.veloxq_solve(ctx, R, 70, sched, seed=5)
        if path == AUTO:
            assert B.veloxq_last_timing(ctx).path == DENSE
        g = torch.Generator(device="cuda").manual_seed(n)
        S = torch.rand(R, n, generator=g, device="cuda") * 2 - 1
        Y = torch.rand(R, n, generator=g, device="cuda") * 2 - 1
        F = torch.zeros_like(S)
        B.veloxq_steps_dev(ctx, R, 3, 4, 20, sched, S, Y, F)
        torch.cuda.synchronize()
        out.append((res, S, Y, F))
    (a, *ta), (b, *tb) = out
    assert np.array_equal(a["x"], b["x"]) and a["E"] == b["E"]
    assert np.array_equal(a["E_per_replica"], b["E_per_replica"])
    assert all(torch.equal(x, y) for x, y in zip(ta, tb))


@pytest.mark.parametrize("n,sigma0", [(320, 0.1), (256, 1e-30)])     # asked for: tensor cores; SGEMM
def test_chosen_and_asked_dense_path_take_turns(B, n, sigma0):
    """The captured loop of one is not replayed for the other: each solve launches what it launches on a new context
    and gives that context's energies."""
    ctx = _ctx(B, n, False)
    for path in (AUTO, DENSE, AUTO, DENSE):
        sched = B.make_schedule(readout_every=20, path=path, sigma0=sigma0)
        new = _ctx(B, n, False)
        a, b = (B.veloxq_solve(c, 17, 60, sched, seed=2) for c in (ctx, new))
        assert B.veloxq_last_timing(ctx).path == DENSE
        assert B.veloxq_last_timing(ctx).launches == B.veloxq_last_timing(new).launches
        assert np.array_equal(a["E_per_replica"], b["E_per_replica"])
