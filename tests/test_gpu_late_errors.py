"""A bounded wait that gives up after its call has returned is reported once,
by whichever entry point comes next or by veloxq_synchronize, and the calls
after the report are valid again. The wait is the self-test's, made to run out
on the context's own error words."""
import numpy as np
import pytest

from paper_2501_19221_gb300 import instances as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, R = 300, 16


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    J, _ = I.sk_qubo(N, seed=0)
    return B.veloxq_create_ising_dense(J)


def _steps(B, ctx):
    g = torch.Generator(device="cuda").manual_seed(1)
    S = torch.rand(R, N, generator=g, device="cuda") * 2 - 1
    Y = torch.zeros_like(S)
    B.veloxq_steps_dev(ctx, R, 0, 4, 20, B.make_schedule(c0=1.0, prec=1), S, Y)
    return S, Y


def _energy(B, ctx, call):
    X = torch.zeros((4, N), dtype=torch.uint8, device="cuda")
    call(ctx, X, torch.empty(4, dtype=torch.float64, device="cuda"))


CALLS = {
    "synchronize": lambda B, c: B.veloxq_synchronize(c),
    "steps": _steps,
    "solve": lambda B, c: B.veloxq_solve(c, R, 10, B.make_schedule(prec=1), seed=0),
    "batch": lambda B, c: B.veloxq_solve_batch([c], R, 10, B.make_schedule(prec=1, readout_every=0), seed=0),
    "energy_dev": lambda B, c: _energy(B, c, B.veloxq_energy_dev),
    "energy_noalloc": lambda B, c: _energy(B, c, B.veloxq_energy_dev_noalloc),
}


@pytest.mark.parametrize("name", list(CALLS))
def test_reported_once_and_clean_afterwards(B, ctx, name):
    want = _steps(B, ctx)
    B.veloxq_synchronize(ctx)
    B.veloxq_selftest_timeout_async(ctx, 2_000)
    torch.cuda.synchronize()
    with pytest.raises(B.VeloxqError) as e:
        CALLS[name](B, ctx)
    assert e.value.status == B.VELOXQ_ETIMEDOUT and "code 8" in e.value.message
    got = _steps(B, ctx)
    B.veloxq_synchronize(ctx)
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    CALLS[name](B, ctx)


def test_last_call_is_asked_for(B, ctx):
    """The wait still runs when the caller asks, and steps issued behind it are among the invalid calls."""
    side = torch.cuda.Stream()
    want = _steps(B, ctx)
    B.veloxq_synchronize(ctx)
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)
        B.veloxq_selftest_timeout_async(ctx, 2_000_000)
        _steps(B, ctx)
        with pytest.raises(B.VeloxqError) as e:
            B.veloxq_synchronize(ctx)
        assert e.value.status == B.VELOXQ_ETIMEDOUT
        got = _steps(B, ctx)
        B.veloxq_synchronize(ctx)
    assert all(torch.equal(a, b) for a, b in zip(want, got))


def test_bad_arguments(B, ctx):
    for call in (lambda: B.veloxq_selftest_timeout_async(ctx, 10),):
        with pytest.raises(B.VeloxqError) as e:
            call()
        assert e.value.status == B.VELOXQ_EINVAL
    assert B._lib.veloxq_synchronize(None) == B.VELOXQ_EINVAL
