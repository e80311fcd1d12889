"""Calls on one context from several streams. A call that returns before its
kernels end leaves them on the context's scratch (the second state buffer,
operand copies, partial fields, transposed states), so a call on another
stream is ordered behind it. The first stream is held up by a timed sleep:
when the second call's work has ended, the first call's must have ended too."""
import numpy as np
import pytest

from paper_2501_19221_gb300 import instances as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HOLD = 100_000_000        # SM cycles, about 50 ms
STREAM, DENSE = 2, 3


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2501_19221_gb300 import binding
    return binding


def _dense(B, n):
    J, _ = I.sk_qubo(n, seed=n)
    return B.veloxq_create_ising_dense(J), n


def _sparse(B):
    sp = I.chimera_ising(4, 4, 4, seed=1)
    return B.veloxq_create_ising_csr(sp.n, sp.rowptr, sp.col, sp.val, sp.lin), sp.n


def _state(R, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(R, n, generator=g, device="cuda") * 2 - 1, torch.rand(R, n, generator=g, device="cuda") * 2 - 1


# the exits of a step call: in the resident kernel's order of sums, FP32 sums of products, FP32 tensor-core form,
# BF16, and sparse rows
STEPS = [("ordered", 300, {}), ("sgemm", 150, {"path": DENSE}), ("terms", 300, {"path": DENSE}),
         ("bf16", 300, {"prec": 1}), ("rows", 0, {"path": STREAM})]


@pytest.mark.parametrize("form,n,kw", STEPS, ids=[s[0] for s in STEPS])
def test_steps_on_two_streams(B, form, n, kw):
    ctx, n = _dense(B, n) if n else _sparse(B)
    R, odd = 17, 5
    sched = B.make_schedule(c0=1.0, **kw)

    def steps(S, Y):
        B.veloxq_steps_dev(ctx, R, 0, odd, 20, sched, S, Y)

    want = []
    for seed in (1, 2):                              # in turn (and everything allocated, the schedule uploaded)
        S, Y = _state(R, n, seed)
        steps(S, Y)
        torch.cuda.synchronize()
        want += [S, Y]
    (S1, Y1), (S2, Y2) = _state(R, n, 1), _state(R, n, 2)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        if form != "terms":                          # that form waits for its stream (the range of S)
            torch.cuda._sleep(HOLD)
        steps(S1, Y1)
        e1 = s1.record_event()
    with torch.cuda.stream(s2):
        steps(S2, Y2)
        e2 = s2.record_event()
    e2.synchronize()
    assert e1.query()
    assert all(torch.equal(a, b) for a, b in zip(want, (S1, Y1, S2, Y2)))


@pytest.mark.parametrize("n,prec", [(150, 0), (300, 0), (300, 1), (0, 0)])
def test_fields_on_two_streams(B, n, prec):
    ctx, n = _dense(B, n) if n else _sparse(B)
    R = 17
    S, _ = _state(R, n, 1)
    want, got = [], []
    for x in (S, -S):
        F = torch.empty_like(S)
        B.veloxq_field_dev(ctx, R, prec, x, F)
        torch.cuda.synchronize()
        want.append(F)
    streams, ends = [torch.cuda.Stream(), torch.cuda.Stream()], []
    xs = [S, -S]
    got = [torch.empty_like(S), torch.empty_like(S)]
    torch.cuda.synchronize()
    for q, st in enumerate(streams):
        with torch.cuda.stream(st):
            if q == 0:
                torch.cuda._sleep(HOLD)
            B.veloxq_field_dev(ctx, R, prec, xs[q], got[q])
            ends.append(st.record_event())
    ends[1].synchronize()
    assert ends[0].query()
    assert all(torch.equal(a, b) for a, b in zip(want, got))


def _held_steps(ctx, B, stream, R, S, Y, sched):
    """A step call behind the sleep; its end as an event."""
    with torch.cuda.stream(stream):
        torch.cuda._sleep(HOLD)
        B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, S, Y)
        return stream.record_event()


@pytest.mark.parametrize("default_first", [True, False])
def test_default_stream_and_another(B, default_first):
    """The legacy default stream orders itself only behind streams that ask for it; these do not."""
    ctx, n = _dense(B, 300)
    R, sched = 17, B.make_schedule(c0=1.0)
    states = [_state(R, n, s) for s in (1, 2)]
    B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, *_state(R, n, 1))
    torch.cuda.synchronize()
    pair = [torch.cuda.default_stream(), torch.cuda.Stream()]
    first, second = pair if default_first else pair[::-1]
    e1 = _held_steps(ctx, B, first, R, *states[0], sched)
    with torch.cuda.stream(second):
        B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, *states[1])
        e2 = second.record_event()
    e2.synchronize()
    assert e1.query()


def test_third_stream_waits_too(B):
    """A call in between that leaves nothing on the scratch does not end the wait for the first one."""
    ctx, n = _dense(B, 300)
    R, sched = 17, B.make_schedule(c0=1.0)
    states = [_state(R, n, s) for s in (1, 2, 3)]
    B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, *_state(R, n, 1))
    torch.cuda.synchronize()
    s1, s2, s3 = (torch.cuda.Stream() for _ in range(3))
    e1 = _held_steps(ctx, B, s1, R, *states[0], sched)
    with torch.cuda.stream(s2):
        B.veloxq_init_state_dev(ctx, R, 1, 0.1, *states[1])
    with torch.cuda.stream(s3):
        B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, *states[2])
        e3 = s3.record_event()
    e3.synchronize()
    assert e1.query()


def test_captured_call_waits_at_capture(B):
    ctx, n = _dense(B, 300)
    R, sched = 17, B.make_schedule(c0=1.0)
    S, F = _state(R, n, 1)[0], torch.empty(R, n, device="cuda")
    B.veloxq_field_dev(ctx, R, 0, S, F)              # buffers, so that the capture allocates nothing
    want = F.clone()
    X, Y = _state(R, n, 2)
    B.veloxq_steps_dev(ctx, R, 0, 1, 20, sched, X, Y)
    torch.cuda.synchronize()
    F.zero_()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    e1 = _held_steps(ctx, B, s1, R, X, Y, sched)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s2):
        graph.capture_begin()
        B.veloxq_field_dev(ctx, R, 0, S, F)
        graph.capture_end()
        assert e1.query()
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(F, want)


def test_batch_waits_for_steps_left_on_another_stream(B):
    """The contexts' streams were changed after the steps were left there; the batch takes their operand copies, state
    buffers and schedules."""
    ctxs = [_dense(B, n)[0] for n in (200, 300, 260)]
    R, n = 16, 260
    sched = B.make_schedule(c0=1.0, prec=1, readout_every=0)
    S, Y = _state(R, n, 1)
    B.veloxq_steps_dev(ctxs[2], R, 0, 3, 20, sched, S, Y)
    torch.cuda.synchronize()
    want = (S, Y, B.veloxq_solve_batch(ctxs, R, 20, sched, seed=4))
    S, Y = _state(R, n, 1)
    torch.cuda.synchronize()
    s1 = torch.cuda.Stream()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(HOLD)
        B.veloxq_steps_dev(ctxs[2], R, 0, 3, 20, sched, S, Y)
        e1 = s1.record_event()
    # not the default stream, which would wait for every other one
    s2 = torch.cuda.Stream()
    for c in ctxs:
        B.veloxq_set_stream(c, s2.cuda_stream)
    got = B.veloxq_solve_batch(ctxs, R, 20, sched, seed=4)
    assert e1.query()
    assert torch.equal(S, want[0]) and torch.equal(Y, want[1])
    assert np.array_equal(got["E"], want[2]["E"])
    assert all(np.array_equal(a, b) for a, b in zip(got["x"], want[2]["x"]))
