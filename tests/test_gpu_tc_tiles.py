"""The tensor-core step's tile widths (256, 128 or 64 replicas, chosen by the
sizes): a replica's field and steps have the same bits whichever width its
run takes."""
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


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("n,wide,parts", [(2300, 2560, [1, 63, 64, 65, 128, 200, 640]), (530, 300, [16, 64, 129])])
def test_widths_agree(B, n, wide, parts, prec):
    J, _ = I.sk_qubo(n, seed=4)
    ctx = B.veloxq_create_ising_dense(J)
    g = torch.Generator(device="cuda").manual_seed(n)
    S = torch.rand(wide, n, generator=g, device="cuda") * 2 - 1
    Y = torch.rand(wide, n, generator=g, device="cuda") * 0.2 - 0.1
    sched = B.make_schedule(prec=prec, c0=1.0)

    def run(R):
        F, s, y = torch.empty(R, n, device="cuda"), S[:R].clone(), Y[:R].clone()
        B.veloxq_field_dev(ctx, R, prec, s, F)
        B.veloxq_steps_dev(ctx, R, 0, 5, 40, sched, s, y)
        torch.cuda.synchronize()
        return F, s, y

    ref = run(wide)
    for R in parts:
        assert all(torch.equal(a, b[:R]) for a, b in zip(run(R), ref))
