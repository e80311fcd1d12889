"""The FP32 field of dense contexts where a sum has few terms: rows of one,
two and six couplings, and states of few variables on full rows (split and
fused form of the tensor-core kernel).

Tolerance per element, against FP64: a sum of k products in FP32 rounds k
times, each by at most 2^-24 of the sum of magnitudes; one more such unit
covers the term product that is left out (2^-29 of each product) and what the
accumulators cut off the small products (at most 2^-23 of these, which are
2^-5 of the whole)."""
import pytest

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


def _check(B, Q, S, k):
    ctx = B.veloxq_create_dense(Q.cpu().numpy())
    F = torch.empty_like(S)
    B.veloxq_field_dev(ctx, S.shape[0], B.VELOXQ_PREC_FP32, S, F)
    torch.cuda.synchronize()
    ref, mag = S.double() @ Q.double(), S.double().abs() @ Q.double().abs()
    assert float(((F.double() - ref).abs() / mag)[mag > 0].max()) <= (k + 1) * 2.0 ** -24
    assert bool((F[mag == 0] == 0).all())


@pytest.mark.parametrize("n,R", [(700, 100), (701, 40), (2600, 520)])
@pytest.mark.parametrize("k", [1, 2, 6])
def test_rows_of_few_couplings(B, n, R, k):
    g = torch.Generator(device="cuda").manual_seed(10 * n + k)
    Q = torch.zeros(n, n, device="cuda")
    for _ in range(k):                           # pairs of variables, k times
        p = torch.randperm(n, generator=g, device="cuda")
        a, b = p[:n // 2], p[n // 2:2 * (n // 2)]
        v = torch.randn(n // 2, generator=g, device="cuda")
        Q[a, b] = v
        Q[b, a] = v
    _check(B, Q, torch.rand(R, n, generator=g, device="cuda") * 2 - 1, k)


@pytest.mark.parametrize("n,R", [(700, 100), (2600, 520)])
def test_states_of_one_variable(B, n, R):
    g = torch.Generator(device="cuda").manual_seed(n)
    Q = torch.randn(n, n, generator=g, device="cuda").triu(1)
    S = torch.zeros(R, n, device="cuda")
    S[torch.arange(R), torch.randint(0, n, (R,), generator=g, device="cuda").cpu()] = \
        torch.rand(R, generator=g, device="cuda") * 2 - 1
    _check(B, Q + Q.T, S, 1)
