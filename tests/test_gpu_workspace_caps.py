"""GPU: calls under a workspace cap that holds what they cannot do without: partial
sums in fewer chunks, scratch of one phase in the place of another's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    return rbfkr


def test_evaluate(R):
    n, m = 1000, 2000
    rng = np.random.default_rng(1)
    X, P = (torch.as_tensor(rng.uniform(0, 1, (3, k)), device="cuda") for k in (n, m))
    co = torch.as_tensor(rng.normal(size=n), device="cuda")
    out = []
    for c in (0, 70 * 1024):  # room for four chunks
        ctx = R.Context(0, workspace_cap=c)
        op = ctx.rbf_operator_init(X, n, n // 2, 0.2, 1.0, R.RBF_MATRIX_FREE, R.RBF_MIXED)
        u = torch.empty(m, dtype=torch.float64, device="cuda")
        ctx.rbf_evaluate(op, co, P, m, u)
        out.append(u)
        torch.cuda.synchronize()
        ctx.close()
    # another order of the same sum: n roundings of at most the sum of magnitudes (|co| < 5, Phi < 2)
    assert (out[0] - out[1]).abs().max() <= n * 2.0**-53 * 10 * n


def test_gradient(R):
    g = torch.Generator(device="cuda").manual_seed(1)
    p = 0.1 * torch.randn(19458, generator=g, device="cuda")
    x, y = torch.randn((512, 20), generator=g, device="cuda"), torch.randn((512, 2), generator=g, device="cuda")
    out = []
    for c in (0, 1700 * 1024):
        ctx = R.Context(0, workspace_cap=c)
        grad = torch.empty_like(p)
        ctx.rbf_mlp_grad(p, x, y, 512, grad)
        out.append(grad)
        ctx.close()
    # both are exact sums but for one FP32 rounding
    assert (out[0] - out[1]).abs().max() <= 2.0**-23 * out[0].abs().max()


def test_full_svd(R):
    n = 1000
    rng = np.random.default_rng(2)
    D = torch.zeros((n, R.padded_lda(n, R.RBF_FP64)), dtype=torch.float64, device="cuda")
    D[:, :n] = torch.as_tensor(rng.normal(size=(n, n)), device="cuda")
    f = torch.as_tensor(rng.normal(size=n), device="cuda")
    out = []
    for c in (0, 88_200_000):
        ctx = R.Context(0, workspace_cap=c)
        op = ctx.rbf_operator_init(torch.zeros((3, n), dtype=torch.float64, device="cuda"), n, n // 2, 1.0, 1.0, A=D,
                                   lda=D.shape[1])
        coef = torch.empty(n, dtype=torch.float64, device="cuda")
        ctx.rbf_tikhonov(op, f, R.RBF_GCV, 0.0, coef)
        out.append(coef)
        ctx.close()
    assert torch.equal(out[0], out[1])
