"""GPU: full-SVD path at the edges of its bidiagonalization (pieces of 256 rows
of a column, blocks of 4 rows, one column per CTA) and of the blocked
application of the right reflectors (blocks of 32), on matrices with a known
answer.

Tolerances: backward-stable singular values agree with LAPACK's to a small
multiple of n eps sigma_1; with lambda a fraction t of sigma_1 the Tikhonov
solution moves by about n eps / t relative (1e3 times that allowed, as for the
other full-SVD tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    return rbfkr


@pytest.fixture(scope="module")
def ctx(R):
    c = R.Context(0)
    yield c
    c.close()


def _op(ctx, R, A):
    n = A.shape[0]
    lda = R.padded_lda(n, R.RBF_FP64) + 2
    D = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
    D[:, :n] = torch.as_tensor(A, device="cuda")
    return ctx.rbf_operator_init(torch.zeros((3, n), dtype=torch.float64, device="cuda"), n, n // 2, 1.0, 1.0, A=D,
                                 lda=lda)


@pytest.mark.parametrize("n", [2, 3, 4, 5, 31, 32, 33, 34, 63, 65, 151, 152, 153, 255, 257, 511, 516, 611])
def test_tikhonov_edges(ctx, R, n):
    rng = np.random.default_rng(n)
    A = rng.normal(size=(n, n)) * 10.0 ** -np.linspace(0, 6, n)
    f = rng.normal(size=n)
    op = _op(ctx, R, A)
    sig = torch.empty(n, dtype=torch.float64, device="cuda")
    fh = torch.empty(n, dtype=torch.float64, device="cuda")
    V = torch.empty((n, n), dtype=torch.float64, device="cuda")
    ctx.rbf_svd_full(op, sig, torch.as_tensor(f, device="cuda"), fh, V)
    U, s, Vt = np.linalg.svd(A)
    assert np.max(np.abs(sig.cpu().numpy() - s)) <= 8 * n * EPS * s[0]
    assert abs(np.linalg.norm(fh.cpu().numpy()) - np.linalg.norm(f)) <= 50 * n * EPS * np.linalg.norm(f) + 1e-13
    Vn = V.cpu().numpy().T
    assert np.max(np.abs(Vn.T @ Vn - np.eye(n))) <= max(1e-12, 40 * n * EPS / 1e-3)
    coef = torch.empty(n, dtype=torch.float64, device="cuda")
    t = 1e-3
    ctx.rbf_tikhonov(op, torch.as_tensor(f, device="cuda"), R.RBF_FIXED, t * s[0], coef)
    ref = Vt.T @ (s / (s**2 + (t * s[0]) ** 2) * (U.T @ f))
    assert np.linalg.norm(coef.cpu().numpy() - ref) <= 1e3 * n * EPS / t * np.linalg.norm(ref)


@pytest.mark.parametrize("kind", ["zero", "identity", "rank1", "bidiagonal"])
def test_degenerate_reflectors(ctx, R, kind):
    n = 70
    rng = np.random.default_rng(9)
    A = {"zero": np.zeros((n, n)), "identity": np.eye(n), "rank1": np.outer(rng.normal(size=n), rng.normal(size=n)),
         "bidiagonal": np.diag(np.arange(1.0, n + 1)) + np.diag(np.ones(n - 1), 1)}[kind]
    sig = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.rbf_svd_full(_op(ctx, R, A), sig)
    s = np.linalg.svd(A, compute_uv=False)
    assert np.max(np.abs(sig.cpu().numpy() - s)) <= 8 * n * EPS * max(s[0], 1.0)
