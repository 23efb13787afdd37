"""GPU: solutions through the full SVD of matrices with exactly or numerically
zero singular values (the vector of a zero singular value may have no part to
normalise; a reflector of nothing but roundings).

Tolerances, with |dA| = n eps sigma_1 the backward error: a computed zero singular
value of up to |dA| adds at most |dA| / lambda^2 |f| to a Tikhonov solution, the
others move by less; eight times that is allowed.  A truncated solution moves by
|dA| / sigma_r^2 |f|, with the factor 1e3 of the other full-SVD tests."""
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


def _matrix(kind, n):
    g = np.random.default_rng(n).normal(size=(n, n))
    i = np.arange(n)
    if kind == "zero columns":
        g[:, n // 2:] = 0.0
    elif kind == "zero rows":
        g[n // 2:] = 0.0
    elif kind == "zero column":
        g[:, n // 3] = 0.0
    elif kind == "diagonal, some zero":
        g = np.diag(np.where(i % 3 == 0, 0.0, i + 1.0))
    elif kind == "diagonal, last zero":
        g = np.diag(np.where(i == n - 1, 0.0, i + 1.0))
    elif kind == "bidiagonal":
        g = np.diag(np.where(i == n // 2, 0.0, i + 1.0)) + np.diag(np.ones(n - 1), 1)
    elif kind == "equal columns":
        g = np.repeat(g[:, :(n + 1) // 2], 2, axis=1)[:, :n]
    return g


def _check(ctx, R, A):
    n = A.shape[0]
    lda = R.padded_lda(n, R.RBF_FP64)
    D = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
    D[:, :n] = torch.as_tensor(A, device="cuda")
    op = ctx.rbf_operator_init(torch.zeros((3, n), dtype=torch.float64, device="cuda"), n, n // 2, 1.0, 1.0, A=D,
                               lda=lda)
    f = np.random.default_rng(1).normal(size=n)
    fd = torch.as_tensor(f, device="cuda")
    U, s, Vt = np.linalg.svd(A)
    sig, coef = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    ctx.rbf_svd_full(op, sig)
    assert np.max(np.abs(sig.cpu().numpy() - s)) <= 8 * n * EPS * s[0]
    lam = 1e-3 * s[0]
    ctx.rbf_tikhonov(op, fd, R.RBF_FIXED, lam, coef)
    ref = Vt.T @ (s / (s**2 + lam**2) * (U.T @ f))
    assert np.linalg.norm(coef.cpu().numpy() - ref) <= 8 * n * EPS * s[0] / lam**2 * np.linalg.norm(f)
    r = int(np.sum(s > n * EPS * s[0]))
    ctx.rbf_tsvd(op, fd, r, coef)
    ref = Vt[:r].T @ ((U.T @ f)[:r] / s[:r])
    assert np.linalg.norm(coef.cpu().numpy() - ref) <= 1e3 * n * EPS * s[0] / s[r - 1] ** 2 * np.linalg.norm(f)


@pytest.mark.parametrize("n", [2, 33, 70, 160])
@pytest.mark.parametrize("kind", ["zero columns", "zero rows", "zero column", "diagonal, some zero",
                                  "diagonal, last zero", "bidiagonal", "equal columns"])
def test_zero_singular_values(ctx, R, kind, n):
    _check(ctx, R, _matrix(kind, n))


@pytest.mark.parametrize("n", [33, 160, 300])
def test_reflectors_of_roundings(ctx, R, n):
    """Rank 1 exactly: every step divides what is left by another 1e16, down to
    columns whose squares underflow."""
    _check(ctx, R, np.ones((n, n)))
    _check(ctx, R, np.outer(1.0 + np.arange(n) % 3, 2.0 ** (np.arange(n) % 5)))


@pytest.mark.parametrize("k", [-505, -470, 470, 500])
def test_ends_of_the_range(ctx, R, k):
    """Norms near the square roots of the smallest and the largest double."""
    g = np.random.default_rng(2).normal(size=(40, 40))
    n = 40
    lda = R.padded_lda(n, R.RBF_FP64)
    out = []
    for scale in (1.0, 2.0**k):
        D = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
        D[:, :n] = torch.as_tensor(g * scale, device="cuda")
        op = ctx.rbf_operator_init(torch.zeros((3, n), dtype=torch.float64, device="cuda"), n, n // 2, 1.0, 1.0, A=D,
                                   lda=lda)
        sig = torch.empty(n, dtype=torch.float64, device="cuda")
        V = torch.empty((n, n), dtype=torch.float64, device="cuda")
        ctx.rbf_svd_full(op, sig, None, None, V)
        V = V.cpu().numpy()
        assert np.max(np.abs(V @ V.T - np.eye(n))) <= 40 * n * EPS / 1e-3
        out.append(sig.cpu().numpy() / scale)
    assert np.max(np.abs(out[0] - out[1])) <= 8 * n * EPS * out[0][0]
