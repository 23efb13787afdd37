"""GPU: reconstruction in fixed point against extended precision, at the edges of
its tiles (128 points, 128 nodes, 1 to 8 vectors) and on both sides of the rule
that takes it (c against the largest coordinate; non-finite values).

Tolerance: a term of the fixed-point form is off by at most 2^-57 of the largest
Phi times the coefficient (2^-57.8 in Phi, 2^-61 in coordinates and
coefficients), of the FP64 form by about 4 ulps of itself; sums add one rounding
per chunk or term: n 2^-53 of the sum of magnitudes is never exceeded."""
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


@pytest.fixture(scope="module")
def ctx(R):
    c = R.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _eval(ctx, R, X, P, co, c, form=0):
    n, m = X.shape[0], P.shape[0]
    op = ctx.rbf_operator_init(_dev(X.T), n, n // 2, c, 1.0, R.RBF_MATRIX_FREE, R.RBF_MIXED, form)
    u = torch.full((co.shape[0], m), float("nan"), dtype=torch.float64, device="cuda")
    if co.shape[0] == 1:
        ctx.rbf_evaluate(op, _dev(co[0]), _dev(P.T), m, u[0])
    else:
        ctx.rbf_evaluate_many(op, _dev(co), n, co.shape[0], _dev(P.T), m, u)
    return u.cpu().numpy()


def _ref(X, P, co, c, scale=1.0):
    L = np.longdouble
    d = P[:, None, :].astype(L) - X[None].astype(L)
    phi = np.sqrt((d * d).sum(-1) + L(c) * L(c)) * L(scale)
    return co.astype(L) @ phi.T, np.abs(co).astype(L) @ np.ones_like(phi).T * phi.max(), np.abs(co).astype(L) @ phi.T


@pytest.mark.parametrize("n,m,q", [(1, 1, 1), (2, 127, 1), (127, 128, 2), (128, 129, 3), (129, 1, 4), (255, 33, 5),
                                   (257, 200, 8), (700, 300, 9), (1000, 131, 17)])
@pytest.mark.parametrize("form", [0, 1])
def test_sizes(ctx, R, n, m, q, form):
    rng = np.random.default_rng(n + m)
    X, P = rng.uniform(-1, 1, (n, 3)), rng.uniform(-1, 1, (m, 3))
    co = rng.normal(size=(q, n)) * 10.0 ** rng.uniform(-8, 8, (q, n))
    c = 0.21
    u = _eval(ctx, R, X, P, co, c, form)
    ref, big, mag = _ref(X, P, co, c, 1.0 / c if form else 1.0)
    # 2^-57 per term; a few roundings of the partials and of the scaled sum, none
    # of which is larger than the sum of magnitudes
    assert np.all(np.abs(u - ref) <= big * 2.0**-57 + mag * 2.0**-50)


@pytest.mark.parametrize("scale", [1.0, 3.0, 1e-150, 1e140])
@pytest.mark.parametrize("ratio", [8.0, 1.0, 2.0**-4.9, 2.0**-5.1, 2.0**-6.1, 1e-4])
def test_both_sides_of_the_rule(ctx, R, ratio, scale):
    rng = np.random.default_rng(3)
    n, m = 300, 150
    X, P = rng.uniform(-1, 1, (n, 3)) * scale, rng.uniform(-1, 1, (m, 3)) * scale
    X[0, 0] = scale  # the largest coordinate
    P[:40] = X[:40]  # the smallest distances
    co = rng.normal(size=(1, n))
    c = ratio * scale
    u = _eval(ctx, R, X, P, co, c)
    ref, _, mag = _ref(X, P, co, c)
    assert np.all(np.abs(u - ref) <= n * 2.0**-53 * mag)


def test_domain_far_from_the_origin(ctx, R):
    rng = np.random.default_rng(4)
    X, P = rng.uniform(0, 1, (400, 3)) + 1000.0, rng.uniform(0, 1, (90, 3)) + 1000.0
    co = rng.normal(size=(2, 400))
    u = _eval(ctx, R, X, P, co, 0.2)
    ref, _, mag = _ref(X, P, co, 0.2)
    assert np.all(np.abs(u - ref) <= 400 * 2.0**-53 * mag)


@pytest.mark.parametrize("where", ["node", "point", "coef"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite(ctx, R, where, bad):
    rng = np.random.default_rng(5)
    X, P, co = rng.uniform(0, 1, (200, 3)), rng.uniform(0, 1, (140, 3)), rng.normal(size=(1, 200))
    ref = _ref(X, P, co, 0.3)[0]
    if where == "node":
        X[7, 1] = bad
    elif where == "point":
        P[3, 2] = bad
    else:
        co[0, 9] = bad
    u = _eval(ctx, R, X, P, co, 0.3)
    if where == "point":
        ok = np.arange(140) != 3
        assert not np.isfinite(u[0, 3]) and np.all(np.abs(u[0, ok] - ref[0, ok]) < 1e-11)
    else:
        assert not np.isfinite(u).any()


def test_zero_coefficients(ctx, R):
    rng = np.random.default_rng(6)
    u = _eval(ctx, R, rng.uniform(0, 1, (150, 3)), rng.uniform(0, 1, (20, 3)), np.zeros((3, 150)), 0.3)
    assert np.all(u == 0.0)
