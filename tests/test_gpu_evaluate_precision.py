"""GPU: the precision of the fixed-point reconstruction where its bounds are tightest:
c at the smallest share of the coordinates that the rule admits, domains off the
origin, coefficients of very different size in one CTA.

One term is off by at most 1 unit in N (N >= 2^53 where c is 2^-5 of the coordinates'
power of two, and twice that for every doubling of c), by a quarter of a unit of
2^64 in the product (with the largest coefficient of its stage at 2^61 or above)
and by the roundings to FP64: with N0 = 2^53 c / (2^-5 max) that is 2^-53 (1 + 2^53 / N0
+ 2 x 2^53 / N0) of itself."""
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


def _eval(ctx, R, X, P, co, c):
    n, m = X.shape[0], P.shape[0]
    op = ctx.rbf_operator_init(_dev(X.T), n, n // 2, c, 1.0, R.RBF_MATRIX_FREE, R.RBF_MIXED)
    u = torch.empty(m, dtype=torch.float64, device="cuda")
    ctx.rbf_evaluate(op, _dev(co), _dev(P.T), m, u)
    L = np.longdouble
    d = P[:, None, :].astype(L) - X[None].astype(L)
    phi = np.sqrt((d * d).sum(-1) + L(c) * L(c))
    return u.cpu().numpy(), phi @ co.astype(L), phi @ np.abs(co).astype(L)


def test_small_coefficients_beside_cancelling_ones(ctx, R):
    """64 pairs of equal nodes (two apart) with coefficients +1 and -1, which cancel
    exactly, then 128 nodes with coefficients of about 1e-12, all in one CTA (enough
    points that the nodes are not split): the small ones at full precision."""
    rng = np.random.default_rng(1)
    X = rng.uniform(0, 1, (256, 3))
    X[2:128:4], X[3:128:4] = X[0:128:4], X[1:128:4]
    co = np.r_[np.tile([1.0, 1.0, -1.0, -1.0], 32), 2.0**-40 * rng.normal(size=128)]
    P, m = rng.uniform(0, 1, (300000, 3)), 300000
    op = ctx.rbf_operator_init(_dev(X.T), 256, 128, 0.2, 1.0, R.RBF_MATRIX_FREE, R.RBF_MIXED)
    u = torch.empty(m, dtype=torch.float64, device="cuda")
    ctx.rbf_evaluate(op, _dev(co), _dev(P.T), m, u)
    L = np.longdouble
    d = P[:200, None, :].astype(L) - X[None, 128:].astype(L)
    phi = np.sqrt((d * d).sum(-1) + L(0.2) * L(0.2))
    ref, mag = phi @ co[128:].astype(L), phi @ np.abs(co[128:]).astype(L)
    assert np.all(np.abs(u[:200].cpu().numpy() - ref) <= 4 * 2.0**-53 * mag)


@pytest.mark.parametrize("n", [1, 2, 63])
@pytest.mark.parametrize("ratio", [2.0**-4.99, 2.0**-4, 0.4])
def test_one_term(ctx, R, n, ratio):
    """One coefficient of 1 (the others zero): the term itself, and no more roundings
    than those of the stage and of the sum over the partials."""
    rng = np.random.default_rng(2)
    X = rng.uniform(-0.9, 0.9, (n, 3))
    X[-1] = 0.9
    P = X[-1] + 1e-3 * rng.normal(size=(500, 3))
    co = np.zeros(n)
    co[-1] = 1.0
    c = 0.5 * ratio  # the coordinates are in [0.5, 1)
    u, ref, _ = _eval(ctx, R, X, P, co, c)
    edge = 2.0**-5 / ratio  # 2^53 / N0
    assert np.all(np.abs(u - ref) <= 2.0**-53 * (1 + 3 * edge) * ref)


@pytest.mark.parametrize("where,size,c", [(10.0, 0.5, 0.5), (1.0, 0.01, 1 / 32), (-3.0, 1.0, 0.13)])
def test_domain_off_the_origin(ctx, R, where, size, c):
    rng = np.random.default_rng(3)
    X, P = where + size * rng.uniform(-1, 0, (3000, 3)), where + size * rng.uniform(-1, 0, (140, 3))
    u, ref, mag = _eval(ctx, R, X, P, rng.normal(size=3000), c)
    # per term the bound at the edge of the rule, a rounding per stage and per partial
    # of sums that are well below the sum of magnitudes
    assert np.all(np.abs(u - ref) <= 2.0**-53 * 4 * mag)


@pytest.mark.parametrize("n,m,q", [(1, 70000, 1), (65, 70000, 9), (515, 70000, 17), (20001, 3, 1), (1025, 257, 2)])
def test_chunks(ctx, R, n, m, q):
    """Both ends of the rule for the centre chunks: more CTAs than one wave holds, and
    hundreds of chunks for a few points."""
    rng = np.random.default_rng(n)
    X, P, co = rng.uniform(0, 1, (n, 3)), rng.uniform(0, 1, (m, 3)), rng.normal(size=(q, n))
    op = ctx.rbf_operator_init(_dev(X.T), n, n // 2, 0.2, 1.0, R.RBF_MATRIX_FREE, R.RBF_MIXED)
    u = torch.full((q, m), float("nan"), dtype=torch.float64, device="cuda")
    ctx.rbf_evaluate_many(op, _dev(co), n, q, _dev(P.T), m, u)
    assert torch.isfinite(u).all()
    at = rng.choice(m, min(m, 40), replace=False)
    L = np.longdouble
    d = P[at][:, None, :].astype(L) - X[None].astype(L)
    phi = np.sqrt((d * d).sum(-1) + L(0.2) * L(0.2))
    ref, mag = co.astype(L) @ phi.T, np.abs(co).astype(L) @ phi.T
    assert np.all(np.abs(u.cpu().numpy()[:, at] - ref) <= 4 * 2.0**-53 * mag)
