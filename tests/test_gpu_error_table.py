"""GPU: the labelling error table at the edges of its tiles (points per CTA,
lambdas per CTA, l per row), against a direct solve of the projected problem.

Tolerance: y = (B^T B + lambda^2 I)^-1 B^T b.  An SVD with backward error
C eps sigma_1 moves y by at most C eps (sigma_1 / lambda)^2 |b| / sigma_1; the
direct solve is a least-squares solve of [B; lambda I], whose error has the same
bound.  C = 100 covers both.  Compared for lambda >= 1e-4 sigma_1.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
L = 70


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    rng = np.random.default_rng(3)
    ctx = rbfkr.Context(0)
    st, _, _, alpha, beta = rbfkr.make_state(torch, 4, L)
    a = rng.uniform(0.2, 1.0, L) * np.logspace(0, -3, L)
    b = rng.uniform(0.2, 1.0, L + 1) * np.logspace(0, -3, L + 1)
    alpha.copy_(torch.as_tensor(a))
    beta.copy_(torch.as_tensor(b))
    st.steps_done = L
    yield ctx, st, a, b
    ctx.close()


def _table(setup, m, ells, stride, uref, G):
    ctx, st, _, _ = setup
    jp = (321 - 1) // stride + 1
    err = torch.full((len(ells), jp), -1.0, dtype=torch.float64, device="cuda")
    ctx.rbf_hkt_error_table(st, torch.as_tensor(G, device="cuda"), G.shape[1], m, torch.as_tensor(uref, device="cuda"),
                            ells, stride, err)
    return err.cpu().numpy()


@pytest.mark.parametrize("m", [1, 127, 128, 129, 333, 8193])
@pytest.mark.parametrize("ells,stride", [([1], 320), ([70, 1, 33], 64), ([2, 69, 70], 23)])
def test_tiles(setup, m, ells, stride):
    _, _, a, b = setup
    rng = np.random.default_rng(m)
    G = rng.normal(size=(L, m + 3))
    uref = rng.normal(size=m)
    E = _table(setup, m, ells, stride, uref, G)
    for e, l in enumerate(ells):
        B = np.zeros((l + 1, l))
        B[np.arange(l), np.arange(l)] = a[:l]
        B[np.arange(1, l + 1), np.arange(l)] = b[1:l + 1]
        s1 = np.linalg.svd(B, compute_uv=False)[0]
        for q in range(E.shape[1]):
            t = -16.0 + 16.0 * q * stride / 320
            if t < -4.0:
                continue
            lam = s1 * 10.0 ** t
            rhs = np.zeros(2 * l + 1)
            rhs[0] = b[0]
            y = np.linalg.lstsq(np.vstack([B, lam * np.eye(l)]), rhs, rcond=None)[0]
            ref = np.max(np.abs(G[:l, :m].T @ y - uref)) / np.max(np.abs(uref))
            gmax = np.max(np.linalg.norm(G[:l, :m], axis=0))
            dy = 100 * EPS * (s1 / lam) ** 2 * b[0] / s1 + l * EPS * np.linalg.norm(y)
            tol = gmax * dy / np.max(np.abs(uref)) + 4 * EPS * ref
            assert abs(E[e, q] - ref) <= tol, (l, q, E[e, q], ref)


@pytest.mark.parametrize("m", [100, 300])
def test_zero_reference(setup, m):
    """u = 0: a nonzero reconstruction anywhere gives infinity, none at all NaN."""
    G = np.zeros((L, m))
    uref = np.zeros(m)
    assert np.all(np.isnan(_table(setup, m, [5], 64, uref, G)))
    G[0, m - 1] = 1.0
    assert np.all(np.isinf(_table(setup, m, [5], 64, uref, G)))
