"""GPU: singular values and vectors of bidiagonals through the Golub-Kahan
tridiagonal, at the edges of its kernels (groups of 8 minors, warps of 32, 8 or
32 lanes per value) and on bidiagonals that stress the brackets: equal, tiny and
decoupled entries.

Tolerances, from first principles: a Sturm count is exact for a matrix whose
entries differ by a few eps relative, which moves a singular value of an
l-dimensional bidiagonal by at most about 4 l eps sigma; LAPACK's own error is
about l eps sigma_1.  Vectors of values a relative gap of 1e-3 or more apart
are orthogonal to about l eps / 1e-3, closer ones are orthogonalised."""
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


def _bidiagonal(kind, l, rng):
    """alpha[l], beta[l + 1] (beta[0] = beta_1) of the lower bidiagonal."""
    a, b = rng.uniform(0.2, 1.0, l), rng.uniform(0.2, 1.0, l + 1)
    if kind == "equal":
        a[:], b[:] = 0.5, 0.5
    elif kind == "graded":
        s = 10.0 ** -np.linspace(0.0, 14.0, l)
        a, b[1:] = a * s, b[1:] * s
    elif kind == "tail":  # breakdown in beta: the last coupling is zero
        b[l] = 0.0
    elif kind == "split":  # decoupled blocks with the same values
        a[:], b[1:] = 0.7, 0.3
        b[1 + l // 2] = 0.0
    return a, b


def _dense(a, b):
    l = a.size
    C = np.zeros((l + 1, l))
    C[np.arange(l), np.arange(l)] = a
    C[np.arange(1, l + 1), np.arange(l)] = b[1:]
    return C


@pytest.mark.parametrize("kind", ["random", "equal", "graded", "tail", "split"])
@pytest.mark.parametrize("l", [1, 2, 3, 4, 7, 8, 15, 16, 17, 31, 33, 64, 129, 300])
def test_projected_svd_edges(ctx, R, kind, l):
    a, b = _bidiagonal(kind, l, np.random.default_rng(100 * l + len(kind)))
    st, W, Z, al, be = R.make_state(torch, l + 1, l)
    al.copy_(torch.as_tensor(a))
    be.copy_(torch.as_tensor(b))
    st.steps_done = l
    sig = torch.empty(l, dtype=torch.float64, device="cuda")
    ft = torch.empty(l + 1, dtype=torch.float64, device="cuda")
    V = torch.empty((l, l), dtype=torch.float64, device="cuda")
    ctx.rbf_projected_svd(st, sig, ft, V, l)
    torch.cuda.synchronize()
    C = _dense(a, b)
    ref = np.linalg.svd(C, compute_uv=False)
    s, Vn = sig.cpu().numpy(), V.cpu().numpy().T
    assert np.all(np.diff(s) <= 0.0)
    assert np.max(np.abs(s - ref)) <= 8 * (l + 1) * EPS * ref[0]
    assert np.max(np.abs(Vn.T @ Vn - np.eye(l))) <= max(1e-12, 40 * l * EPS / 1e-3)
    assert np.max(np.abs(np.linalg.norm(C @ Vn, axis=0) - s)) <= 40 * (l + 1) * EPS * ref[0] / 1e-3
    assert abs(np.sum(ft.cpu().numpy() ** 2) - b[0] ** 2) <= 1e-11 * b[0] ** 2


# the last size with 32 lanes per value on 152 SMs, the first with 8; shared tables of just under 48 KB
@pytest.mark.parametrize("n", [1823, 1825, 2045])
def test_singular_values_lane_split(ctx, R, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    lda = R.padded_lda(n, R.RBF_FP64)
    A = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
    A[:, :n] = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda")
    A[:, :n] *= 10.0 ** -torch.linspace(0, 9, n, dtype=torch.float64, device="cuda")
    nodes = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    op = ctx.rbf_operator_init(nodes, n, n // 2, 1.0, 1.0, A=A, lda=lda)
    sig = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.rbf_svd_full(op, sig)
    ref = np.linalg.svd(A[:, :n].cpu().numpy(), compute_uv=False)
    assert np.max(np.abs(sig.cpu().numpy() - ref)) <= 4 * n * EPS * ref[0]
