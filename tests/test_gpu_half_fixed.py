"""GPU: the cluster half-step's fixed-point form (slabs of at least 4096 entries of
Q) against the grid form in FP64, on both sides of its rule: the slab size, an
entry of Q of 2 or more (FP64), and columns scaled far apart.

Tolerance as for the cluster form: 1e-11 of the largest entry over the run.  The
scaled operators are A and 2^k A (the same run up to powers of two: bitwise, since
every scale is one)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def both():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    a, b = rbfkr.Context(0), rbfkr.Context(0, wait_budget=4000)
    yield rbfkr, a, b
    a.close()
    b.close()


def _run(R, ctx, n, steps, more=0, scale=1.0, poke=None):
    rng = np.random.default_rng(n)
    nodes = torch.as_tensor(rng.uniform(0, 1, (3, n)), device="cuda")
    lda = R.padded_lda(n, R.RBF_FP64)
    D = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
    op = ctx.rbf_operator_init(nodes, n, (2 * n) // 3, 0.2, 3.0, A=D, lda=lda)
    # a well-conditioned matrix, so that one rounding stays one
    D[:, :n] = scale * (torch.eye(n, device="cuda", dtype=torch.float64) * 3 +
                        torch.as_tensor(rng.normal(size=(n, n)) / np.sqrt(n), device="cuda"))
    f = torch.as_tensor(rng.normal(size=n), device="cuda")
    st, W, Z, al, be = R.make_state(torch, n, steps + more)
    ctx.rbf_gkb(op, f, steps, st)
    if poke is not None:
        W[0, 0] = poke
        Z[1, 1] = -poke
        ctx.rbf_gkb_resume(op, st, more)
    assert st.steps_done == steps + (more if poke is not None else 0)
    return W, Z, al, be


@pytest.mark.parametrize("n,steps", [(1008, 66), (1500, 60), (2161, 140), (3000, 45), (4096, 30), (8192, 25)])
def test_fixed_matches_grid(both, n, steps):
    R, a, b = both
    for x, y in zip(_run(R, a, n, steps), _run(R, b, n, steps)):
        assert torch.max(torch.abs(x - y)).item() <= 1e-11 * torch.max(torch.abs(y)).item()


@pytest.mark.parametrize("k", [-300, 200])
def test_scaled_operator(both, k):
    R, a, _ = both
    x, y = _run(R, a, 1500, 60), _run(R, a, 1500, 60, scale=2.0 ** k)
    assert torch.equal(x[0], y[0]) and torch.equal(x[1], y[1])
    assert torch.equal(x[2] * 2.0 ** k, y[2])


@pytest.mark.parametrize("poke", [1.5, 2.0, 2.5])
def test_large_entries(both, poke):
    R, a, b = both
    for x, y in zip(_run(R, a, 2000, 50, 2, poke=poke), _run(R, b, 2000, 50, 2, poke=poke)):
        assert torch.max(torch.abs(x - y)).item() <= 1e-11 * torch.max(torch.abs(y)).item()
