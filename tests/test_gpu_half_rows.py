"""GPU: the cluster half-step's fixed-point form on a basis whose rows differ in size by
12 decades, side by side in every CTA, against the grid form in FP64.

Rows of the new basis vector scale with the rows of the basis; FP64 keeps each to
a few roundings of its own size (50 terms: 1e-14), 1e-11 is allowed as in the other
comparisons of the two forms."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _step(R, ctx, n, steps):
    rng = np.random.default_rng(7)
    size = 10.0 ** (-12.0 * (np.arange(n) % 8) / 7.0)
    lda = R.padded_lda(n, R.RBF_FP64)
    D = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
    D[:, :n] = torch.as_tensor(rng.normal(size=(n, n)) / np.sqrt(n) * size[None], device="cuda")
    nodes = torch.as_tensor(rng.uniform(0, 1, (3, n)), device="cuda")
    op = ctx.rbf_operator_init(nodes, n, n // 2, 0.2, 3.0, A=D, lda=lda)
    st, W, Z, al, be = R.make_state(torch, n, steps + 1)
    Wq = np.linalg.qr(rng.normal(size=(n, steps + 1)))[0].T
    Zq = np.linalg.qr(size[:, None] * rng.normal(size=(n, steps)))[0].T
    ctx.rbf_gkb_restore(st, dict(W=Wq.copy(), Z=Zq.copy(), alpha=np.ones(steps), beta=np.full(steps + 1, 1e-3),
                                 steps_done=steps, breakdown=0, c_hat=1.0))
    ctx.rbf_gkb_resume(op, st, 1)
    assert st.steps_done == steps + 1
    return Z[steps, :n].cpu().numpy()


@pytest.mark.parametrize("n,steps", [(2000, 50), (1009, 100), (4096, 20)])
def test_rows_of_different_size(n, steps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr as R
    a, b = R.Context(0), R.Context(0, wait_budget=4000)
    x, y = _step(R, a, n, steps), _step(R, b, n, steps)
    for k in range(8):
        assert np.max(np.abs(x[k::8] - y[k::8])) <= 1e-11 * np.max(np.abs(y[k::8])), k
    a.close()
    b.close()
