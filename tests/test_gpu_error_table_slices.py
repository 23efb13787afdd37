"""GPU: the error table on a long lambda grid: its coefficients take the place of the
SVD's scratch, in slices where they do not all fit, so that the workspace does not
grow with the grid."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _table(L, ells, J, stride, m, **opts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    ctx = rbfkr.Context(0, grid_j=J, **opts)
    rng = np.random.default_rng(L)
    st, _, _, alpha, beta = rbfkr.make_state(torch, 4, L)
    alpha.copy_(torch.as_tensor(rng.uniform(0.2, 1.0, L) * np.logspace(0, -3, L)))
    beta.copy_(torch.as_tensor(rng.uniform(0.2, 1.0, L + 1) * np.logspace(0, -3, L + 1)))
    st.steps_done = L
    G = torch.as_tensor(rng.normal(size=(L, m)), device="cuda")
    uref = torch.as_tensor(rng.normal(size=m), device="cuda")
    err = torch.full((len(ells), (J - 1) // stride + 1), -1.0, dtype=torch.float64, device="cuda")
    ctx.rbf_hkt_error_table(st, G, m, m, uref, ells, stride, err)
    out = err.cpu().numpy()
    ctx.close()
    return out


@pytest.mark.parametrize("L,ells", [(1, [1]), (3, [1, 3]), (20, [20, 7, 1])])
def test_slices_match_a_short_table(L, ells):
    """The same lambdas, all of them and every 40th (which fit in one slice)."""
    J = 40 * 300 + 1
    full, some = _table(L, ells, J, 1, 150), _table(L, ells, J, 40, 150)
    assert np.all(full >= 0.0)
    assert np.array_equal(full[:, ::40], some)


def test_workspace_does_not_grow_with_the_grid():
    """1.2 MB of SVD results and scratch under a cap of 2 MB; all coefficients would take 34 MB."""
    out = _table(70, [70, 33, 5], 20001, 1, 40, workspace_cap=2 << 20)
    assert np.all(np.isfinite(out)) and np.all(out >= 0.0)
