"""GPU: the cluster form of the GKB half-step against the grid form, at the edges
of its rule (16 CTAs, n = 4096 and 8192, the n x basis limits) and through
breakdowns, resumes and concurrent runs.  A context with a small wait budget
takes the grid form throughout.

Both forms compute the same sums in another order: scalars and vectors agree to
the growth of one rounding over the run (1e-11 here; the oracle's own two
Gram-Schmidt orders differ by up to 2e-12 on such runs)."""
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
def both(R):
    a, b = R.Context(0), R.Context(0, wait_budget=4000)
    yield a, b
    a.close()
    b.close()


def _problem(ctx, R, n, seed, A=None):
    rng = np.random.default_rng(seed)
    nodes = torch.as_tensor(rng.uniform(0, 1, (3, n)), device="cuda")
    lda = R.padded_lda(n, R.RBF_FP64)
    D = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
    op = ctx.rbf_operator_init(nodes, n, (2 * n) // 3, 0.2, 3.0, A=D, lda=lda)
    if A is None:
        ctx.rbf_assemble(op)
    else:
        D[:, :n] = torch.as_tensor(A, device="cuda")
    return op, torch.as_tensor(rng.normal(size=n), device="cuda")


def _run(ctx, R, op, f, n, steps, cap=None):
    st, W, Z, al, be = R.make_state(torch, n, cap or steps)
    ctx.rbf_gkb(op, f, steps, st)
    return st, W, Z, al, be


@pytest.mark.parametrize("n,steps", [(1, 1), (2, 2), (15, 10), (16, 16), (17, 9), (31, 12), (33, 33), (500, 60),
                                     (1024, 30), (4095, 40), (4096, 104), (4097, 53), (6000, 40), (8192, 28),
                                     (8193, 6)])
def test_cluster_matches_grid(both, R, n, steps):
    out = []
    for ctx in both:
        op, f = _problem(ctx, R, n, n)
        st, W, Z, al, be = _run(ctx, R, op, f, n, steps)
        out.append((st.steps_done, st.breakdown, W, Z, al, be))
    a, b = out
    assert a[:2] == b[:2]
    l = a[0]
    for x, y in ((a[2][:l], b[2][:l]), (a[3][:l], b[3][:l])):
        assert (x - y).abs().max() <= 1e-11
        assert (x @ x.T - torch.eye(l, dtype=torch.float64, device="cuda")).abs().max() <= 1e-12
    assert ((a[4] - b[4])[:l].abs() <= 1e-11 * b[4][:l].abs()).all()


@pytest.mark.parametrize("rank", [1, 5, 23])
def test_breakdowns(both, R, rank):
    n = 300
    rng = np.random.default_rng(rank)
    A = rng.normal(size=(n, rank)) @ rng.normal(size=(rank, n))
    got = []
    for ctx in both:
        op, f = _problem(ctx, R, n, 3, A)
        st, W, *_ = _run(ctx, R, op, f, n, 40)
        got.append((st.steps_done, st.breakdown, bool((W[st.steps_done] == 0).all())))
    assert got[0] == got[1] and got[0][1] in (1, 2)


def test_zero_and_nonfinite_rhs(both, R):
    ctx = both[0]
    op, f = _problem(ctx, R, 200, 1)
    for bad, code in ((0.0, 1), (float("nan"), 3), (float("inf"), 3)):
        g = torch.zeros_like(f) if bad == 0.0 else f.clone()
        if bad != 0.0:
            g[7] = bad
        st, *_ = _run(ctx, R, op, g, 200, 5)
        assert (st.steps_done, st.breakdown) == (0, code)


def test_resume_and_lanes_take_the_same_path(both, R):
    ctx, n = both[0], 4200  # crosses the limit of the cluster form within the run
    op, f = _problem(ctx, R, n, 5)
    st, W, Z, al, be = _run(ctx, R, op, f, n, 70)
    s2, W2, Z2, al2, be2 = _run(ctx, R, op, f, n, 33, cap=70)
    ctx.rbf_gkb_resume(op, s2, 37)
    assert (al - al2).abs().max() <= 1e-11 * al.max() and (Z - Z2).abs().max() <= 1e-11
    sts = [R.make_state(torch, n, 70) for _ in range(3)]
    ctx.rbf_gkb_many([op] * 3, [f] * 3, 70, [s[0] for s in sts])
    for s in sts:
        assert torch.equal(s[1], W) and torch.equal(s[2], Z) and torch.equal(s[3], al)


def test_launch_timing_keeps_results(R):
    """Launch timing puts events between the launches: no programmatic launches,
    the same results."""
    outs = []
    for opts in ({}, {"timing": 2}):
        ctx = R.Context(0)
        if opts:
            ctx.close()
            o = R.Options()
            o.timing = 2
            import ctypes as C
            ctx = R.Context.__new__(R.Context)
            ctx.lib, h = R.load(), C.c_void_p()
            assert ctx.lib.rbf_create(C.byref(h), 0, None, C.byref(o)) == 0
            ctx.h, ctx.grid_j, ctx.grid_t_lo, ctx.grid_t_hi = h, 321, -16.0, 0.0
        op, f = _problem(ctx, R, 900, 2)
        outs.append(_run(ctx, R, op, f, 900, 30)[1:])
        ctx.close()
    for x, y in zip(*outs):
        assert torch.equal(x, y)
