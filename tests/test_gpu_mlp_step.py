"""GPU: training step of the stop network at the edges of its tiles (4 or 8
samples per CTA, chunks of 16 samples, at most 64 chunks), against FP64 autograd;
the paired FP32 sums on cancelling and on overflowing terms.

Tolerances: the activations carry FP32 rounding over dot products of 128 terms
(about 1e-6 relative of the gradient's largest entry; 2e-5 allowed, the bound of
FP32 results); the sum over the batch adds no more than one FP32 rounding."""
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


def _layers(p):
    i = 0
    for fi, fo in ((20, 128), (128, 128), (128, 2)):
        yield p[i:i + fi * fo].reshape(fi, fo), p[i + fi * fo:i + fi * fo + fo]
        i += fi * fo + fo


def _ref(p, x, y):
    p = p.double().requires_grad_(True)
    h = x.double()
    for q, (w, b) in enumerate(_layers(p)):
        h = h @ w + b
        h = torch.nn.functional.gelu(h) if q < 2 else h
    loss = ((h - y.double()) ** 2).sum() / (2 * x.shape[0])
    loss.backward()
    return h.detach(), p.grad, float(loss.detach())


def _inputs(batch, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    p = 0.1 * torch.randn(19458, generator=g, device="cuda")
    return p, torch.randn((batch, 20), generator=g, device="cuda"), torch.randn((batch, 2), generator=g, device="cuda")


@pytest.mark.parametrize("offset", [0, 1])  # a parameter vector off 16-byte alignment
@pytest.mark.parametrize("batch", [1, 3, 4, 5, 15, 16, 17, 96, 513, 1025, 1041, 7297])
def test_step_sizes(ctx, R, batch, offset):
    p0, x, y = _inputs(batch, batch)
    p = torch.empty(19458 + offset, device="cuda")[offset:]
    p.copy_(p0)
    h, gref, lref = _ref(p, x, y)
    out = torch.empty((batch, 2), device="cuda")
    ctx.rbf_mlp_forward(p, x, batch, out)
    assert (out.double() - h).abs().max() <= 2e-5 * h.abs().max()
    g, g2 = torch.empty(19458, device="cuda"), torch.empty(19458, device="cuda")
    loss = ctx.rbf_mlp_grad(p, x, y, batch, g)
    assert abs(loss - lref) <= 2e-5 * abs(lref)
    assert (g.double() - gref).abs().max() <= 2e-5 * gref.abs().max()
    m, v = torch.zeros_like(g), torch.zeros_like(g)
    q = p.clone()
    ctx.rbf_mlp_train_step(q, m, v, 1, 1e-3, x, y, batch, g2)
    assert torch.equal(g, g2)  # the fused update sums in the same order
    m2, v2, q2 = torch.zeros_like(g), torch.zeros_like(g), p.clone()
    ctx.rbf_mlp_adam(q2, m2, v2, g, 1, 1e-3)
    assert torch.equal(q, q2) and torch.equal(m, m2) and torch.equal(v, v2)


def test_cancelling_and_overflowing_terms(ctx, R):
    batch = 64
    p, x, y = _inputs(batch, 5)
    x[1::2] = x[::2]  # pairs of samples whose output errors nearly cancel
    h, _, _ = _ref(p, x, y)
    y = (h + 1000.0 * torch.tensor([1.0, -1.0], device="cuda").repeat(batch // 2)[:, None]).float()
    y[1::2] += 1e-3
    g = torch.empty(19458, device="cuda")
    ctx.rbf_mlp_grad(p, x, y, batch, g)
    # the same activations summed in FP64: what the batch sum itself may lose is
    # bounded by the FP32 activations' own error on terms of size 1000 / 64
    _, gref, _ = _ref(p, x, y)
    assert (g.double() - gref).abs().max() <= 2e-5 * 1000.0
    big = p.clone()
    big[-2:] = 3e38  # output errors near FP32's largest value: sums leave its range
    ctx.rbf_mlp_grad(big, x, y, batch, g)
    b3 = g[-2:]
    assert torch.isfinite(b3).all() and (b3 / 3e38 - 1.0).abs().max() < 1e-5  # mean of the errors
