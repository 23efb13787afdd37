"""GPU: the stop network's forward pass and gradient at the batch sizes where the
number of samples per CTA changes (4, 8, 32 or 48 forward, 4 or 16 with gradients; 152
SMs) and where CTAs take several tiles, against FP64 autograd.

Tolerance: FP32 activations, 2e-5 of the largest as in the other network tests."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ref(p, x, y):
    p = p.double().requires_grad_(True)
    h, i = x.double(), 0
    for fi, fo in ((20, 128), (128, 128), (128, 2)):
        w, b = p[i:i + fi * fo].reshape(fi, fo), p[i + fi * fo:i + fi * fo + fo]
        i += fi * fo + fo
        h = h @ w + b
        h = torch.nn.functional.gelu(h) if fo == 128 else h
    loss = ((h - y.double()) ** 2).sum() / (2 * x.shape[0])
    loss.backward()
    return h.detach(), p.grad, float(loss.detach())


@pytest.mark.parametrize("batch", [7, 608, 609, 1825, 2432, 2433, 4863, 4865, 7295, 7297, 9729, 20011, 50000])
def test_batches(batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    ctx = rbfkr.Context(0)
    g = torch.Generator(device="cuda").manual_seed(batch)
    p = 0.1 * torch.randn(19458, generator=g, device="cuda")
    x = torch.randn((batch, 20), generator=g, device="cuda")
    y = torch.randn((batch, 2), generator=g, device="cuda")
    h, gref, lref = _ref(p, x, y)
    out = torch.full((batch, 2), float("nan"), device="cuda")
    ctx.rbf_mlp_forward(p, x, batch, out)
    assert (out.double() - h).abs().max() <= 2e-5 * h.abs().max()
    grad = torch.empty(19458, device="cuda")
    loss = ctx.rbf_mlp_grad(p, x, y, batch, grad)
    assert abs(loss - lref) <= 2e-5 * lref
    assert (grad.double() - gref).abs().max() <= 2e-5 * gref.abs().max()
    ctx.close()
