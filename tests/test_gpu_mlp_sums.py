"""GPU: the weight gradients' sums over the batch at the precision they are documented
with (twice FP32's), on batches whose terms are known exactly.

With W2 = 0 and W3 = b3 = 0 the output is 0 and the second hidden layer is the same
for every sample: dY = -T / B in FP32, the gradient of b3 is sum dY and that of W3 is h
sum dY with h = gelu(b2), read off with a forward pass through a unit W3.  The exact
sums are taken with Python's fractions; the kernel's may be one FP32 rounding off
(one unit in the last place).  The targets hold large values that cancel and
small ones that do not; a plain FP32 sum in any order of this kind is thousands of
units off, which is checked too."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NP, B2, W3, B3 = 19458, 20 * 128 + 128 + 128 * 128, 19458 - 258, 19458 - 2


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    return rbfkr


def _exact(terms):
    return sum((Fraction(float(a)) for a in terms), Fraction(0))


@pytest.mark.parametrize("scale", [0, 60, -60, -110, -125])  # powers of two on the targets
@pytest.mark.parametrize("batch", [8, 64, 1024, 4096])  # one chunk to 64 chunks
def test_cancelling_sums(R, batch, scale):
    ctx = R.Context(0)
    rng = np.random.default_rng(batch)
    big = (2.0**18 * (1 + rng.random((batch // 4, 2)))).astype(np.float32)
    small = rng.normal(size=(batch // 2, 2)).astype(np.float32)
    t = np.concatenate([big, -big, small])[rng.permutation(batch)].astype(np.float32) * np.float32(2.0**scale)
    dy = -t / np.float32(batch)  # (a power of two: exact above the subnormal numbers)
    p = np.zeros(NP, np.float32)
    p[:20 * 128] = 0.1 * rng.normal(size=20 * 128)
    p[B2:B2 + 128] = rng.uniform(0.2, 2.0, 128)
    x = torch.as_tensor(rng.normal(size=(batch, 20)).astype(np.float32), device="cuda")
    h = np.zeros(128, np.float32)
    y = torch.empty((batch, 2), device="cuda")
    for j in range(0, 128, 2):
        q = p.copy()
        q[W3 + 2 * j] = q[W3 + 2 * (j + 1) + 1] = 1.0
        ctx.rbf_mlp_forward(torch.as_tensor(q, device="cuda"), x, batch, y)
        h[j:j + 2] = y[0].cpu().numpy()
    g = torch.empty(NP, device="cuda")
    ctx.rbf_mlp_grad(torch.as_tensor(p, device="cuda"), x, torch.as_tensor(t, device="cuda"), batch, g)
    g = g.cpu().numpy()
    plain_off = 0.0
    for o in range(2):
        e = _exact(dy[:, o])
        ref = np.float32(float(e))
        assert abs(Fraction(float(g[B3 + o])) - e) <= Fraction(float(np.spacing(abs(ref)))), (o, g[B3 + o], ref)
        plain = np.float32(0)
        for v in dy[:, o]:
            plain = np.float32(plain + v)
        plain_off = max(plain_off, float(abs(Fraction(float(plain)) - e) / Fraction(float(np.spacing(abs(ref))))))
        for j in range(128):
            ej = e * Fraction(float(h[j]))
            ref = np.float32(float(ej))
            assert abs(Fraction(float(g[W3 + 2 * j + o])) - ej) <= Fraction(float(np.spacing(abs(ref)))), (o, j)
    if batch >= 64 and scale > -110:
        assert plain_off > 1000
    ctx.close()


def test_units_without_response(R):
    """All-zero factors (an unused input, dead units) give exactly zero."""
    ctx = R.Context(0)
    g = torch.Generator(device="cuda").manual_seed(1)
    p = 0.1 * torch.randn(NP, generator=g, device="cuda")
    x = torch.randn((512, 20), generator=g, device="cuda")
    x[:, 3] = 0.0
    grad = torch.empty(NP, device="cuda")
    ctx.rbf_mlp_grad(p, x, torch.randn((512, 2), generator=g, device="cuda"), 512, grad)
    assert torch.all(grad[3 * 128:4 * 128] == 0.0) and torch.all(grad[:3 * 128] != 0.0)
    ctx.close()
