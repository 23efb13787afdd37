"""GPU: the batched half-step's two ways of adding dot partials (an instance on at
most 128 CTAs, and beyond) against the basis they produce.

The reorthogonalized basis vectors have |W^T W - I| at FP64 rounding: two passes
of classical Gram-Schmidt leave a few n eps per entry at most, 1e-12 for n < 1e4
(4500 x 2.2e-16).  A partial left out or read before it is written leaves the
first pass's error, 1e-8 or more with products in FP32.
"""
import numpy as np
import pytest

import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(8200,), (8100, 64), (9000, 300, 65), (3000, 2999, 70)])
def test_basis_is_orthonormal(sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr
    rng = np.random.Generator(np.random.PCG64(4))
    sets = [w.cube_faces_random(n, 0.3, rng) for n in sizes]
    fs = [w.plane_wave_rhs(s, 3.0, w.problem.DIAG) for s in sets]
    L = 19
    ctx = rbfkr.Context(0)
    bt, keep = rbfkr.make_batch(torch, sets, [0.3] * len(sets), [3.0] * len(sets), fs, L)
    ctx.rbf_batch_gkb(bt, L)
    for b, s in enumerate(sets):
        n, off, steps = s.n, int(keep["offsets"][b]), bt.steps_done[b]
        assert steps == L, (b, steps)
        W = keep["W"].reshape(-1)[(L + 1) * off:(L + 1) * off + L * n].reshape(L, n)
        Z = keep["Z"].reshape(-1)[L * off:L * off + L * n].reshape(L, n)
        eye = torch.eye(L, dtype=torch.float64, device="cuda")
        for Q in (W, Z):
            assert torch.max(torch.abs(Q @ Q.T - eye)).item() <= 1e-12, b
    ctx.close()
