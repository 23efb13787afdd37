"""Contexts on several host threads (one each): calls at different sizes at the
same time.  A kernel's dynamic shared-memory limit belongs to the function on the
device, so a limit set to one call's size would be lowered under another
thread's launch; limits are raised once, in one place, and never lowered."""
import os
import re
import threading

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09798_gb300", "csrc")


def test_limits_are_raised_in_one_place():
    found = []
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        found += [f] * text.count("cudaFuncAttributeMaxDynamicSharedMemorySize")
    assert found == ["internal.h"]


@pytest.mark.gpu
def test_two_threads_at_two_sizes():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09798_gb300 import rbfkr as R

    steps = 30

    def problem(n):  # A z by rows: 42 and 58 KB of shared memory
        rng = np.random.default_rng(n)
        ctx = R.Context(0, stream=torch.cuda.Stream())
        lda = R.padded_lda(n, R.RBF_FP64)
        A = torch.zeros((n, lda), dtype=torch.float64, device="cuda")
        nodes = torch.as_tensor(rng.uniform(0, 1, (3, n)), device="cuda")
        op = ctx.rbf_operator_init(nodes, n, n // 2, 0.2, 3.0, A=A, lda=lda)
        ctx.rbf_assemble(op)
        st, W, Z, al, be = R.make_state(torch, n, steps)
        return ctx, op, torch.as_tensor(rng.normal(size=n), device="cuda"), st, (W, Z, al, be), nodes, A

    probs = [problem(3500), problem(4800)]
    torch.cuda.synchronize()
    refs = []
    for ctx, op, f, st, out, *_ in probs:
        ctx.rbf_gkb(op, f, steps, st)
        refs.append([t.clone() for t in out])
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(2)

    def work(ctx, op, f, st, *_):
        try:
            start.wait()
            for _ in range(40):
                ctx.rbf_gkb(op, f, steps, st)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=p) for p in probs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for p, ref in zip(probs, refs):
        for x, y in zip(p[4], ref):
            assert torch.equal(x, y)
        p[0].close()
