"""Small calls start each kernel while the one before it finishes. Steps queued back to back on
reused buffers, their inputs rewritten by copies in between and read out by copies after, give
bit for bit what the same steps give with the device idle before and after each."""
import numpy as np
import pytest
import torch

from paper_2604_01622_gb300.layer import ECMoELayer, TCMoELayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["f32", "bf16", "bf16_shared", "tc"])
def test_queued_steps_equal_separate_ones(kind):
    torch.manual_seed(11)
    N, d, E, F, steps = 480, 128, 24, 128, 12
    td = torch.float32 if kind == "f32" else torch.bfloat16
    mk = lambda *s: (torch.randn(*s, device="cuda") / s[-2] ** 0.5).to(td)
    Xs, dYs = [mk(N, d) for _ in range(steps)], [mk(N, d) for _ in range(steps)]
    W = (mk(d, E), torch.randn(E, device="cuda"), mk(E, d, F), mk(E, d, F), mk(E, F, d))
    shared = (mk(d, 192), mk(d, 192), mk(192, d)) if kind == "bf16_shared" else None
    if kind == "tc":
        lay = TCMoELayer(N, d, E, F, 3, 80)
    else:
        lay = ECMoELayer(N, d, E, F, np.array([0, 200, 200, N]), np.array([30, 0, 41]),
                         dtype="f32" if kind == "f32" else "bf16",
                         d_ff_shared=192 if shared else 0)
    X, dY = torch.empty_like(Xs[0]), torch.empty_like(dYs[0])

    def run(sync):
        kept, grads = [], None
        for x, dy in zip(Xs, dYs):
            X.copy_(x)
            dY.copy_(dy)
            if sync:
                torch.cuda.synchronize()
            out = lay.forward(X, *W, shared=shared)
            grads = lay.backward(dY, grads=grads, with_bias=True)
            if sync:
                torch.cuda.synchronize()
            kept.append([t.clone() for t in (*out, *(grads[k] for k in sorted(grads)))])
        lay.check()
        return kept

    want = run(True)
    for _ in range(3):
        for a, b in zip(run(False), want):
            for x, y in zip(a, b):
                assert torch.equal(x, y)
