"""Two contexts used from two host threads at once, each on its own stream, with sizes that take
the same kernel with different amounts of shared memory. Neither call may disturb the other: every
call succeeds and gives what it gives alone."""
import threading

import numpy as np
import pytest
import torch

from paper_2604_01622_gb300 import ECError, ec_route
from paper_2604_01622_gb300.layer import ECMoELayer

pytestmark = pytest.mark.gpu


class Caller:
    """One context with its arrays and stream: routes X and Wr (given E > 0) or given scores."""

    def __init__(self, N, E, from_scores):
        g = torch.Generator(device="cuda").manual_seed(N + E)
        d = 64
        self.lay = ECMoELayer(N, d, E, 64, np.array([0, N], np.int32), np.array([5], np.int32),
                              dtype="f32")
        self.X = torch.randn(N, d, device="cuda", generator=g)
        self.Wr = torch.randn(d, E, device="cuda", generator=g)
        self.S = torch.rand(E, N, device="cuda", generator=g) if from_scores else None
        self.idx = torch.empty(E, 5, dtype=torch.int32, device="cuda")
        self.gate = torch.empty(E, 5, device="cuda")
        self.stream = torch.cuda.Stream()
        self.errors = []

    def calls(self, n):
        s = self.S is not None
        args = (None if s else self.X.data_ptr(), None if s else self.Wr.data_ptr(), None,
                self.S.data_ptr() if s else None, None, self.idx.data_ptr(), self.gate.data_ptr(),
                self.stream.cuda_stream)
        for _ in range(n):
            try:
                ec_route(self.lay.ctx, *args)
            except ECError as e:
                self.errors.append(str(e))
        self.stream.synchronize()


@pytest.mark.parametrize("sizes,from_scores", [
    (((20000, 2), (49152, 2)), True),      # one CTA per column: 144 and 208 KB
    (((120000, 1), (300000, 1)), True),    # a cluster of CTAs per column: 64 and 160 KB each
    (((2000, 130), (2000, 512)), False),   # fp32 router: the logits of 130 and of 512 experts
], ids=["topk_block", "topk_cluster", "router_f32"])
def test_calls_of_two_threads(sizes, from_scores):
    callers = [Caller(N, E, from_scores) for N, E in sizes]
    torch.cuda.synchronize()
    want = []
    for c in callers:
        c.calls(1)
        want.append((c.idx.clone(), c.gate.clone()))
    torch.cuda.synchronize()
    threads = [threading.Thread(target=c.calls, args=(3000,)) for c in callers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for c, (idx, gate) in zip(callers, want):
        assert not c.errors, (len(c.errors), c.errors[0])
        c.lay.check(c.stream)
        assert torch.equal(c.idx, idx) and torch.equal(c.gate, gate)
