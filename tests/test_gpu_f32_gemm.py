"""The fp32 path's GEMMs at the sizes where a tile shape or a load form changes, against the
oracle (relative max-norm 1e-4, the fp32 parity bound of the other tests). Every tile that a product
can take runs with ragged row, column and k edges; the comments say which the choice by the busiest
of 152 SMs gives. Also an expert count that is not a multiple of 4 (scalar loads and stores in the
router products), more than 64 experts (the router's widest tile), fewer than 64 tokens (one split
of X^T dZ) and more rows than a grid of the smallest tiles can have."""
import numpy as np
import pytest
import torch

from paper_2604_01622_gb300 import inputs as I
from paper_2604_01622_gb300.layer import ECMoELayer
from tests.test_gpu_parity import _check_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,d,E,d_ff,k", [
    (337, 252, 65, 124, 117),     # 128 x 128 (gate/up, down, dH, weight gradients), 64 x 128 (dU)
    (1421, 196, 7, 116, 1029),    # the same with 5 rows past a tile; 64 x 128 weight gradients
    (406, 100, 16, 332, 262),     # 128 x 128 (dU, weight gradients), 64 x 64 (gate/up)
    (4100, 252, 124, 4, 30),      # X^T dZ 128 x 128
    (867, 360, 67, 4, 469),       # X^T dZ 64 x 128
    (3000, 260, 24, 132, 700),    # 128 x 64 (gate/up, down, dH, dZ Wr^T): a 60-row tail
    (2000, 260, 16, 132, 260),    # 64 x 64, 4 columns past a tile
    (900, 132, 14, 132, 130),     # 128 x 64 (gate/up) and 64 x 64, 14 experts
    (130, 68, 6, 36, 33),         # 32 x 32: one row past a tile
    (1000, 36, 70, 20, 40),       # 70 experts: one 128-column tile of the router
    (60, 4, 3, 8, 9),             # the smallest width: the second half of dWd has no columns
    (40, 516, 5, 4, 7),           # 40 tokens, k loop of 516 = 32 slices and 4; d_ff one chunk
])
def test_f32_layer_tile_edges(L, d, E, d_ff, k):
    w = I.scaled(I.WORKLOADS["tiny_f32"], G=1, L=L, d=d, E=E, d_ff=d_ff, k_base=k, seed=31,
                 router_bias=True)
    _check_layer(I.make_inputs(w))


def test_more_rows_than_a_grid_of_the_smallest_tiles():
    """2.1 million rows per expert and d_ff 4: the smallest tile (32 rows) would need more than the
    65535 tile rows a launch can have. Against the layer in 64 bits on the same selection."""
    N, M, d, E, F = 2_100_200, 2_100_100, 4, 2, 4
    g = torch.Generator(device="cuda").manual_seed(5)
    X, dY, Wr, Wg, Wu, Wd = (torch.randn(s, device="cuda", generator=g) for s in
                             ((N, d), (N, d), (d, E), (E, d, F), (E, d, F), (E, F, d)))
    lay = ECMoELayer(N, d, E, F, np.array([0, N], np.int32), np.array([M], np.int32), dtype="f32")
    Y, idx, gate, S = lay.forward(X, Wr, None, Wg, Wu, Wd)
    got = lay.backward(dY)
    lay.check()
    x, dy, wg, wu, wd = (t.double() for t in (X, dY, Wg, Wu, Wd))
    y = torch.zeros_like(x)
    for e in range(E):
        rows = idx[e].long()
        h, do, gt = x[rows], dy[rows], gate[e].double()[:, None]
        a, b = h @ wg[e], h @ wu[e]
        s = torch.sigmoid(a)
        u = a * s * b
        y.index_add_(0, rows, gt * (u @ wd[e]))
        du = (gt * do) @ wd[e].T
        ref = {"dWg": h.T @ (du * b * s * (1 + a * (1 - s))), "dWu": h.T @ (du * a * s),
               "dWd": u.T @ (gt * do)}
        for k, want in ref.items():
            err = ((got[k][e].double() - want).abs().max() / want.abs().max()).item()
            assert err <= 1e-4, (k, e, err)
    assert ((Y.double() - y).abs().max() / y.abs().max()).item() <= 1e-4
