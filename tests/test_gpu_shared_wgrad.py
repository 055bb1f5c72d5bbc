"""The shared experts' weight gradients on each side of their tile rules: few tiles as blocks of the
tokens (the most and the fewest blocks, a short last one), one list of tiles, the down gradient as two
halves of the tokens (narrow and wide tiles, token counts whose half is and is not a multiple of
the 64-row k-step), and one list where only one of the two problems has columns for wide ones. Against the SwiGLU FFN in 64 bits, 2e-2 relative max-norm (the
bf16 parity bound of the other tests)."""
import numpy as np
import pytest
import torch

from paper_2604_01622_gb300 import EC_TILES_256, EC_TILES_512, EC_TILES_AUTO
from paper_2604_01622_gb300.layer import ECMoELayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,Fs", [
    (8192, 832, 1600),     # halves, narrow tiles
    (8196, 1600, 832),     # halves of 4098 tokens
    (8193, 1600, 832),     # an odd count has no halves: one list
    (16384, 4096, 1024),   # halves, wide tiles
    (13000, 64, 64),       # 2 tiles: 23 blocks of 9 k-slices, the last of 6
    (4097, 256, 256),      # blocks, one token in the last slice
    (3900, 1536, 384),     # 30 tiles: two blocks
    (3840, 1536, 384),     # ... of 30 slices each, one list
    (8192, 2048, 896),     # wide columns for the down gradient alone, few tiles
])
def test_shared_weight_gradients(N, d, Fs):
    E, F = 4, 64
    g = torch.Generator(device="cuda").manual_seed(N + d)

    def r(*s, scale=1.0):
        return (torch.randn(*s, device="cuda", generator=g) * scale).to(torch.bfloat16)

    X, dY = r(N, d), r(N, d)
    Wr, Wg, Wu, Wd = r(d, E, scale=.1), r(E, d, F), r(E, d, F), r(E, F, d)
    sh = (r(d, Fs, scale=d ** -.5), r(d, Fs, scale=d ** -.5), r(Fs, d, scale=Fs ** -.5))
    layer = ECMoELayer(N, d, E, F, np.array([0, N], np.int32), np.array([8], np.int32),
                       d_ff_shared=Fs)
    layer.forward(X, Wr, None, Wg, Wu, Wd, shared=sh)
    got = layer.backward(dY)
    layer.check()
    x, dy, wg, wu, wd = (t.double() for t in (X, dY, *sh))
    a, b = x @ wg, x @ wu
    s = torch.sigmoid(a)
    du = dy @ wd.T
    ref = {"dWg_s": x.T @ (du * b * s * (1 + a * (1 - s))), "dWu_s": x.T @ (du * a * s),
           "dWd_s": (a * s * b).T @ dy}
    for k, want in ref.items():
        err = ((got[k].double() - want).abs().max() / want.abs().max()).item()
        assert err <= 2e-2, (k, err)


def _shared_grads(N, d, Fs, policy):
    """Gradients of a layer with shared experts under one tile policy, and the launches of its
    backward pass."""
    E, F = 4, 64
    g = torch.Generator(device="cuda").manual_seed(N + d + Fs)

    def r(*s, scale=1.0):
        return (torch.randn(*s, device="cuda", generator=g) * scale).to(torch.bfloat16)

    layer = ECMoELayer(N, d, E, F, np.array([0, N], np.int32), np.array([200], np.int32),
                       d_ff_shared=Fs)
    layer.set_tiles(policy)
    layer.forward(r(N, d), r(d, E, scale=.1), None, r(E, d, F), r(E, d, F), r(E, F, d),
                  shared=(r(d, Fs, scale=d ** -.5), r(d, Fs, scale=d ** -.5),
                          r(Fs, d, scale=Fs ** -.5)))
    before = layer.launches
    got = layer.backward(r(N, d))
    launches = layer.launches - before
    layer.check()
    layer.close()
    return got, launches


@pytest.mark.parametrize("N,d,Fs", [
    (4097, 256, 256),      # blocks of the tokens, wide columns for the gate/up gradients
    (13000, 512, 512),     # blocks, wide columns for all three
    (3900, 512, 320),      # blocks, wide columns for the down gradient alone
    (8192, 832, 1600),     # halves, no wide columns
    (16384, 4096, 1024),   # halves, wide columns for all three
    (8192, 2048, 896),     # one list, wide columns for the down gradient alone
])
def test_tile_policies_agree_with_shared_experts(N, d, Fs):
    """The number of partial sums over the tokens follows from the sizes, not from the tile policy:
    every gradient has the same bits under the three policies."""
    want, _ = _shared_grads(N, d, Fs, EC_TILES_AUTO)
    for policy in (EC_TILES_256, EC_TILES_512):
        got, _ = _shared_grads(N, d, Fs, policy)
        for k, t in want.items():
            if t is not None:
                assert torch.equal(got[k], t), (policy, k)


def test_wide_tiles_where_one_of_the_two_problems_fills_them():
    """d 2048 fills wide tiles of the down gradient, the gate/up columns of d_ff 896 (shared) and 64
    (routed) do not: EC_TILES_512 runs the two apart, each with its own tiles, where EC_TILES_256
    has one list of narrow ones."""
    narrow = _shared_grads(8192, 2048, 896, EC_TILES_256)[1]
    assert _shared_grads(8192, 2048, 896, EC_TILES_512)[1] == narrow + 2
