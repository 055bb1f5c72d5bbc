"""The fp32 router at the token and expert counts where its tile changes. The tile must not show in
the result: the scores of the first and last tokens of a call have the bits that a call with those
tokens alone gives (the smallest tile), and all scores are within the rounding bound of a float64
softmax."""
import numpy as np
import pytest
import torch

from paper_2604_01622_gb300.layer import ECMoELayer

pytestmark = pytest.mark.gpu


def _scores(X, Wr, br, Wg, Wd):
    N, E = X.shape[0], Wr.shape[1]
    layer = ECMoELayer(N, X.shape[1], E, Wg.shape[2], np.array([0, N], np.int32),
                       np.array([1], np.int32), dtype="f32")
    S = layer.forward(X, Wr, br, Wg, Wg, Wd)[3]
    layer.check()
    return S.cpu()


@pytest.mark.parametrize("E", [16, 17, 32, 33, 64, 65, 130])
@pytest.mark.parametrize("N", [1216, 1217, 4864, 4865, 9728, 9729])
def test_router_tile_changes_no_bit(E, N):
    g = torch.Generator(device="cuda").manual_seed(7 * N + E)
    X, Wr, br, Wg, Wd = (torch.randn(s, device="cuda", generator=g) for s in
                         ((N, 132), (132, E), (E,), (E, 132, 4), (E, 4, 132)))
    S = _scores(X, Wr, br, Wg, Wd)
    assert torch.equal(S[:, :40], _scores(X[:40].contiguous(), Wr, br, Wg, Wd))
    assert torch.equal(S[:, -41:], _scores(X[-41:].contiguous(), Wr, br, Wg, Wd))
    x, w, b = (t.cpu().double() for t in (X, Wr, br))
    ref = torch.softmax(x @ w + b, 1).T
    # a logit is a chain of 132 FMAs and the bias; twice its error in the exponent (the entry and
    # the row maximum or sum), then exp, the sum and the division
    u = 2.0 ** -24
    bound = 2 * 134 * u * (x.abs() @ w.abs() + b.abs()).max(1).values + (E + 8) * u
    assert bool(((S.double() - ref).abs() <= bound * ref + 1e-37).all())
