"""Row widths around the limits of the warp-per-token gather and sums (48, 64 and 96 16-byte
units), with token counts that leave the last CTA short, tokens no expert picks, the residual form
and shared experts (every optional term of the sums). Against the oracle."""
import numpy as np
import pytest
import torch

from paper_2604_01622_gb300 import inputs as I
from tests._util import dev, gpu_layer
from tests.test_gpu_parity import _check_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("bf16", 256), ("bf16", 320), ("bf16", 384),
                                     ("bf16", 448), ("bf16", 768), ("bf16", 832), ("f32", 4),
                                     ("f32", 128), ("f32", 252), ("f32", 256), ("f32", 260)])
def test_widths(dtype, d):
    w = I.scaled(I.WORKLOADS["tiny_f32" if dtype == "f32" else "ec_d2048_e64"], G=1, L=181, d=d,
                 E=37, d_ff=64, k_base=11, seed=61, router_bias=True, layers=1)
    _check_layer(I.make_inputs(w))


@pytest.mark.parametrize("d", [128, 512])
def test_residual_and_shared_terms(d):
    """Y and dX with the residual equal those without it plus X or dY, to the rounding of one
    bf16 addition each way; unpicked tokens get exactly X and dY."""
    w = I.scaled(I.WORKLOADS["ec_d2048_e64"], G=1, L=150, d=d, E=9, d_ff=64, k_base=10, seed=62,
                 layers=1)
    inp = I.make_inputs(w)
    L = inp.layers[0]
    X, dY = dev(inp.X), dev(inp.dY)
    args = (dev(L.Wr), None, dev(L.Wg), dev(L.Wu), dev(L.Wd))
    lay, plain = gpu_layer(inp)
    lay.set_residual(True)
    Y, idx, _, _ = lay.forward(X, *args)
    g = lay.backward(dY)
    lay.check()
    for got, part, base in ((Y, plain["Y"], X), (g["dX"], plain["dX"], dY)):
        want = part.double() + base.double()
        assert torch.all((got.double() - want).abs()
                         <= 2.0 ** -8 * (want.abs() + part.double().abs()) + 1e-30)
    rest = np.setdiff1d(np.arange(w.N), idx.cpu().numpy().ravel())
    assert len(rest) and torch.equal(Y[rest], X[rest]) and torch.equal(g["dX"][rest], dY[rest])
