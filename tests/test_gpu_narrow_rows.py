"""Row widths around the limits of the warp-per-token gather and sums (48, 64 and 96 16-byte
units), with token counts that leave the last CTA short and tokens no expert picks, and narrow and
wide sums with the residual form and shared experts (every optional term). Against the oracle."""
import numpy as np
import pytest
import torch

from oracle import ecmoe as O
from paper_2604_01622_gb300 import inputs as I
from paper_2604_01622_gb300.layer import ECMoELayer
from tests._util import dev, gpu_layer, host, relmax, tol
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
def test_residual_term(d):
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


@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 512), ("f32", 128), ("f32", 512)])
def test_shared_and_residual_terms(dtype, d, residual):
    """Y and dX with shared experts, with and without the residual, for tokens that some expert
    picks and for tokens that none does."""
    w = I.scaled(I.WORKLOADS["tiny_f32" if dtype == "f32" else "ec_d2048_e64"], G=1, L=150, d=d, E=9,
                 d_ff=64, k_base=10, seed=63, layers=1)
    inp = I.make_inputs(w)
    L, sh = inp.layers[0], I.make_shared(w, 0, 2, 64)
    lay = ECMoELayer(w.N, d, w.E, w.d_ff, inp.group_off, inp.k_g, dtype=dtype, d_ff_shared=128)
    lay.set_residual(residual)
    Y, idx, _, _ = lay.forward(dev(inp.X), dev(L.Wr), None, dev(L.Wg), dev(L.Wu), dev(L.Wd),
                               shared=(dev(sh.Wg), dev(sh.Wu), dev(sh.Wd)))
    dX = lay.backward(dev(inp.dY))["dX"]
    lay.check()
    idx = idx.cpu().numpy()
    fwd = O.forward(inp.X.f64(), L.Wr.f64(), None, L.Wg.f64(), L.Wu.f64(), L.Wd.f64(),
                    inp.group_off, inp.k_g, forced_idx=idx, shared=[sh.expert(s) for s in range(2)])
    bwd = O.backward(fwd, inp.dY.f64(), L.Wr.f64(), L.Wg.f64(), L.Wu.f64(), L.Wd.f64())
    picked = np.isin(np.arange(w.N), idx)
    assert picked.any() and not picked.all()
    for got, want, base in ((Y, fwd["Y"], inp.X), (dX, bwd["dX"], inp.dY)):
        want = want + base.f64() if residual else want
        for rows in (picked, ~picked):
            assert relmax(host(got)[rows], want[rows]) <= tol(w)
