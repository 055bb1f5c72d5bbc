"""The router's weight gradient at the edges of its split over the tokens: one block (written
straight into dWr), blocks of whole 64-token k-slices with a short last one, token counts around
multiples of 64; 8, 12, 72 and 100 experts (weights read in place or from the padded copy, one or
two column halves per tile), d with a ragged last row tile. Against the oracle."""
import pytest

from paper_2604_01622_gb300 import inputs as I
from tests.test_gpu_parity import _check_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [8, 12, 72, 100])
@pytest.mark.parametrize("N", [63, 65, 129, 256, 321, 1000])
def test_router_gradient_splits(N, E):
    w = I.scaled(I.WORKLOADS["ec_many_small_e128"], G=1, L=N, d=192, E=E, d_ff=64,
                 k_base=max(1, N // 6), seed=51, router_bias=True, layers=1)
    _check_layer(I.make_inputs(w))
