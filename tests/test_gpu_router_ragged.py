"""The router's scores where a row of S or of S^T is not a multiple of 16 bytes, so the epilogue
stores that array itself: expert counts and token counts around multiples of 4 and of the 32-token
blocks, one and both 64-expert halves, with a bias. Forward and backward against the oracle."""
import pytest

from paper_2604_01622_gb300 import inputs as I
from tests.test_gpu_parity import _check_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [3, 33, 64, 66, 127])
@pytest.mark.parametrize("N", [31, 132, 257, 1001])
def test_ragged_score_rows(E, N):
    w = I.scaled(I.WORKLOADS["ec_many_small_e128"], G=1, L=N, d=128, E=E, d_ff=64,
                 k_base=max(1, N // 6), seed=77, router_bias=True, layers=1)
    _check_layer(I.make_inputs(w))
