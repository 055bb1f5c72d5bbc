"""Up to 128 rows per expert the expert GEMMs take one-CTA tiles of 128 rows: at the edges of that
range (1, 127, 128 rows, and 129 on the other side) and with column tails of every tile (d and
d_ff not multiples of 128 or 256), the layer matches the oracle and equals 256 x 256 tiles bit
for bit. Also expert counts that are multiples of 8 but not of 64, whose router weights are read
in place with the missing columns filled by the loads."""
import pytest
import torch

from paper_2604_01622_gb300 import EC_TILES_256
from paper_2604_01622_gb300 import inputs as I
from tests._util import gpu_layer
from tests.test_gpu_parity import _check_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d,d_ff,E", [(1, 64, 64, 8), (127, 320, 192, 3), (128, 192, 320, 72),
                                        (129, 192, 320, 16), (33, 576, 576, 40)])
def test_short_rows(M, d, d_ff, E):
    w = I.scaled(I.WORKLOADS["ec_d2048_e64"], G=1, L=2 * M + 40, d=d, E=E, d_ff=d_ff, k_base=M,
                 seed=41, router_bias=True, layers=1)
    inp = I.make_inputs(w)
    _check_layer(inp)
    _, a = gpu_layer(inp)
    _, b = gpu_layer(inp, tiles=EC_TILES_256)
    for k in ("Y", "idx", "gate", "S", "dX", "dWr", "dbr", "dWg", "dWu", "dWd"):
        assert torch.equal(a[k], b[k]), k
