"""Order of the dense contraction's output tiles at the edges of its bands: a row tile left over that joins the band
above it (13 pair rows, 25 row tiles), and all rows in one band (SM pairs, 16 column tiles and more). The same check
and bound as in test_gpu_tile_order.py."""

import pytest

from test_gpu_tile_order import lib, test_partial_band as check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("math_mode", ["x3", "bf16"])
@pytest.mark.parametrize("policy,B,N_in,N_out", [(1, 104, 40, 300), (1, 64, 40, 2050), (1, 66, 72, 1930),
                                                 (2, 4, 40, 3150), (2, 4, 72, 1665)])
def test_bands(math_mode, policy, B, N_in, N_out):
    check(math_mode, policy, B, N_in, N_out)
