"""Upsampling layers (a skip tensor concatenated with an upsampled one) at the
edges of their 256-column tiles, as layers of the joint network (d0a at W, d1a at
W / 2): widths a few columns into a tile, heights cut at 2 of 4 rows, several
images, each with as many tiles as the dispatch asks for on 152 SMs, and a width
just too narrow for it.

The criterion is the one-ulp one of every layer inside the network (the oracle's
sums of the same BF16 operands, rounded once).
"""
import pytest

from test_gpu_unet import spp, test_predict_layerwise_parity as layerwise_parity  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,W,H", [
    (1, 128, 20),                                  # neither layer
    (1, 132, 308), (1, 516, 200), (3, 388, 156),   # d0a: 4, 4 and 132 columns in the last tile
    (2, 260, 308), (1, 520, 416),                  # d1a: 2 and 4 columns
])
def test_upsampling_layers_at_tile_edges(spp, B, W, H):  # noqa: F811
    layerwise_parity(spp, B, W, H)
