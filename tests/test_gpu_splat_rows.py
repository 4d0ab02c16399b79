"""Splat and pyramid at the widths that choose its kernels (multiples of 4 and
others) and at the edges of their tiles, against the oracle as in
the other splat tests."""
import pytest

from test_gpu_parity import spp, test_render_and_splat_parity as splat_parity  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,L", [(4, 2, 2), (128, 16, 5), (132, 17, 1), (144, 48, 5), (260, 36, 3),
                                   (2, 2, 2), (62, 18, 2), (66, 30, 2), (130, 6, 2), (3, 5, 1),
                                   (33, 19, 1)])
def test_splat_widths(spp, W, H, L):  # noqa: F811
    splat_parity(spp, W, H, L, 0.5)
