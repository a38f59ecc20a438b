"""Tensor-core core convolution in every geometry (k, stride) it takes, against the oracle: tiles of 128 consecutive
output pixels with a ragged last one, images wider than a tile, one row or one pixel, tap classes of a strided data
gradient of unequal (or no) taps and of unequal size, ranks on both sides of the fused 1 x 1 product's limit of 256."""
import pytest

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl
from test_gpu_tucker import MASKS, check_tucker

pytestmark = pytest.mark.gpu

GEOMS = [  # B, H, W, C, S, r1, r2, k, stride
    (1, 3, 140, 16, 16, 16, 16, 3, 1), (1, 139, 5, 16, 24, 16, 8, 3, 2), (3, 7, 7, 64, 80, 40, 72, 3, 2), (5, 1, 1, 16, 16, 8, 16, 3, 2),
    (2, 1, 6, 16, 16, 16, 8, 5, 1), (3, 8, 9, 16, 16, 8, 8, 7, 2), (5, 7, 7, 64, 72, 33, 41, 3, 2), (2, 14, 14, 512, 512, 320, 264, 3, 2),
    (2, 9, 9, 64, 256, 64, 192, 5, 2), (6, 16, 15, 32, 32, 16, 16, 1, 2), (4, 12, 12, 40, 24, 24, 16, 1, 1), (9, 28, 28, 64, 64, 32, 48, 3, 2),
    (2, 12, 12, 256, 200, 192, 192, 3, 2), (1, 8, 9, 8, 24, 4, 20, 3, 1)]


@pytest.mark.parametrize("geom", GEOMS, ids=["x".join(map(str, g)) for g in GEOMS])
@pytest.mark.parametrize("freeze", MASKS)
def test_core_geometry(geom, freeze):
    B, H, W, C, S, r1, r2, k, stride = geom
    case = wl.random_tucker_case(B, H, W, C, S, r1, r2, k, "bf16", 900 + H + W + k, stride=stride)
    check_tucker(case, freeze)
    check_tucker(case, freeze, path=b.LRD_PATH_UNFUSED)
