"""The general fp32-FMA product in every tile and split it takes: reductions shorter than a k-tile, split over 1 to 8 blocks
with empty shares, ragged edges of the 32, 64 and 128-row tiles, and the bias gradient that rides on the weight gradient."""
import pytest

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl
from test_gpu_tucker import check_tucker

from helpers import check_linear

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1, 1), (33, 31, 65, 7), (256, 512, 512, 40), (1023, 97, 130, 33), (2500, 40, 515, 17), (6000, 128, 64, 64), (300, 1100, 1090, 260)]


@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_linear_layer(shape, dtype):
    M, K, N, r = shape
    for freeze in (b.LRD_FREEZE_NONE, b.LRD_FREEZE_U, b.LRD_FREEZE_V):
        check_linear(wl.random_factor_case(M, K, N, r, dtype, 820 + M), freeze, path=b.LRD_PATH_GENERAL)


@pytest.mark.parametrize("geom", [(9, 14, 13, 33, 40, 17, 25, 3, 2), (2, 30, 31, 64, 64, 64, 48, 3, 1), (40, 9, 9, 8, 8, 4, 8, 5, 1)])
def test_convolution(geom):
    B, H, W, C, S, r1, r2, k, stride = geom
    check_tucker(wl.random_tucker_case(B, H, W, C, S, r1, r2, k, "f32", 830 + H, stride=stride), b.LRD_TK_FREEZE_NONE)
