"""GPU parity of the tensor-core variant's row boxes on planes that leave many lanes of a 32-pixel segment empty (4 to 44 pixels a
row), against the fp64 oracle: one and two segments a row, a last row block that ends inside a tile, narrow, resident and streamed
filter banks, pairs of pixel tiles, both strides, pointwise layers."""
import pytest

from paper_2006_09791_b200 import build as gbuild
from paper_2006_09791_b200 import gconv
from paper_2006_09791_b200.workloads import Layer

from gpu_util import check_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    gbuild.build()


CASES = [  # N, C_in, H, W, C_out, filter, stride, groups
    (3, 64, 10, 4, 64, 3, 1, 4), (5, 64, 9, 8, 64, 3, 1, 8), (2, 128, 9, 8, 128, 3, 2, 8), (2, 96, 13, 12, 96, 3, 1, 1),
    (9, 64, 12, 12, 64, 3, 1, 4), (4, 32, 15, 16, 32, 3, 1, 2), (64, 128, 20, 20, 128, 3, 1, 1), (70, 256, 12, 12, 256, 3, 1, 1),
    (3, 64, 41, 36, 64, 3, 1, 1), (5, 64, 40, 40, 64, 3, 1, 16), (4, 48, 30, 44, 48, 3, 1, 1), (11, 16, 15, 16, 80, 3, 1, 1),
    (3, 64, 30, 20, 96, 1, 1, 1), (5, 128, 12, 12, 64, 1, 2, 2), (2, 64, 21, 40, 64, 1, 2, 1), (3, 64, 9, 8, 64, 1, 2, 1),
]


@pytest.mark.parametrize("cfg", CASES)
def test_sparse_row_boxes(cfg):
    N, C, H, W, K, k, stride, g = cfg
    err, used = check_layer(Layer("rowbox", N, C, H, W, K, k, k, stride, k // 2, 1, g), seed=13)
    assert used == gconv.GCONV_VARIANT_IGEMM_TF32


# tall planes 4 and 8 wide whose row-box tiles would take several times the waves: flat tiles (rows straddle the warps' quarters)
@pytest.mark.parametrize("cfg", [(36, 256, 13, 4, 256, 1), (26, 64, 146, 8, 128, 1), (60, 96, 77, 4, 32, 4)])
def test_tall_narrow_planes(cfg):
    N, Ci, H, W, Co, g = cfg
    err, used = check_layer(Layer("tall", N, Ci, H, W, Co, groups=g), seed=23)
    assert used == gconv.GCONV_VARIANT_IGEMM_TF32
