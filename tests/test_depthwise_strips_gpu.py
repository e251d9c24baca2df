"""GPU parity of the depthwise kernels against the fp64 oracle, whole tensor, where the geometry that is chosen per shape changes:
the shortest and the longest strips, strips that end inside a plane's last rows, one wave and a little more than one."""
import pytest

from paper_2006_09791_b200 import build as gbuild
from paper_2006_09791_b200 import gconv
from paper_2006_09791_b200.workloads import Layer

from gpu_util import check_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    gbuild.build()


STRIPS = [  # N, C, H, W, filter, stride
    # one plane (strips of one pipeline block: 4, 2 or 1 rows), every alignment of the rows
    (1, 1, 61, 60, 3, 1), (1, 1, 23, 22, 3, 1), (1, 1, 60, 61, 3, 2), (1, 1, 33, 30, 5, 1), (1, 1, 61, 44, 5, 2),
    # a plane of a single output row, of one row more than a block
    (2, 3, 1, 40, 3, 1), (2, 3, 2, 40, 3, 2), (1, 5, 5, 17, 5, 1), (2, 3, 1, 17, 5, 2), (3, 2, 29, 31, 3, 1),
    # many planes: whole planes per thread, and strips whose last one is short
    (40, 200, 9, 9, 3, 1), (24, 160, 13, 13, 5, 2), (16, 48, 54, 54, 3, 2), (10, 72, 55, 55, 3, 1), (9, 96, 25, 25, 5, 1), (6, 40, 97, 96, 5, 2),
]


@pytest.mark.parametrize("cfg", STRIPS)
def test_depthwise_strips(cfg):
    N, C, H, W, k, stride = cfg
    err, used = check_layer(Layer("dw", N, C, H, W, C, k, k, stride, k // 2, 1, C), seed=47)
    assert used == gconv.GCONV_VARIANT_DIRECT_TILED and err <= 2e-6      # sums of at most 25 products: 2^-24 x 25 is 1.5e-6


BATCHES = [  # N, C, H, W, filter, stride: enough small planes for batches in shared memory; N * C and H * W leave a short last batch
    # whose floats end 1, 2 or 3 past a multiple of four, one plane in the last batch, whole batches only
    # (filters copied one by one), one plane in the last batch, whole batches only, fewer channels than a batch has planes
    (1, 2049, 7, 7, 3, 1), (1, 6151, 7, 7, 5, 1), (3, 1367, 5, 7, 3, 1), (97, 64, 7, 7, 5, 1), (11, 2235, 7, 7, 3, 2), (3, 4099, 7, 7, 5, 2),
    (9, 1367, 14, 14, 3, 1), (7, 1999, 13, 14, 3, 2), (1, 6151, 14, 14, 5, 1), (5, 1231, 14, 14, 5, 2), (1, 4251, 27, 28, 5, 1),
    (1, 6149, 28, 28, 5, 2), (3, 5667, 27, 28, 3, 2), (2100, 3, 7, 7, 5, 1), (1600, 4, 7, 7, 3, 1), (2500, 1, 14, 14, 5, 1),
]


@pytest.mark.parametrize("cfg", BATCHES)
def test_depthwise_batches_of_planes(cfg):
    test_depthwise_strips(cfg)
