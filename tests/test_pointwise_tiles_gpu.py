"""GPU parity of pointwise layers on the tensor-core variant against the fp64 oracle: planes re-cut into segments of 32 pixels (whole,
short last segment, several images per tile, straddled tiles), stride 2 on even rows only (one and two segments a row, 64 wide,
odd heights), filter tiles of 192 and 256."""
import pytest

from paper_2006_09791_b200 import build as gbuild
from paper_2006_09791_b200 import gconv
from paper_2006_09791_b200.workloads import Layer

from gpu_util import check_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    gbuild.build()


CASES = [  # N, C_in, H, W, C_out, stride, groups
    (5, 64, 6, 6, 64, 1, 1), (7, 64, 12, 12, 128, 1, 1), (3, 32, 14, 14, 32, 1, 1), (9, 64, 8, 4, 64, 1, 2), (4, 48, 5, 20, 80, 1, 1),
    (2, 64, 56, 56, 128, 1, 1), (3, 64, 9, 100, 64, 1, 1), (130, 32, 6, 6, 32, 1, 4), (1, 64, 1, 36, 64, 1, 1), (2, 16, 64, 63, 24, 1, 1),
    (3, 64, 56, 56, 96, 2, 1), (2, 64, 64, 64, 64, 2, 1), (5, 32, 7, 8, 32, 2, 1), (4, 64, 13, 28, 64, 2, 2), (2, 256, 31, 60, 512, 2, 1),
    (6, 320, 14, 14, 512, 1, 1), (9, 512, 10, 10, 384, 1, 1), (3, 192, 16, 16, 256, 1, 1), (40, 512, 14, 14, 768, 1, 1), (3, 96, 32, 32, 192, 2, 1),
]


@pytest.mark.parametrize("cfg", CASES)
def test_pointwise_tiles(cfg):
    N, C, H, W, K, stride, g = cfg
    err, used = check_layer(Layer("pw", N, C, H, W, K, 1, 1, stride, 0, 1, g), seed=19)
    assert used == gconv.GCONV_VARIANT_IGEMM_TF32


@pytest.mark.parametrize("cfg", [(3, 16, 4, 4, 16), (2, 16, 50, 200, 16)])
def test_planes_that_stay_on_the_fp32_variants(cfg):
    N, C, H, W, K = cfg
    err, used = check_layer(Layer("pw32", N, C, H, W, K, 1, 1, 1, 0, 1, 1), seed=19)
    assert used != gconv.GCONV_VARIANT_IGEMM_TF32


ONE_ROW = [  # N, C_in, H, W, C_out, stride, groups: planes copied to one row each (1, 2 or 3 floats of padding, one segment or many, images
    # that share a tile); stride 2 on odd, even and single-row planes, a last odd row or column; groups; every filter tile width
    (5, 64, 7, 7, 64, 1, 1), (3, 96, 5, 5, 160, 1, 1), (2, 64, 9, 9, 72, 1, 1), (1, 128, 13, 13, 512, 1, 2), (2, 48, 25, 30, 64, 1, 1), (1, 40, 57, 57, 48, 1, 1),
    (1, 64, 1, 127, 64, 1, 1), (4, 256, 3, 3, 256, 1, 1), (130, 512, 7, 7, 512, 1, 1), (2, 320, 5, 7, 320, 1, 1), (3, 32, 3, 33, 32, 1, 1),
    (5, 64, 7, 7, 128, 2, 1), (3, 96, 15, 15, 96, 2, 1), (2, 256, 29, 29, 512, 2, 1), (1, 64, 50, 50, 128, 2, 1), (2, 128, 13, 26, 64, 2, 2), (1, 64, 1, 90, 64, 2, 1),
    (2, 72, 58, 57, 200, 2, 1), (4, 512, 5, 5, 512, 2, 1), (1, 48, 33, 35, 48, 2, 1), (2, 64, 127, 127, 64, 2, 1),
]


@pytest.mark.parametrize("cfg", ONE_ROW)
def test_pointwise_planes_of_one_row(cfg):
    test_pointwise_tiles(cfg)


# narrow groups with 512 filters and more on such planes: the gather producer's tiles of at most 128 filters, no workspace
@pytest.mark.parametrize("cfg", [(5, 128, 7, 7, 2048, 1, 4), (3, 64, 7, 3, 1024, 1, 2), (2, 48, 17, 7, 1024, 2, 2), (4, 32, 14, 14, 512, 2, 1)])
def test_gathered_pointwise_planes(cfg):
    N, C, H, W, K, stride, g = cfg
    d = gconv.gconv_desc_create(N, C, H, W, K, 1, 1, stride, 0, 1, g)
    assert gconv.gconv_workspace_bytes(d) == 0
    gconv.gconv_desc_destroy(d)
    test_pointwise_tiles(cfg)
