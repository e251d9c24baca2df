"""GPU parity of the staged FP32 kernel (filters of any size, stride, padding and dilation; wide or odd groups the tensor cores
do not take) against the fp64 oracle, whole tensor, at the sizes where its tiles, chunks and splits end."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_09791_b200 import build as gbuild
from paper_2006_09791_b200 import gconv, synth

from gpu_util import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    gbuild.build()


CASES = [  # N, C_in, H, W, C_out, (filter), (stride), (pad), (dilation), groups
    # one filter per group, two and three (less than a register tile), five, and one more than a block of 16 and of 64
    (2, 6, 19, 21, 6, (7, 7), (1, 1), (3, 3), (1, 1), 6), (3, 6, 12, 12, 6, (5, 5), (1, 1), (2, 2), (1, 1), 3),
    (2, 4, 17, 24, 6, (3, 5), (2, 1), (1, 2), (1, 1), 2), (1, 7, 30, 30, 5, (4, 4), (2, 2), (1, 1), (1, 1), 1),
    (4, 8, 14, 14, 17, (5, 5), (1, 1), (2, 2), (1, 1), 1), (2, 16, 20, 28, 65, (3, 3), (1, 1), (2, 2), (2, 2), 1),
    # first layers on images: several column tiles, column phases of stride 2 and 3, a patch narrower than its tile
    (2, 3, 97, 131, 32, (7, 7), (2, 2), (3, 3), (1, 1), 1), (1, 3, 224, 224, 64, (7, 7), (2, 2), (3, 3), (1, 1), 1),
    (3, 5, 33, 70, 12, (3, 3), (3, 3), (0, 1), (1, 2), 1), (1, 4, 5, 2100, 8, (1, 9), (1, 1), (0, 4), (1, 1), 1),
    # tiny planes with many channels (tiles of several images, channels split over a cluster, the last chunk short), one pixel
    (5, 512, 4, 4, 512, (3, 3), (1, 1), (1, 1), (1, 1), 1), (3, 250, 2, 2, 96, (3, 3), (1, 1), (1, 1), (1, 1), 1),
    (1, 96, 1, 1, 130, (3, 3), (1, 1), (1, 1), (1, 1), 1), (9, 72, 3, 5, 40, (5, 5), (1, 1), (2, 2), (1, 1), 2),
    # rows staged as 16-byte vectors from an unaligned first column, odd padding, wide dilation
    (2, 32, 40, 60, 24, (3, 3), (1, 1), (3, 5), (3, 5), 4), (1, 48, 28, 28, 48, (1, 7), (1, 1), (0, 3), (1, 1), 3),
    (2, 48, 28, 28, 48, (7, 1), (2, 1), (3, 0), (1, 1), 3),
    # no tile holds a patch of this dilation: the one-thread-per-output kernel
    (1, 2, 560, 560, 3, (3, 3), (1, 1), (0, 0), (270, 270), 1), (1, 2, 40, 40, 2, (35, 35), (1, 1), (17, 17), (1, 1), 2),
    # column strides far beyond the width: whole column phases of a staged row would be millions of columns
    (1, 1, 5000, 1, 1, (3, 1), (1, 3000000), (0, 0), (1, 1), 1), (2, 8, 30, 5, 8, (3, 3), (1, 2147483647), (1, 1), (1, 1), 1),
    (2, 6, 9, 40, 4, (3, 3), (2, 50), (1, 1), (1, 1), 2),
    # groups of one filter whose patches are mostly halo: the one-thread-per-output kernel, one channel a group and two
    (3, 21, 6, 6, 21, (11, 11), (3, 3), (15, 15), (3, 3), 21), (5, 30, 14, 14, 30, (5, 5), (2, 2), (8, 8), (4, 4), 30),
    (7, 14, 28, 6, 14, (1, 7), (1, 1), (0, 9), (1, 3), 14), (6, 20, 7, 7, 10, (7, 7), (2, 2), (9, 9), (3, 3), 10),
]


@pytest.mark.parametrize("cfg", CASES)
def test_staged_fp32_kernel(cfg):
    N, C_in, H, W, C_out, k, st, pd, dl, g = cfg
    dev = torch.device("cuda:0")
    x, w = synth.make_layer_tensors(N, C_in, H, W, C_out, k[0], k[1], g, synth.layer_seed(91, N, C_in, H, C_out, g))
    d = gconv.gconv_desc_create_2d(N, C_in, H, W, C_out, k[0], k[1], st[0], st[1], pd[0], pd[1], dl[0], dl[1], g)
    try:
        gconv.gconv_desc_set_variant(d, gconv.GCONV_VARIANT_DIRECT_GENERIC)
        Ho, Wo = gconv.gconv_out_shape(d)
        n = N * C_out * Ho * Wo
        guard, sentinel = 64, float(np.float32(-1.2345678e30))
        y_full = torch.full((n + 2 * guard,), sentinel, dtype=torch.float32, device=dev)
        wp = torch.empty(gconv.gconv_packed_bytes(d) // 4, dtype=torch.float32, device=dev)
        gconv.gconv_pack_weights(d, torch.from_numpy(w).to(dev), wp)
        gconv.gconv_forward(d, torch.from_numpy(x).to(dev), wp, y_full[guard:guard + n])
        assert gconv.gconv_last_status(d) == gconv.GCONV_OK
        assert bool((y_full[:guard] == sentinel).all()) and bool((y_full[guard + n:] == sentinel).all())
        ref = oracle.gconv_ref(x, w, st, pd, dl, g, threads=oracle.max_threads())
        got = y_full[guard:guard + n].cpu().numpy().reshape(ref.shape)
        assert rel_err(got, ref) <= 1e-5          # FP32 sums of at most 4608 products: 2^-24 x sqrt(4608) is 4e-6
    finally:
        gconv.gconv_desc_destroy(d)


@pytest.mark.parametrize("cfg", [(2, 3, 29, 37, 20, (7, 7), (2, 2), (3, 3), (1, 1), 1), (3, 250, 2, 2, 96, (3, 3), (1, 1), (1, 1), (1, 1), 1),
                                 (2, 8, 20, 28, 17, (3, 5), (1, 1), (2, 4), (2, 2), 1), (9, 72, 3, 5, 40, (5, 5), (1, 1), (2, 2), (1, 1), 2)])
def test_weights_that_are_not_finite(cfg):
    """Taps outside the image are left out, whatever their weight; packing finite weights into the same buffer afterwards is as ever."""
    N, C_in, H, W, C_out, k, st, pd, dl, g = cfg
    dev = torch.device("cuda:0")
    x, w = synth.make_layer_tensors(N, C_in, H, W, C_out, k[0], k[1], g, 17)
    x[x == 0] = 0.5
    bad = w.copy()
    bad[0, 0, 0, 0], bad[1, -1, -1, -1], bad[C_out - 1, 0, 0, -1] = np.inf, -np.inf, np.nan
    d = gconv.gconv_desc_create_2d(N, C_in, H, W, C_out, k[0], k[1], st[0], st[1], pd[0], pd[1], dl[0], dl[1], g)
    try:
        gconv.gconv_desc_set_variant(d, gconv.GCONV_VARIANT_DIRECT_GENERIC)
        Ho, Wo = gconv.gconv_out_shape(d)
        wp = torch.empty(gconv.gconv_packed_bytes(d) // 4, dtype=torch.float32, device=dev)
        for weights in (bad, w):
            y = torch.empty(N, C_out, Ho, Wo, device=dev)
            gconv.gconv_pack_weights(d, torch.from_numpy(weights).to(dev), wp)
            gconv.gconv_forward(d, torch.from_numpy(x).to(dev), wp, y)
            assert gconv.gconv_last_status(d) == gconv.GCONV_OK
            ref, got = oracle.gconv_ref(x, weights, st, pd, dl, g, threads=oracle.max_threads()), y.cpu().numpy().astype(np.float64)
            fin = np.isfinite(ref)
            assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
            assert 0 < fin.sum() and rel_err(got[fin], ref[fin]) <= 1e-5
    finally:
        gconv.gconv_desc_destroy(d)
