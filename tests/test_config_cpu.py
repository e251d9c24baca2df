"""The host side's choices, without a GPU: every shape the tensor-core variant takes has a kernel that runs its configuration, and the
staged FP32 kernel's buffers hold what it puts there."""
import math
import os
import random
import subprocess

import pytest

from paper_2006_09791_b200 import build as gbuild
from paper_2006_09791_b200 import gconv

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    lib = gbuild.build()
    exe = str(tmp_path_factory.mktemp("probe") / "config_probe")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-o", exe, os.path.join(HERE, "config_probe.cu"), lib,
                           "-Xlinker", "-rpath=" + os.path.dirname(lib)])

    def run(shapes):
        out = subprocess.run([exe], input="\n".join(" ".join(str(v) for v in s) for s in shapes), capture_output=True, text=True, check=True)
        rows = [tuple(int(v) for v in line.split()) if line != "refused" else None for line in out.stdout.splitlines()]
        assert len(rows) == len(shapes)
        return rows

    return run


def _square(N, Ci, H, W, Co, k, stride, g, pad=None):
    p = k // 2 if pad is None else pad
    return (N, Ci, H, W, Co, k, k, stride, stride, p, p, 1, 1, g)


def _drawn(count, seed=11):
    """Shapes around the tensor-core variant's range: pointwise and 3x3, both strides, all alignments, few tiles and many."""
    rng = random.Random(seed)

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    for _ in range(count):
        H = log_int(4, 130)
        W = H if rng.random() < 0.4 else log_int(4, 128)
        cg = rng.choice([2, 4, 8, 12, 16, 24, 32, 40, 48, 64, 72, 96, 128, 192, 256, 320, 512])
        kg = rng.choice([cg, cg, 2 * cg, 4 * cg, 8, 16, 32, 64, 128, 256, 512])
        g = rng.choice([1, 1, 2, 3, 4, 6, 8, 16, 32])
        yield _square(log_int(1, 256), g * cg, H, W, g * kg, rng.choice([3, 3, 1]), rng.choice([1, 1, 2]), g)


# stride 2 on odd planes, wide groups, one pixel tile each and more (group, filter tile) pairs than count as few
ONE_TILE = [(2, 64, 7, 7, 256, 4), (1, 64, 9, 9, 256, 4), (2, 32, 9, 9, 256, 2), (1, 128, 7, 7, 512, 8), (2, 256, 10, 10, 1024, 8)]


def test_every_supported_shape_has_a_kernel(probe):
    shapes = [_square(N, Ci, H, W, Co, 3, 2, g) for N, Ci, H, W, Co, g in ONE_TILE] + list(_drawn(60000))
    rows = probe(shapes)
    assert sum(r is not None and r[0] == gconv.GCONV_VARIANT_IGEMM_TF32 for r in rows) > 20000
    bad = [s for s, r in zip(shapes, rows) if r is not None and r[1] != 1]
    assert not bad, (len(bad), bad[:5])


def test_gathered_pointwise_layers_need_no_workspace(probe):
    """Narrow groups with many filters on planes the tiled copies cannot address: the gather producer, whatever the filter tile."""
    shapes = [_square(31, 128, 7, 7, 2048, 1, 1, 4), _square(14, 512, 7, 3, 8192, 1, 1, 16), _square(23, 48, 117, 7, 1024, 1, 2, 2),
              _square(19, 72, 195, 2, 1536, 1, 1, 3), _square(64, 32, 14, 14, 512, 1, 2, 1)]
    assert [(r[0], r[2]) for r in probe(shapes)] == [(gconv.GCONV_VARIANT_IGEMM_TF32, 0)] * len(shapes)


def test_staged_fp32_buffers_in_64_bits(probe):
    """Column strides up to 2^31 - 1: a staged row is whole column phases, however few columns of it the patch has."""
    huge = [(1, 1, 5000, 1, 1, 3, 1, 1, 3000000, 0, 0, 1, 1, 1), (1, 1, 8, 1, 1, 4, 1, 1, 1 << 30, 0, 0, 1, 1, 1), (2, 8, 30, 5, 8, 3, 3, 1, 2147483647, 1, 1, 1, 1, 1),
            (1, 4, 40, 3, 4, 3, 3, 2, 2147483646, 0, 0, 1, 1, 2), (1, 2, 9, 200000, 2, 3, 3, 1, 70000, 1, 1, 1, 1, 1), (3, 4, 64, 7, 4, 5, 7, 1, 65536, 2, 0, 1, 1, 4)]
    rng = random.Random(3)
    drawn = []
    while len(drawn) < 1500:
        sw = int(math.exp(rng.uniform(0, math.log(2.0 ** 31 - 1))))
        kh, kw, W = rng.randint(1, 9), rng.randint(1, 9), rng.choice([1, 3, 4, 7, 12, 28, 33, 224, 3000])
        pw = rng.randint(0, 4)
        if W + 2 * pw >= kw:
            g = rng.choice([1, 2, 4])
            drawn.append((rng.randint(1, 40), g * rng.randint(1, 9), rng.choice([9, 16, 33, 500]), W, g * rng.randint(1, 20), kh, kw, rng.choice([1, 1, 2, 3]),
                          sw if rng.random() < 0.7 else rng.randint(1, 4), rng.randint(0, 4), pw, 1, 1, g))
    rows = probe(huge + drawn)
    bad = [s for s, r in zip(huge + drawn, rows) if r is None or r[3] == 0]
    assert not bad, (len(bad), bad[:5])
    assert sum(r[3] == 1 for r in rows) > 600, sum(r[3] == 1 for r in rows)
    # more output pixels than 31 bits count: still staged
    assert probe([(70000, 1, 180, 180, 1, 7, 7, 1, 1, 3, 3, 1, 1, 1)])[0][3] == 1


def test_host_batches_are_cut_for_the_variant_that_runs(probe):
    """A batch whose tensor-core layout allows no parts is cut once the descriptor runs the generic variant."""
    rows = probe([_square(8, 576, 16, 16, 2304, 1, 1, 3), _square(92, 6144, 20, 20, 512, 3, 1, 32), _square(27, 384, 42, 42, 32, 3, 1, 2)])
    assert [r[4] for r in rows] == [0, 0, 0] and [r[5] for r in rows] == [4, 5, 5]


def test_groups_of_one_filter_take_the_faster_fp32_kernel(probe):
    """Patches that are mostly halo: one thread per output; wide planes, several filters: staged."""
    plain = [(51, 121, 6, 6, 121, 11, 11, 3, 3, 15, 15, 3, 3, 121), (113, 224, 14, 14, 224, 5, 5, 2, 2, 8, 8, 4, 4, 224), (65, 140, 28, 6, 140, 1, 7, 1, 1, 0, 9, 3, 3, 140),
             (125, 158, 14, 14, 79, 1, 7, 2, 2, 0, 3, 1, 1, 79)]
    staged = [(105, 22, 56, 56, 22, 7, 7, 1, 1, 6, 6, 2, 2, 22), (4, 64, 29, 29, 128, 7, 7, 1, 1, 3, 3, 1, 1, 64), (2, 6, 19, 21, 6, 7, 7, 1, 1, 3, 3, 1, 1, 6)]
    assert [r[3] for r in probe(plain + staged)] == [-1] * 4 + [1] * 3


def test_stride_2_splits_only_where_they_pay(probe):
    """Channels a CTA is spared: too few on row tiles of one segment and on the gather producer's pair tiles, enough, and row tiles of two segments."""
    whole = [(3, 256, 20, 12, 512, 3, 2, 4), (1, 192, 36, 16, 192, 3, 2, 1), (11, 128, 16, 18, 512, 3, 2, 8), (21, 128, 9, 27, 256, 3, 2, 4)]
    split = [(1, 256, 36, 24, 64, 3, 2, 1), (1, 64, 56, 56, 128, 3, 2, 1), (2, 512, 27, 19, 1024, 3, 2, 8), (1, 768, 5, 5, 768, 3, 2, 1)]
    assert [r[6] > 0 for r in probe([_square(*s) for s in whole + split])] == [False] * 4 + [True] * 4


def test_pointwise_stride_2_filter_tiles_follow_the_tiles_there_are(probe):
    """Even rows only, a tile four segments of one row each: on 8- and 16-wide planes more tiles than pixels / 128, so wider filter tiles."""
    rows = probe([_square(30, 256, 8, 8, 512, 1, 2, 1, 0), _square(32, 1024, 16, 16, 128, 1, 2, 2, 0), _square(64, 256, 56, 56, 512, 1, 2, 1, 0)])
    assert [r[8] for r in rows] == [128, 64, 256] and all(r[7] for r in rows)


def test_tall_narrow_planes_are_flat_where_row_boxes_take_many_more_waves(probe):
    flat = [(122, 128, 77, 4, 256, 3, 1, 2), (26, 64, 146, 8, 128, 3, 1, 1), (36, 256, 13, 4, 256, 3, 1, 1)]
    boxes = [(91, 64, 11, 8, 128, 3, 1, 1), (70, 32, 49, 4, 32, 3, 1, 1), (2, 32, 18, 4, 32, 3, 1, 1), (64, 256, 12, 12, 256, 3, 1, 1)]
    assert [r[7] for r in probe([_square(*s) for s in flat + boxes])] == [0] * 3 + [1] * 4
