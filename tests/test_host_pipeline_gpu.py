"""gconv_forward_host where it overlaps the copies and kernels of parts of the batch: against the device-resident call on the same
inputs, for batches that do not divide into parts, planes that are not a multiple of 16 bytes, a layer with a workspace, FP32
variants, repeated calls with other buffers, several threads, and a captured stream."""
import threading

import numpy as np
import pytest
import torch

from paper_2006_09791_b200 import build as gbuild
from paper_2006_09791_b200 import gconv, synth
from paper_2006_09791_b200.torch_util import attach_workspace

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    gbuild.build()


class _Host:
    def __init__(self, N, C, H, W, K, k, stride, g, seed=3):
        dev = torch.device("cuda:0")
        x, w = synth.make_layer_tensors(N, C, H, W, K, k, k, g, seed)
        self.d = gconv.gconv_desc_create(N, C, H, W, K, k, k, stride, k // 2, 1, g)
        self.ws = attach_workspace(self.d, dev)
        ho, wo = gconv.gconv_out_shape(self.d)
        self.wp = torch.empty(gconv.gconv_packed_bytes(self.d) // 4, device=dev)
        gconv.gconv_pack_weights(self.d, torch.from_numpy(w).to(dev), self.wp)
        self.xh = torch.from_numpy(x).pin_memory()
        self.xs, self.ys = torch.empty(x.shape, device=dev), torch.empty((N, K, ho, wo), device=dev)
        self.want = torch.empty((N, K, ho, wo), device=dev)
        xd = self.xh.to(dev)
        gconv.gconv_forward(self.d, xd, self.wp, self.want)
        assert gconv.gconv_last_status(self.d) == gconv.GCONV_OK
        self.want = self.want.cpu().numpy()
        # a part's kernel may take another tiling than the whole batch's: the same products in another order of FP32 sums
        self.tol = 2e-5 * float(np.max(np.abs(self.want)))

    def run(self, stream, pinned=True):
        yh = torch.full(self.want.shape, float("nan"))
        yh = yh.pin_memory() if pinned else yh
        gconv.gconv_forward_host(self.d, self.xh, self.wp, yh, self.xs, self.ys, stream)
        return yh

    def check(self, yh):
        assert float(np.max(np.abs(yh.numpy() - self.want))) <= self.tol

    def close(self):
        gconv.gconv_desc_destroy(self.d)


@pytest.mark.parametrize("cfg", [(64, 64, 28, 28, 64, 3, 1, 8), (37, 64, 32, 32, 64, 3, 1, 2), (61, 60, 15, 15, 60, 3, 1, 60), (50, 64, 13, 13, 64, 3, 2, 1),
                                 (33, 128, 10, 54, 128, 3, 1, 4), (40, 16, 30, 31, 16, 5, 1, 2), (2, 64, 112, 112, 64, 3, 1, 4),
                                 (1, 64, 112, 112, 64, 3, 1, 4), (128, 32, 8, 8, 32, 3, 1, 4), (64, 128, 56, 56, 32, 1, 1, 1),
                                 # no workspace for the whole batch, one for a shorter part
                                 (103, 64, 19, 19, 256, 3, 1, 8), (88, 192, 19, 19, 512, 3, 1, 4)])
def test_host_parts(cfg):
    L = _Host(*cfg)
    try:
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        for pinned in (True, True, False):
            yh = L.run(s, pinned)
            assert gconv.gconv_last_status(L.d, s) == gconv.GCONV_OK     # synchronises the stream: y is complete
            L.check(yh)
    finally:
        L.close()


@pytest.mark.parametrize("cfg,shift", [((64, 32, 56, 56, 128, 3, 1, 4), 0), ((64, 64, 56, 56, 64, 3, 1, 4), -1000), ((64, 64, 56, 56, 64, 3, 1, 4), 1 << 20)])
def test_host_buffers_that_share_memory(cfg, shift):
    """y in the place of x, before it and behind it: the whole input is read before any output is written."""
    L = _Host(*cfg)
    try:
        s = torch.cuda.Stream()
        at_x, at_y = max(0, -shift), max(0, shift)
        both = torch.empty(max(at_x + L.xh.numel(), at_y + L.want.size)).pin_memory()
        x, y = both[at_x:at_x + L.xh.numel()], both[at_y:at_y + L.want.size]
        torch.cuda.synchronize()
        for _ in range(3):
            x.copy_(L.xh.view(-1))
            gconv.gconv_forward_host(L.d, x, L.wp, y, L.xs, L.ys, s)
            assert gconv.gconv_last_status(L.d, s) == gconv.GCONV_OK
            L.check(y.view(L.want.shape))
    finally:
        L.close()


def test_calls_of_several_streams_move_whole_batches():
    """A call that finds another stream's call in flight copies x and y whole (the callers overlap by themselves); alone, it copies parts."""
    L = _Host(64, 64, 28, 28, 64, 3, 1, 8)
    try:
        streams = [torch.cuda.Stream() for _ in range(3)]
        stages = [(torch.empty_like(L.xs), torch.empty_like(L.ys)) for _ in streams]
        ys = [torch.full(L.want.shape, float("nan")).pin_memory() for _ in streams]

        def copies(body):
            torch.cuda.synchronize()
            with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU, torch.profiler.ProfilerActivity.CUDA]) as prof:
                body()
                torch.cuda.synchronize()
            names = [e.name for e in prof.events()]
            return sum("Memcpy HtoD" in n for n in names), sum("Memcpy DtoH" in n for n in names)

        def call(k):
            gconv.gconv_forward_host(L.d, L.xh, L.wp, ys[k], *stages[k], streams[k])

        def overlapped():
            with torch.cuda.stream(streams[0]):
                torch.cuda._sleep(400_000_000)                  # 0.2 s: the first call is in flight until the others are enqueued
            call(0)                                             # (nothing of the library's is in flight yet: parts)
            call(1)
            call(2)
            call(1)

        alone = copies(lambda: call(0))
        assert alone[0] > 1 and alone[0] == alone[1], alone
        assert copies(overlapped) == (alone[0] + 3, alone[1] + 3)
        assert copies(lambda: call(2)) == alone
        for y in ys:
            L.check(y)
    finally:
        L.close()


def test_host_parts_from_several_threads_and_in_a_graph():
    L = _Host(48, 64, 32, 32, 64, 3, 1, 4)
    other = [(torch.empty_like(L.xs), torch.empty_like(L.ys)) for _ in range(2)]
    errors = []
    try:
        torch.cuda.synchronize()

        def work(k):
            try:
                s = torch.cuda.Stream()
                for _ in range(4):
                    yh = torch.full(L.want.shape, float("nan")).pin_memory()
                    gconv.gconv_forward_host(L.d, L.xh, L.wp, yh, other[k][0], other[k][1], s)
                    s.synchronize()
                    L.check(yh)
            except Exception as e:      # noqa: BLE001
                errors.append(e)

        threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors, errors
        s = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        yh = torch.full(L.want.shape, float("nan")).pin_memory()
        with torch.cuda.graph(g, stream=s):
            gconv.gconv_forward_host(L.d, L.xh, L.wp, yh, L.xs, L.ys, s)
        g.replay()
        torch.cuda.synchronize()
        L.check(yh)
    finally:
        L.close()
