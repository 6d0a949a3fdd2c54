"""FP32 products and convolutions whose last tile is mostly empty: rows past M
and columns past N are zeros that nobody reads, so a tile with 8 columns
gives exact results in every layout and costs no more than a full one."""
import numpy as np
import pytest
import torch

import oracle.nk_oracle as O
from paper_2307_16080_gb300 import synth
from tests.gpu_util import DEV, Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    import paper_2307_16080_gb300.nk as m
    m.lib()
    return m


def _layout(x, transposed, pad):
    """x on the device, row- or column-major, with `pad` elements between rows."""
    r, c = x.shape
    t = torch.full((c, r + pad) if transposed else (r, c + pad), float("inf"), device=DEV)
    t = t[:, :r].t() if transposed else t[:, :c]
    t.copy_(dev(x))
    return t


@pytest.mark.parametrize("at", [False, True])
@pytest.mark.parametrize("bt", [False, True])
@pytest.mark.parametrize("M,N,K", [(1, 1, 16), (8, 8, 144), (72, 4, 320), (200, 92, 336), (129, 63, 33)])
def test_ragged_tiles_in_every_layout(nk, M, N, K, at, bt):
    A, B = synth.small_ints(911, 0, (M, K)), synth.small_ints(911, 1, (K, N))
    want = (A.astype(np.float64) @ B).astype(np.float32)
    for pad in (0, 4, 3):   # what lies between the rows is infinite
        a, b = _layout(A, at, pad), _layout(B, bt, pad)
        for sched in (None, (64, 64, 16, 1, 2, 1), (64, 64, 16, 1, 2, 3), (128, 128, 16, 1, 2, 1)):
            C = Canary((M, N), strides=(N + 1, 1))
            nk.nk_matmul(a, b, C.t, "f32", schedule=sched)
            nk.nk_sync_status()
            assert np.array_equal(host(C.t), want), (pad, sched)
            C.check()


@pytest.mark.parametrize("n,h,w,c,f,k,stride", [(1, 5, 5, 4, 8, 3, 1), (2, 9, 7, 16, 16, 3, 2), (1, 3, 3, 3, 5, 3, 1)])
def test_ragged_convolutions(nk, n, h, w, c, f, k, stride):
    I, W = synth.small_ints(912, 0, (n, h, w, c)), synth.small_ints(912, 1, (k, k, c, f))
    want = O.conv2d_nhwc_hwcf(I, W, stride=(stride,) * 2, pad=(1,) * 4)
    for sched in (None, (64, 64, 16, 1, 2, 1), (128, 128, 16, 1, 2, 1)):
        out = torch.empty(*want.shape, device=DEV)
        nk.nk_conv2d_nhwc_hwcf(dev(I), dev(W), out, (stride,) * 2, (1, 1), (1,) * 4, "f32", schedule=sched)
        nk.nk_sync_status()
        assert np.array_equal(host(out), want)


@pytest.mark.parametrize("M,N,K", [(700, 700, 700), (8192, 64, 576), (2500, 130, 400)])
def test_built_in_tile_is_no_slower_than_plain_64(nk, M, N, K):
    A, B, C = torch.ones(M, K, device=DEV), torch.ones(K, N, device=DEV), torch.empty(M, N, device=DEV)
    t = []
    for sched in (None, (64, 64, 16, 1, 2, 1)):
        g = torch.cuda.CUDAGraph()
        nk.nk_matmul(A, B, C, "f32", schedule=sched)
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            for _ in range(8):
                nk.nk_matmul(A, B, C, "f32", schedule=sched)
        t.append(_time(g.replay))
    assert t[0] <= 1.05 * t[1]


def _time(call):
    for _ in range(3):
        call()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        a.record()
        for _ in range(50):
            call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("narrow", [8, 16])
def test_narrow_product_costs_no_more_than_a_full_tile(nk, narrow):
    """One 64-column tile either way, and the reads of the narrow one are fewer
    (reading the last columns again for those that do not exist took 2.7 times
    as long)."""
    t = {}
    for N in (narrow, 64):
        A, B, C = torch.ones(8192, 144, device=DEV), torch.ones(144, N, device=DEV), torch.empty(8192, N, device=DEV)
        g = torch.cuda.CUDAGraph()
        nk.nk_matmul(A, B, C, "f32")
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            for _ in range(8):
                nk.nk_matmul(A, B, C, "f32")
        t[N] = _time(g.replay)
    assert t[narrow] <= 1.3 * t[64]
