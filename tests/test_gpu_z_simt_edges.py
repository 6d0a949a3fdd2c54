"""FP32 products and convolutions at the edges of the CUDA-core kernel: every
copy mode (odd and 16-byte row strides, row- and column-major operands, the
im2col gather with and without 16-byte channels), tiles of one to several,
reductions shorter than a cluster's slices, and tall outputs.  Small-integer
operands make every sum exact, so any order of addition gives the same bits."""
import numpy as np
import pytest
import torch

import oracle.nk_oracle as O
from paper_2307_16080_gb300 import synth
from tests.gpu_util import DEV, Canary, dev, host

pytestmark = pytest.mark.gpu


def _view(x, major, pad):
    """x on the device, row- or column-major, with `pad` spare elements per row."""
    src = x if major == "row" else x.T
    buf = torch.full((src.shape[0], src.shape[1] + pad), float("nan"), device=DEV)
    buf[:, :src.shape[1]] = dev(src)
    v = buf[:, :src.shape[1]]
    return v if major == "row" else v.t()


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (3, 5, 15), (64, 64, 64), (65, 63, 17), (129, 260, 100), (300, 4, 1000),
                                   (4, 500, 33), (200, 300, 129), (1000, 1000, 48)])
@pytest.mark.parametrize("am,bm,pad", [("row", "row", 0), ("row", "row", 1), ("col", "row", 4), ("row", "col", 3),
                                       ("col", "col", 4), ("col", "col", 1)])
def test_matmul_edges_bitwise(M, N, K, am, bm, pad):
    from paper_2307_16080_gb300 import nk
    A, B = synth.small_ints(911, 0, (M, K)), synth.small_ints(911, 1, (K, N))
    bias, C0 = synth.small_ints(911, 2, (N,)), synth.small_ints(911, 3, (M, N))
    want = np.maximum(A.astype(np.float64) @ B + C0 + bias, 0).astype(np.float32)
    for sched in (None, (128, 128, 16, 1, 2, 1), (64, 64, 16, 1, 2, 1)):
        C = Canary((M, N), strides=(N + pad, 1))
        C.t.copy_(dev(C0))
        nk.nk_matmul(_view(A, am, pad), _view(B, bm, pad), C.t, "f32", bias=dev(bias), relu=True, accumulate=True,
                     schedule=sched)
        nk.nk_sync_status()
        assert np.array_equal(host(C.t), want)
        C.check()


@pytest.mark.parametrize("n,h,w,c,f,k,s,d,p", [(1, 1, 1, 1, 1, 1, 1, 1, 0), (2, 9, 7, 3, 5, 3, 1, 1, 1),
                                               (3, 14, 15, 20, 70, 3, 2, 1, 1), (1, 20, 20, 64, 130, 3, 1, 2, 2),
                                               (5, 8, 8, 12, 64, 5, 1, 1, 4), (2, 40, 33, 8, 9, 1, 2, 1, 0)])
def test_conv_edges_bitwise(n, h, w, c, f, k, s, d, p):
    from paper_2307_16080_gb300 import nk
    I, W, b = synth.small_ints(912, 0, (n, h, w, c)), synth.small_ints(912, 1, (k, k, c, f)), synth.small_ints(912, 2, (f,))
    want = O.conv2d_nhwc_hwcf(I, W, stride=(s, s), dilation=(d, d), pad=(p,) * 4) + b
    C = Canary(want.shape)
    nk.nk_conv2d_nhwc_hwcf(dev(I), dev(W), C.t, (s, s), (d, d), (p,) * 4, "f32", bias=dev(b))
    nk.nk_sync_status()
    assert np.array_equal(host(C.t), want.astype(np.float32))
    C.check()


def test_tall_output_keeps_its_grid():
    """More 64-row tiles than a grid has rows."""
    from paper_2307_16080_gb300 import nk
    M = 65535 * 64 + 129
    A = torch.arange(M, device=DEV, dtype=torch.float32).remainder(31).view(M, 1)
    C = torch.empty(M, 1, device=DEV)
    nk.nk_matmul(A, torch.full((1, 1), 2.0, device=DEV), C, "f32")
    nk.nk_sync_status()
    assert torch.equal(C, A * 2)
