"""FP32 convolutions on both sides of the extent (32000) from which positions no
longer fit the gather's 16 bits: exact on small integers, and as fast for each
pixel as the short ones."""
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


@pytest.mark.parametrize("sched", [None, (64, 64, 16, 1, 2, 1), (128, 128, 16, 1, 2, 1), (64, 64, 16, 1, 2, 2)])
@pytest.mark.parametrize("h,w,c,f,kh,kw,stride,dil", [
    (1, 31990, 4, 8, 1, 5, 1, 1), (1, 32100, 4, 8, 1, 5, 1, 1), (1, 40001, 3, 70, 1, 3, 1, 1),
    (2, 33000, 8, 5, 3, 3, 2, 1), (33001, 2, 4, 66, 3, 2, 1, 1), (1, 40000, 4, 8, 1, 3, 1, 7), (66000, 1, 4, 4, 4, 1, 3, 2)])
def test_either_side_of_the_packed_positions(nk, h, w, c, f, kh, kw, stride, dil, sched):
    I, W = synth.small_ints(921, 0, (1, h, w, c), -3, 3), synth.small_ints(921, 1, (kh, kw, c, f), -3, 3)
    pad = (1 if kh > 1 else 0,) * 2 + (1 if kw > 1 else 0,) * 2
    st, dl = (stride, stride), (dil, dil)
    want = O.conv2d_nhwc_hwcf(I, W, stride=st, dilation=dl, pad=pad)
    out = Canary(want.shape)
    nk.nk_conv2d_nhwc_hwcf(dev(I), dev(W), out.t, st, dl, pad, "f32", schedule=sched)
    nk.nk_sync_status()
    assert np.array_equal(host(out.t), want)
    out.check()


def test_a_long_signal_costs_what_two_short_ones_do(nk):
    """The same pixels as one signal or two: 3.5 times as long through the
    kernel that loads one value at a time."""
    W, best = torch.ones(1, 3, 64, 64, device=DEV), {}
    for n, w in ((1, 40000), (2, 20000)):
        I, out = torch.ones(n, 1, w, 64, device=DEV), torch.empty(n, 1, w, 64, device=DEV)
        run = lambda: nk.nk_conv2d_nhwc_hwcf(I, W, out, (1, 1), (1, 1), (0, 0, 1, 1), "f32")  # noqa: E731
        for _ in range(3):
            run()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best[n] = float("inf")
        for _ in range(5):
            a.record()
            for _ in range(20):
                run()
            b.record()
            b.synchronize()
            best[n] = min(best[n], a.elapsed_time(b))
    assert best[1] <= 1.4 * best[2]
