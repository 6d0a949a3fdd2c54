"""The single-input-channel NCHW kernel where a row's alignment, its end and
the run of rows per thread can go wrong: widths around a warp's 128 and a
block's 512 outputs, rows that start at every 4-byte offset, one output row to
more than a run, one to five output channels, padding, accumulate and ReLU;
bitwise on small integers, canary-padded outputs."""
import numpy as np
import pytest
import torch

from paper_2307_16080_gb300 import synth
from tests.gpu_util import DEV, Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ow", [1, 3, 4, 127, 128, 129, 130, 131, 511, 514])
@pytest.mark.parametrize("oh,co,k,pad,gap", [(1, 1, 3, 0, 0), (9, 3, 3, 0, 0), (17, 3, 3, 1, 1), (26, 5, 5, 2, 3),
                                             (6, 4, 1, 0, 2), (8, 2, 3, 0, 5)])
def test_rows_bitwise(ow, oh, co, k, pad, gap):
    from paper_2307_16080_gb300 import nk
    n, h, w = 2, oh + k - 1 - 2 * pad, ow + k - 1 - 2 * pad
    if h < 1 or w < 1:
        pytest.skip("the padding alone covers the filter")
    I, K = synth.small_ints(921, 0, (n, 1, h, w)), synth.small_ints(921, 1, (co, 1, k, k))
    b, C0 = synth.small_ints(921, 2, (co,)), synth.small_ints(921, 3, (n, co, oh, ow))
    xp = np.pad(I[:, 0].astype(np.float64), ((0, 0), (pad, pad), (pad, pad)))
    want = np.zeros((n, co, oh, ow)) + b[None, :, None, None]
    for i in range(k):
        for j in range(k):
            want += K[None, :, 0, i, j, None, None] * xp[:, None, i:i + oh, j:j + ow]
    for acc, relu in ((False, False), (True, True)):
        O = Canary((n, co, oh, ow), strides=(co * oh * (ow + gap) + gap, oh * (ow + gap), ow + gap, 1), pad=4097)
        O.t.copy_(dev(C0))
        nk.nk_conv2d_nchw_fchw(dev(I), dev(K), O.t, pad=(pad,) * 4, bias=dev(b), relu=relu, accumulate=acc)
        nk.nk_sync_status()
        ref = np.maximum(want + C0, 0) if acc else want
        assert np.array_equal(host(O.t), ref.astype(np.float32))
        O.check()
