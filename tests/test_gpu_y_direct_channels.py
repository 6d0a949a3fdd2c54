"""NCHW kernels over several input channels: exact channel counts, rows and
channels that start at every 4-byte offset, widths around a warp's and a block's
outputs, a last block of fewer than four rows; bitwise on small integers,
canary-padded outputs."""
import pytest
import torch

from paper_2307_16080_gb300 import synth
from tests.gpu_util import DEV, Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ow", [1, 4, 127, 130, 512, 515])
@pytest.mark.parametrize("oh,ci,co,k,pad,gap,igap", [(1, 2, 1, 3, 0, 0, 0), (9, 3, 3, 3, 0, 0, 1), (6, 3, 2, 3, 1, 1, 0),
                                                     (5, 2, 5, 5, 2, 3, 2), (7, 3, 4, 1, 0, 2, 0), (4, 5, 6, 3, 0, 5, 4)])
def test_channels_bitwise(ow, oh, ci, co, k, pad, gap, igap):
    from paper_2307_16080_gb300 import nk
    n, h, w = 2, oh + k - 1 - 2 * pad, ow + k - 1 - 2 * pad
    if h < 1 or w < 1:
        pytest.skip("the padding alone covers the filter")
    I, K = dev(synth.small_ints(931, 0, (n, ci, h, w))), dev(synth.small_ints(931, 1, (co, ci, k, k)))
    b, C0 = dev(synth.small_ints(931, 2, (co,))), dev(synth.small_ints(931, 3, (n, co, oh, ow)))
    # input rows igap floats apart, channels another igap, all from an odd offset
    sc = h * (w + igap) + igap
    Ip = torch.empty(n * ci * sc + igap + 1, device=DEV).as_strided((n, ci, h, w), (ci * sc, sc, w + igap, 1), igap)
    Ip.copy_(I)
    want = torch.nn.functional.conv2d(I.double(), K.double(), b.double(), padding=pad)
    for acc, relu in ((False, False), (True, True)):
        O = Canary((n, co, oh, ow), strides=(co * oh * (ow + gap) + gap, oh * (ow + gap), ow + gap, 1), pad=4097)
        O.t.copy_(C0)
        nk.nk_conv2d_nchw_fchw(Ip, K, O.t, pad=(pad,) * 4, bias=b, relu=relu, accumulate=acc)
        nk.nk_sync_status()
        ref = (want + C0.double()).relu() if acc else want
        assert torch.equal(O.t, ref.float())
        O.check()
