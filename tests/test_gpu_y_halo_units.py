"""Unit indices of the window convolution: launches small enough for the exact
multiply-high and launches past it (tiles x units >= 2^32) split their index the
same way, so repeated images give repeated outputs, bit for bit."""
import pytest
import torch

from tests.gpu_util import DEV, Canary

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,f", [(7, 9, 72), (3, 57, 136), (40000, 8, 16), (131072, 8, 16)])
@pytest.mark.parametrize("sched", [(128, 64, 192, 1, 2, 1), (256, 64, 192, 1, 4, 1), (128, 64, 576, 1, 2, 1)])
def test_repeated_images(n, h, f, sched):
    from paper_2307_16080_gb300 import nk
    c, reps = 16, 8 if n > 8 else 1
    g = torch.Generator(device=DEV).manual_seed(h + f)
    base = torch.randn(n // reps if reps == 1 else reps, h, h, c, generator=g, device=DEV).bfloat16()
    I = base if reps == 1 else base.repeat(n // reps, 1, 1, 1)
    W = torch.randn(3, 3, c, f, generator=g, device=DEV)
    Wp = nk.nk_conv2d_pack_weights(W)
    O = Canary((n, h, h, f))
    nk.nk_conv2d_nhwc_hwcf(I, Wp, O.t, (1, 1), (1, 1), (1,) * 4, "bf16", schedule=sched)
    nk.nk_sync_status()
    O.check()
    if reps > 1:
        small = torch.empty(reps, h, h, f, device=DEV)
        nk.nk_conv2d_nhwc_hwcf(base, Wp, small, (1, 1), (1, 1), (1,) * 4, "bf16", schedule=sched)
        nk.nk_sync_status()
        assert torch.equal(O.t.reshape(n // reps, -1), small.reshape(1, -1).expand(n // reps, -1))
        got = small
    else:
        got = O.t
    x, w = base.double().permute(0, 3, 1, 2), W.bfloat16().double().permute(3, 2, 0, 1)
    want = torch.nn.functional.conv2d(x, w, padding=1).permute(0, 2, 3, 1)
    mag = torch.nn.functional.conv2d(x.abs(), w.abs(), padding=1).permute(0, 2, 3, 1)
    # 144 products summed in FP32 in any order: error at most 144 * 2^-23 of the sum of magnitudes
    assert ((got.double() - want).abs() <= 144 * 2.0 ** -23 * mag + 1e-30).all()
