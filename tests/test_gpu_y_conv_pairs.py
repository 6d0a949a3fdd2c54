"""Convolutions large enough for the built-in CTA-pair tiles: the same bits as
one CTA per tile (each output sums its taps and channels in the same order),
ragged tails of tiles and filters included, and small-integer sums equal to the
reference bit for bit."""
import pytest
import torch

from tests.gpu_util import DEV, Canary

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,c,f,k,s,out16", [(64, 28, 128, 256, 3, 2, True), (65, 28, 128, 136, 3, 1, True),
                                               (33, 33, 72, 72, 3, 1, False), (150, 14, 256, 264, 3, 2, True),
                                               (170, 7, 512, 520, 1, 1, False)])
def test_pairs_against_single_tiles(n, h, c, f, k, s, out16):
    from paper_2307_16080_gb300 import nk
    from paper_2307_16080_gb300 import nk_tune as nt
    pad, oh = k // 2, (h + 2 * (k // 2) - k) // s + 1
    p = nt.conv_problem(n, h, h, c, f, k, k, s, pad)
    assert nt.nk_default_schedule(p) == (256, 128, 64, 2, 3, 1)
    g = torch.Generator(device=DEV).manual_seed(n)
    dt = torch.bfloat16 if out16 else torch.float32
    b = torch.randint(-4, 5, (f,), generator=g, device=DEV).float()
    for ints in (False, True):
        if ints:
            I = torch.randint(-2, 3, (n, h, h, c), generator=g, device=DEV).bfloat16()
            W = torch.randint(-2, 3, (k, k, c, f), generator=g, device=DEV).float()
        else:
            I = torch.randn(n, h, h, c, generator=g, device=DEV).bfloat16()
            W = torch.randn(k, k, c, f, generator=g, device=DEV)
        Wp = nk.nk_conv2d_pack_weights(W)
        O, R = Canary((n, oh, oh, f), dt), Canary((n, oh, oh, f), dt)
        nk.nk_conv2d_nhwc_hwcf(I, Wp, O.t, (s, s), (1, 1), (pad,) * 4, "bf16", bias=b, relu=True)
        nk.nk_conv2d_nhwc_hwcf(I, Wp, R.t, (s, s), (1, 1), (pad,) * 4, "bf16", bias=b, relu=True,
                               schedule=(128, 64, 64, 1, 3, 1))
        nk.nk_sync_status()
        assert torch.equal(O.t, R.t)
        O.check()
        if ints:
            want = torch.nn.functional.conv2d(I.float().permute(0, 3, 1, 2).double(), W.double().permute(3, 2, 0, 1),
                                              b.double(), stride=s, padding=pad).relu().permute(0, 2, 3, 1)
            assert torch.equal(O.t, want.float().to(dt))
