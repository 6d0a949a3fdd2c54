"""Operand conversions at the edges of their tiles and words: rows and columns
around 8, 64 and 128, unaligned inputs and outputs, both orientations, every
kind.  BF16 and the hi / lo split are compared with torch's conversions bit for
bit, E4M3 (a scale of 448 / 3.5 = 128, exact codes) likewise."""
import pytest
import torch

from tests.gpu_util import DEV, Canary, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1, 1), (1, 7), (3, 8), (9, 15), (63, 65), (64, 64), (127, 129), (130, 63),
                                       (300, 2049)])
@pytest.mark.parametrize("pad_in,pad_out", [(0, 0), (1, 1), (4, 8), (3, 16)])
@pytest.mark.parametrize("transpose", [False, True])
def test_casts_bitwise(rows, cols, pad_in, pad_out, transpose):
    from paper_2307_16080_gb300 import nk
    g = torch.Generator(device=DEV).manual_seed(rows * 10007 + cols)
    buf = torch.full((rows, cols + pad_in), float("nan"), device=DEV)
    x = buf[:, :cols]
    x.copy_(torch.randn(rows, cols, generator=g, device=DEV))
    shape = (cols, rows) if transpose else (rows, cols)
    ld = shape[1] + pad_out
    want = x.t() if transpose else x
    out = Canary(shape, torch.bfloat16, strides=(ld, 1))
    nk.nk_cast_bf16(x, out.t, transpose)
    assert torch.equal(out.t, want.bfloat16())
    out.check()
    hi, lo = Canary(shape, torch.bfloat16, strides=(ld, 1)), Canary(shape, torch.bfloat16, strides=(ld, 1))
    nk.nk_split_bf16x3(x, hi.t, lo.t, transpose)
    assert torch.equal(hi.t, want.bfloat16()) and torch.equal(lo.t, (want - want.bfloat16().float()).bfloat16())
    hi.check(), lo.check()
    y = torch.randint(-7, 8, (rows, cols), generator=g, device=DEV).float() / 2
    y[0, 0] = 3.5
    x.copy_(y)
    q, amax, scale = Canary(shape, torch.uint8, strides=(ld, 1)), torch.empty(1, device=DEV), torch.empty(1, device=DEV)
    flat = y.reshape(-1)
    nk.nk_amax(flat, amax)
    nk.nk_cast_fp8(x, amax, q.t, transpose, scale_out=scale)
    nk.nk_sync_status()
    assert host(amax)[0] == 3.5 and host(scale)[0] == 128.0
    ref = ((y.t() if transpose else y) * 128).to(torch.float8_e4m3fn).contiguous().view(torch.uint8)
    assert torch.equal(q.t, ref)
    q.check()


@pytest.mark.parametrize("n", [1, 4, 1000, 4 * 1024 * 256 * 7 + 4, 4 * 1024 * 256 * 8 + 1024, 3 * 10**6 + 1])
def test_amax_finds_the_last_element_and_keeps_nan(n):
    from paper_2307_16080_gb300 import nk
    x, out = torch.zeros(n, device=DEV), torch.empty(1, device=DEV)
    for at in (0, n // 2, n - 1):
        x[at] = -5.0 - at
        assert host(nk.nk_amax(x, out))[0] == x.abs().max().item()
    x[n // 3] = float("nan")
    assert torch.isnan(nk.nk_amax(x, out)).item()
