"""Conversions of narrow and of few-row matrices, of dense matrices whose rows
do not end on words, and amax of short runs: bit for bit, with NaN and the last
element in every position class, and no slower than the kernels for whole tiles
(3 x 1000000 took nearly as long as 24 rows)."""
import pytest
import torch

from paper_2307_16080_gb300 import nk
from tests.gpu_util import DEV, Canary, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1, 300), (300, 1), (16, 16), (16, 17), (17, 16), (32, 33), (33, 32), (5, 1000),
                                       (1000, 5), (1000, 16), (1000, 17), (31, 2000)])
@pytest.mark.parametrize("pad_in,pad_out", [(0, 0), (1, 0), (0, 1), (5, 16)])
@pytest.mark.parametrize("transpose", [False, True])
def test_narrow_casts_bitwise(rows, cols, pad_in, pad_out, transpose):
    g = torch.Generator(device=DEV).manual_seed(rows * 101 + cols)
    x = torch.full((rows, cols + pad_in), float("nan"), device=DEV)[:, :cols]
    x.copy_(torch.randint(-14, 15, (rows, cols), generator=g, device=DEV).float() / 4)
    shape = (cols, rows) if transpose else (rows, cols)
    want = x.t() if transpose else x
    outs = [Canary(shape, torch.bfloat16, strides=(shape[1] + pad_out, 1)) for _ in range(3)]
    nk.nk_cast_bf16(x, outs[0].t, transpose)
    x.add_(2.0 ** -9)   # low parts that are not zero
    nk.nk_split_bf16x3(x, outs[1].t, outs[2].t, transpose)
    assert torch.equal(outs[1].t, want.bfloat16())
    assert torch.equal(outs[2].t, (want - want.bfloat16().float()).bfloat16())
    x.sub_(2.0 ** -9)
    assert torch.equal(outs[0].t, want.bfloat16())
    q, scale = Canary(shape, torch.uint8, strides=(shape[1] + pad_out, 1)), torch.empty(1, device=DEV)
    nk.nk_cast_fp8(x, torch.full((1,), 3.5, device=DEV), q.t, transpose, scale_out=scale)
    nk.nk_sync_status()
    assert host(scale)[0] == 128.0
    assert torch.equal(q.t, (want * 128).to(torch.float8_e4m3fn).contiguous().view(torch.uint8))
    for o in outs + [q]:
        o.check()


@pytest.mark.parametrize("n", [4, 1020, 1024, 1028, 4096, 1024 * 1024, 7 * 1024 * 1024 + 4])
def test_amax_of_short_runs(n):
    x, out = torch.zeros(n, device=DEV), torch.empty(1, device=DEV)
    for i, at in enumerate((0, n // 2, n - 1)):
        x[at] = -5.0 - i
        assert host(nk.nk_amax(x, out))[0] == 5.0 + i
    x[n - 2] = float("nan")
    assert torch.isnan(nk.nk_amax(x, out)).item()


def _time(run):
    for _ in range(3):
        run()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        a.record()
        for _ in range(20):
            run()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_few_rows_cost_a_fraction_of_a_tile():
    t = {}
    for rows in (3, 24):
        x, q = torch.ones(rows, 1000000, device=DEV), torch.empty(1000000, 32, dtype=torch.uint8, device=DEV)
        am = torch.ones(1, device=DEV)
        t[rows] = _time(lambda: nk.nk_cast_fp8(x, am, q[:, :rows], True))
    assert t[3] <= 0.6 * t[24]
