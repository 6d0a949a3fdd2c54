"""BF16x3 without a schedule at a size whose tiles are the 256 x 256 pairs, through
every epilogue -- accumulate, bias and ReLU, programs, a residual that is the
output, column-major C with a bias per row, odd C: the bits of the 128 x 128 tiles
(the same products in the same order)."""
import pytest
import torch

from paper_2307_16080_gb300 import nk
from tests.gpu_util import DEV, Canary

pytestmark = pytest.mark.gpu
M, N, K = 3841, 4100, 3100


@pytest.mark.parametrize("what", ["accumulate", "bias_relu", "gelu", "residual", "column", "odd"])
def test_every_epilogue(what):
    g = torch.Generator(device=DEV).manual_seed(7)
    n = N - 3 if what == "odd" else N
    A, B = torch.randn(M, K, generator=g, device=DEV), torch.randn(K, n, generator=g, device=DEV)
    C0, bias = torch.randn(M, n, generator=g, device=DEV), torch.randn(n, generator=g, device=DEV)
    out = []
    for sched in ((128, 128, 64, 1, 3, 1), None):
        C = Canary((M, n), strides=(1, M + 3) if what == "column" else (n, 1))
        C.t.copy_(C0)
        kw = {"accumulate": dict(accumulate=True, bias=bias), "gelu": dict(bias=bias, ew=[("gelu",)]),
              "residual": dict(ew=[("add", C.t), ("relu",)])}.get(what, dict(bias=bias, relu=True))
        nk.nk_matmul(A, B, C.t, "bf16x3", schedule=sched, **kw)
        nk.nk_sync_status()
        C.check()
        out.append(C.t.clone())
    assert torch.equal(out[0], out[1])
