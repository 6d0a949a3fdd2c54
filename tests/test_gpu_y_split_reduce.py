"""Split-K partials and their reduce pass at ragged columns: two to sixteen
slices, every precision, outputs whose rows take 16-byte stores and ones that
do not, with the whole epilogue; bitwise on small integers, canary-padded
outputs, and a workspace of exactly the size asked for."""
import numpy as np
import pytest
import torch

from paper_2307_16080_gb300 import synth
from tests.gpu_util import Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "bf16", "fp8", "bf16x3"])
@pytest.mark.parametrize("split", [2, 3, 4, 8, 16])
@pytest.mark.parametrize("M,N,ldc", [(1, 1, 1), (129, 70, 72), (300, 133, 133), (128, 256, 260), (5, 1027, 1027)])
def test_slices(prec, split, M, N, ldc):
    from paper_2307_16080_gb300 import nk
    tk = {"fp8": 128, "f32": 16}.get(prec, 64)
    K = 3 * tk * split - 8
    A, B = synth.small_ints(931, 0, (M, K), -7, 7) / 2, synth.small_ints(931, 1, (K, N), -7, 7) / 2
    A[0, 0] = B[0, 0] = 3.5
    bias, C0 = synth.small_ints(931, 2, (N,)), synth.small_ints(931, 3, (M, N))
    want = np.maximum(A.astype(np.float64) @ B + C0 + bias, 0)
    sched = (64, 64, 16, 1, 2, split) if prec == "f32" else (128, 64, tk, 1, 3, split)
    C = Canary((M, N), strides=(ldc, 1))
    C.t.copy_(dev(C0))
    a, b = dev(A), dev(B)
    need = nk.nk_matmul_workspace_size(a, b, C.t, prec, sched)
    ws = Canary((need,), torch.uint8)
    nk.nk_matmul(a, b, C.t, prec, bias=dev(bias), relu=True, accumulate=True, schedule=sched, ws=ws.t)
    nk.nk_sync_status()
    assert np.array_equal(host(C.t), want.astype(np.float32))
    C.check(), ws.check()
