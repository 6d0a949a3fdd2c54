"""Split-K summed inside a cluster: products of 2, 4 and 8 slices at ragged
edges, every precision, with the whole epilogue; bitwise on small integers,
canary-padded outputs."""
import numpy as np
import pytest

from paper_2307_16080_gb300 import synth
from tests.gpu_util import Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp8", "bf16x3"])
@pytest.mark.parametrize("split", [2, 4, 8])
@pytest.mark.parametrize("M,N,ldc", [(1, 1, 1), (129, 70, 72), (300, 133, 133), (128, 256, 260)])
def test_matmul_slices(prec, split, M, N, ldc):
    from paper_2307_16080_gb300 import nk
    tk = 128 if prec == "fp8" else 64
    K = 9 * tk * split - 24
    A, B = synth.small_ints(931, 0, (M, K), -7, 7) / 2, synth.small_ints(931, 1, (K, N), -7, 7) / 2
    A[0, 0] = B[0, 0] = 3.5
    bias, C0 = synth.small_ints(931, 2, (N,)), synth.small_ints(931, 3, (M, N))
    want = np.maximum(A.astype(np.float64) @ B + C0 + bias, 0) * 0.5 + 1
    for tn in (64, 128):
        C = Canary((M, N), strides=(ldc, 1))
        C.t.copy_(dev(C0))
        nk.nk_matmul(dev(A), dev(B), C.t, prec, bias=dev(bias), relu=True, accumulate=True, ew=[("affine", 0.5, 1.0)],
                     schedule=(128, tn, tk, 1, 3 if prec == "bf16x3" and tn == 128 else 4, split))
        nk.nk_sync_status()
        assert np.array_equal(host(C.t), want.astype(np.float32))
        C.check()
