"""The reduce pass of K slices over short and long rows: a block takes several
short rows (as many as fill it), one of middling length, or a part of a long
one; exact on small integers, and in proportion to the outputs."""
import numpy as np
import pytest
import torch

from paper_2307_16080_gb300 import nk, synth
from tests.gpu_util import DEV, Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [2, 3, 8])
@pytest.mark.parametrize("M,N", [(1, 4), (3, 8), (8193, 16), (130, 20), (33, 100), (70, 512), (70, 516), (9, 1024),
                                 (9, 1028), (66001, 4), (5, 2052)])
def test_rows_of_every_length(M, N, split):
    K = 32 * split
    A, B = synth.small_ints(941, 0, (M, K)), synth.small_ints(941, 1, (K, N))
    bias = synth.small_ints(941, 2, (N,))
    C = Canary((M, N), strides=(N + 4, 1))
    nk.nk_matmul(dev(A), dev(B), C.t, "f32", bias=dev(bias), schedule=(64, 64, 16, 1, 2, split))
    nk.nk_sync_status()
    assert np.array_equal(host(C.t), (A.astype(np.float64) @ B + bias).astype(np.float32))
    C.check()


def test_short_rows_cost_what_their_outputs_do():
    """A million outputs as 65536 rows of 16 or 4096 of 256 (a block for each
    short row took ten times as long)."""
    t = {}
    for M, N in ((65536, 16), (4096, 256)):
        A, B, C = torch.ones(M, 32, device=DEV), torch.ones(32, N, device=DEV), torch.empty(M, N, device=DEV)
        ws = nk.workspace(nk.nk_matmul_workspace_size(A, B, C, "f32", (64, 64, 16, 1, 2, 2)), C.device)
        run = lambda: nk.nk_matmul(A, B, C, "f32", schedule=(64, 64, 16, 1, 2, 2), ws=ws)  # noqa: E731
        for _ in range(3):
            run()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t[M] = float("inf")
        for _ in range(5):
            a.record()
            for _ in range(20):
                run()
            b.record()
            b.synchronize()
            t[M] = min(t[M], a.elapsed_time(b))
    assert t[65536] <= 4 * t[4096]
