"""A wait budget of one poll runs out in the shortest kernels too: the poll
does not sleep until the awaited copy has landed, so the timeout is reported
every time, and the next call is exact."""
import numpy as np
import pytest
import torch

import oracle.nk_oracle as O
from paper_2307_16080_gb300 import synth
from tests.gpu_util import DEV, dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    import paper_2307_16080_gb300.nk as m
    m.lib()
    return m


@pytest.mark.parametrize("hw,sched", [(8, (128, 64, 576, 1, 2, 1)), (8, (128, 64, 192, 1, 2, 1)),
                                      (24, (128, 64, 192, 1, 2, 1))])
def test_one_poll_always_runs_out(nk, hw, sched):
    I = synth.small_ints(83, 0, (1, hw, hw, 64))
    W = synth.small_ints(83, 1, (3, 3, 64, 64))
    i, w, out = dev(I), dev(W), torch.empty(1, hw, hw, 64, device=DEV)
    call = lambda: nk.nk_conv2d_nhwc_hwcf(i, w, out, pad=(1, 1, 1, 1), precision="bf16", schedule=sched)  # noqa: E731
    call()   # loads the kernel
    nk.nk_sync_status()
    try:
        nk.nk_set_wait_budget(1)
        for _ in range(10):
            call()
            with pytest.raises(nk.NkError) as e:
                nk.nk_sync_status()
            assert e.value.status == -6
    finally:
        nk.nk_set_wait_budget(0)
    call()
    nk.nk_sync_status()
    np.testing.assert_array_equal(host(out), O.conv2d_nhwc_hwcf(I, W, pad=(1, 1, 1, 1)))
