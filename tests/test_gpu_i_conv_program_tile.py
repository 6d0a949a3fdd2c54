"""An FP32 convolution with a program and no schedule takes a tile that its
filters fill: no slower than the 64 x 64 one that a schedule asks for."""
import pytest
import torch

from tests.gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    import paper_2307_16080_gb300.nk as m
    m.lib()
    return m


@pytest.mark.parametrize("which", ["ew", "pro_i"])
def test_built_in_tile_of_a_convolution_with_a_program(nk, which):
    I, W = torch.rand(8, 56, 56, 64, device=DEV), torch.rand(3, 3, 64, 64, device=DEV)
    out, t = [], []
    for sched in (None, (64, 64, 16, 1, 2, 1)):
        o = torch.empty(8, 56, 56, 64, device=DEV)
        run = lambda: nk.nk_conv2d_nhwc_hwcf(I, W, o, (1, 1), (1, 1), (1,) * 4, "f32", schedule=sched,  # noqa: E731
                                             **{which: [("relu",)]})
        for _ in range(3):
            run()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(5):
            a.record()
            for _ in range(10):
                run()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        out.append(o)
        t.append(best)
    assert torch.equal(out[0], out[1])
    assert t[0] <= 1.15 * t[1]
