"""The built-in convolution rule at the borders between its kernels (measured
times of each stand beside the rule)."""
import pytest

nt = pytest.importorskip("paper_2307_16080_gb300.nk_tune")


@pytest.mark.parametrize("n,h,c,f,sched", [
    (128, 28, 128, 128, (256, 128, 64, 2, 3, 1)),    # many units, many tiles: CTA pairs
    (512, 4, 128, 256, (128, 64, 64, 1, 3, 1)),      # many window units, few per-tap tiles: one CTA per tile
    (80, 10, 128, 256, (128, 64, 64, 1, 3, 1)),
    (32, 56, 64, 64, (256, 64, 192, 1, 2, 1)),       # one channel block: kernel rows stacked, two buffers
    (8, 28, 128, 128, (128, 64, 192, 1, 2, 1))])     # few units: one buffer
def test_convolution_rule(n, h, c, f, sched):
    assert nt.nk_default_schedule(nt.conv_problem(n, h, h, c, f, 3, 3, 1, 1)) == sched
