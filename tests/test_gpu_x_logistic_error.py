"""SiLU, sigmoid and the tanh form of GELU are as exact as y / (1 + e^-u) with
an exact division: the relative error of e^-u (one unit in the last place,
2^-23), of 1 + e^-u and of the quotient (2^-24 each) add up to 2^-22.  The
argument u of GELU's tanh form carries at most five roundings of 2^-24."""
import numpy as np
import pytest
import torch

from tests.gpu_util import DEV, dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    import paper_2307_16080_gb300.nk as m
    m.lib()
    return m


@pytest.mark.parametrize("name", ["silu", "sigmoid", "gelu_tanh"])
def test_relative_error(nk, name):
    rng = np.random.default_rng(11)
    end = 9.0 if name == "gelu_tanh" else 87.0     # results stay normal numbers
    x = np.concatenate([np.linspace(-end, end, 200001), rng.uniform(-12, 12, 400000).clip(-end, end),
                        np.float64(1.37) * 2.0 ** np.arange(-120, 3), -np.float64(1.37) * 2.0 ** np.arange(-120, 3)])
    x = x[x != 0].astype(np.float32)
    y = torch.empty(x.size, device=DEV)
    nk.nk_elementwise(dev(x), y, [(name,)])
    nk.nk_sync_status()
    v = x.astype(np.float64)
    u = 2 * np.sqrt(2 / np.pi) * (v + 0.044715 * v ** 3) if name == "gelu_tanh" else v
    want = (1.0 if name == "sigmoid" else v) / (1 + np.exp(-u))
    rel = np.abs(host(y).astype(np.float64) - want) / np.abs(want)
    tol = 2.0 ** -22 * (1 + 2.0 ** -18) + (np.abs(u) * 5 * 2.0 ** -24 if name == "gelu_tanh" else 0.0)
    assert (rel <= tol).all(), (name, rel.max(), v[rel.argmax()])
