"""Cost-model forward and gradient at batches around its block structure: one
row, ragged eight-row steps, one step and several steps per block.  The
reference is the same network in FP64.  Sums over at most 4,000 rows or 128
units of FP32 products: relative Frobenius error well under 1e-5."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 7, 8, 9, 255, 1216, 1217, 3000])
def test_forward_and_gradient(B):
    from paper_2307_16080_gb300 import nk
    from paper_2307_16080_gb300 import nk_tune as nt
    g = torch.Generator(device="cuda").manual_seed(B)
    n = nt.nk_mlp_param_count()
    P = torch.randn(n, generator=g, device="cuda") * 0.1
    X, t = torch.rand(B, 16, generator=g, device="cuda"), torch.randn(B, generator=g, device="cuda")
    grad, loss = torch.full_like(P, float("nan")), torch.empty(1, device="cuda")
    nt.nk_mlp_grad(P, X, t, grad, loss)
    again = torch.empty_like(P)
    nt.nk_mlp_grad(P, X, t, again)
    y = nt.nk_mlp_forward(P, X)
    nk.nk_sync_status()
    assert torch.equal(grad, again)
    p = P.double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = p.split([2048, 128, 128 * 128, 128, 128, 1])
    gelu = lambda z: 0.5 * z * torch.erfc(-z / math.sqrt(2.0))  # noqa: E731
    want = gelu(gelu(X.double() @ W1.view(128, 16).t() + b1) @ W2.view(128, 128).t() + b2) @ W3 + b3
    L = ((want - t.double()) ** 2).mean()
    L.backward()
    assert (y.double() - want).norm() <= 1e-5 * want.norm()
    assert abs(loss.item() - L.item()) <= 1e-5 * L.item()
    for a, b in zip(grad.double().split([2048, 128, 128 * 128, 128, 128, 1]),
                    p.grad.split([2048, 128, 128 * 128, 128, 128, 1])):
        assert (a - b).norm() <= 1e-5 * b.norm()
