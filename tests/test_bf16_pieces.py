"""The arithmetic of the FP32 path's tensor-core products, restated on the CPU: three BF16 pieces per value, six of the nine products."""
import pytest

# relative 2-norm error that every gradient tensor of the FP32 path keeps to (test_gpu_grad_step.py), about four times what it has
PRECISION_FP32 = 6e-7

PRODUCTS = [(0, 0), (0, 1), (1, 0), (0, 2), (1, 1), (2, 0)]


def _pieces(x):
    import torch
    h = x.bfloat16()
    m = (x - h.float()).bfloat16()
    return [t.double() for t in (h, m, (x - h.float() - m.float()).bfloat16())]


def _error(products, K):
    import torch
    gen = torch.Generator().manual_seed(K)
    a = torch.randn((256, K), generator=gen).clamp(min=0)
    w = 0.05 * torch.randn((K, 64), generator=gen)
    A, B, exact = _pieces(a), _pieces(w), a.double() @ w.double()
    return float((sum(A[i] @ B[j] for i, j in products) - exact).norm() / exact.norm())


@pytest.mark.parametrize("K", [16, 144, 512, 1568])
def test_six_products_hold_single_precision_and_no_five_do(K):
    assert _error(PRODUCTS, K) <= 2.0 ** -24
    for p in PRODUCTS:
        assert _error([q for q in PRODUCTS if q != p], K) > 2 * PRECISION_FP32, p
