"""Arguments that stand for others: scalars of NumPy and torch in place of integers, and a
gradient that is a negating view."""
import numpy as np
import pytest
import torch

import paper_1411_2860_gb300 as pj

pytestmark = pytest.mark.gpu


def _operands(dtype=torch.float32):
    g = torch.Generator(device="cuda").manual_seed(5)
    return (torch.randn(60, 200, device="cuda", generator=g).to(dtype),
            torch.randn(200, 72, device="cuda", generator=g).to(dtype))


@pytest.mark.parametrize("scalar", [np.int64, np.array, torch.tensor])
def test_index_like_sizes(scalar):
    A, B = _operands()
    want = pj.proj_gemm(A, B, 16, 8, "dct2", 8, split=2)
    assert torch.equal(pj.proj_gemm(A, B, scalar(16), scalar(8), "dct2", scalar(8), split=scalar(2)), want)
    Xb, Wb = _operands(torch.bfloat16)
    dY = torch.randn(60, 72, device="cuda")
    got = pj.proj_gemm_backward(Xb, Wb, dY, scalar(16), scalar(8), "dct2", scalar(8))
    for g, w in zip(got, pj.proj_gemm_backward(Xb, Wb, dY, 16, 8, "dct2", 8)):
        assert torch.equal(g, w)


def test_sizes_that_change_in_place():
    """Nothing is remembered of an object that can change its value."""
    A, B = _operands()
    block, R, L = torch.tensor(16), torch.tensor(4), torch.tensor(8)
    assert torch.equal(pj.proj_gemm(A, B, block, R, "dct2", L), pj.proj_gemm(A, B, 16, 4, "dct2", 8))
    R.fill_(16)     # more components: a larger workspace
    L.fill_(4)
    assert torch.equal(pj.proj_gemm(A, B, block, R, "dct2", L), pj.proj_gemm(A, B, 16, 16, "dct2", 4))


def test_negated_gradient():
    """A contiguous FP32 view that negates its memory when it is read."""
    X, W = _operands(torch.bfloat16)
    dY = torch.randn(60, 72, device="cuda")
    neg = torch._neg_view(dY)
    assert neg.is_neg() and neg.is_contiguous()
    for g, w in zip(pj.proj_gemm_backward(X, W, neg, 16, 8), pj.proj_gemm_backward(X, W, -dY, 16, 8)):
        assert torch.equal(g, w)
    X.requires_grad_()
    W.requires_grad_()
    for save in (False, True):
        Y = pj.proj_matmul(X, W, 16, 8, save_projections=save)
        for g, w in zip(torch.autograd.grad(Y, (X, W), neg, retain_graph=not save),
                        pj.proj_gemm_backward(X.detach(), W.detach(), -dY, 16, 8)):
            assert torch.equal(g, w)
