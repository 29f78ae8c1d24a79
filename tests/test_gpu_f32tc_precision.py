"""Rounding of the fp32 routes.  A product of less than one 32-element chunk of
K is a chain of round-to-nearest multiply-adds: its errors have no bias, also
where every term has the same sign (the tensor cores' truncation has one of
0.7 u to 1 u).  From one chunk on the tensor cores' error is no larger than such
a chain's.  A sum of one term is exact on either.

Tolerances: a chain's k-th rounding is uniform within half an ulp of the
partial sum, at most u of it, so its rms is at most u / sqrt(3) times the sum of
the partial sums' squares, (k / K)^2 each for terms of like size; its mean is 0,
and over 10^8 elements the estimate of the mean stays far below 0.05 u."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _relative_error(M, N, K, level):
    """Errors of C over the sum of |a b|, in u, on operands of one sign."""
    import torch
    import paper_2305_01024_gb300 as ft
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    A = torch.rand(M, K, generator=g, device="cuda") * 0.5 + 0.75
    B = torch.rand(K, N, generator=g, device="cuda") * 0.5 + 0.75
    C = torch.zeros(M, N, device="cuda")
    h = ft.Handle(0)
    rep = h.gemm(A, B, C, level=level)
    h.close()
    assert rep.detected == 0
    d = C.double()
    S = A.double() @ B.double()
    return (d - S).div_(S).div_(U)


@pytest.mark.parametrize("level", ["off", "block"])
@pytest.mark.parametrize("M,N,K", [(16384, 16384, 8), (16384, 16384, 16), (12288, 8192, 31)])
def test_less_than_a_chunk_has_no_bias(M, N, K, level):
    assert abs(_relative_error(M, N, K, level).mean().item()) < 0.05


@pytest.mark.parametrize("level", ["off", "block"])
@pytest.mark.parametrize("M,N,K", [(8192, 8192, 32), (8192, 8192, 33), (8192, 8192, 63), (2048, 2048, 512)])
def test_from_a_chunk_on_no_worse_than_a_chain(M, N, K, level):
    rms = _relative_error(M, N, K, level).square_().mean().sqrt().item()
    chain = np.sqrt(sum((k / K) ** 2 for k in range(1, K + 1)) / 3)
    assert rms <= chain


@pytest.mark.parametrize("level", ["off", "warp", "block"])
def test_sums_of_one_term_are_exact(level):
    """A = I and full 24-bit mantissas over a range of exponents in B: the three
    planes of every element come together again."""
    import torch
    import paper_2305_01024_gb300 as ft
    K, N = 1000, 1500
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    B = torch.randn(K, N, generator=g, device="cuda") * torch.exp2(torch.randint(-90, 50, (K, N), generator=g, device="cuda").float())
    C = torch.zeros(K, N, device="cuda")
    h = ft.Handle(0)
    h.gemm(torch.eye(K, device="cuda"), B, C, level=level)
    h.close()
    assert torch.equal(C, B)
