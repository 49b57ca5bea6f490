"""The block reflectors and trailing updates on the split-BF16 products, at the
edges of their blocks (64 reflectors: FP64 below; 256 a block), of the 128-wide
tiles, of the K chunks and of the slabs.  Q from bdc_geqrf / bdc_orgqr and
bdc_ormbr (both sides) against A = Q R, Q^T Q = I and the product with a dense
matrix.  Bound: n reflectors, each applied with a few ulp of each entry (1e-15
n is 4.5 ulp a reflector; the FP64 path measures 4e-17 n)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _rand(m, n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()


@pytest.mark.parametrize("m,n", [(63, 63), (64, 64), (129, 127), (255, 255), (300, 257), (513, 512), (5000, 70),
                                 (1000, 385), (20000, 130)])
def test_qr_and_explicit_q(m, n):
    from paper_2508_11467_gb300 import bdc
    A = _rand(m, n, m + n)
    Ar, tau, info = bdc.geqrf(A)
    assert info == 0
    R = torch.triu(Ar[:n]).clone()
    Q = bdc.orgqr(Ar, tau)
    assert float((Q @ R - A).norm()) <= 1e-15 * n * float(A.norm())
    assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device="cuda")).norm()) <= 1e-15 * n


@pytest.mark.parametrize("n,cdim", [(64, 64), (65, 300), (256, 129), (257, 1000), (700, 70), (1600, 20000)])
def test_back_transformation_keeps_products(n, cdim):
    """Q1 C and C P1^T keep C's Gram matrix (norms of sums of columns) and are
    undone by the explicit transposes."""
    from paper_2508_11467_gb300 import bdc
    Ar, _, _, tauq, taup, info = bdc.gebrd(_rand(n, n, n))
    assert info == 0
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    Q = bdc.ormbr(0, Ar, tauq, eye.clone().t())
    C = _rand(n, cdim, 1)
    X = bdc.ormbr(0, Ar, tauq, C.t().clone().t())
    assert float((Q.t() @ X - C).norm()) <= 1e-15 * n * float(C.norm())
    P = bdc.ormbr(1, Ar, taup, eye.clone().t())
    D = _rand(cdim, n, 2)
    Y = bdc.ormbr(1, Ar, taup, D.t().clone().t())
    assert float((Y @ P.t() - D).norm()) <= 1e-15 * n * float(D.norm())
