"""The on-chip bidiagonalization (k_gebd2_resident) where it can go wrong:
fewer rows than SMs, one row more than a multiple of the grid, more rows per
CTA than it handles at once, more columns than threads, the largest size that
fits and the first that does not (blocked panels first, then the rest on
chip).  A = Q1 B P1^T with Q1, P1 applied by bdc_ormbr; bound: n products of
reflectors, each with a few ulp of backward error (1e-15 n sqrt(n) ||A||_F is
above the sum of their worst cases at n >= 1)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(3, 2), (151, 151), (153, 40), (305, 128), (1300, 7), (1217, 129), (2500, 257),
                                 (20000, 60), (1650, 1650), (1960, 1960)])
def test_resident_reduction(m, n):
    from paper_2508_11467_gb300 import bdc
    g = torch.Generator("cuda").manual_seed(m + n)
    A = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    Ar, d, e, tauq, taup, info = bdc.gebrd(A)
    assert info == 0
    C = torch.zeros(n, m, dtype=torch.float64, device="cuda").t()
    C[:n].copy_(torch.diag(d) + (torch.diag(e, 1) if n > 1 else 0.0))
    bdc.ormbr(0, Ar, tauq, C)
    bdc.ormbr(1, Ar, taup, C)
    assert float((C - A).norm()) <= 1e-15 * n * n ** 0.5 * float(A.norm())
    assert float(taup[-1]) == 0.0


@pytest.mark.parametrize("m,n", [(1, 1), (32, 32), (33, 31), (64, 1), (352, 32), (705, 33), (9729, 32)])
def test_resident_qr_panel(m, n):
    """Panels held on chip: fewer rows than CTAs have, a column alone, the
    smallest grid, one more row than a full share, the next panel's first
    column.  Bound: n reflectors of a few ulp each, as above."""
    from paper_2508_11467_gb300 import bdc
    g = torch.Generator("cuda").manual_seed(m + 3 * n)
    A = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    Ar, tau, info = bdc.geqrf(A.clone())   # (factors a column-major matrix of one column in place)
    assert info == 0
    R = torch.triu(Ar[:n])
    Q = bdc.orgqr(Ar.clone().t().contiguous().t(), tau)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    assert float((Q @ R - A).norm()) <= 1e-15 * (n + 1) * (n + 1) ** 0.5 * float(A.norm())
    assert float((Q.t() @ Q - eye).norm()) <= 1e-15 * (n + 1) * (n + 1) ** 0.5 * n ** 0.5
