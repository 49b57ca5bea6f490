"""Dense reductions too large for the chip (blocked panels and a trailing
update) on matrices whose columns differ in scale: the panel's first column far
below or above the rest, or zero, at several norms, and a block-diagonal input
whose second block begins a panel with a tiny column.

A = Q1 B P1^T with Q1, P1 applied by bdc_ormbr.  No row reflector touches
column 0, so column 0 and the other columns are each judged against their own
norm.  Bound: 2 n reflectors act on a column, each leaving a few ulp of it in
directions of its own, so sqrt(2 n) 4 ulp = 6e-14 at n = 2000: 1e-13."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-13


def _gauss(m, n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()


def _rebuilt(A):
    from paper_2508_11467_gb300 import bdc
    m, n = A.shape
    Ar, d, e, tauq, taup, info = bdc.gebrd(A)
    assert info == 0
    C = torch.zeros(n, m, dtype=torch.float64, device="cuda").t()
    C[:n].copy_(torch.diag(d) + torch.diag(e, 1))
    bdc.ormbr(0, Ar, tauq, C)
    bdc.ormbr(1, Ar, taup, C)
    return C


def _check(A):
    C = _rebuilt(A)
    for s in (slice(0, 1), slice(1, None)):
        assert float((C[:, s] - A[:, s]).norm()) <= TOL * float(A[:, s].norm())


@pytest.mark.parametrize("norm", [1e-8, 1.0, 1e8])
@pytest.mark.parametrize("first", [0.0, 1e-16, 1e-8, 1e-4, 1e8])
def test_first_column_of_another_scale(first, norm):
    A = _gauss(1900, 1900, 5) * norm
    A[:, 0] *= first
    _check(A)


@pytest.mark.parametrize("first", [0.0, 1e-12, 1e8])
def test_rectangular(first):
    A = _gauss(2500, 2000, 6)
    A[:, 0] *= first
    _check(A)


def test_second_panel_begins_with_a_tiny_column():
    A = torch.zeros(1900, 1900, dtype=torch.float64, device="cuda").t()
    A[:32, :32] = _gauss(32, 32, 7)
    A[32:, 32:] = _gauss(1868, 1868, 8)
    A[32:, 32] *= 1e-12
    C = _rebuilt(A)
    for s in (slice(0, 32), slice(32, 33), slice(33, None)):
        assert float((C[:, s] - A[:, s]).norm()) <= TOL * float(A[:, s].norm())


@pytest.mark.parametrize("first,norm", [(0.0, 1e8), (1e-16, 1.0), (1e8, 1.0)])
def test_gesvd(first, norm):
    from paper_2508_11467_gb300 import bdc
    A = _gauss(1900, 1900, 9) * norm
    A[:, 0] *= first
    S, U, VT, info = bdc.gesvd(A)
    assert info == 0
    assert float((U * S[None, :] @ VT - A).norm()) <= TOL * float(A.norm())
    eye = torch.eye(1900, dtype=torch.float64, device="cuda")
    assert float((U.t() @ U - eye).norm()) <= TOL * 1900 ** 0.5
    assert float((VT @ VT.t() - eye).norm()) <= TOL * 1900 ** 0.5
