"""Dense calls with more rows than a product's tile list can index (32767 row
blocks of 128): the trailing update of a reduction, the rows of C in a
back-transformation, and the product Q U_R of a tall SVD.

Bounds: sqrt(2 n) 4 ulp a column as for any reduction (n <= 66), on top of the
norms' own rounding: 1e-13."""
import pytest
import torch

pytestmark = pytest.mark.gpu
ROWS = 32767 * 128


@pytest.fixture(autouse=True)
def _release():
    yield
    torch.cuda.empty_cache()


def _gauss(m, n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()


def test_reduction_of_more_rows_than_tiles():
    from paper_2508_11467_gb300 import bdc
    m, n = ROWS + 500, 40
    A = _gauss(m, n, 1)
    Ar, d, e, tauq, taup, info = bdc.gebrd(A)
    assert info == 0
    C = torch.zeros(n, m, dtype=torch.float64, device="cuda").t()
    C[:n].copy_(torch.diag(d) + torch.diag(e, 1))
    bdc.ormbr(0, Ar, tauq, C)
    PT = bdc.ormbr(1, Ar, taup, torch.eye(n, dtype=torch.float64, device="cuda").t())
    assert float((C @ PT - A).norm()) <= 1e-13 * float(A.norm())


def test_back_transformation_of_more_rows_than_tiles():
    from paper_2508_11467_gb300 import bdc
    n, cdim = 66, ROWS + 300
    Ar, _, _, _, taup, info = bdc.gebrd(_gauss(n, n, 2))
    assert info == 0
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    P = bdc.ormbr(1, Ar, taup, eye.clone().t())
    C = _gauss(cdim, n, 3)
    X = bdc.ormbr(1, Ar, taup, C.t().clone().t())
    assert float((X - C @ P).norm()) <= 1e-13 * float(C.norm())
    assert float((X[ROWS:] - C[ROWS:] @ P).norm()) <= 1e-13 * float(C[ROWS:].norm())


def test_svd_of_more_rows_than_tiles():
    from paper_2508_11467_gb300 import bdc
    m, n = ROWS + 200, 64
    A = _gauss(m, n, 4)
    S, U, VT, info = bdc.gesvd(A)
    assert info == 0
    for rows in (slice(0, ROWS), slice(ROWS, m)):
        assert float((U[rows] * S[None, :] @ VT - A[rows]).norm()) <= 1e-13 * float(A[rows].norm())
    assert float((U.t() @ U - torch.eye(n, dtype=torch.float64, device="cuda")).norm()) <= 1e-13
