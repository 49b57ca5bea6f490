"""QR of matrices whose panels are longer than one product's K (16384) times
the number of products the trailing update is cut into by its tiles alone: the
smallest such widths and one between.  Bound: n reflectors of a few ulp each in
directions of their own, sqrt(n) 4 ulp = 3e-14 at n = 1000, on A and on the
orthogonality of Q's columns (times sqrt(n) over all of them)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(320000, 1000), (500000, 640), (450000, 700)])
def test_long_panels(m, n):
    from paper_2508_11467_gb300 import bdc
    g = torch.Generator("cuda").manual_seed(m)
    A = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    Ar, tau, info = bdc.geqrf(A)
    assert info == 0
    R = torch.triu(Ar[:n]).clone()
    Q = bdc.orgqr(Ar, tau)
    assert float((Q @ R - A).norm()) <= 3e-14 * float(A.norm())
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    assert float((Q.t() @ Q - eye).norm()) <= 3e-14 * n ** 0.5
    del A, Ar, Q, R
    torch.cuda.empty_cache()
