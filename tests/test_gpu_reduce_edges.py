"""The reduction on both sides of what fits on chip (from the device's SM
count and shared memory), and blocked to the matrix's last column (panels so
long that not even their last columns fit: a full last panel, a short one, a
column alone).  Bound: sqrt(2 n) 4 ulp of ||A||, 6e-14 at n = 2000: 1e-13."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _largest_on_chip():
    """n of the largest n x n matrix whose rows fit (a block per SM, at most 160):
    own rows, two vectors of a column each, 13 rows of 136 sums, four of own rows."""
    p = torch.cuda.get_device_properties(0)
    most = p.shared_memory_per_block_optin - 128

    def fits(n):
        rows = -(-n // min(p.multi_processor_count, 160, n))
        return 8 * (rows * n + 2 * n + 13 * 136 + 4 * rows + 2) <= most

    return max(n for n in range(1, 2201) if fits(n))


def _check(m, n):
    from paper_2508_11467_gb300 import bdc
    g = torch.Generator("cuda").manual_seed(m + n)
    A = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    Ar, d, e, tauq, taup, info = bdc.gebrd(A)
    assert info == 0 and float(taup[-1]) == 0.0
    C = torch.zeros(n, m, dtype=torch.float64, device="cuda").t()
    C[:n].copy_(torch.diag(d) + torch.diag(e, 1))
    bdc.ormbr(0, Ar, tauq, C)
    PT = bdc.ormbr(1, Ar, taup, torch.eye(n, dtype=torch.float64, device="cuda").t())
    assert float((C @ PT - A).norm()) <= 1e-13 * float(A.norm())


@pytest.mark.parametrize("more", [0, 1, 33])
def test_edge_of_the_chip(more):
    n = _largest_on_chip() + more
    _check(n, n)
    _check(n + 100, n - 100)


@pytest.mark.parametrize("n", [33, 60, 64])
def test_blocked_to_the_last_column(n):
    _check(200000, n)
