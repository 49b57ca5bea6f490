"""Operands below the normal range in the block reflectors: C of subnormal
entries comes back rotated (compared with the same C scaled up by a power of
two), to the rounding of the subnormal grid: n products of reflectors, each
entry rounded to 2^-1074 a few times a block; 16 n units bound it."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vect", [0, 1])
@pytest.mark.parametrize("n", [64, 300])
def test_subnormal_c(n, vect):
    from paper_2508_11467_gb300 import bdc
    g = torch.Generator("cuda").manual_seed(n)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g).t()
    Ar, _, _, tauq, taup, info = bdc.gebrd(A)
    assert info == 0
    tau = tauq if vect == 0 else taup
    C = torch.randint(-2 ** 40, 2 ** 40, (n, n), device="cuda", generator=g).double().t().contiguous().t()
    big = bdc.ormbr(vect, Ar, tau, C.t().clone().t())             # entries up to 2^40 units of 2^-1074
    small = bdc.ormbr(vect, Ar, tau, (C * 2.0 ** -537 * 2.0 ** -537).t().clone().t())
    back = small * 2.0 ** 537 * 2.0 ** 537
    assert float((back - big).abs().max()) <= 16 * n
