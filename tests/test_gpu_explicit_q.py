"""The explicit Q of bdc_orgqr, and Q1 C of bdc_ormbr, against the product of
the stored reflectors in twice the precision (double-double).

Bounds: what the block reflectors in FP64 leave (blocks of 64, FP64 products)
on these shapes, 6.3e-16 of ||Q|| for a square Q, 3.1e-16 for 2000 x 600,
1.54e-16 for 10000 x 300, and 9.4e-16 for Q C of a Gaussian C (2000 x 600:
5.6e-16, 10000 x 300: 2.6e-16), two per cent above: the sliced products may not
be further off."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _split(a):
    c = 134217729.0 * a
    h = c - (c - a)
    return h, a - h


def _mul(h, l, b):
    """(h + l) b for doubles b."""
    p = h * b
    ah, al = _split(h)
    bh, bl = _split(b)
    e = ((ah * bh - p) + ah * bl + al * bh) + al * bl + l * b
    s = p + e
    return s, e - (s - p)


def _add(ah, al, bh, bl):
    s = ah + bh
    t = s - ah
    e = (ah - (s - t)) + (bh - t) + (al + bl)
    h = s + e
    return h, e - (h - s)


def _column_sums(h, l):
    while h.shape[0] > 1:
        k = h.shape[0] // 2
        a, b = _add(h[:k], l[:k], h[k:2 * k], l[k:2 * k])
        if h.shape[0] % 2:
            a, b = torch.cat([a, h[2 * k:]]), torch.cat([b, l[2 * k:]])
        h, l = a, b
    return h[0], l[0]


def _apply(Ar, tau, C):
    """H_1 ... H_n C, one reflector after the other."""
    H, L = C.contiguous().clone(), torch.zeros_like(C).contiguous()
    for j in range(tau.numel() - 1, -1, -1):
        v = Ar[j:, j].clone()
        v[0] = 1.0
        v = v[:, None].expand_as(H[j:])
        w = _mul(*_column_sums(*_mul(H[j:], L[j:], v)), tau[j].expand(C.shape[1]))
        q = _mul(w[0][None].expand_as(v), w[1][None].expand_as(v), v)
        H[j:], L[j:] = _add(H[j:], L[j:], -q[0], -q[1])
    return H, L


@pytest.mark.parametrize("m,n,q_fp64,c_fp64", [(64, 64, 5.9e-16, 9.0e-16), (257, 257, 6.3e-16, 9.4e-16),
                                               (333, 333, 6.3e-16, 9.4e-16), (600, 600, 6.5e-16, 9.5e-16),
                                               (2000, 600, 3.1e-16, 5.6e-16), (10000, 300, 1.54e-16, 2.6e-16)])
def test_no_further_off_than_fp64(m, n, q_fp64, c_fp64):
    from paper_2508_11467_gb300 import bdc
    g = torch.Generator("cuda").manual_seed(m + n)
    A = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    Ar, tau, info = bdc.geqrf(A)
    assert info == 0
    C = torch.randn(min(n, 300), m, dtype=torch.float64, device="cuda", generator=g).t()
    for X, bound, call in ((torch.eye(m, n, dtype=torch.float64, device="cuda"), q_fp64,
                            lambda: bdc.orgqr(Ar.t().clone().t(), tau)),
                           (C, c_fp64, lambda: bdc.ormbr(0, Ar, tau, C.t().clone().t()))):
        h, l = _apply(Ar, tau, X)
        assert float(((call() - h) - l).norm() / h.norm()) <= 1.02 * bound
