"""The scalars of one reflector, through the QR of a matrix of one column with
two entries (alpha, x): beta, tau and v = x / (alpha - beta) against extended
precision, over random and extreme pairs.

Bounds in units of 2^-52.  s = alpha^2 + x^2 carries 1 (two roundings), its
square root half of that and one of its own: beta 1.5.  alpha - beta (no
cancellation: opposite signs) adds 0.5 to at most beta's error: 2, its quotient
by beta with beta's own error and one rounded quotient: tau 4.5.  The reciprocal
1 and the product 0.5: v 3.5."""
import math
import random
from fractions import Fraction

import pytest
import torch

pytestmark = pytest.mark.gpu


def _pairs():
    r = random.Random(11)
    out = [(1.0, 1.0), (-1.0, 1.0), (0.0, 1.0), (-0.0, 1.0), (0.0, -2.5), (3.0, 4.0), (1.0, 1e-9), (1e-9, 1.0),
           (1.0, 2.0 ** -26), (1.0, 2.0 ** -27), (-1.0, 2.0 ** -300)]
    # both sides of the range in which s = alpha^2 + x^2 takes the short way (2^-900, 2^900)
    for e in (-460, -452, -451, -450, -449, -448, 0, 448, 449, 450, 451, 452, 460, 500, -500):
        for _ in range(3):
            out.append((math.ldexp(r.uniform(-2, 2), e), math.ldexp(r.uniform(-2, 2), e)))
    for _ in range(150):
        out.append((r.uniform(-2, 2), math.ldexp(r.uniform(-2, 2), r.randint(-40, 40))))
    return out


def _sqrt(q):
    """sqrt of a Fraction to 2^-200 relative."""
    k = 2 * (400 - (q.numerator.bit_length() - q.denominator.bit_length()) // 2)
    n = q * Fraction(2) ** k
    return Fraction(math.isqrt(n.numerator // n.denominator)) / Fraction(2) ** (k // 2)


def _reflector(alpha, x):
    from paper_2508_11467_gb300 import bdc
    A = torch.tensor([[alpha], [x]], dtype=torch.float64, device="cuda")
    Ar, tau, info = bdc.geqrf(A)
    assert info == 0
    return float(Ar[0, 0]), float(tau[0]), float(Ar[1, 0])


def test_scalars():
    for alpha, x in _pairs():
        beta, tau, v = _reflector(alpha, x)
        a, b = Fraction(alpha), Fraction(x)
        nrm = _sqrt(a * a + b * b)
        want = -nrm if a >= 0 else nrm
        unit = Fraction(1, 2 ** 52)
        assert abs(Fraction(beta) - want) <= Fraction(3, 2) * unit * nrm, (alpha, x)
        assert abs(Fraction(tau) - (want - a) / want) <= Fraction(9, 2) * unit * abs((want - a) / want), (alpha, x)
        assert abs(Fraction(v) - b / (a - want)) <= Fraction(7, 2) * unit * abs(b / (a - want)), (alpha, x)


@pytest.mark.parametrize("alpha", [0.0, -0.0])
def test_zero_of_either_sign_reflects_alike(alpha):
    """A zero alpha counts as positive whatever its sign bit: beta = -||x||, in
    the panels of QR and in the reduction."""
    from paper_2508_11467_gb300 import bdc
    assert _reflector(alpha, 2.0) == (-2.0, 1.0, 1.0)
    A = torch.tensor([[alpha], [2.0]], dtype=torch.float64, device="cuda")
    _, d, _, tauq, _, info = bdc.gebrd(A)
    assert info == 0 and float(d[0]) == -2.0 and float(tauq[0]) == 1.0


@pytest.mark.parametrize("alpha", [0.0, -0.0, 1.5, -1.5])
def test_nothing_to_annihilate(alpha):
    beta, tau, v = _reflector(alpha, 0.0)
    assert beta == alpha and tau == 0.0 and v == 0.0
