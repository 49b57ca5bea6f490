"""NaN and infinity in the operands of the sliced products (block reflectors
of ormbr, orgqr and geqrf): a column of C, or of A, that holds one comes back
without a finite entry where FP64 arithmetic leaves none, and the others come
back as if it were not there, to the bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu
BAD = [float("nan"), float("inf"), float("-inf")]


def _gauss(m, n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("n", [100, 300])
def test_back_transformation(n, bad):
    from paper_2508_11467_gb300 import bdc
    Ar, _, _, tauq, taup, info = bdc.gebrd(_gauss(n, n, n))
    assert info == 0
    for vect, tau in ((0, tauq), (1, taup)):
        C = _gauss(n, 200, 1) if vect == 0 else _gauss(200, n, 1)
        D = C.t().clone().t()
        cols = D if vect == 0 else D.t()       # vectors that the reflectors act on: columns of this view
        cols[n - 3, 5] = bad                   # below the first blocks' unit entries
        cols[7, 130] = bad
        X, Y = bdc.ormbr(vect, Ar, tau, C), bdc.ormbr(vect, Ar, tau, D)
        X, Y = (X, Y) if vect == 0 else (X.t(), Y.t())
        hit = torch.zeros(200, dtype=torch.bool, device="cuda")
        hit[[5, 130]] = True
        assert not bool(torch.isfinite(Y[1:, hit]).any())     # (row 0: P1 leaves the first entry alone)
        assert bool((Y[:, ~hit] == X[:, ~hit]).all())


@pytest.mark.parametrize("bad", BAD)
def test_qr_trailing_column(bad):
    from paper_2508_11467_gb300 import bdc
    A = _gauss(700, 600, 3)
    Ar, tau, info = bdc.geqrf(A)
    assert info == 0
    B = A.t().clone().t()
    B[650, 400] = bad
    Br, taub, _ = bdc.geqrf(B)
    assert bool((Br[:, :384] == Ar[:, :384]).all()) and bool((taub[:384] == tau[:384]).all())
    assert not bool(torch.isfinite(Br[:384, 400]).any())
    assert bool((Br[:384, 401:] == Ar[:384, 401:]).all())


@pytest.mark.parametrize("bad", BAD)
def test_explicit_q_of_a_broken_reflector(bad):
    """Reflector 100 of 300 broken: every column of Q from it on, and by the
    reflectors before it every row, is lost; nothing may look like a result."""
    from paper_2508_11467_gb300 import bdc
    Ar, tau, info = bdc.geqrf(_gauss(500, 300, 4))
    assert info == 0
    Ar[450, 100] = bad
    Q = bdc.orgqr(Ar, tau)
    assert not bool(torch.isfinite(Q[:, 100:]).any())
