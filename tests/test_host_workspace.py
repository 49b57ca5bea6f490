"""Workspaces of the dense calls, sized on the host: each call asks for what
its shape can reach.

* calls that never take the sliced products (fewer than 64 reflectors or
  vectors, more rows than they allow) need no slices, blocks of reflectors or
  partial products of them: their figures are those of the FP64 path;
* a reduction needs its panels, not a back-transformation's blocks;
* the vectors a back-transformation acts on, and the columns of a wide QR, add
  to the workspace no faster than linearly;
* a workspace serves every smaller shape too (gesvd: with fewer rows; its
  R exists for tall shapes only).
"""
import ctypes
import random

import pytest


@pytest.fixture(scope="module")
def ws():
    from paper_2508_11467_gb300 import bdc as b
    from paper_2508_11467_gb300 import build
    build.build()
    L = b.lib()
    for name in ("bdc_gebrd_workspace", "bdc_geqrf_workspace", "bdc_gesvd_workspace", "bdc_ormbr_workspace"):
        getattr(L, name).restype = ctypes.c_size_t
    o = b.make_opts("exact", 0)
    return {"gebrd": L.bdc_gebrd_workspace, "geqrf": L.bdc_geqrf_workspace, "ormbr": L.bdc_ormbr_workspace,
            "gesvd": lambda m, n: L.bdc_gesvd_workspace(m, n, ctypes.byref(o)), "bdc": lambda n: b.workspace_bytes(n, o)}


# bytes: per row 16 partial products of 64 vectors, the copied reflectors and
# the vectors' products, 10.3 KB in all, and 1 MB of fixed size
@pytest.mark.parametrize("m,n", [(3, 2), (60, 60), (1000, 63), (1000000, 50)])
def test_small_widths_take_no_slices(ws, m, n):
    most = 10300 * m + (1 << 20)
    assert ws["geqrf"](m, n) <= most and ws["ormbr"](m, n, n) <= most
    assert ws["gesvd"](m, n) <= most + ws["bdc"](n) + 32 * n + 16 * n * n + 4096


@pytest.mark.parametrize("m,n", [(3, 2), (1000, 1000), (4096, 4096), (16384, 16384), (10000, 600), (4194500, 40)])
def test_reduction_is_linear(ws, m, n):
    """Panels V, X, Y, U of 32 columns, partial sums (32 a row and column), two
    operands of 32 in seven slices of two bytes: 1.9 KB a row or column; the
    on-chip exchange: 2.7 KB a column, up to 2200."""
    assert ws["gebrd"](m, n) <= 1900 * (m + n) + 2700 * min(n, 2200) + (1 << 20)


@pytest.mark.parametrize("m,n", [(100, 100), (700, 66), (1600, 1600)])
def test_vectors_add_linearly(ws, m, n):
    a, b, c = (ws["ormbr"](m, n, k) for k in (1 << 16, 1 << 17, 1 << 18))
    assert b <= 2.1 * a and c <= 2.1 * b
    assert c <= (1 << 18) * 8 * 1600 + (1 << 30)


def test_wide_qr_is_linear(ws):
    a, b, c = (ws["geqrf"](100, n) for n in (50000, 100000, 200000))
    assert b <= 2.1 * a and c <= 2.1 * b and c <= 200000 * 1024


def test_square_sizes(ws):
    """Reflectors (8 bytes an entry), their slices and the vectors' (14 each)
    and partial products (8 each, up to three): at most 60 bytes an entry and
    12 MB of block triangles and fixed sizes."""
    for n in (64, 100, 333, 1000, 2048):
        assert ws["ormbr"](n, n, n) <= 60 * n * n + (12 << 20)
        assert ws["geqrf"](n, n) <= 60 * n * n + (12 << 20)


def test_serves_smaller_shapes(ws):
    r = random.Random(7)
    size = lambda a, b: int(round(a * (b / a) ** r.random()))
    for _ in range(4000):
        top = r.choice([300, 3000, 30000, 300000, 5000000])
        m = size(1, top)
        n, c, wide = size(1, min(m, 20000)), size(1, top), size(1, 20000)
        less = (lambda x: max(1, x - r.randint(0, 3))) if r.random() < 0.5 else (lambda x: size(1, x))
        m2, c2, wide2 = less(m), less(c), less(wide)
        n2 = min(m2, less(n))
        assert ws["gebrd"](m2, n2) <= ws["gebrd"](m, n), (m, n, m2, n2)
        assert ws["ormbr"](m2, n2, c2) <= ws["ormbr"](m, n, c), (m, n, c, m2, n2, c2)
        assert ws["geqrf"](m2, wide2) <= ws["geqrf"](m, wide), (m, wide, m2, wide2)
        if n <= m2 and n <= 3000:
            assert ws["gesvd"](m2, n) <= ws["gesvd"](m, n), (m, n, m2)


@pytest.mark.parametrize("edge", [64, 2048, 131072, 32767 * 128])
def test_serves_smaller_shapes_at_edges(ws, edge):
    """Where the path changes: reflectors or vectors from 64 on, two sides at
    once up to 2048, rows of the sliced reflectors, rows of a product."""
    for k in range(-3, 4):
        x = edge + k
        for n in (50, 63, 64, 65, 300, 1000):
            if n < x:
                assert ws["gebrd"](x - 1, n) <= ws["gebrd"](x, n) and ws["geqrf"](x - 1, n) <= ws["geqrf"](x, n)
                assert ws["ormbr"](x - 1, n, n) <= ws["ormbr"](x, n, n) and ws["gesvd"](x - 1, n) <= ws["gesvd"](x, n)
                assert ws["ormbr"](1000, n, x - 1) <= ws["ormbr"](1000, n, x)
            if edge <= 2048:
                assert ws["ormbr"](3000, x - 1, n) <= ws["ormbr"](3000, x, n)
                assert ws["geqrf"](3000, x - 1) <= ws["geqrf"](3000, x) and ws["gebrd"](3000, x - 1) <= ws["gebrd"](3000, x)
