"""The area of bodies far below one cell, relative to itself: corners cut off at
the domain's four corners, and single vertices of the reference phase (four
corner triangles each) with legs over many decades, alone in their tile of the
fields kernel (64 x 32 cells), several to a tile, and beside ordinary ones.

Against the exact sum of the fractions' products (rational arithmetic): 1e-12,
far above the rounding of a double sum of the at most 2500 triangles (2^-50
each way) and of the tiles' partials."""
from fractions import Fraction

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402


def area_of(S, prec):
    ctx = ebit.ebit_create(S.nx, S.ny, S.dx, prec)
    try:
        ebit.ebit_load_state(ctx, S.K, S.Z, S.sH, S.sV)
        area = ebit.ebit_fraction(ctx)
        return area, ebit.ebit_diagnostics(ctx)["area"]
    finally:
        ebit.ebit_destroy(ctx)


def empty(nx, ny, prec):
    S = oracle.State(nx, ny, 1.0, prec)
    S.K[...] = 0
    S.Z[...] = 0
    S.sH[...] = 0.5
    S.sV[...] = 0.5
    return S


def stored(x, prec):
    return float(np.float32(x)) if prec == 1 else float(x)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("leg", [0.9, 0.06, 1e-3, 1e-5, 1e-9, 1e-15])
@pytest.mark.parametrize("nx,ny", [(5, 4), (64, 32), (65, 33), (130, 70)])
def test_domain_corner(nx, ny, leg, prec):
    for ci, cj in ((0, 0), (nx, 0), (0, ny), (nx, ny)):
        S = empty(nx, ny, prec)
        S.K[cj, ci] = 1
        top = 1 - 2.0 ** -24 if prec == 1 else 1 - 2.0 ** -53
        a, b = stored(leg, prec), stored(0.7 * leg, prec)
        a = min(stored(1 - a, prec), top) if ci else a
        b = min(stored(1 - b, prec), top) if cj else b
        S.sH[cj, max(ci - 1, 0)], S.sV[max(cj - 1, 0), ci] = a, b
        want = Fraction(1 - a if ci else a) * Fraction(1 - b if cj else b) / 2
        for got in area_of(S, prec):
            assert abs(Fraction(got) - want) <= Fraction(10) ** -12 * want


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("lo,hi", [(-1.0, -0.1), (-4.0, -1.0), (-12.0, -3.0), (-20.0, -8.0), (-18.0, -0.3)])
@pytest.mark.parametrize("nx,ny,every", [(64, 32, 3), (200, 100, 2), (200, 100, 30), (140, 70, 66)])
def test_single_vertices(nx, ny, every, lo, hi, prec):
    rng = np.random.default_rng(int(1000 * hi) + nx + every + 50000)
    S = empty(nx, ny, prec)
    want = Fraction(0)
    for j in range(1, ny, every):
        for i in range(1, nx, every):
            S.K[j, i] = 1
            legs = [stored(10.0 ** rng.uniform(lo, hi), prec) for _ in range(2)]  # right, up
            back = [stored(1 - 10.0 ** rng.uniform(-5.0, -1.0), prec) for _ in range(2)]  # left, down
            S.sH[j, i], S.sV[j, i] = legs
            S.sH[j, i - 1], S.sV[j - 1, i] = back
            x = Fraction(legs[0]) + 1 - Fraction(back[0])
            y = Fraction(legs[1]) + 1 - Fraction(back[1])
            want += x * y / 2  # the four triangles together
    for got in area_of(S, prec):
        assert abs(Fraction(got) - want) <= Fraction(10) ** -12 * want
