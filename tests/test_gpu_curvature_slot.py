"""Curvature where the second difference of three column heights is largest: a
slot one cell wide and five deep (a finger, with the colours exchanged) whose
walls lie on the grid lines but for 1e-6 cell, with one vertex of the other
phase in its middle cell.  Heights of 5.5, 1 and 5.5 cells: the second
difference is 9, in any orientation.

Against the oracle: the same cells have a curvature, kappa equal in FP32, kappa
dx within 1e-12 in FP64 (a height is a sum of seven fractions, within 7 * 2^-50,
and kappa dx changes by at most four times the heights' difference)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402


def slot(n, i, j, turned, flipped, swapped, prec):
    """Cell (i, j) is the slot's middle one; arrays are indexed [y, x]."""
    t = 1e-6
    K = np.zeros((n + 1, n + 1), np.uint8)
    K[: j + 3, :] = 1
    K[j - 1 : j + 3, i : i + 2] = 0
    K[j, i] = 1
    sH, sV = np.full((n + 1, n), 0.5), np.full((n, n + 1), 0.5)
    sV[j + 2, :] = 1 - t             # the surface, just below the vertices of row j + 3
    sV[j - 2, i : i + 2] = t         # the slot's bottom
    sH[j - 1 : j + 3, i - 1] = 1 - t  # its walls
    sH[j - 1 : j + 3, i + 1] = t
    sV[j - 1, i], sV[j, i], sH[j, i] = 1 - t, t, 2 * t  # the vertex in the middle cell
    if flipped:  # upside down
        K, sH, sV = K[::-1], sH[::-1], 1 - sV[::-1]
    if turned:
        K, sH, sV = K.T, sV.T, sH.T
    S = oracle.State(n, n, 1.0 / n, prec)
    S.K[...] = K ^ 1 if swapped else K
    S.Z[...] = 0
    for a, b in ((S.sH, sH), (S.sV, sV)):
        a[...] = b.astype(np.float32) if prec == 1 else b
    return S


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("swapped", [False, True], ids=["slot", "finger"])
@pytest.mark.parametrize("flipped", [False, True], ids=["up", "down"])
@pytest.mark.parametrize("turned", [False, True], ids=["heights-y", "heights-x"])
def test_slot(turned, flipped, swapped, prec):
    n, i, j = 12, 5, 5
    S = slot(n, i, j, turned, flipped, swapped, prec)
    ctx = ebit.ebit_create(n, n, S.dx, prec)
    try:
        ebit.ebit_load_state(ctx, S.K, S.Z, S.sH, S.sV)
        kappa = torch.empty((n, n), dtype=torch.float64 if prec == 0 else torch.float32, device="cuda")
        invalid = ebit.ebit_curvature(ctx, kappa)
    finally:
        ebit.ebit_destroy(ctx)
    kappa = kappa.double().cpu().numpy()
    C0, _ = oracle.fraction(S)
    kappa0, invalid0 = oracle.curvature(S, C0)[:2]
    j = n - 1 - j if flipped else j
    mid = kappa0[(i, j) if turned else (j, i)]
    assert abs(abs(mid * S.dx) - 9.0) < 0.01, "the state is the one described"
    assert invalid == invalid0
    assert np.array_equal(np.isnan(kappa), np.isnan(kappa0))
    ok = ~np.isnan(kappa0)
    if prec == 1:
        assert np.array_equal(kappa[ok], kappa0[ok])
    else:
        assert np.max(np.abs(kappa - kappa0)[ok] * S.dx) <= 1e-12
