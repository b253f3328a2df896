"""Fractions and curvature of states at the edges of the fields kernel's tiles
(64 x 32 cells with a 3-cell halo) with fractions a flow rarely gives: zeros,
values far below the spacing of doubles near 1, the largest below 1, so that
interface cells come out exactly full, exactly empty or almost so.

Against the oracle: which cells have a curvature is equal; C and kappa are
equal in FP32; in FP64 C agrees to 1e-12 and kappa dx to 1e-12: heights are sums
of seven fractions, in double (the oracle, within 7 * 2^-50 of the exact sum) or
in units of 2^-60 (the kernel), and kappa dx changes by at most four times
their difference, below 1e-13."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("turned", [False, True], ids=["heights-y", "heights-x"])
@pytest.mark.parametrize("nx,ny", [(7, 7), (64, 32), (65, 33), (61, 70), (131, 64), (200, 100)])
def test_fractions_and_curvature(nx, ny, turned, prec):
    rng = np.random.default_rng(nx + 1000 * ny + turned)
    S = oracle.State(nx, ny, 1.0 / nx, prec)
    a, b = (ny, nx) if turned else (nx, ny)
    level = b // 2 + np.cumsum(rng.integers(-1, 2, a + 1) * (rng.random(a + 1) < 0.3))
    K = np.arange(b + 1)[:, None] <= np.clip(level, 0, b)[None, :]
    K ^= rng.random(K.shape) < 0.002
    if rng.random() < 0.5:
        K = ~K
    S.K[...] = K.T if turned else K
    S.Z[...] = rng.random(S.Z.shape) < 0.5
    top = 1 - 2.0 ** -24 if prec == 1 else 1 - 2.0 ** -53
    for s in (S.sH, S.sV):
        s[...] = rng.random(s.shape)
        kind = rng.integers(0, 12, s.shape)
        s[kind == 0], s[kind == 1], s[kind == 2], s[kind == 3] = 0.0, 2.0 ** -70, top, 2.0 ** -30
        if prec == 1:
            s[...] = np.minimum(s.astype(np.float32), np.float32(top))
    ctx = ebit.ebit_create(nx, ny, S.dx, prec)
    try:
        ebit.ebit_load_state(ctx, S.K, S.Z, S.sH, S.sV)
        dt = torch.float64 if prec == 0 else torch.float32
        C, kappa = (torch.empty((ny, nx), dtype=dt, device="cuda") for _ in range(2))
        area = ebit.ebit_fraction(ctx, C)
        invalid = ebit.ebit_curvature(ctx, kappa)
    finally:
        ebit.ebit_destroy(ctx)
    C, kappa = C.double().cpu().numpy(), kappa.double().cpu().numpy()
    C0, area0 = oracle.fraction(S)
    kappa0, invalid0 = oracle.curvature(S, C0)[:2]
    assert invalid == invalid0
    assert np.array_equal(np.isnan(kappa), np.isnan(kappa0))
    ok = ~np.isnan(kappa0)
    assert ok.any() or min(nx, ny) < 8
    if prec == 1:
        assert np.array_equal(C, C0) and np.array_equal(kappa[ok], kappa0[ok])
    else:
        assert np.max(np.abs(C - C0)) <= 1e-12
        assert np.max(np.abs(kappa - kappa0)[ok] * S.dx, initial=0.0) <= 1e-12
    assert abs(area - area0) <= 1e-12 * max(1.0, abs(area0))
