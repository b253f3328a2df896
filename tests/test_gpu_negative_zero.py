"""Sweeps from FP32 fractions at the low end of their range: -0.0 is 0, and
values below 2^-26 (down to the smallest denormal) are themselves.  Bit-exact
against the oracle started from the same values, and -0.0 and +0.0 markers step
to the same state."""
import numpy as np
import pytest

import oracle
from paper_2309_00338_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402
from tests.test_gpu_parity import COMPARED, assert_same_state, dev, gpu_from  # noqa: E402


@pytest.mark.parametrize("small", [-0.0, 0.0, 2.0 ** -27, 2.0 ** -60, 2.0 ** -149], ids=str)
@pytest.mark.parametrize("n", [48, 130])
def test_small_fractions(n, small):
    wl = W.vortex_workload(n, period=2.0, cfl=0.5)
    S = oracle.init(n, n, wl.dx, wl.scene, prec=oracle.FP32)
    rng = np.random.default_rng(n)
    for s in (S.sH, S.sV):
        s[rng.random(s.shape) < 0.5] = small
    u, v = (a.astype(np.float32).astype(np.float64) for a in (wl.field.u, wl.field.v))
    ctx = gpu_from(S)
    for s in (S.sH, S.sV):
        s[...] = np.abs(s)  # the oracle starts from +0
    try:
        for k in range(2):  # x then y, y then x
            ebit.ebit_step(ctx, dev(u, 1), dev(v, 1), wl.dt)
            r = oracle.step(S, u, v, wl.dt)
            c = ebit.ebit_diagnostics(ctx)["counters"]
            for q in COMPARED:
                assert c[q] == r["counters"][q], f"counter {q}"
            assert_same_state(ebit.ebit_get_state(ctx, n, n), S, 1)
    finally:
        ebit.ebit_destroy(ctx)
