"""The tiled sweep on states far denser in markers than any flow makes: random
colours (half, a fifth, a tenth of the vertices) and fractions, so that tiles
hold more markers than shared memory keeps, just about as many, and more
candidates than the list.  Bit-exact against the oracle, as everywhere else:
colours, presence and counters, and fractions exactly in FP32 and to 1e-12 in
FP64 (the path's tolerance)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402
from tests.test_gpu_parity import COMPARED, assert_same_state, dev, gpu_from  # noqa: E402


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("share", [0.5, 0.2, 0.1])
@pytest.mark.parametrize("nx,ny", [(64, 32), (65, 97), (200, 66), (2, 90), (2050, 600)])
def test_random_states(nx, ny, share, prec):
    rng = np.random.default_rng(nx * 100 + ny)
    S = oracle.State(nx, ny, 1.0 / nx, prec)
    S.K[...] = rng.random(S.K.shape) < share
    S.Z[...] = rng.random(S.Z.shape) < 0.5
    for a in (S.sH, S.sV):
        a[...] = rng.random(a.shape).astype(np.float32).clip(0, np.float32(1 - 2.0 ** -24))
    u, v = (rng.uniform(-1.0, 1.0, (ny + 1, nx + 1)) for _ in range(2))
    if prec == 1:
        u, v = u.astype(np.float32).astype(np.float64), v.astype(np.float32).astype(np.float64)
    ctx = gpu_from(S)
    try:
        for _ in range(2):  # x then y, y then x
            ebit.ebit_step(ctx, dev(u, prec), dev(v, prec), 0.75 * S.dx)
            r = oracle.step(S, u, v, 0.75 * S.dx)
            c = ebit.ebit_diagnostics(ctx)["counters"]
            for q in COMPARED:
                assert c[q] == r["counters"][q], f"counter {q}"
            assert_same_state(ebit.ebit_get_state(ctx, nx, ny), S, prec)
    finally:
        ebit.ebit_destroy(ctx)
