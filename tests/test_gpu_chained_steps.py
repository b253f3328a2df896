"""Steps whose launches overlap: many steps queued without a host
synchronisation in between, the counters read after each run of them, one sweep
alone between steps, and a step captured once and replayed.  Everything equals
the oracle's step by step (counters and colours exactly, FP64 fractions to the
path's 1e-12)."""
import numpy as np
import pytest

import oracle
from paper_2309_00338_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402
from tests.test_gpu_parity import COMPARED, assert_same_fields, assert_same_state, dev, gpu_from  # noqa: E402


def _scene(n):
    dx = 1.0 / n
    rng = W.Rng(n)
    circles = W.place_circles(rng, n // 4, 2 * dx, 9 * dx, 2 * dx, lambda x, y, r: True)
    f = W.cellular_field(n, n, dx)
    return oracle.init(n, n, dx, W.circle_scene(circles), 0), f, 0.6 * dx


@pytest.mark.parametrize("n", [48, 300])
def test_queued_steps_and_counters(n):
    S, f, dt = _scene(n)
    ctx = gpu_from(S)
    u, v = dev(f.u, 0), dev(f.v, 0)
    try:
        for run in (1, 7, 2):
            for _ in range(run):
                ebit.ebit_step(ctx, u, v, dt)
                r = oracle.step(S, f.u, f.v, dt)
            c = ebit.ebit_diagnostics(ctx)
            for q in COMPARED:
                assert c["counters"][q] == r["counters"][q], f"counter {q}"
            assert abs(c["max_cfl"] - r["max_cfl"]) <= 1e-12
            assert_same_fields(ctx, S, r, 0)
        # one sweep alone counts by itself, and leaves nothing to the next step
        ebit.ebit_sweep(ctx, 0, u, dt)
        one, _ = oracle.sweep(S, 0, f.u, dt / S.dx)
        c = ebit.ebit_diagnostics(ctx)["counters"]
        for q in COMPARED:
            assert c[q] == one[q], f"counter {q} of a sweep"
        ebit.ebit_step(ctx, u, v, dt)
        r = oracle.step(S, f.u, f.v, dt)
        c = ebit.ebit_diagnostics(ctx)["counters"]
        for q in COMPARED:
            assert c[q] == r["counters"][q], f"counter {q} after a sweep"
        assert_same_state(ebit.ebit_get_state(ctx, n, n), S, 0)
    finally:
        ebit.ebit_destroy(ctx)


def test_captured_step_replays():
    """A step captured in a graph advances by the same split order each time it
    is replayed, and its counters are those of its last replay alone."""
    n = 130
    S, f, dt = _scene(n)
    stream = torch.cuda.Stream()
    u, v = dev(f.u, 0), dev(f.v, 0)
    torch.cuda.synchronize()
    ctx = ebit.ebit_create(n, n, S.dx, 0, stream=stream)
    try:
        ebit.ebit_load_state(ctx, S.K, S.Z, S.sH, S.sV, S.step_index)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            ebit.ebit_step(ctx, u, v, dt)
        with torch.cuda.stream(stream):
            for _ in range(5):
                g.replay()
        stream.synchronize()
        for _ in range(5):
            S.step_index = 0  # x first, as captured
            r = oracle.step(S, f.u, f.v, dt)
        c = ebit.ebit_diagnostics(ctx)["counters"]
        for q in COMPARED:
            assert c[q] == r["counters"][q], f"counter {q}"
        assert_same_fields(ctx, S, r, 0)
        assert_same_state(ebit.ebit_get_state(ctx, n, n), S, 0)
    finally:
        ebit.ebit_destroy(ctx)
