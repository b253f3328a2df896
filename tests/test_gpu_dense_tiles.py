"""Sweeps of closely packed small drops (a cell apart, as close as the input may
be), whose tiles hold about as many markers as shared memory keeps moved fractions
of or more, and of a checkerboard, where every edge holds a marker.  Against the
oracle, bit for bit as in the other sweep tests, one grid at a time and in the
batched launches; and such a sweep costs in proportion to its markers: 1.7 to 1.8
times the time of drops that the tiles hold easily, for 1.8 times the markers, and
3 allowed (7.5 and 14 in FP32 and FP64 when every answer was recomputed from global
memory)."""
import math

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
from tests.test_gpu_server import _run  # noqa: E402


def lattice(nx, ny, radius, pitch, dx):
    """Drops on a lattice, none nearer than two cells to a wall."""
    x, y = (pitch * (np.arange(int((m - 4 - 2 * radius) / pitch) + 1)) + radius + 2.1 for m in (nx, ny))
    return [(a * dx, b * dx, radius * dx) for b in y for a in x]


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("radius,pitch", [(2.0, 5.0), (1.5, 4.0), (1.45, 3.9)])
@pytest.mark.parametrize("nx,ny", [(100, 40), (65, 97), (193, 130)])
def test_packed_drops(nx, ny, radius, pitch, prec):
    dx = 1.0 / max(nx, ny)
    S = oracle.init(nx, ny, dx, W.circle_scene(lattice(nx, ny, radius, pitch, dx)), prec)
    f = W.rotation_field(nx, ny, dx, 2 * math.pi, (0.5 * nx * dx, 0.5 * ny * dx), (0.3, 0.1))
    run_steps(S, f.u, f.v, 0.5 * dx / f.umax, prec)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(1, 70), (64, 32), (70, 33), (131, 99)])
def test_checkerboard(nx, ny, prec):
    rng = np.random.default_rng(nx + ny)
    S = oracle.State(nx, ny, 1.0 / nx, prec)
    S.K[...] = np.add.outer(np.arange(ny + 1), np.arange(nx + 1)) & 1
    S.Z[...] = rng.random(S.Z.shape) < 0.5
    for a in (S.sH, S.sV):
        a[...] = rng.random(a.shape).astype(np.float32).clip(0, np.float32(1 - 2.0 ** -24))
    u, v = (rng.uniform(-1.0, 1.0, (ny + 1, nx + 1)).astype(np.float32).astype(np.float64) for _ in range(2))
    run_steps(S, u, v, 0.75 * S.dx, prec)


def run_steps(S, u, v, dt, prec):
    if prec == 1:
        u, v = (a.astype(np.float32).astype(np.float64) for a in (u, v))
    ctx = gpu_from(S)
    try:
        for _ in range(2):  # x then y, y then x
            ebit.ebit_step(ctx, dev(u, prec), dev(v, prec), dt)
            r = oracle.step(S, u, v, dt)
            c = ebit.ebit_diagnostics(ctx)["counters"]
            for q in COMPARED:
                assert c[q] == r["counters"][q], f"counter {q}"
            assert_same_state(ebit.ebit_get_state(ctx, S.nx, S.ny), S, prec)
    finally:
        ebit.ebit_destroy(ctx)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
def test_batched(prec):
    """Every schedule of the server (a launch per sweep, or one persistent
    launch) gives what one grid at a time gives."""
    specs = []
    for n, radius, pitch in ((100, 1.5, 4.0), (131, 2.0, 5.0), (64, 1.45, 3.9)):
        specs.append(dict(n=n, circles=lattice(n, n, radius, pitch, 1.0 / n), field=ebit.EBIT_FIELD_ROTATION, prec=prec,
                          steps=4, cfl=0.5, period=1.0, omega=2 * math.pi, centre=(0.5, 0.5), drift=(0.3, 0.1)))
    alone = []
    for sp in specs:
        n = sp["n"]
        dx = 1.0 / n
        f = W.rotation_field(n, n, dx, sp["omega"], sp["centre"], sp["drift"])
        ctx = ebit.ebit_init(n, n, dx, W.circle_scene(sp["circles"]), prec)
        for _ in range(sp["steps"]):
            ebit.ebit_step(ctx, dev(f.u, prec), dev(f.v, prec), 0.5 * dx / f.umax)
        C = torch.empty((n, n), dtype=torch.float64 if prec == 0 else torch.float32, device="cuda")
        ebit.ebit_fraction(ctx, C)
        alone.append(C.cpu().numpy().ravel())
        ebit.ebit_destroy(ctx)
    for schedule in (0, ebit.EBIT_SCHED_PERSISTENT_LARGEST_FIRST):
        res, outs, _ = _run(specs, 8 << 30, autotune=False, schedule=schedule)
        for r, got, want in zip(res, outs, alone):
            assert r["status"] == 0 and r["counters"][ebit.D_INVARIANT] == 0
            assert np.array_equal(got, want)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
def test_cost(prec):
    n = 1024
    dx = 1.0 / n
    f = W.rotation_field(n, n, dx, 2 * math.pi, (0.5, 0.5), (0.3, 0.1))
    u, v = dev(f.u, prec), dev(f.v, prec)

    def sweep_ms(radius, pitch):
        ctx = ebit.ebit_init(n, n, dx, W.circle_scene(lattice(n, n, radius, pitch, dx)), prec)
        try:
            best = math.inf
            ebit.ebit_set_timing(ctx)
            for _ in range(8):
                ebit.ebit_step(ctx, u, v, 0.25 * dx / f.umax)
                ms, launches = ebit.ebit_timings(ctx)["sweep"]
                best = min(best, ms / launches)
            return best
        finally:
            ebit.ebit_destroy(ctx)

    assert sweep_ms(1.5, 4.0) < 3.0 * sweep_ms(2.0, 6.2)
