"""The work a program that uses this library has it do, as cases to be timed.

A case is one pass through the public entry points on one grid (or one set of
requests):

  step      a solver's time step: the interface advected by vertex velocities,
            then its fractions C and curvature kappa taken into the caller's
            own dense tensors
  coupled   the same step handed to a one-fluid flow solver: density and
            viscosity per cell, surface-tension force per face
  host      a step whose velocities come from pinned host memory and whose
            fractions go back there (a solver that runs on the host)
  noalloc   fractions, area and marker counts of a state held in the caller's
            own buffers, without a context
  served    a set of requests (grids of uneven sizes, many steps each) handed
            to the batching server and waited for

Scenes are disks on a jittered lattice (one per lattice cell, at least four
cells apart), optionally with the Fourier curve of the 4096^2 workload across
the middle.  A stepping state moves with the flow for TURN passes and back
for as many, as the time-reversed tests of the method do, so that it can be
stepped for as long as one likes and still holds the same kind of interface.
"""
import math

import numpy as np
import torch

from paper_2309_00338_gb300 import ebit
from paper_2309_00338_gb300 import workloads as W

TURN = 16           # passes in one direction before the flow is turned round
CFL = 0.5
FLUIDS = dict(rho1=1000.0, rho2=1.2, mu1=1.0e-3, mu2=1.8e-5, sigma=0.0728)
EXACT_CELLS = 5_000_000   # the 64-bit evaluation of a step takes about a second per million cells


def _grid(name, kind, nx, ny, fp64, flow, rmin, rmax, pitch, curve=False, line=False, ghf=False):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "fp64": fp64, "flow": flow, "rmin": rmin, "rmax": rmax,
            "pitch": pitch, "curve": curve, "line": line, "ghf": ghf}


def listed():
    return [
        # the smallest call: one disk in the single vortex on the 64^2 grid of the accuracy tests, double
        _grid("step_fp64_64", "step", 64, 64, True, "vortex", 9.6, 9.6, 64.0),
        # a small ragged grid with the straight-line fit (EBIT-SL), as the method's comparison runs take it
        _grid("step_fp32_193x257_line", "step", 193, 257, False, "cellular", 3.0, 12.0, 29.0, line=True),
        # an ordinary grid: many small disks in solid rotation, as the 1024^2 workload
        _grid("step_fp32_1024", "step", 1024, 1024, False, "rotation", 2.0, 9.0, 20.0),
        # an ordinary ragged grid in double with little interface: most tiles hold none
        _grid("step_fp64_1021x771", "step", 1021, 771, True, "vortex", 20.0, 60.0, 170.0),
        # the large grid of the benchmark, both precisions
        _grid("step_fp32_4096", "step", 4096, 4096, False, "cellular", 3.0, 12.0, 29.0, curve=True),
        _grid("step_fp64_4096", "step", 4096, 4096, True, "cellular", 3.0, 12.0, 29.0, curve=True),
        # a flow solver's step, curvature with the generalised height functions
        _grid("coupled_fp32_2048_ghf", "coupled", 2048, 2048, False, "cellular", 3.0, 12.0, 29.0, curve=True, ghf=True),
        # the same in double on a ragged grid, standard height functions
        _grid("coupled_fp64_1100x1501", "coupled", 1100, 1501, True, "rotation", 4.0, 24.0, 54.0),
        # a solver on the host: velocities up and fractions down every step
        _grid("host_fp32_2048", "host", 2048, 2048, False, "cellular", 3.0, 12.0, 29.0, curve=True),
        # the allocation-free fraction entry at a large size and at a ragged one in double
        _grid("noalloc_fp32_4096", "noalloc", 4096, 4096, False, "cellular", 3.0, 12.0, 29.0),
        _grid("noalloc_fp64_1283x777", "noalloc", 1283, 777, True, "cellular", 3.0, 12.0, 29.0),
        # the batched workload: grids of 32..512 cells a side, 1-64 disks, hundreds of steps, single precision
        {"name": "served_fp32_64", "kind": "served", "grids": 64, "fp64": False, "smin": 200, "smax": 600},
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "coupled", "host", "noalloc", "served"])
    fp64 = rng.random() < 0.5
    if kind == "served":
        smin = rng.randint(40, 130)
        return {"kind": kind, "grids": int(round(math.exp(rng.uniform(math.log(6), math.log(60))))), "fp64": fp64,
                "smin": smin, "smax": smin * 2}
    top = 2900 if kind in ("noalloc", "host", "coupled") or fp64 else 3600  # times the aspect: at most 4096^2 cells
    nx = int(round(math.exp(rng.uniform(math.log(40), math.log(top)))))
    ny = max(33, int(round(nx * math.exp(rng.uniform(-0.25, 0.25)))))
    rmin = rng.uniform(2.0, 6.0)
    rmax = min(rmin + rng.uniform(0.5, 24.0), 0.2 * min(nx, ny))
    rmin = min(rmin, rmax)
    case = _grid("", kind, nx, ny, fp64, rng.choice(["vortex", "cellular", "rotation"]), round(rmin, 3), round(rmax, 3),
                 round(2.0 * rmax + rng.uniform(3.0, 30.0), 3), curve=rng.random() < 0.3 and min(nx, ny) > 200,
                 line=kind == "step" and rng.random() < 0.2, ghf=kind == "coupled" and rng.random() < 0.5)
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _disks(case, seed):
    """Disks in cell units on a lattice of cells of `pitch`: arrays (ly, lx) of centre x, y and radius (0: none)."""
    rng = np.random.RandomState(seed % (1 << 31))
    p = case["pitch"]
    lx, ly = max(1, int(case["nx"] // p)), max(1, int(case["ny"] // p))
    r = rng.uniform(case["rmin"], case["rmax"], (ly, lx))
    room = np.maximum(0.0, 0.5 * (p - 4.0) - r)
    xc = (np.arange(lx)[None, :] + 0.5) * p + rng.uniform(-1.0, 1.0, (ly, lx)) * room
    yc = (np.arange(ly)[:, None] + 0.5) * p + rng.uniform(-1.0, 1.0, (ly, lx)) * room
    r = np.where((xc - r < 2.0) | (yc - r < 2.0) | (xc + r > case["nx"] - 2.0) | (yc + r > case["ny"] - 2.0), 0.0, r)
    curve = None
    if case["curve"]:
        curve = W.fourier_curve(W.Rng(seed), y0=0.5 * case["ny"] / case["nx"])
        xs = np.linspace(0.0, case["nx"], 2048)
        h = W.curve_height(curve, xs / case["nx"]) * case["nx"]
        near = np.zeros_like(r, bool)
        for a in range(0, 2048, 4):
            near |= (xc - xs[a]) ** 2 + (yc - h[a]) ** 2 < (r + 3.0) ** 2
        r = np.where(near, 0.0, r)
    return xc, yc, r, curve


def _flow(case, device, dtype):
    """Vertex velocities of the flow on [0,1] x [0,ny/nx], and the largest component."""
    nx, ny = case["nx"], case["ny"]
    a = ny / nx
    X = torch.arange(nx + 1, dtype=torch.float64, device=device)[None, :] / nx
    Y = torch.arange(ny + 1, dtype=torch.float64, device=device)[:, None] / ny
    s = lambda t: torch.sin(math.pi * t)  # noqa: E731
    c = lambda t: torch.cos(math.pi * t)  # noqa: E731
    if case["flow"] == "cellular":
        u, v = s(X) * c(Y), -a * c(X) * s(Y)
    elif case["flow"] == "vortex":
        u, v = -s(X) ** 2 * s(2.0 * Y), a * s(Y) ** 2 * s(2.0 * X)
    else:
        u, v = -2.0 * math.pi * (a * Y - 0.5 * a) + 0.3 + 0.0 * X, 2.0 * math.pi * (X - 0.5) + 0.1 + 0.0 * Y
    umax = float(max(u.abs().max(), v.abs().max()))
    return u.to(dtype).contiguous(), v.to(dtype).contiguous(), umax


def _state64(case, seed):
    """The scene's colours and marker fractions in double, dense: the disk of a vertex's lattice cell decides it."""
    xc, yc, r, _ = _disks(case, seed)
    nx, ny, p = case["nx"], case["ny"], case["pitch"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T = [torch.from_numpy(np.ascontiguousarray(t)).to(dev) for t in (xc, yc, r)]
    ly, lx = r.shape

    def owner(x, y):  # the disk of the lattice cell of each point of a grid x, y (1-D coordinates)
        ci = torch.clamp((x / p).floor().long(), 0, lx - 1)
        cj = torch.clamp((y / p).floor().long(), 0, ly - 1)
        return [t[cj[:, None], ci[None, :]] for t in T]

    def inside(x, y):
        ox, oy, o = owner(x, y)
        return ((x[None, :] - ox) ** 2 + (y[:, None] - oy) ** 2 <= o * o) & (o > 0)

    xi = torch.arange(nx + 1, dtype=torch.float64, device=dev)
    yj = torch.arange(ny + 1, dtype=torch.float64, device=dev)
    K, Z = inside(xi, yj), inside(xi[:-1] + 0.5, yj[:-1] + 0.5)
    ox, oy, o = owner(xi, yj)

    def root(at, low, c, other, oc, rad):  # fraction along an edge whose `low` end is inside (or its other end is)
        half = torch.sqrt(torch.clamp(rad * rad - (other - oc) ** 2, min=0.0))
        return torch.where(low, c + half, c - half) - at

    pick = lambda t, k: torch.where(k, t[:, :-1], t[:, 1:])  # noqa: E731
    k = K[:, :-1]
    sH = root(xi[None, :-1], k, pick(ox, k), yj[:, None], pick(oy, k), pick(o, k))
    pick = lambda t, k: torch.where(k, t[:-1], t[1:])  # noqa: E731
    k = K[:-1]
    sV = root(yj[:-1, None], k, pick(oy, k), xi[None, :], pick(ox, k), pick(o, k))
    top = 1.0 - 2.0 ** -24
    sH = torch.where(K[:, 1:] ^ K[:, :-1], torch.clamp(sH, 0.0, top), torch.full_like(sH, 0.5))
    sV = torch.where(K[1:] ^ K[:-1], torch.clamp(sV, 0.0, top), torch.full_like(sV, 0.5))
    return K, Z, sH, sV


class _Context:
    """A context handle that is given back with the state."""

    def __init__(self, case, seed):
        xc, yc, r, curve = _disks(case, seed)
        n = case["nx"]
        circles = np.stack([xc[r > 0], yc[r > 0], r[r > 0]], 1) / n
        scene = {"circles": circles} | ({"curve": curve} if curve else {})
        flags = (ebit.EBIT_FIT_LINE if case["line"] else 0) | (ebit.EBIT_CURV_GHF if case["ghf"] else 0)
        self.h = ebit.ebit_init(n, case["ny"], 1.0 / n, scene, _prec(case), flags)

    def __del__(self):
        ebit.ebit_destroy(self.h)


class _Server:
    def __init__(self):
        self.h = ebit.ebit_server_create(16 << 30)

    def __del__(self):
        ebit.ebit_server_destroy(self.h)


def _prec(case):
    return ebit.EBIT_FP64 if case["fp64"] else ebit.EBIT_FP32


def _requests(case, seed):
    """(side, disks, vortex or cellular flow, steps) of each request: the sizes are the case's, the disks the seed's
    (the distributions of the batched workload)."""
    size, rng, out = W.Rng(case["grids"] + case["smin"]), W.Rng(seed), []
    for _ in range(case["grids"]):
        n = int(round(math.exp(size.uniform(math.log(32), math.log(512)))))
        lo = max(0.05, 3.0 / n)
        disks = W.place_circles(rng, size.integer(1, 64), lo, max(0.15, lo), 2.0 / n, lambda x, y, r: True, max_tries=50)
        out.append((n, disks, size.uniform() < 0.5, size.integer(case["smin"], case["smax"])))
    return out


def prepare(case, seed):
    dtype = torch.float64 if case["fp64"] else torch.float32
    if case["kind"] == "served":
        made = _requests(case, seed)
        C = np.zeros(sum(n * n for n, *_ in made), np.float64 if case["fp64"] else np.float32)
        reqs, at = [], 0
        for n, disks, vortex, steps in made:  # the vortex turns round once within the request's steps
            reqs.append(ebit.make_request(n, disks, ebit.EBIT_FIELD_VORTEX if vortex else ebit.EBIT_FIELD_CELLULAR,
                                          steps, CFL, _prec(case), steps * CFL / n, C_out=C[at:at + n * n]))
            at += n * n
        return {"case": case, "server": _Server(), "reqs": reqs, "C": C}
    nx, ny = case["nx"], case["ny"]
    new = lambda *shape: torch.empty(shape, dtype=dtype, device="cuda")  # noqa: E731
    if case["kind"] == "noalloc":
        K, Z, sH, sV = _state64(case, seed)
        return {"case": case, "K": K.to(torch.uint8), "Z": Z.to(torch.uint8), "sH": sH.to(dtype), "sV": sV.to(dtype),
                "C": new(ny, nx), "area": torch.empty(1, dtype=torch.float64, device="cuda"),
                "counts": torch.empty(2, dtype=torch.int64, device="cuda")}
    u, v, umax = _flow(case, "cuda", dtype)
    st = {"case": case, "ctx": _Context(case, seed), "u": u, "v": v, "dt": CFL / nx / umax, "pass": 0}
    if case["kind"] == "step":
        st |= {"C": new(ny, nx), "kappa": new(ny, nx)}
    elif case["kind"] == "coupled":
        st |= {"rho": new(ny, nx), "mu": new(ny, nx), "fx": new(ny, nx + 1), "fy": new(ny + 1, nx)}
    else:
        pin = lambda t: torch.empty(t.shape, dtype=dtype, pin_memory=True).copy_(t)  # noqa: E731
        st |= {"u_host": pin(u), "v_host": pin(v), "C_host": torch.empty((ny, nx), dtype=dtype, pin_memory=True),
               "area": torch.empty(1, dtype=torch.float64, pin_memory=True)}
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "served":
        tickets = [ebit.ebit_submit(st["server"].h, r) for r, _ in st["reqs"]]
        done = ebit.wait_all(st["server"].h, tickets)
        return {"C": st["C"], "area": np.array([done[t]["area"] for t in tickets]),
                "status": np.array([done[t]["status"] for t in tickets])}
    if kind == "noalloc":
        ebit.ebit_fraction_noalloc(case["nx"], case["ny"], 1.0 / case["nx"], _prec(case), st["K"], st["Z"], st["sH"],
                                   st["sV"], st["C"], st["area"], st["counts"])
        return {"C": st["C"], "area": st["area"], "counts": st["counts"]}
    ctx = st["ctx"].h
    dt = st["dt"] if (st["pass"] // TURN) % 2 == 0 else -st["dt"]
    st["pass"] += 1
    if kind == "host":
        st["u"].copy_(st["u_host"], non_blocking=True)
        st["v"].copy_(st["v_host"], non_blocking=True)
        ebit.ebit_step(ctx, st["u"], st["v"], dt)
        ebit.ebit_fraction_to_host(ctx, st["C_host"])
        ebit.ebit_area_async(ctx, st["area"])
        return {"C": st["C_host"], "area": st["area"]}
    ebit.ebit_step(ctx, st["u"], st["v"], dt)
    if kind == "coupled":
        out = {k: st[k] for k in ("rho", "mu", "fx", "fy")}
        ebit.ebit_coupling(ctx, **FLUIDS, **out)
        return out
    ebit.ebit_fraction(ctx, st["C"], want_area=False)
    ebit.ebit_curvature(ctx, st["kappa"], want_invalid=False)
    return {"C": st["C"], "kappa": st["kappa"]}


def _markers(case):
    """About how many markers of one orientation the case's interface has."""
    lattice = max(1, int(case["nx"] // case["pitch"])) * max(1, int(case["ny"] // case["pitch"]))
    return 4.0 * 0.5 * (case["rmin"] + case["rmax"]) * lattice + (case["nx"] if case["curve"] else 0)


def work(case):
    e = 8 if case["fp64"] else 4
    if case["kind"] == "served":
        # per request and step: the colours read and written, C and kappa written, the analytic velocity read;
        # sizes and steps at their means (log-uniform sides of 32..512 cells)
        cells = (512.0 ** 2 - 32.0 ** 2) / (2.0 * math.log(16.0)) * 0.5 * (case["smin"] + case["smax"]) * case["grids"]
        return {"bytes": cells * (0.5 + 4 * e), "flops": cells * 8.0}
    nx, ny = case["nx"], case["ny"]
    cells, verts, m = nx * ny, (nx + 1) * (ny + 1), _markers(case)
    if case["kind"] == "noalloc":
        return {"bytes": verts + cells + e * ((ny + 1) * nx + ny * (nx + 1)) + e * cells + 24, "flops": 16.0 * m}
    # colours and markers read and written, velocities read, the outputs written; per marker and sweep about a
    # move (8) and, for the unaligned half, two circle fits (81)
    base = 0.5 * cells + 4 * e * m + 2 * e * verts
    out = {"step": 2 * cells, "coupled": 2 * cells + nx * (ny + 1) + ny * (nx + 1), "host": cells}[case["kind"]]
    return {"bytes": base + e * out, "flops": m * (4 * 8 + 2 * (4 if case["line"] else 81) + 2 * 40)}


# ---------------------------------------------------------------------------
# the first pass in 64 bits, in plain numpy
# ---------------------------------------------------------------------------
def _partner_table():
    """partner[q, z, e]: the edge joined to edge e of a cell with corner mask q and centre colour z (-1: none);
    edges 0 bottom, 1 right, 2 top, 3 left, corners counter-clockwise from the lower left."""
    t = np.full((16, 2, 4), -1)
    for q in range(16):
        c = [(q >> b) & 1 for b in range(4)]
        on = [e for e in range(4) if c[e] != c[(e + 1) % 4]]
        for z in (0, 1):
            pairs = [on] if len(on) == 2 else [] if not on else [(b, (b + 3) % 4) for b in range(4) if c[b] != z]
            for a, b in pairs:
                t[q, z, a], t[q, z, b] = b, a
    return t


_PARTNER = _partner_table()
_DI, _DJ = np.array([0, 1, 0, 0]), np.array([0, 0, 1, 0])  # edge e of cell (i, j) is edge (i + DI, j + DJ)


def _masks(K):
    return K[:-1, :-1] + 2 * K[:-1, 1:] + 4 * K[1:, 1:] + 8 * K[1:, :-1]


def _crossing(A, B, P, have):
    """Where the circle through A, B and P (arrays of x, y; the grid line is x = 0) meets the line on the arc from A
    to B without P; valid where the circle is usable and the crossing lies on the edge."""
    qx, qy, rx, ry = B[0] - A[0], B[1] - A[1], P[0] - A[0], P[1] - A[1]
    q2, r2, t2 = qx * qx + qy * qy, rx * rx + ry * ry, (P[0] - B[0]) ** 2 + (P[1] - B[1]) ** 2
    x0 = -A[0]
    kap = qx * ry - qy * rx
    al, be = r2 * qy - q2 * ry, q2 * rx - r2 * qx
    c0 = x0 * (kap * x0 + al)
    disc = be * be - 4 * kap * c0
    h = -0.5 * (be + np.copysign(np.sqrt(np.maximum(disc, 0)), be))
    ok = have & (r2 >= 1e-4) & (t2 >= 1e-4) & (disc >= 0) & (h != 0)
    with np.errstate(all="ignore"):
        near, far = c0 / h, h / kap
        side = lambda y: (qx * y - qy * x0) * np.sign(kap) > 0  # noqa: E731
        y = np.where((kap != 0) & side(near) & ~side(far), far, near)
    y = A[1] + y
    return y, ok & (y >= 0) & (y <= 1)


def _sweep64(K, Z, sH, sV, w, lam, line):
    """One split sweep along x: vertex colours, centre colours and marker fractions after it."""
    ny, nx = Z.shape
    below = np.nextafter(1.0, 0.0)
    mH, mV = K[:, 1:] != K[:, :-1], K[1:] != K[:-1]
    I, J = np.arange(nx)[None, :], np.arange(nx + 1)[None, :]
    t = sH + np.clip(((1 - sH) * w[:, :-1] + sH * w[:, 1:]) * lam, -1, 1)
    aX = I + np.floor(t).astype(int)
    aF = np.minimum(t - np.floor(t), below)
    aF = np.where(aX < 0, 0.0, np.where(aX > nx - 1, below, aF))
    aX = np.clip(aX, 0, nx - 1)
    t = np.clip(((1 - sV) * w[:-1] + sV * w[1:]) * lam, -1, 1)
    t[:, [0, -1]] = 0.0
    uX, uF = J + np.floor(t).astype(int), np.minimum(t - np.floor(t), below)
    N = K.copy()
    for d, at in ((1, I + 1), (-1, I)):
        j, i = np.nonzero(mH & (aX == I + d))
        np.logical_xor.at(N, (j, at[0, i]), True)
    # landings: the median of those on an edge that keeps a marker
    pos = np.full((3, ny + 1, nx), np.inf)
    for q in range(3):
        lo, hi = max(0, 1 - q), nx - max(0, q - 1)
        src = slice(lo + q - 1, hi + q - 1)
        pos[q, :, lo:hi] = np.where(mH[:, src] & (aX[:, src] == I[:, lo:hi]), aF[:, src], np.inf)
    n = np.isfinite(pos).sum(0)
    rank = np.argsort(pos, axis=0, kind="stable")
    q = np.take_along_axis(rank, np.minimum(n // 2, 2)[None], 0)[0]
    present = N[:, 1:] != N[:, :-1]
    kept = np.where(present & (n % 2 == 1), I - 1 + q, -9)
    nH = np.where(kept >= -1, np.take_along_axis(pos, q[None], 0)[0], 0.5)
    # chords of the old segments
    M = _masks(K.astype(int))
    em = M ^ ((M >> 1) | ((M & 1) << 3))
    j, i = np.nonzero(em)
    a = np.array([[(m >> e) & 1 for e in range(4)] for m in range(16)]).argmax(1)[em[j, i]]
    two = em[j, i] == 15
    # (the two segments of a four-marker cell are those of its edges 0 and 2)
    seg = np.r_[np.zeros(len(j), int), np.ones(two.sum(), int)]
    j, i, a = np.r_[j, j[two]], np.r_[i, i[two]], np.r_[a, np.full(two.sum(), 2)]
    b = _PARTNER[M[j, i], Z[j, i].astype(int), a]

    def moved(kind, mi, mj):  # grid line index, fraction along the sweep, y
        h = kind == 0
        hi, vj = np.where(h, mi, 0), np.where(h, 0, mj)
        return (np.where(h, aX[mj, hi], uX[vj, mi]), np.where(h, aF[mj, hi], uF[vj, mi]),
                mj + np.where(h, 0.0, sV[vj, mi]))

    def edge(ci, cj, e):
        return e % 2, ci + _DI[e], cj + _DJ[e]

    def beyond(mk, ci, cj):  # the marker next along the interface on the far side of mk's edge, and its cell
        kind, mi, mj = mk
        oi = np.where((kind == 1) & (ci == mi), mi - 1, mi)
        oj = np.where((kind == 0) & (cj == mj), mj - 1, mj)
        oe = np.where(kind == 0, np.where(cj == mj, 2, 0), np.where(ci == mi, 1, 3))
        ok = (oi >= 0) & (oj >= 0) & (oi < nx) & (oj < ny)
        oi, oj = np.where(ok, oi, 0), np.where(ok, oj, 0)
        pe = np.where(ok, _PARTNER[M[oj, oi], Z[oj, oi].astype(int), oe], -1)
        return edge(oi, oj, np.maximum(pe, 0)), oi, oj, pe >= 0

    cand = []
    ea, eb = edge(i, j, a), edge(i, j, b)
    xa, xb = moved(*ea)[0], moved(*eb)[0]
    lo, hi = np.minimum(xa, xb), np.maximum(xa, xb)
    for s in range(1, 5):
        k = lo + s
        at = np.nonzero((k <= hi) & (k >= 1) & (k <= nx - 1))[0]
        left = xa[at] < k[at]
        pick = lambda f, x, y: tuple(np.where(f, p[at], r[at]) for p, r in zip(x, y))  # noqa: E731
        mA, mB = pick(left, ea, eb), pick(left, eb, ea)
        ci, cj, k = i[at], j[at], k[at]

        def xy(mk):
            X, F, Y = moved(*mk)
            return X - k + F, Y - cj

        A, B = xy(mA), xy(mB)
        far = []
        for near, mk in ((A, mA), (B, mB)):
            p, oi, oj, ok = beyond(mk, ci, cj)
            p2, _, _, ok2 = beyond(p, oi, oj)
            P, P2 = xy(p), xy(p2)
            close = (P[0] - near[0]) ** 2 + (P[1] - near[1]) ** 2 < 1e-4
            far.append((tuple(np.where(close, y, x) for x, y in zip(P, P2)), ok & (~close | ok2), p, ok))
        y1, v1 = _crossing(A, B, far[0][0], far[0][1])
        y4, v4 = _crossing(A, B, far[1][0], far[1][1])
        use = ((B[0] - A[0]) ** 2 + (B[1] - A[1]) ** 2 >= 1e-4) & (not line)
        v1, v4 = v1 & use, v4 & use
        with np.errstate(all="ignore"):
            chord = A[1] - A[0] * (B[1] - A[1]) / (B[0] - A[0])
        y = np.where(v1 & v4, 0.5 * (y1 + y4), np.where(v1, y1, np.where(v4, y4, chord)))
        y = np.where(B[0] == 0, B[1], y)
        g = lambda m, ok: np.stack([np.where(ok, m[0], -1), m[1], m[2]], 1)  # noqa: E731
        one = np.ones(len(k), bool)
        cand.append((cj * (nx + 1) + k, y, (ci - k + 2) * 2 + seg[at],
                     g(mA, one), g(mB, one), g(far[0][2], far[0][3]), g(far[1][2], far[1][3])))
    key, y, order, cA, cB, c1, c4 = (np.concatenate(t) for t in zip(*cand))
    by = np.lexsort((order, y, key))
    key, y = key[by], y[by]
    first = np.r_[True, key[1:] != key[:-1]]
    start = np.nonzero(first)[0]
    count = np.diff(np.r_[start, len(key)])
    mid = start + count // 2
    ej, ek = key[start] // (nx + 1), key[start] % (nx + 1)
    keep = (N[ej, ek] != N[ej + 1, ek]) & (count % 2 == 1)
    nV = np.where((J == 0) | (J == nx), sV, 0.5)
    nV[ej[keep], ek[keep]] = np.clip(y[mid[keep]], 0.0, below)
    # centre colours of the cells with four markers afterwards
    slot = {int(t): int(by[m]) for t, m in zip(key[start][keep], mid[keep])}
    NZ = Z.copy()
    m = _masks(N.astype(int))

    def verdict(j, k, right):
        s = slot.get(j * (nx + 1) + k)
        for mk in (() if s is None else (cB[s], c4[s]) if right else (cA[s], c1[s])):
            kind, mi, mj = (int(t) for t in mk)
            if kind < 0 or (aX[mj, mi] if kind == 0 else uX[mj, mi]) != (k if right else k - 1):
                return None
            if kind == 0:
                col = k if right else k - 1
                return (not N[mj, k]) if kept[mj, col] == mi else None
        return None

    for j, i in np.argwhere((m == 5) | (m == 10)):
        z = verdict(j, i, True) if i >= 1 else None
        if z is None and i + 1 <= nx - 1:
            z = verdict(j, i + 1, False)
        if z is not None:
            NZ[j, i] = z
    return N, NZ, nH, nV


def _fields64(K, Z, sH, sV, dx):
    """Fractions and 7x3 height-function curvature (NaN where there is none)."""
    M = _masks(K.astype(int))
    em = M ^ ((M >> 1) | ((M & 1) << 3))
    s = [sH[:-1], sV[:, 1:], sH[1:], sV[:, :-1]]
    legs = [s[3] * s[0], (1 - s[0]) * s[1], (1 - s[1]) * (1 - s[2]), s[2] * (1 - s[3])]
    C = np.where(M == 15, 1.0, 0.0)
    for c in range(4):
        cut = em == ((1 << c) | (1 << ((c + 3) % 4)))
        C = np.where(cut, np.where((M >> c) & 1, 0.5 * legs[c], 1 - 0.5 * legs[c]), C)
    for e, x, y in ((5, s[0], s[2]), (10, s[3], s[1])):
        C = np.where(em == e, np.where(M & 1, 0.5 * (x + y), 0.5 * ((1 - x) + (1 - y))), C)
    pair = np.where((M & 1) == Z, legs[1] + legs[3], legs[0] + legs[2])
    C = np.where(em == 15, np.where(Z, 1 - 0.5 * pair, 0.5 * pair), C)
    kap = np.full(C.shape, np.nan)
    ny, nx = C.shape
    j, i = np.nonzero(em)
    e, z = em[j, i], Z[j, i].astype(int)
    q = [t[j, i] for t in s]
    px, py = [q[0], 1.0 + 0 * q[0], q[2], 0 * q[0]], [0 * q[0], q[1], 1.0 + 0 * q[0], q[3]]
    ax = ay = 0.0
    for a in range(4):
        b = _PARTNER[M[j, i], z, a]
        for t in range(a + 1, 4):
            ax = ax + np.where(b == t, abs(px[t] - px[a]), 0.0)
            ay = ay + np.where(b == t, abs(py[t] - py[a]), 0.0)
    for ycol in (True, False):
        use = (ax >= ay) == ycol
        a, b = (i[use], j[use]) if ycol else (j[use], i[use])
        D = C if ycol else C.T
        inside = (a >= 1) & (a + 1 < D.shape[1]) & (b >= 3) & (b + 3 < D.shape[0])
        a, b = a[inside], b[inside]
        cols = [np.stack([D[b + t, a + m] for t in range(-3, 4)]) for m in (-1, 0, 1)]
        o = [np.where((c[0] == 1) & (c[6] == 0), 1, np.where((c[0] == 0) & (c[6] == 1), -1, 0)) for c in cols]
        h = [c.sum(0) for c in cols]
        hp, hpp = 0.5 * (h[2] - h[0]), h[2] - 2 * h[1] + h[0]
        ok = (o[0] != 0) & (o[0] == o[1]) & (o[1] == o[2])
        out = kap if ycol else kap.T
        out[b, a] = np.where(ok, -hpp / (dx * (1 + hp * hp) ** 1.5), np.nan)
    return C, kap


def _coupling64(C, kap, dx):
    f = FLUIDS
    rho, mu = (C * f[a] + (1 - C) * f[b] for a, b in (("rho1", "rho2"), ("mu1", "mu2")))

    def force(C, kap):  # faces along x, walls included
        a, b = kap[:, :-1], kap[:, 1:]
        k = np.where(np.isnan(a), np.where(np.isnan(b), 0.0, b), np.where(np.isnan(b), a, 0.5 * (a + b)))
        return np.pad(f["sigma"] / dx * k * (C[:, 1:] - C[:, :-1]), ((0, 0), (1, 1)))

    return rho, mu, force(C, kap), force(C.T, kap.T).T


def exact(case, seed):
    if case["kind"] == "served" or case["nx"] * case["ny"] > EXACT_CELLS * (4 if case["kind"] == "noalloc" else 1) \
            or case["curve"]:
        return None  # hundreds of steps of many grids; a large grid's step; the curve's markers are bisected
    dtype = torch.float64 if case["fp64"] else torch.float32
    K, Z, sH, sV = _state64(case, seed)
    if case["kind"] == "noalloc":  # the state is the input, in the precision it is given in
        sH, sV = sH.to(dtype).double(), sV.to(dtype).double()
    K, Z, sH, sV = (t.cpu().numpy() for t in (K, Z, sH, sV))
    dx = 1.0 / case["nx"]
    if case["kind"] != "noalloc":
        u, v, umax = _flow(case, "cuda" if torch.cuda.is_available() else "cpu", dtype)
        lam = CFL / case["nx"] / umax / dx
        K, Z, sH, sV = _sweep64(K, Z, sH, sV, u.double().cpu().numpy(), lam, case["line"])
        T = _sweep64(K.T.copy(), Z.T.copy(), sV.T.copy(), sH.T.copy(), v.double().cpu().numpy().T.copy(), lam, case["line"])
        K, Z, sV, sH = (t.T for t in T)
    C, kap = _fields64(K, Z, sH, sV, dx)
    area = np.array([C.sum() * dx * dx])
    if case["kind"] == "noalloc":
        return {"C": C, "area": area, "counts": None}
    if case["kind"] == "host":
        return {"C": C, "area": area}
    if case["kind"] == "coupled":
        rho, mu, fx, fy = _coupling64(C, kap, dx)
        return {"rho": rho, "mu": mu} | ({"fx": None, "fy": None} if case["ghf"] else {"fx": fx, "fy": fy})
    return {"C": C, "kappa": kap}
