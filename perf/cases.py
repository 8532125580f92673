"""What this library is timed on: runs of the HWFV1 model through its public
entry points, from the smallest grids to the largest ones its workloads use.

A simulation case is one forecast cycle of a program that keeps its handle:
put a state in (hwfv1_set_fields, hwfv1_set_time), take some steps
(hwfv1_advance, hwfv1_advance_uniform or hwfv1_batch_advance), read the fields
back (hwfv1_get_fields).  Each pass therefore starts from the same state and
does the same work.  The other cases are a whole run from host buffers (init,
steps, fields to the host), the multiresolution analysis on its own, and one
gradient of the subtree network.

The scenes are the model's usual ones: a circular dam-break on a flat bed, a
dam-break over Gaussian humps with wet/dry fronts, water columns on a flat
bed, a wet mound in a closed basin, and a terrain flood (spectral DEM, carved
channel, inflow, Manning friction).  Their sizes are those of the benchmark
and the tests; the seed draws the beds, positions and depths.

`exact` restates the method in plain float64 torch on row-major arrays.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2206_05761_gb300 import hwfv1 as H

G = 9.80665
INF = float("inf")


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _sim(name, scene, L, steps, eps=1e-3, precision=64, mode="plain"):
    """mode: plain, uniform (every finest cell), matched (conservative
    fluxes), store (exact leaf-value store)."""
    return dict(name=name, kind="cycle", scene=scene, L=L, steps=steps, eps=eps, precision=precision, mode=mode)


def listed():
    return [
        # the smallest runs: a 64 x 64 grid, 100 steps (launches and latency)
        _sim("circular_L6", "circular", 6, 100),
        # an ordinary adaptive run over an uneven, wet bed with dry humps;
        # the step count is not a multiple of the steps per graph
        _sim("bumpy_L10", "bumpy", 10, 37),
        # the flagship: the terrain flood at its hydrograph peak, mostly dry
        _sim("flood_L12", "flood", 12, 40),
        # the same problem one size down in the 32-bit path
        _sim("flood_L11_f32", "flood", 11, 40, precision=32),
        # smooth water on a flat bed: coarse leaves, encode and decode count
        _sim("columns_L11", "columns", 11, 20),
        # the same with the exact leaf-value store
        _sim("columns_L11_store", "columns", 11, 20, mode="store"),
        # the comparison solver: uniform FV1 on the finest grid
        _sim("uniform_L10", "bumpy", 10, 17, mode="uniform"),
        # the conservative variant in a closed, wet basin
        _sim("basin_L9_matched", "basin", 9, 48, mode="matched"),
        # a batch of independent dam-breaks of mixed depth, one graph per step
        dict(name="ensemble_16", kind="ensemble", levels="7,8,9,10", members=16, steps=10, eps=1e-3, precision=64),
        # the multiresolution analysis alone, phase by phase: new fields in,
        # encode, flag, traverse, the leaf list and one coarse level out
        dict(name="mra_L12", kind="mra", scene="flood", L=12, eps=1e-3, precision=64),
        # a whole short run from pinned host buffers to pinned host buffers
        dict(name="host_run_L10", kind="host", scene="flood", L=10, steps=32, eps=1e-3, precision=64),
        # forward and backward of the subtree network on a training batch
        dict(name="skipnet_gradients", kind="gradients", images=8, rows=128, cols=128),
    ]


def draw(rng):
    kind = rng.choice(["cycle"] * 7 + ["ensemble", "mra", "host", "gradients"])
    eps = 10.0 ** rng.uniform(-4.0, -2.0)
    if kind == "gradients":
        # ragged images as well as the square ones of a domain
        rows, cols = (int(2 ** rng.uniform(4, 7)) for _ in range(2))
        return dict(kind=kind, images=rng.randint(1, 8), rows=rows, cols=cols)
    if kind == "ensemble":
        lv = sorted(rng.sample([6, 7, 8, 9], rng.randint(1, 4)))
        return dict(kind=kind, levels=",".join(map(str, lv)), members=rng.randint(2, 16),
                    steps=rng.randint(1, 10), eps=eps, precision=rng.choice([64, 64, 32]))
    if kind == "mra":
        return dict(kind=kind, scene=rng.choice(["flood", "bumpy", "columns"]), L=rng.randint(6, 12), eps=eps,
                    precision=rng.choice([64, 64, 32]))
    scene = rng.choice(["circular", "bumpy", "flood", "columns", "basin"])
    precision = rng.choice([64, 64, 64, 32])
    if kind == "host":
        return dict(kind=kind, scene=scene, L=rng.randint(5, 10), steps=rng.randint(1, 24), eps=eps,
                    precision=precision)
    mode = rng.choice(["plain"] * 4 + ["uniform", "matched", "store"])
    top = {"uniform": 10, "matched": 9}.get(mode, 12 if scene == "flood" else 10)
    L = rng.randint(5, top)
    steps = int(round(2 ** rng.uniform(0, 5)))
    if L >= 10 and not (scene == "flood" and mode == "plain"):
        steps = min(steps, 15)
    return dict(kind=kind, scene=scene, L=L, steps=steps, eps=eps, precision=precision, mode=mode)


# ---------------------------------------------------------------------------
# Scenes: a problem description and its fields (row-major [j, i], float64)
# ---------------------------------------------------------------------------

def _problem(L, lx, eps, bc, manning_n=0.0, inflow=None, matched=False):
    return dict(L=L, lx=lx, ly=lx, x0=0.0, y0=0.0, eps=eps, cfl=0.5, g=G, manning_n=manning_n, tol_h=1e-3,
                dt_max=1.0, bc=bc, inflow=inflow, flux_match=matched)


def _f64(v, dev):
    return torch.tensor(v, dtype=torch.float64, device=dev)


def _humps(x, y, r, lo, hi):
    z = torch.zeros_like(x)
    for _ in range(8):
        a, s, cx, cy = r.uniform(lo, hi), r.uniform(0.02, 0.08), r.random(), r.random()
        z += a * torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2.0 * s * s))
    return z


def _scene(scene, L, eps, seed, dev, matched=False):
    """(problem, {z, h, qx, qy}, t0)."""
    r = random.Random(seed)
    n = 1 << L
    side = 10_000.0 if scene == "flood" else 1.0
    c = (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) * (side / n)
    x, y = c[None, :].expand(n, n), c[:, None].expand(n, n)
    qx, qy = torch.zeros(n, n, dtype=torch.float64, device=dev), torch.zeros(n, n, dtype=torch.float64, device=dev)
    t0, n_m, inflow, bc = 0.0, 0.0, None, ("closed",) * 4
    if scene == "circular":
        bc = ("transmissive",) * 4
        z = torch.zeros_like(qx)
        cx, cy, rad, hin = r.uniform(0.45, 0.55), r.uniform(0.45, 0.55), r.uniform(0.22, 0.28), r.uniform(1.8, 2.2)
        eta = torch.where((x - cx) ** 2 + (y - cy) ** 2 < rad * rad, _f64(hin, dev), _f64(1.0, dev))
    elif scene == "bumpy":
        z = _humps(x, y, r, 0.1, 0.6)
        eta = torch.where(x < 0.3, _f64(r.uniform(0.9, 1.1), dev), _f64(0.5, dev))
    elif scene == "columns":
        z = torch.zeros_like(qx)
        eta = torch.ones_like(qx)
        for _ in range(3):
            cx, cy, rad, hin = r.uniform(0.2, 0.8), r.uniform(0.2, 0.8), r.uniform(0.05, 0.15), r.uniform(1.3, 2.0)
            eta = torch.where((x - cx) ** 2 + (y - cy) ** 2 < rad * rad, eta.clamp(min=hin), eta)
    elif scene == "basin":
        z = _humps(x, y, r, 0.1, 0.6)
        eta = 1.0 + 0.3 * torch.exp(-((x - r.uniform(0.3, 0.7)) ** 2 + (y - r.uniform(0.3, 0.7)) ** 2) / 0.01)
    elif scene == "flood":
        gen = torch.Generator(device=dev).manual_seed(seed)
        f = torch.fft.fftfreq(n, dtype=torch.float64, device=dev)
        f2 = f[None, :] ** 2 + f[:, None] ** 2
        f2[0, 0] = INF
        noise = torch.complex(*(torch.randn(n, n, generator=gen, dtype=torch.float64, device=dev) for _ in range(2)))
        z = torch.fft.ifft2(noise / f2).real
        z = (z - z.min()) / (z.max() - z.min()) * 50.0 + 1e-3 * (side - x)
        width = max(60.0, 4.0 * side / n)
        yc = 0.5 * side + 0.1 * side * torch.sin(2.0 * math.pi * x / (r.uniform(0.45, 0.55) * side))
        inside = (y - yc).abs() < 0.5 * width
        z = torch.where(inside, z - 4.0, z)
        fill = r.uniform(0.9, 1.1)
        h, qx = inside * _f64(3.45 * fill, dev), inside * _f64(8.33 * fill, dev)
        dy = side / n
        inflow = dict(a0=int(math.floor((0.5 * side - 0.5 * width) / dy)),
                      a1=int(math.ceil((0.5 * side + 0.5 * width) / dy)), t=[0.0, 1800.0, 3600.0],
                      Q=[0.0, 500.0, 0.0])
        bc, n_m, t0 = ("inflow", "closed", "closed", "closed"), 0.03, 1800.0
        return (_problem(L, side, eps, bc, n_m, inflow, matched),
                dict(z=z.contiguous(), h=h.contiguous(), qx=qx.contiguous(), qy=qy), t0)
    h = (eta - z).clamp(min=0.0)
    return _problem(L, side, eps, bc, n_m, inflow, matched), dict(z=z.contiguous(), h=h.contiguous(), qx=qx, qy=qy), t0


def _members(case, seed):
    r = random.Random(seed)
    lv = [int(v) for v in case["levels"].split(",")]
    # every level occurs, so that a case's work does not depend on the seed
    return [(lv[d % len(lv)], r.randrange(1 << 30)) for d in range(case["members"])]


def _net_inputs(case, seed, dev):
    n, r, c = case["images"], case["rows"], case["cols"]
    gen = torch.Generator(device="cpu").manual_seed(seed)
    h = torch.rand(n, r, c, 1, generator=gen)
    q = 0.3 * torch.randn(n, r, c, 2, generator=gen)
    z = torch.rand(n, r, c, 1, generator=gen) * 0.6
    x = torch.cat([h, q, z], dim=-1).to(torch.bfloat16)
    y = torch.randint(0, 5, (n, r, c), generator=gen, dtype=torch.uint8)
    ws = []
    for co, ci in ((16, 4), (16, 16), (5, 16)):
        ws.append(torch.randn(co, ci, 3, 3, generator=gen) * math.sqrt(2.0 / (9 * ci)))
        ws.append(0.1 * torch.randn(co, generator=gen))
    par = torch.cat([w.reshape(-1) for w in ws]).to(torch.bfloat16).float().numpy()
    return x.to(dev), y.to(dev), par


# ---------------------------------------------------------------------------
# prepare, run, work
# ---------------------------------------------------------------------------

class _Handle:
    """A simulation (or batch, or network) handle freed with its state."""

    def __init__(self, hd, free):
        self.hd, self._free = hd, free

    def __del__(self):
        try:
            self._free(self.hd)
        except Exception:
            pass


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "gradients":
        x, y, par = _net_inputs(case, seed, dev)
        net = H.hwfv1_skipnet_create(0)
        H.hwfv1_skipnet_set_params(net, par)
        return dict(case=case, net=_Handle(net, H.hwfv1_skipnet_destroy), x=x, y=y)
    if kind == "ensemble":
        probs, fields = [], []
        for L, s in _members(case, seed):
            p, f, _ = _scene("bumpy", L, case["eps"], s, dev)
            probs.append(p)
            fields.append(f)
        torch.cuda.synchronize()
        specs = [H.make_problem(p, case["precision"]) for p in probs]
        bt = H.hwfv1_batch_init(specs, *[[f[k] for f in fields] for k in ("z", "h", "qx", "qy")])
        hds = [H.hwfv1_batch_member(bt, d) for d in range(len(specs))]
        return dict(case=case, batch=_Handle(bt, H.hwfv1_batch_destroy), members=hds,
                    start=[(0.0, H.hwfv1_get_time(hd)[1]) for hd in hds], fields=fields,
                    out=[[torch.empty_like(f["h"]) for _ in range(3)] for f in fields])
    p, f, t0 = _scene(case["scene"], case["L"], case["eps"], seed, dev, case.get("mode") == "matched")
    spec = H.make_problem(p, case["precision"])
    if kind == "host":
        f = {k: v.cpu().pin_memory() for k, v in f.items()}
        out = [torch.empty_like(f["h"]).pin_memory() for _ in range(3)]
        return dict(case=case, spec=spec, fields=f, out=out, t0=t0)
    torch.cuda.synchronize()
    hd = H.hwfv1_init(spec, f["z"], f["h"], f["qx"], f["qy"])
    if case.get("mode") == "store":
        H.hwfv1_set_leaf_store(hd, True)
    state = dict(case=case, sim=_Handle(hd, H.hwfv1_destroy), fields=f, start=(t0, H.hwfv1_get_time(hd)[1]))
    if kind == "mra":
        L = case["L"]
        state["leaves"] = torch.zeros(1 << (2 * L), dtype=torch.int32, device=dev)
        state["levels"] = [torch.empty(1 << (2 * (L - 2)), dtype=torch.float64, device=dev) for _ in range(3)]
    else:
        state["out"] = [torch.empty_like(f["h"]) for _ in range(3)]
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gradients":
        return H.hwfv1_skipnet_gradients(state["net"].hd, state["x"], state["y"], case["images"], case["rows"],
                                         case["cols"])
    if kind == "ensemble":
        for hd, f, (t, dt) in zip(state["members"], state["fields"], state["start"]):
            H.hwfv1_set_fields(hd, f["h"], f["qx"], f["qy"])
            H.hwfv1_set_time(hd, t, dt)
        H.hwfv1_batch_advance(state["batch"].hd, INF, case["steps"])
        for hd, out in zip(state["members"], state["out"]):
            H.hwfv1_get_fields(hd, *out)
        return state["out"]
    f = state["fields"]
    if kind == "host":
        hd = H.hwfv1_init(state["spec"], f["z"], f["h"], f["qx"], f["qy"])
        try:
            if state["t0"]:
                H.hwfv1_set_time(hd, state["t0"], H.hwfv1_get_time(hd)[1])
            H.hwfv1_advance(hd, INF, case["steps"])
            H.hwfv1_get_fields(hd, *state["out"])
        finally:
            H.hwfv1_destroy(hd)
        return state["out"]
    hd = state["sim"].hd
    H.hwfv1_set_fields(hd, f["h"], f["qx"], f["qy"])
    if kind == "mra":
        H.hwfv1_encode(hd)
        H.hwfv1_flag(hd)
        H.hwfv1_traverse(hd)
        n = H.hwfv1_get_leaves(hd, state["leaves"])
        for q, out in enumerate(state["levels"]):
            H.hwfv1_get_level(hd, q, case["L"] - 2, out)
        return {"n": n, "leaves": state["leaves"], "levels": state["levels"]}     # entries past n stay 0
    H.hwfv1_set_time(hd, *state["start"])
    if case["mode"] == "uniform":
        H.hwfv1_advance_uniform(hd, INF, case["steps"])
    else:
        H.hwfv1_advance(hd, INF, case["steps"])
    H.hwfv1_get_fields(hd, *state["out"])
    return state["out"]


# Leaves that hold or meet water, as a share of the finest cells, at the start
# of a run with eps = 1e-3 (the other leaves are dry and stay as they are).
_WET_SHARE = {"circular": 0.25, "bumpy": 0.3, "columns": 0.06, "basin": 0.1, "flood": 0.008}
# Additions, multiplications, square roots and divisions of one leaf update
# with every face formed once: two HLL faces (56 each), the velocities, the
# bed source, the update, the CFL bound.
_FLOP_LEAF = 152
# Per finest cell and step: three parents' sums over the levels (4/3 x 3/4 x 3).
_FLOP_CELL = 3


def work(case):
    kind = case["kind"]
    if kind == "gradients":
        px = case["images"] * case["rows"] * case["cols"]
        mac = 9 * (4 * 16 + 16 * 16 + 16 * 5)
        # forward, weight gradients of all layers, input gradients of two
        return {"bytes": px * (4 * 2 + 1), "flops": 2 * px * (2 * mac + 9 * (16 * 16 + 16 * 5))}
    if kind == "ensemble":
        lv = [int(v) for v in case["levels"].split(",")]
        cells = sum(1 << (2 * lv[d % len(lv)]) for d in range(case["members"]))
        return {"bytes": 7 * 8 * cells,
                "flops": case["steps"] * cells * (_WET_SHARE["bumpy"] * _FLOP_LEAF + _FLOP_CELL)}
    cells = 1 << (2 * case["L"])
    if kind == "mra":
        return {"bytes": (3 * 8 * 17 // 16 + 4) * cells, "flops": cells * 3 * 3}
    if case.get("mode") == "uniform":
        per = _FLOP_LEAF
    elif case["scene"] == "flood":
        per = _WET_SHARE["flood"] * (_FLOP_LEAF + _FLOP_CELL)     # dry ground is at rest
    else:
        per = _WET_SHARE[case["scene"]] * _FLOP_LEAF + _FLOP_CELL
    return {"bytes": 7 * 8 * cells, "flops": case["steps"] * cells * per}


# ---------------------------------------------------------------------------
# The method in plain float64 torch
# ---------------------------------------------------------------------------

def _kids(a):
    """Children [0]..[3] of every parent: (2i,2j) (2i+1,2j) (2i,2j+1) (2i+1,2j+1)."""
    return a[0::2, 0::2], a[0::2, 1::2], a[1::2, 0::2], a[1::2, 1::2]


def _parent(a):
    c0, c1, c2, c3 = _kids(a)
    p, q, d, e = c0 + c2, c1 + c3, c0 - c2, c1 - c3
    return 0.25 * (p + q), 0.25 * torch.maximum(torch.maximum((d + e).abs(), (p - q).abs()), (d - e).abs())


def _up(a):
    return a.repeat_interleave(2, 0).repeat_interleave(2, 1)


def _pyramid(a, L, eps):
    """Levels 0..L of one quantity and the threshold flags of levels 0..L-1."""
    s = max(1.0, float(a.abs().max()))
    lev, flags = [a], []
    for n in range(L - 1, -1, -1):
        p, d = _parent(lev[0])
        lev.insert(0, p)
        flags.insert(0, d >= math.ldexp(eps, n - L) * s)
    return lev, flags


def _tree(flags, L):
    """Regularised significance: ancestors and children of every flag."""
    close = [f.clone() for f in flags]
    for n in range(L - 2, -1, -1):
        c0, c1, c2, c3 = _kids(close[n + 1])
        close[n] |= c0 | c1 | c2 | c3
    return [close[n] | _up(flags[n - 1]) if n else close[0] for n in range(L)]


def _leaf_masks(sig, L):
    alive, out = torch.ones(1, 1, dtype=torch.bool, device=sig[0].device), []
    for n in range(L):
        out.append(alive & ~sig[n])
        alive = _up(alive & sig[n])
    return out + [alive]


def _hll(g, tol, hl, zl, ul, tl, hr, zr, ur, tr):
    zf = torch.maximum(zl, zr)
    dl, dr = (hl + zl) - zf, (hr + zr) - zf
    hl, hr = torch.where(dl >= tol, dl, 0.0), torch.where(dr >= tol, dr, 0.0)
    al, ar = torch.sqrt(g * hl), torch.sqrt(g * hr)
    us, cs = 0.5 * (ul + ur) + al - ar, 0.5 * (al + ar) + 0.25 * (ul - ur)
    sl, sr = torch.minimum(ul - al, us - cs), torch.maximum(ur + ar, us + cs)
    dryl, dryr = hl == 0.0, hr == 0.0
    sl = torch.where(dryl, ur - 2.0 * ar, torch.where(dryr, ul - al, sl))
    sr = torch.where(dryl, ur + ar, torch.where(dryr, ul + 2.0 * al, sr))
    qnl, qtl, qnr, qtr = hl * ul, hl * tl, hr * ur, hr * tr
    fl = (qnl, qnl * ul + 0.5 * g * hl * hl, qnl * tl)
    fr = (qnr, qnr * ur + 0.5 * g * hr * hr, qnr * tr)
    inv = 1.0 / (sr - sl)
    out = []
    for a, b, d in zip(fl, fr, (hr - hl, qnr - qnl, qtr - qtl)):
        m = (sr * a - sl * b + sl * sr * d) * inv
        v = torch.where(sl >= 0.0, a, torch.where(sr <= 0.0, b, m))
        out.append(torch.where(dryl & dryr, 0.0, v))
    return out, hl, hr


def _velocity(c, tol):
    wet = c[0] >= tol
    rh = 1.0 / torch.where(wet, c[0], 1.0)
    return torch.where(wet, c[1] * rh, 0.0), torch.where(wet, c[2] * rh, 0.0)


def _side_face(p, s, C, X):
    """Flux (h, normal, tangential) and the cell's own squared face depth on
    side s (0 W, 1 E, 2 S, 3 N) between the cell C and the state X."""
    (uc, vc), (ux, vx) = _velocity(C, p["tol_h"]), _velocity(X, p["tol_h"])
    if s >= 2:
        uc, vc, ux, vx = vc, uc, vx, ux
    if s in (0, 2):
        f, _, own = _hll(p["g"], p["tol_h"], X[0], X[3], ux, vx, C[0], C[3], uc, vc)
    else:
        f, own, _ = _hll(p["g"], p["tol_h"], C[0], C[3], uc, vc, X[0], X[3], ux, vx)
    return f + [own * own]


def _neighbour(lev, n, j, i, s, p):
    """State across side s of the cells (j, i) of level n; ghosts at the edge."""
    last = (1 << n) - 1
    dj, di = ((0, -1), (0, 1), (-1, 0), (1, 0))[s]
    jn, im = j + dj, i + di
    out = (jn < 0) | (jn > last) | (im < 0) | (im > last)
    jn, im = jn.clamp(0, last), im.clamp(0, last)
    X = [a[jn, im] for a in lev]
    if p["bc"][s] != "transmissive":
        k = 1 if s < 2 else 2
        X[k] = torch.where(out, -X[k], X[k])
    return X, jn, im, out


def _matched_faces(p, levels, sig, L):
    """Per level and side, the faces of every cell with the finer halves
    averaged toward refined neighbours."""
    faces = [None] * (L + 1)
    halves = ((0, 2), (1, 3), (0, 1), (2, 3))       # children on the W, E, S, N side
    for n in range(L, -1, -1):
        r = torch.arange(1 << n, device=sig[0].device)
        j, i = r[:, None].expand(1 << n, 1 << n), r[None, :].expand(1 << n, 1 << n)
        C = list(levels[n])
        faces[n] = []
        for s in range(4):
            X, jn, im, out = _neighbour(levels[n], n, j, i, s, p)
            f = _side_face(p, s, C, X)
            if n < L:
                refined = sig[n][jn, im] & ~out
                for q in range(4):
                    k = _kids(faces[n + 1][s][q])
                    f[q] = torch.where(refined, 0.5 * (k[halves[s][0]] + k[halves[s][1]]), f[q])
            faces[n].append(f)
    return faces


def _update(p, C, F, n, j, i, t, dt):
    """New (h, qx, qy) of the cells and their CFL bound."""
    L, g, tol = p["L"], p["g"], p["tol_h"]
    dx, dy = math.ldexp(p["lx"], -n), math.ldexp(p["ly"], -n)
    rx, ry = dt / dx, dt / dy
    W, E, S, N = F
    h = C[0] - rx * (E[0] - W[0]) - ry * (N[0] - S[0])
    qx = C[1] - rx * ((E[1] - W[1]) + 0.5 * g * (W[3] - E[3])) - ry * (N[2] - S[2])
    qy = C[2] - rx * (E[2] - W[2]) - ry * ((N[1] - S[1]) + 0.5 * g * (S[3] - N[3]))
    inf = p["inflow"]
    if inf:                                          # on the west side
        Q = float(np.interp(t, inf["t"], inf["Q"]))
        w = 1 << (L - n)
        cover = ((j + 1) * w).clamp(max=inf["a1"]) - (j * w).clamp(min=inf["a0"])
        cover = torch.where(i == 0, cover, 0).clamp(min=0)
        h = h + torch.where(cover > 0, (Q * dt) * (cover / (inf["a1"] - inf["a0"])) / (dx * dy), 0.0)
    h = h.clamp(min=0.0)
    wet = h >= tol
    qx, qy = torch.where(wet, qx, 0.0), torch.where(wet, qy, 0.0)
    hs = torch.where(wet, h, 1.0)
    if p["manning_n"] > 0.0:
        u, v = qx * (1.0 / hs), qy * (1.0 / hs)
        D = 1.0 + dt * g * p["manning_n"] * p["manning_n"] * torch.sqrt(u * u + v * v) / (hs * hs ** (1.0 / 3.0))
        qx, qy = qx * (1.0 / D), qy * (1.0 / D)
    return [h, qx, qy], _cfl(p, h, qx, qy)


def _cfl(p, h, qx, qy):
    wet = h >= p["tol_h"]
    hs = torch.where(wet, h, 1.0)
    a = torch.sqrt(p["g"] * hs)
    bx = math.ldexp(p["lx"], -p["L"]) / ((qx * (1.0 / hs)).abs() + a)
    by = math.ldexp(p["ly"], -p["L"]) / ((qy * (1.0 / hs)).abs() + a)
    b = torch.where(wet, torch.minimum(bx, by), INF)
    return float(b.min()) if b.numel() else INF


def _simulate(p, fields, t, steps, uniform=False):
    L, tol = p["L"], p["tol_h"]
    st = [fields["h"], fields["qx"], fields["qy"]]
    z = fields["z"]
    dev = z.device
    zl, zflags = _pyramid(z, L, p["eps"])
    dt = min(p["cfl"] * _cfl(p, *st), p["dt_max"])
    for _ in range(steps):
        if uniform:
            levels = [None] * L + [(*st, z)]
            sig = None
            masks = [torch.zeros(1, 1, dtype=torch.bool, device=dev)] * L + [torch.ones_like(z, dtype=torch.bool)]
        else:
            pyr = [_pyramid(a, L, p["eps"]) for a in st]
            flags = [zflags[n] | pyr[0][1][n] | pyr[1][1][n] | pyr[2][1][n] for n in range(L)]
            levels = [(pyr[0][0][n], pyr[1][0][n], pyr[2][0][n], zl[n]) for n in range(L + 1)]
            sig = _tree(flags, L)
            masks = _leaf_masks(sig, L)
        matched = _matched_faces(p, levels, sig, L) if p["flux_match"] and not uniform else None
        bound = INF
        carry = None                     # value handed down by a coarser leaf: h, qx, qy, eta or -inf, mask
        for n in range(L + 1):
            size = (1 << n, 1 << n)
            if carry is not None:
                carry = [_up(a) for a in carry]
            j, i = torch.nonzero(masks[n], as_tuple=True)
            if j.numel():
                C = [a[j, i] for a in levels[n]]
                if matched is not None:
                    F = [[q[j, i] for q in matched[n][s]] for s in range(4)]
                else:
                    F = [_side_face(p, s, C, _neighbour(levels[n], n, j, i, s, p)[0]) for s in range(4)]
                new, b = _update(p, C, F, n, j, i, t, dt)
                bound = min(bound, b)
                if carry is None:
                    carry = [torch.zeros(size, dtype=torch.float64, device=dev) for _ in range(4)]
                eta = new[0] + C[3] if n < L else new[0]
                eta = torch.where(new[0] >= tol, eta, -INF) if n < L else torch.full_like(new[0], -INF)
                for a, v in zip(carry, (*new, eta)):
                    a[j, i] = v
        h = torch.where(carry[3] > -INF, (carry[3] - z).clamp(min=0.0), carry[0])
        st = [h, carry[1], carry[2]]
        t += dt
        dt = min(p["cfl"] * bound, p["dt_max"])
    return st


def _exact_gradients(case, seed, dev):
    x, y, par = _net_inputs(case, seed, dev)
    x = x.double().permute(0, 3, 1, 2)
    shapes = [(16, 4, 3, 3), (16,), (16, 16, 3, 3), (16,), (5, 16, 3, 3), (5,)]
    flat = torch.from_numpy(par).double().to(dev)
    ws, o = [], 0
    for s in shapes:
        k = math.prod(s)
        ws.append(flat[o:o + k].reshape(s).clone().requires_grad_(True))
        o += k

    def conv(a, w, b):
        n, c, hh, ww = a.shape
        cols = torch.nn.functional.unfold(a, 3, padding=1)
        return (torch.einsum("ok,nkp->nop", w.reshape(w.shape[0], -1), cols)
                + b[None, :, None]).reshape(n, w.shape[0], hh, ww)

    a = torch.relu(conv(x, ws[0], ws[1]))
    a = torch.relu(conv(a, ws[2], ws[3]))
    logits = conv(a, ws[4], ws[5]).permute(0, 2, 3, 1).reshape(-1, 5)
    loss = torch.nn.functional.cross_entropy(logits, y.reshape(-1).long())
    loss.backward()
    return float(loss.detach()), torch.cat([w.grad.reshape(-1) for w in ws]).cpu().numpy()


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind = case["kind"]
    if kind == "gradients":
        return _exact_gradients(case, seed, dev)
    if kind == "ensemble":
        out = []
        for L, s in _members(case, seed):
            p, f, t = _scene("bumpy", L, case["eps"], s, dev)
            out.append(_simulate(p, f, t, case["steps"]))
        return out
    p, f, t = _scene(case["scene"], case["L"], case["eps"], seed, dev, case.get("mode") == "matched")
    if kind == "mra":
        lv = []
        for k in ("h", "qx", "qy"):
            a = _parent(_parent(f[k])[0])[0]
            n = a.shape[0]
            code = np.arange(n * n, dtype=np.int64)
            i, j = np.zeros_like(code), np.zeros_like(code)
            for b in range(case["L"]):
                i |= ((code >> (2 * b)) & 1) << b
                j |= ((code >> (2 * b + 1)) & 1) << b
            lv.append(a.reshape(-1)[torch.from_numpy(j * n + i).to(dev)])
        return {"n": None, "leaves": None, "levels": lv}
    out = _simulate(p, f, t, case["steps"], case.get("mode") == "uniform")
    return [a.cpu() for a in out] if kind == "host" else out
