"""The measured cases: what a user of the solver has it do, through the public
entry points of ``paper_1909_13086_gb300.lbm``.

Kinds of a case:
  * ``solo``   -- one lattice advanced ``steps`` steps, then its diagnostics and
                  all six fields read into pinned host arrays (a study's sample,
                  a request's result); with ``history`` also the ring of every
                  step's heated-wall inflow;
  * ``batch``  -- lattices advanced together, ``calls`` quanta of ``steps`` steps
                  (the serving loop), then every member's diagnostics and fields;
  * ``resume`` -- a checkpoint uploaded, ``steps`` steps, a checkpoint read back;
  * ``static`` -- one allocation-free step on the caller's own device buffers.

Every lattice starts in the middle of a run: a melt pool over the heated strip
(or ahead of the heated wall), a mushy rim, the solid at its seeded
perturbation, and a pair of convection rolls in the liquid.  Such a state is
uploaded as FP64 populations; the library rounds it to its storage type.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1909_13086_gb300 import lbm, workloads

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
FIELDS = ("H", "T", "fl", "ux", "uy", "rho")
DIAG = ("step", "melt_fraction", "H_total", "Q_strip", "Q_cum", "Nu", "front_x", "max_u")
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2, "fp16sr": 2, "bf16sr": 2}
TILE = 128  # column tile of the population layout that lbm_step_static takes


def listed():
    return [
        # The repository's reference cavity, advanced a few steps between
        # looks: the smallest calls, where launches and latency count.
        dict(name="solo_64x32_fp32", kind="solo", nx=64, ny=32, precision="fp32", problem="cavity", Ra=1e4,
             Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=10, diag_every=0, history=0),
        # One-dimensional melting (the Stefan study): periodic, no flow, FP64,
        # many steps between reads.
        dict(name="stefan_1024x4_fp64", kind="solo", nx=1024, ny=4, precision="fp64", problem="stefan", Ra=0.0,
             Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=500, diag_every=0, history=0),
        # A small request solved alone, one quantum.
        dict(name="solo_256x128_fp32", kind="solo", nx=256, ny=128, precision="fp32", problem="cavity", Ra=1e6,
             Pr=1.0, Ste=1.0, center=0.35, width=0.25, steps=100, diag_every=0, history=0),
        # The cavity study of the paper's parameters at 512 x 512: one sample.
        dict(name="solo_512x512_fp32", kind="solo", nx=512, ny=512, precision="fp32", problem="cavity", Ra=1e8,
             Pr=6.2, Ste=0.125, center=0.375, width=0.5, steps=200, diag_every=0, history=0),
        # A ragged, odd-sized cavity in BF16 storage with stochastic rounding.
        dict(name="solo_1001x701_bf16sr", kind="solo", nx=1001, ny=701, precision="bf16sr", problem="cavity",
             Ra=1e7, Pr=1.0, Ste=1.0, center=0.65, width=0.25, steps=99, diag_every=0, history=0),
        # The production cavity, the benchmark's workload: diagnostics every
        # 100 steps and the history of every step.
        dict(name="solo_2048x1024_fp32", kind="solo", nx=2048, ny=1024, precision="fp32", problem="cavity",
             Ra=1e8, Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=200, diag_every=100, history=200),
        # The same with 16-bit storage (the serving precision family).
        dict(name="solo_2048x1024_fp16sr", kind="solo", nx=2048, ny=1024, precision="fp16sr", problem="cavity",
             Ra=1e8, Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=200, diag_every=100, history=200),
        # The FP64 reference run of the precision study.
        dict(name="solo_2048x1024_fp64", kind="solo", nx=2048, ny=1024, precision="fp64", problem="cavity",
             Ra=1e8, Pr=1.0, Ste=1.0, center=0.25, width=0.25, steps=10, diag_every=0, history=0),
        # A serving group: 32 small requests, BF16-SR, five quanta, results read.
        dict(name="batch_32x256x128_bf16sr", kind="batch", nx=256, ny=128, members=32, mixed=False,
             precision="bf16sr", problem="cavity", Ra=1e7, Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=100,
             calls=5),
        # A group of unlike members in FP32 (sizes ragged, strips elsewhere).
        dict(name="batch_12_mixed_fp32", kind="batch", nx=512, ny=256, members=12, mixed=True, precision="fp32",
             problem="cavity", Ra=1e6, Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=100, calls=2),
        # Resume from a checkpoint, advance, write the next checkpoint.
        dict(name="resume_1024x512_fp32", kind="resume", nx=1024, ny=512, precision="fp32", problem="cavity",
             Ra=1e7, Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=100),
        # The allocation-free step of a host program that owns the buffers.
        dict(name="static_2048x1024_fp32", kind="static", nx=2048, ny=1024, precision="fp32", problem="cavity",
             Ra=1e8, Pr=1.0, Ste=1.0, center=0.5, width=0.25, steps=1),
    ]


MAX_CELLS, MAX_STEPS = 2048 * 1024, 500


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solo", "solo", "solo", "batch", "resume", "static"))
    problem = "stefan" if kind == "solo" and rng.random() < 0.25 else "cavity"
    precision = rng.choice(("fp32", "fp32", "bf16sr", "fp16sr", "bf16", "fp16", "fp64"))
    if kind == "static":
        precision = rng.choice(("fp32", "fp64"))
    if problem == "stefan":
        nx, ny = _log_int(rng, 64, 2048), _log_int(rng, 2, 16)
    else:
        nx = _log_int(rng, 48, 2048)
        ny = max(24, min(1024, int(nx * rng.uniform(0.4, 1.1))))
    if kind in ("solo", "resume") and precision == "fp64":
        nx, ny = min(nx, 1024), min(ny, 512)
    case = dict(kind=kind, nx=nx, ny=ny, precision=precision, problem=problem,
                Ra=0.0 if problem == "stefan" else 10.0 ** rng.randint(4, 6), Pr=rng.choice((1.0, 6.2)),
                Ste=rng.choice((0.125, 0.5, 1.0)), center=rng.choice((0.2, 0.35, 0.5, 0.65, 0.8)), width=0.25)
    # work of a pass: at most the largest listed case's cell updates
    budget = MAX_CELLS * (8 if precision == "fp64" else 180)
    if kind == "solo":
        case["steps"] = max(1, min(_log_int(rng, 3, MAX_STEPS), budget // (nx * ny)))
        case["diag_every"] = rng.choice((0, 0, 7, 50))
        case["history"] = rng.choice((0, 256))
    elif kind == "batch":
        case["nx"], case["ny"] = min(nx, 512), min(ny, 256)
        case["members"] = rng.randint(2, 32)
        case["mixed"] = rng.random() < 0.5
        case["calls"] = rng.randint(1, 4)
        cells = case["members"] * case["nx"] * case["ny"]
        case["steps"] = max(1, min(_log_int(rng, 10, 120), budget // (cells * case["calls"])))
    elif kind == "resume":
        case["nx"], case["ny"] = min(nx, 1024), min(ny, 512)
        case["steps"] = max(1, min(_log_int(rng, 3, 200), budget // (case["nx"] * case["ny"])))
    else:
        case["steps"] = 1
    return case


# ---------------------------------------------------------------- the inputs
def _members(case, seed):
    """(nx, ny, parameters, seed) of every lattice of a case."""
    out = []
    for k in range(case.get("members", 1)):
        nx, ny, center, Ra = case["nx"], case["ny"], case["center"], case["Ra"]
        if case.get("members", 1) > 1:
            center = (0.2, 0.35, 0.5, 0.65, 0.8)[k % 5]
            Ra = Ra / 10.0 ** (k % 2)
            if case["mixed"]:
                nx = max(34, int(nx / (1.0, 2.0, 1.37, 2.9)[k % 4]))
                ny = max(18, int(ny / (1.0, 2.0, 1.6)[k % 3]))
        p = dict(Pr=case["Pr"], Ste=case["Ste"], seed=seed + k)
        if case["problem"] == "stefan":
            prm = workloads.stefan_1024x4(Ste=case["Ste"], nx=nx)[2]
            prm.update(p)
        else:
            prm = workloads.params(Ra=Ra, strip_center=center, strip_width=case["width"], **p)
        out.append((nx, ny, prm, 1000003 * seed + k))
    return out


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _initial(nx, ny, p, seed):
    """Post-collision populations (f, g) of a run in its middle, (9, ny, nx) FP64."""
    dev = _device()
    gen = torch.Generator(device="cpu").manual_seed(seed)
    kw = dict(dtype=torch.float64, device=dev)
    size, shift, speed = (torch.rand(3, generator=gen, dtype=torch.float64) + 0.5).tolist()
    x = (torch.arange(nx, **kw) + 0.5)[None, :]
    y = (torch.arange(ny, **kw) + 0.5)[:, None]
    rough = torch.rand(ny, nx, generator=gen, dtype=torch.float64).to(dev) - 0.5
    Lh = 1.0 / p["Ste"]
    if p["problem"] == workloads.STEFAN:
        edge = nx * 0.25 * size
        depth = (edge - x).expand(ny, nx)      # cells inside the liquid
        T = (depth / edge).clamp(0.0, 1.0)
    else:
        cx, rx, ry = nx * (p["strip_center"] + 0.02 * (shift - 1.0)), nx * 0.22 * size, ny * 0.35 * size
        r = torch.sqrt(((x - cx) / rx) ** 2 + (y / ry) ** 2)
        depth = (1.0 - r) * min(rx, ry)
        T = (1.0 - r).clamp(0.0, 1.0) * (1.0 + 0.05 * rough)
    fl = (depth / 2.0 + 0.5 + 0.2 * rough).clamp(0.0, 1.0)
    T = torch.where(fl >= 1.0, T, torch.zeros_like(T))
    H = torch.where(fl > 0.0, T + fl * Lh, 2e-3 * rough)
    T = torch.where(fl > 0.0, T, H.clamp(max=0.0))
    w = torch.tensor(W, **kw)[:, None, None]
    if p["flow_on"]:
        U = 0.02 * speed
        ux = U * fl * torch.sin(2 * math.pi * (x - cx) / rx) * torch.cos(math.pi * y / ry)
        uy = U * fl * torch.cos(2 * math.pi * (x - cx) / rx) * torch.sin(math.pi * y / ry)
    else:
        ux = uy = torch.zeros(ny, nx, **kw)
    ex = torch.tensor(CX, **kw)[:, None, None]
    ey = torch.tensor(CY, **kw)[:, None, None]
    cu = ex * ux + ey * uy
    rho = 1.0 + 1e-4 * rough
    f = w * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
    if not p["flow_on"]:
        f = w.expand(9, ny, nx).clone()
    g = w * T * (1.0 + 3.0 * cu)
    g[0] += H - T
    return f, g


def _lattice(nx, ny, p, seed, precision, stream):
    lat = lbm.Lattice(nx, ny, p, precision=precision, stream=stream)
    f, g = _initial(nx, ny, p, seed)
    lat.set_populations(f.cpu().numpy(), g.cpu().numpy(), 0)
    return lat


def _pinned(*shape):
    return torch.empty(*shape, dtype=torch.float64, pin_memory=torch.cuda.is_available()).numpy()


def _tiles(planes, nx, ny, dtype):
    """(18, ny, nx) planes to the tile-major buffer of lbm_step_static."""
    ntx = -(-nx // TILE)
    pad = torch.zeros(18, ny, ntx * TILE, dtype=planes.dtype, device=planes.device)
    pad[:, :, :nx] = planes
    return pad.view(18, ny, ntx, TILE).permute(2, 1, 0, 3).contiguous().to(dtype)


def prepare(case, seed):
    members = _members(case, seed)
    nx, ny, p, s0 = members[0]
    st = dict(case=case, stream=torch.cuda.Stream())
    raw = st["stream"].cuda_stream
    if case["kind"] == "static":
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        st["src"] = _tiles(torch.cat(_initial(nx, ny, p, s0)), nx, ny, dtype)
        st["dst"] = torch.zeros_like(st["src"])
        st["params"] = p
        torch.cuda.synchronize()
        return st
    if case["kind"] == "resume":
        st["lat"] = lbm.Lattice(nx, ny, p, precision=case["precision"], stream=raw)
        st["in"], st["out"] = _pinned(2, 9, ny, nx), _pinned(2, 9, ny, nx)
        for k, v in enumerate(_initial(nx, ny, p, s0)):
            st["in"][k] = v.cpu().numpy()
        return st
    st["lats"] = [_lattice(a, b, q, s, case["precision"], raw) for a, b, q, s in members]
    st["fields"] = [_pinned(6, b, a) for a, b, _, _ in members]
    if case["kind"] == "batch":
        st["batch"] = lbm.Batch(len(members), raw)
        for lat in st["lats"]:
            st["batch"].add(lat)
    else:
        lbm.lbm_set_diag_every(st["lats"][0].h, case["diag_every"])
        if case["history"]:
            lbm.lbm_set_history(st["lats"][0].h, case["history"])
    return st


def _diag(d):
    return {k: d[k] for k in DIAG}


def run(st):
    case = st["case"]
    if case["kind"] == "static":
        d = lbm.lbm_step_static(st["src"].data_ptr(), st["dst"].data_ptr(), case["nx"], case["ny"],
                                lbm.PRECISIONS[case["precision"]], st["params"], 0, st["stream"].cuda_stream)
        return {"populations": st["dst"], "diag": _diag(d)}
    if case["kind"] == "resume":
        h = st["lat"].h
        lbm.lbm_write_populations(h, st["in"][0], st["in"][1], 0)
        lbm.lbm_step(h, case["steps"])
        lbm.lbm_read_populations(h, st["out"][0], st["out"][1])
        return {"populations": st["out"]}
    if case["kind"] == "batch":
        for _ in range(case["calls"]):
            st["batch"].step(case["steps"])
        diag = []
        for lat, out in zip(st["lats"], st["fields"]):
            d = lat.diagnostics(raise_on_diverged=False)
            diag.append([d[k] for k in DIAG])
            lbm.lbm_read_fields(lat.h, 63, *out)
        return {"fields": st["fields"], "diag": np.array(diag)}
    lat, out = st["lats"][0], st["fields"][0]
    lat.step(case["steps"])
    res = {"diag": _diag(lat.diagnostics(raise_on_diverged=False)), "fields": out}
    if case["history"]:
        res["history"] = lbm.lbm_read_history(lat.h, min(case["steps"], case["history"]))
    lbm.lbm_read_fields(lat.h, 63, *out)
    return res


def work(case):
    """Populations read once and written once, results written once; the
    method's operations on every cell and step (227 with flow, 100 without:
    fields, collisions and their moments, an FMA counted as two)."""
    cells = sum(nx * ny for nx, ny, _, _ in _members(case, 0))
    planes = 9 if case["problem"] == "stefan" else 18
    steps = case["steps"] * case.get("calls", 1)
    state = cells * planes * BYTES[case["precision"]]
    out = cells * (18 * 8 * 2 if case["kind"] == "resume" else 0 if case["kind"] == "static" else 6 * 8)
    return {"bytes": 2 * state + out, "flops": cells * steps * (100 if planes == 9 else 227)}


# ------------------------------------------------------- the same in 64 bits
def _derived(nx, ny, p):
    d = {}
    stefan = p["problem"] == workloads.STEFAN
    d["Href"] = float(nx if stefan else ny)
    if p["alpha_override"] > 0.0:
        d["alpha"] = p["alpha_override"]
        nu = p["Pr"] * d["alpha"]
        d["gbeta"] = p["Ra"] * nu * d["alpha"] / d["Href"] ** 3 if p["Ra"] > 0 else 0.0
    else:
        U = p["Ma"] / math.sqrt(3.0)
        nu = U * d["Href"] * math.sqrt(p["Pr"] / p["Ra"])
        d["alpha"] = nu / p["Pr"]
        d["gbeta"] = U * U / d["Href"]
    d["k"] = (p["k0"], 1.0 / (3.0 * d["alpha"] + 0.5), p["k2"])
    if p["k2"] < 0.0:
        d["k"] = (p["k0"], d["k"][1], 2.0 - d["k"][1])
    d["kf"] = (p["k0f"], p["k1f"], 1.0 / (3.0 * nu + 0.5))
    d["Lh"] = 1.0 / p["Ste"]
    a = nx * (p["strip_center"] - 0.5 * p["strip_width"])
    b = nx * (p["strip_center"] + 0.5 * p["strip_width"])
    d["lo2"], d["hi2"] = math.ceil(2.0 * a), math.floor(2.0 * b)
    d["len"] = float(ny) if stefan else b - a
    return d


def _stream(p, d, f, g):
    """Pull streaming with the wall rules; the heated wall's inflow."""
    nx, ny = g.shape[2], g.shape[1]
    stefan = p["problem"] == workloads.STEFAN
    Q = torch.zeros((), dtype=g.dtype, device=g.device)
    F, G = torch.empty_like(f) if f is not None else None, torch.empty_like(g)
    xs = torch.arange(nx, device=g.device)
    for i in range(9):
        cx, cy, o = CX[i], CY[i], OPP[i]
        for src, dst in ((f, F), (g, G)):
            if src is None:
                continue
            dst[i] = torch.roll(src[i], (cy, cx), (0, 1))
            if cx > 0:
                dst[i][:, 0] = src[o][:, 0]
            if cx < 0:
                dst[i][:, nx - 1] = src[o][:, nx - 1]
            if not stefan and cy > 0:
                dst[i][0] = src[o][0]
            if not stefan and cy < 0:
                dst[i][ny - 1] = src[o][ny - 1]
        if stefan and cx > 0:
            Q = Q + (2.0 * W[i] - 2.0 * g[o][:, 0]).sum()
            G[i][:, 0] = 2.0 * W[i] - g[o][:, 0]
        if not stefan and cy > 0 and p["strip_width"] > 0.0:
            xc2 = 2 * xs + 1 - cx
            hot = (xc2 >= d["lo2"]) & (xc2 <= d["hi2"])
            Q = Q + torch.where(hot, 2.0 * W[i] - 2.0 * g[o][0], torch.zeros_like(g[o][0])).sum()
            G[i][0] = torch.where(hot, 2.0 * W[i] - g[o][0], g[o][0])
    return F, G, Q


def _moments(q):
    s = q.sum(0)
    jx = q[1] - q[3] + q[5] - q[6] - q[7] + q[8]
    jy = q[2] - q[4] + q[5] + q[6] - q[7] - q[8]
    diag = q[5] + q[6] + q[7] + q[8]
    return s, jx, jy, q[1] + q[3] + diag, q[5] - q[6] + q[7] - q[8], q[2] + q[4] + diag


def _collide(q, mom, eq, k, force):
    """q - sum over the blocks of rate x (moment - equilibrium moment), each
    block on its D2Q9 polynomials, plus the forcing's moments: k0 relaxes
    everything, and the first and second moments get the difference of rates."""
    _, jx, jy, xx, xy, yy = mom
    s, ex, ey, exx, exy, eyy = eq
    k0, k1, k2 = k
    F1y, F2xy, F2yy = force
    ax = (k1 - k0) * (jx - ex)
    ay = (k1 - k0) * (jy - ey) - F1y
    bxx, bxy, byy = (k2 - k0) * (xx - exx), (k2 - k0) * (xy - exy) - F2xy, (k2 - k0) * (yy - eyy) - F2yy
    out = torch.empty_like(q)
    third = 1.0 / 3.0
    exx0, eyy0 = exx - s * third, eyy - s * third
    for i in range(9):
        cx, cy = CX[i], CY[i]
        qxx, qxy, qyy = cx * cx - third, cx * cy, cy * cy - third
        eq_i = W[i] * (s + 3.0 * (cx * ex + cy * ey) + 4.5 * (qxx * exx0 + 2.0 * qxy * exy + qyy * eyy0))
        out[i] = (1.0 - k0) * q[i] + k0 * eq_i - W[i] * (
            3.0 * (cx * ax + cy * ay) + 4.5 * (qxx * bxx + 2.0 * qxy * bxy + qyy * byy))
    return out


def _fields(p, d, F, G):
    H = G.sum(0)
    Lh = d["Lh"]
    zero, one = torch.zeros_like(H), torch.ones_like(H)
    T = torch.where(H <= 0, H, torch.where(H >= Lh, H - Lh, zero))
    fl = torch.where(H <= 0, zero, torch.where(H >= Lh, one, H / Lh))
    if F is None:
        return H, T, fl, zero, zero, one, zero, None
    mom = _moments(F)
    Fy = d["gbeta"] * T
    return H, T, fl, fl * mom[1] / mom[0], fl * (mom[2] + 0.5 * Fy) / mom[0], mom[0], Fy, mom


def _advance(nx, ny, p, f, g, steps, diag_at):
    """`steps` steps: (f, g, the last step's fields, inflow and melt fraction of every step)."""
    d = _derived(nx, ny, p)
    flow = bool(p["flow_on"])
    f = f if flow else None
    Qs, melts, fields = [], [], None
    for n in range(1, steps + 1):
        F, G, Q = _stream(p, d, f, g)
        fields = H, T, fl, ux, uy, rho, Fy, mom = _fields(p, d, F, G)
        zero = torch.zeros_like(H)
        g = _collide(G, _moments(G), (T, T * ux, T * uy, T / 3, zero, T / 3), d["k"], (0.0, 0.0, 0.0))
        g[0] += d["k"][0] * (H - T)
        if flow:
            s1, s2 = 1.0 - 0.5 * d["kf"][1], 1.0 - 0.5 * d["kf"][2]
            f = _collide(F, mom, (rho, rho * ux, rho * uy, rho * (1 / 3 + ux * ux), rho * ux * uy,
                                  rho * (1 / 3 + uy * uy)), d["kf"], (s1 * Fy, s2 * ux * Fy, s2 * 2.0 * uy * Fy))
        Qs.append(Q)
        melts.append(fl.mean() if diag_at(n) else torch.full_like(Q, math.nan))
    return d, f, g, torch.stack(fields[:6]), torch.stack(Qs), torch.stack(melts)


def _exact_diag(nx, ny, d, fields, Qs, steps):
    H, _, fl, ux, uy, _ = fields
    Q = Qs[-1].item()
    return dict(step=steps, melt_fraction=fl.mean().item(), H_total=H.sum().item(), Q_strip=Q,
                Q_cum=Qs.sum().item(), Nu=Q * d["Href"] / (d["alpha"] * d["len"]), front_x=fl.sum().item() / ny,
                max_u=torch.sqrt(ux * ux + uy * uy).max().item())


def exact(case, seed):
    steps = case["steps"] * case.get("calls", 1)
    every = case.get("diag_every", 0)
    fields, diags = [], []
    for nx, ny, p, s in _members(case, seed):
        f0, g0 = _initial(nx, ny, p, s)
        d, f, g, F, Qs, melts = _advance(nx, ny, p, f0, g0, steps, lambda n: n == steps or (every and n % every == 0))
        if case["kind"] == "static":
            pop = torch.cat([f if p["flow_on"] else torch.zeros_like(g), g])
            return {"populations": _tiles(pop, nx, ny, torch.float64), "diag": _exact_diag(nx, ny, d, F, Qs, 1)}
        if case["kind"] == "resume":
            return {"populations": torch.stack([f if p["flow_on"] else f0, g])}
        fields.append(F)
        diags.append(_exact_diag(nx, ny, d, F, Qs, steps))
    if case["kind"] == "batch":
        return {"fields": fields, "diag": np.array([[r[k] for k in DIAG] for r in diags])}
    res = {"diag": diags[0], "fields": fields[0]}
    if case["history"]:
        n = min(case["steps"], case["history"])
        Q = Qs[-n:]
        res["history"] = {"step": np.arange(steps - n + 1, steps + 1), "Q": Q,
                          "Nu": Q * d["Href"] / (d["alpha"] * d["len"]), "melt": melts[-n:]}
    return res
