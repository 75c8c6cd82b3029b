"""What a user of this library runs, as cases whose speed and results can be
compared between two states of the code.

Every case is one pass through the public entry points of
``paper_2507_11067_gb300``: a stencil sweep (3D star and box in FP32 and
FP64, the planar kernels, pitched grids and dense ones), a batched acoustic
propagation, the gradient of its records with respect to the velocity, and
one step of the VTI and TTI systems.  Inputs are made on the GPU from a seed;
``exact`` restates each operator in plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_11067_gb300 as mms
from paper_2507_11067_gb300.wave import WaveFunction, WavePropagator

DEV = "cuda"

# Radius-4 (8th-order) central second- and first-derivative weights, offsets 0..4 and 1..4.
FD8 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)
FD1 = (4.0 / 5.0, -1.0 / 5.0, 4.0 / 105.0, -1.0 / 280.0)
W2 = np.array([FD8[abs(d)] for d in range(-4, 5)], np.float32)
W1 = np.array([0.0 if d == 0 else math.copysign(FD1[abs(d) - 1], d) for d in range(-4, 5)], np.float32)
AXES = np.stack([W2, W2, W2])

H, SPONGE, SPONGE_A, CFL, F0, R = 10.0, 20, 0.015, 0.4, 15.0, 4


def listed():
    return [
        # One sweep of a small grid, where the launch and a handful of thread
        # blocks are all there is: the 25-point 8th-order star on 64^3.
        _sweep("star_r4_64", "star", 4, 64, 64, 64),
        # The box sweeps of the benchmark: 27 points (memory) and 125 points
        # (tensor cores) on 512^3.
        _sweep("box_r1_512", "box", 1, 512, 512, 512),
        _sweep("box_r2_512", "box", 2, 512, 512, 512),
        # The widest box (729 points) on a grid whose sizes fit no tile.
        _sweep("box_r4_ragged", "box", 4, 251, 190, 133),
        # The 8th-order star on the largest grid of the sweeps, 1024^3.
        _sweep("star_r4_1024", "star", 4, 1024, 1024, 1024),
        # The one-call entry point on a dense grid of odd row length, as a C
        # program without a pitched allocator has it.
        _sweep("star_r2_dense", "star", 2, 301, 260, 230, layout="dense"),
        # The paper's 49-point planar box on one large plane.
        _sweep("box2d_r3_8192", "box2d", 3, 8192, 8192, 1),
        # Double precision: the 8th-order star on 256^3.
        _sweep("star_r4_f64_256", "star", 4, 256, 256, 256, dtype="f64"),
        # Batched forward modelling for reverse time migration: 8 shots on
        # 512^3, 16 steps of the 500 that a run takes, in one CUDA graph.
        {"name": "rtm_8x512", "op": "forward", "nx": 512, "ny": 512, "nz": 512, "shots": 8, "steps": 16,
         "graph": True},
        # One gradient of a waveform inversion through autograd: 2 shots on
        # 256^3, 40 steps with a checkpoint every 20.
        {"name": "gradient_2x256", "op": "gradient", "nx": 256, "ny": 256, "nz": 256, "shots": 2, "steps": 40,
         "every": 20},
        # One VTI time step on a survey whose sizes fit no tile.
        {"name": "vti_2x250", "op": "vti", "nx": 250, "ny": 230, "nz": 190, "shots": 2},
        # One TTI time step, 2 shots on 512^3.
        {"name": "tti_2x512", "op": "tti", "nx": 512, "ny": 512, "nz": 512, "shots": 2},
    ]


def _sweep(name, shape, r, nx, ny, nz, layout="pitched", dtype="f32"):
    return {"name": name, "op": "sweep", "shape": shape, "r": r, "nx": nx, "ny": ny, "nz": nz, "layout": layout,
            "dtype": dtype}


def _size(rng, lo, hi):
    """A size between lo and hi, even over their logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["sweep"] * 3 + ["dense", "plane", "f64", "forward", "gradient", "vti", "tti"])
    if op in ("sweep", "dense"):
        c = _sweep("", rng.choice(["star", "box"]), rng.randint(1, 4),
                   *(_size(rng, 48, 640 if op == "sweep" else 400) for _ in range(3)),
                   layout="dense" if op == "dense" else "pitched")
    elif op == "plane":
        c = _sweep("", rng.choice(["star2d", "box2d"]), rng.randint(1, 4), _size(rng, 300, 8192),
                   _size(rng, 300, 8192), 1)
    elif op == "f64":
        c = _sweep("", *rng.choice([("star", 2), ("star", 4), ("box", 1), ("box", 2)]),
                   *(_size(rng, 48, 300) for _ in range(3)), dtype="f64")
    elif op == "forward":
        c = {"op": "forward", "nx": _size(rng, 48, 400), "ny": _size(rng, 48, 400), "nz": _size(rng, 48, 400),
             "shots": rng.randint(1, 8), "steps": rng.randint(8, 16), "graph": rng.random() < 0.5}
    elif op == "gradient":
        c = {"op": "gradient", "nx": _size(rng, 48, 256), "ny": _size(rng, 48, 256), "nz": _size(rng, 48, 256),
             "shots": rng.randint(1, 3), "steps": rng.randint(20, 40), "every": rng.choice([10, 15, 20])}
    else:
        c = {"op": op, "nx": _size(rng, 48, 400), "ny": _size(rng, 48, 400), "nz": _size(rng, 48, 400),
             "shots": rng.randint(1, 4)}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs

def _rand(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, shape, lo, hi, dtype=torch.float32):
    return torch.rand(shape, generator=g, device=DEV, dtype=dtype) * (hi - lo) + lo


def _smooth(g, shape, cells=8):
    """A smooth random field in about [-1, 1], varying over `cells` cells."""
    coarse = _uniform(g, [1, 1] + [max(2, -(-n // cells)) for n in shape], -1.0, 1.0)
    return torch.nn.functional.interpolate(coarse, size=list(shape), mode="trilinear", align_corners=True)[0, 0]


def _npts(shape, r):
    return {"star": 6 * r + 1, "box": (2 * r + 1) ** 3, "star2d": 4 * r + 1, "box2d": (2 * r + 1) ** 2}[shape]


def _sweep_inputs(c, seed):
    """(weights, padded dense grid)."""
    shape, r = c["shape"], c["r"]
    dt = torch.float64 if c["dtype"] == "f64" else torch.float32
    g = np.random.default_rng(seed)
    if shape == "star" and r == 4:
        w = AXES.copy()
    else:
        k = 2 * r + 1
        n = {"star": 3 * k, "box": k ** 3, "star2d": 2 * k, "box2d": k * k}[shape]
        w = g.normal(0.0, 1.0 / math.sqrt(_npts(shape, r)), n).astype(np.float32)
    if dt == torch.float64:
        w = w.astype(np.float64)
    rz = 0 if shape.endswith("2d") else r
    return w, _uniform(_rand(seed), (c["nz"] + 2 * rz, c["ny"] + 2 * r, c["nx"] + 2 * r), -1.0, 1.0, dt)


def _velocity(g, rs, nz, ny, nx):
    """Six flat layers, 1500..4500 m/s, with 5 % smooth variation; the layer of each depth."""
    depths = np.sort(rs.choice(np.arange(1, nz), 5, replace=False))
    layer = torch.from_numpy(np.searchsorted(depths, np.arange(nz), side="right")).to(DEV)
    vel = torch.from_numpy(np.sort(np.r_[1500.0, rs.uniform(1500.0, 4500.0, 4), 4500.0])).to(DEV, torch.float32)
    v = vel[layer][:, None, None] * (1.0 + 0.05 * _smooth(g, (nz, ny, nx)))
    return v.contiguous(), layer


def _survey(c, rs):
    """Source points (at the receiver depth, inside the sponge-free box) and that depth."""
    n, z = (c["nx"], c["ny"]), min(SPONGE, c["nz"] - 1)
    at = [[int(rs.integers(SPONGE, k - SPONGE)) if k > 2 * SPONGE else int(rs.integers(0, k)) for k in n] + [z]
          for _ in range(c["shots"])]
    return np.array(at, np.int32), z


def _wavelet(dt, steps, shots):
    t = (np.arange(steps) * dt - 1.0 / F0) * math.pi * F0
    s = dt * dt * (1.0 - 2.0 * t * t) * np.exp(-t * t)
    return torch.from_numpy(np.repeat(s[:, None], shots, 1).astype(np.float32)).to(DEV)


def _wave_inputs(c, seed):
    """(v, src, rec_z, dt, amps, observed records)."""
    g, rs = _rand(seed), np.random.default_rng(seed)
    v, _ = _velocity(g, rs, c["nz"], c["ny"], c["nx"])
    src, rec_z = _survey(c, rs)
    dt = float(np.float32(CFL * H / (4500.0 * 1.05)))
    obs = None
    if c["op"] == "gradient":   # traces smooth in time, of the size of the modelled ones
        obs = torch.stack([2e-7 * _smooth(g, (c["steps"], c["ny"], c["nx"])) for _ in range(c["shots"])], 1)
    return v, src, rec_z, dt, _wavelet(dt, c["steps"], c["shots"]), obs


def _aniso_inputs(c, seed):
    """Interior medium fields, survey, dt and the four fields (shots, nz, ny, nx) at n and n-1."""
    g, rs = _rand(seed), np.random.default_rng(seed)
    n = (c["nz"], c["ny"], c["nx"])
    vp, layer = _velocity(g, rs, *n)

    def per_layer(lo, hi):
        v = torch.from_numpy(rs.uniform(lo, hi, 6)).to(DEV, torch.float32)
        return v[layer][:, None, None].expand(n).contiguous()

    med = {"vp": vp, "eps": per_layer(0.0, 0.3), "delta": per_layer(-0.1, 0.2)}
    if c["op"] == "tti":
        med["vs"] = 0.5 * vp
        med["alpha"] = torch.ones(n, device=DEV)
        med["theta"] = (per_layer(0.0, math.pi / 4) + math.radians(10.0) * _smooth(g, n)).contiguous()
        med["phi"] = (float(rs.uniform(-math.pi, math.pi)) + math.radians(30.0) * _smooth(g, n)).contiguous()
    src, rec_z = _survey(c, rs)
    dt = float(np.float32(CFL * H / (4500.0 * 1.05 * math.sqrt(1.6))))
    fields = [_uniform(g, (c["shots"],) + n, -1.0, 1.0) for _ in range(4)]
    return med, src, rec_z, dt, torch.full((c["shots"],), 0.5, device=DEV), fields


def _padded(c, interior):
    f = mms.padded_empty(c["nx"], c["ny"], c["nz"], R, nshots=c["shots"])
    f[:, R:-R, R:-R, R:-R] = interior
    return f


# ------------------------------------------------------------ prepare, run

def prepare(case, seed):
    c = case
    if c["op"] == "sweep":
        w, grid = _sweep_inputs(c, seed)
        if c["layout"] == "pitched":
            r = c["r"]
            if c["shape"].endswith("2d"):
                inp = mms.padded_empty2d(c["nx"], c["ny"], c["nz"], r, zero=False)
            else:
                inp = mms.padded_empty(c["nx"], c["ny"], c["nz"], r, dtype=grid.dtype, zero=False)
            inp.copy_(grid)
            grid = inp
        out = torch.empty((c["nz"], c["ny"], c["nx"]), device=DEV, dtype=grid.dtype)
        return {"case": c, "w": w, "inp": grid, "out": out}
    if c["op"] in ("forward", "gradient"):
        v, src, rec_z, dt, amps, obs = _wave_inputs(c, seed)
        prop = WavePropagator(c["nx"], c["ny"], c["nz"], src, rec_z, H, dt, SPONGE, SPONGE_A)
        return {"case": c, "prop": prop, "v": v.requires_grad_(c["op"] == "gradient"), "amps": amps, "obs": obs}
    med, src, rec_z, dt, amp, fields = _aniso_inputs(c, seed)
    n = (c["nx"], c["ny"], c["nz"])
    f = [_padded(c, x) for x in fields] + [mms.padded_empty(*n, R, nshots=c["shots"]) for _ in range(2)]
    py, pz, ss = mms.field_geometry(f[0])
    desc, keep = mms.wave_desc(*n, R, c["shots"], py, pz, ss, SPONGE, SPONGE_A, rec_z, src)
    s = {"case": c, "f": f, "desc": desc, "keep": keep, "amp": amp,
         "rec": torch.empty((c["shots"], c["ny"], c["nx"]), device=DEV)}
    if c["op"] == "vti":
        s["mv"], s["rho"] = mms.padded_empty(*n, R), mms.padded_empty(*n, R)
        mms.vti_model(desc, med["vp"], med["eps"], med["delta"], s["mv"], s["rho"], dt, H)
    else:
        s["med"] = torch.empty((8, c["nz"], c["ny"], c["nx"]), device=DEV)
        s["work"] = torch.empty((4, c["shots"], c["nz"], c["ny"], c["nx"]), device=DEV)
        mms.tti_model(desc, *(med[k] for k in ("vp", "vs", "eps", "delta", "alpha", "theta", "phi")), s["med"], dt, H)
    return s


def run(state):
    c = state["case"]
    if c["op"] == "sweep":
        if c["dtype"] == "f64":
            return mms.apply_f64(c["shape"], c["r"], state["w"], state["inp"], state["out"])
        if c["layout"] == "dense":
            return mms.apply_dense(c["shape"], c["r"], state["w"], state["inp"], state["out"])
        return mms.apply(c["shape"], c["r"], state["w"], state["inp"], state["out"])
    if c["op"] == "forward":
        prop = state["prop"]
        rec, _ = prop.forward(state["v"], state["amps"], c["steps"], graph=c["graph"])
        return {"rec": rec, "fields": [prop.p[0], prop.p[1]]}
    if c["op"] == "gradient":
        rec = WaveFunction.apply(state["v"], state["prop"], state["amps"], c["steps"], c["every"])
        grad, = torch.autograd.grad(rec, state["v"], rec.detach() - state["obs"])
        return {"rec": rec.detach(), "grad": grad}
    f = state["f"]
    if c["op"] == "vti":
        mms.vti_step(state["desc"], AXES, state["mv"], state["rho"], *f, state["amp"], state["rec"])
    else:
        mms.tti_step(state["desc"], W2, W1, state["med"], *f, state["work"], state["amp"], state["rec"])
    return {"next": [f[4], f[5]], "rec": state["rec"]}


def work(case):
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    if c["op"] == "sweep":
        r, size = c["r"], 8 if c["dtype"] == "f64" else 4
        rz = 0 if c["shape"].endswith("2d") else r
        padded = (c["nx"] + 2 * r) * (c["ny"] + 2 * r) * (c["nz"] + 2 * rz)
        return {"bytes": size * (padded + n), "flops": 2 * _npts(c["shape"], r) * n}
    s = c["shots"]
    rec = 4 * s * c["nx"] * c["ny"]
    if c["op"] == "forward":   # per step: a^n, a^{n-1} in, a^{n+1} out per shot, m in; records out
        return {"bytes": c["steps"] * ((12 * s + 4) * n + rec), "flops": c["steps"] * s * n * 56}
    if c["op"] == "gradient":
        # forward and recompute (L a^n out too) steps, and adjoint steps with L a^n in
        # and the FP64 gradient in and out
        return {"bytes": c["steps"] * (((12 * s + 4) + (16 * s + 4) + (16 * s + 4 + 16)) * n + 3 * rec),
                "flops": c["steps"] * s * n * 170}
    if c["op"] == "vti":       # two fields at n, n-1 in, at n+1 out per shot; two medium fields in
        return {"bytes": (24 * s + 8) * n + rec, "flops": s * n * 130}
    return {"bytes": (24 * s + 32) * n + rec, "flops": s * n * 300}


# ------------------------------------------------------------------ exact

def _line(f, w, axis, r=R):
    """sum_d w[d] f shifted by d along `axis`: that axis loses its r halo cells on each side."""
    n = f.shape[axis] - 2 * r
    out = torch.zeros_like(f.narrow(axis, r, n))
    for d in range(2 * r + 1):
        if w[d]:
            out.add_(f.narrow(axis, d, n), alpha=float(w[d]))
    return out


def _exact_sweep(c, seed):
    w, grid = _sweep_inputs(c, seed)
    shape, r, k = c["shape"], c["r"], 2 * c["r"] + 1
    grid, w = grid.double(), np.asarray(w, np.float64).reshape(-1)
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    out = torch.zeros((nz, ny, nx), device=DEV, dtype=torch.float64)
    planar = shape.endswith("2d")

    def add(dz, dy, dx, weight):
        z0 = 0 if planar else r + dz
        out.add_(grid[z0:z0 + nz, r + dy:r + dy + ny, r + dx:r + dx + nx], alpha=float(weight))

    offs = range(-r, r + 1)
    if shape.startswith("star"):
        for d in offs:
            add(0, 0, d, w[d + r])
            add(0, d, 0, w[k + d + r])
            if not planar:
                add(d, 0, 0, w[2 * k + d + r])
    else:
        for dz in ([0] if planar else offs):
            for dy in offs:
                for dx in offs:
                    add(dz, dy, dx, w[(((0 if planar else dz + r) * k) + dy + r) * k + dx + r])
    return out


def _damping(c):
    def one(n):
        i = torch.arange(n, device=DEV, dtype=torch.float64)
        d = torch.minimum(i, n - 1 - i)
        t = float(np.float32(SPONGE_A)) * (SPONGE - d)
        return torch.where(d < SPONGE, torch.exp(-t * t), torch.ones_like(t))
    return one(c["nz"])[:, None, None] * one(c["ny"])[None, :, None] * one(c["nx"])[None, None, :]


def _pad(f):
    return torch.nn.functional.pad(f, (R,) * 6)


def _inner(f):
    return f[R:-R, R:-R, R:-R]


def _along(f, axis):
    """The padded field with its halo kept along `axis` only."""
    return f[tuple(slice(None) if a == axis else slice(R, -R) for a in range(3))]


def _lap(f):
    """The three-axis second-derivative star of a padded field, on its interior."""
    return sum(_line(_along(f, a), W2, a) for a in range(3))


def _exact_wave(c, seed):
    v, src, rec_z, dt, amps, obs = _wave_inputs(c, seed)
    v, amps = v.detach().double(), amps.double()
    m, g = v * v * (dt * dt / (H * H)), _damping(c)
    steps = c["steps"]
    recs, last, grad = [], [], torch.zeros_like(m)
    for s in range(c["shots"]):
        x, y, z = (int(k) for k in src[s])
        prev, cur = torch.zeros_like(m), torch.zeros_like(m)
        rec, laps = [], []
        for n in range(steps):
            lap = _lap(_pad(cur))
            if obs is not None:
                laps.append(lap)
            nxt = 2.0 * cur + m * lap - g * prev
            nxt[z, y, x] += amps[n, s]
            prev, cur = cur, nxt.mul_(g)
            rec.append(cur[rec_z].clone())
        recs.append(torch.stack(rec))
        if obs is None:
            # the step buffers alternate, the newest in p[1] after an even count
            last.append((prev, cur) if steps % 2 == 0 else (cur, prev))
            continue
        resid = recs[-1] - obs[:, s].double()
        lam1, lam2 = torch.zeros_like(m), torch.zeros_like(m)   # lam^{n+1}, lam^{n+2}
        for n in range(steps, 0, -1):
            if n < steps:
                grad.add_(g * lam1 * laps[n])
            q = g * lam1
            lam = 2.0 * q + _lap(_pad(m * q)) - g * g * lam2
            lam[rec_z] += resid[n - 1]
            lam1, lam2 = lam, lam1
    rec = torch.stack(recs, 1)
    if obs is not None:
        return {"rec": rec, "grad": grad * 2.0 * v * (dt * dt / (H * H))}
    return {"rec": rec, "fields": [torch.stack([_pad(p[k]) for p in last]) for k in range(2)]}


def _exact_aniso(c, seed):
    med, src, rec_z, dt, amp, fields = _aniso_inputs(c, seed)
    med = {k: t.double() for k, t in med.items()}
    g = _damping(c)
    m = med["vp"] ** 2 * (dt * dt / (H * H))
    fast, root = m * (1.0 + 2.0 * med["eps"]), torch.sqrt(1.0 + 2.0 * med["delta"])
    nxt, rec = ([], []), []
    if c["op"] == "tti":
        ax = (torch.sin(med["theta"]) * torch.cos(med["phi"]), torch.sin(med["theta"]) * torch.sin(med["phi"]),
              torch.cos(med["theta"]))
        vn, vs, al = m * root * root, med["vs"] ** 2 * (dt * dt / (H * H)), med["alpha"]

    def tilted(f):
        """(Laplacian, H1) of a padded field; torch axis 2 - k is the k-th of x, y, z."""
        lap, h1 = 0.0, 0.0
        for i in range(3):
            fii = _line(_along(f, 2 - i), W2, 2 - i)
            lap, h1 = lap + fii, h1 + ax[i] ** 2 * fii
            for j in range(i):
                keep = f[tuple(slice(None) if a in (2 - i, 2 - j) else slice(R, -R) for a in range(3))]
                h1 = h1 + 2.0 * ax[i] * ax[j] * _line(_line(keep, W1, 2 - i), W1, 2 - j)
        return lap, h1

    for s in range(c["shots"]):
        a, b = (_pad(f[s].double()) for f in fields[:2])
        if c["op"] == "vti":
            la, lb = (_line(_along(f, 1), W2, 1) + _line(_along(f, 2), W2, 2) for f in (a, b))
            za, zb = (_line(_along(f, 0), W2, 0) for f in (a, b))
            rhs = (fast * la + m * root * zb, m * root * lb + fast * za)
        else:
            (lp, h1p), (lq, h1q) = tilted(a), tilted(b)
            h2p, h2q = lp - h1p, lq - h1q
            rhs = (fast * h2p + al * m * h1q + vs * (h1p - al * h1q), vn / al * h2p + m * h1q - vs * (h2p / al - h2q))
        x, y, z = (int(k) for k in src[s])
        for k in range(2):
            u = 2.0 * _inner((a, b)[k]) + rhs[k] - g * fields[2 + k][s].double()
            u[z, y, x] += 0.5
            u = u * g
            nxt[k].append(_pad(u))
            if k == 0:
                rec.append(u[rec_z].clone())
    return {"next": [torch.stack(nxt[0]), torch.stack(nxt[1])], "rec": torch.stack(rec)}


def exact(case, seed):
    c = case
    if c["op"] == "sweep":
        return _exact_sweep(c, seed)
    return _exact_wave(c, seed) if c["op"] in ("forward", "gradient") else _exact_aniso(c, seed)
