"""The calls that a user of this framework makes, with the sizes at which they are made.

A case names one path through the public entry points (``paper_1503_01721_gb300.api`` and
``autograd``) and its sizes: voxel grid, control points (CPs), MLC rows and columns, stored
value type, number of apertures.  Sizes come from the repository's own workloads (40^3 with
36 CPs of 20 x 20 beamlets, 128 x 128 x 96 with 180 CPs of 64 x 64, the uneven batch) and
ranges around them.  Inputs are seeded pencil-beam matrices made on the GPU: value
exp(-0.05 depth - rho^2 / 2) in voxel units, dropped below 1% of the unit peak, gantry start
angle, beamlet outputs, structures and vectors drawn from the seed.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1503_01721_gb300 import api, autograd

DEV = "cuda"
LOGCUT = math.log(100.0)  # entries below 1% of a beamlet's peak are dropped
MU = 0.05                 # attenuation per voxel
TRAVEL = 3                # leaf travel, columns per CP step


# ---------------------------------------------------------------------------- the cases

def listed():
    return [
        # pricing of one MLC geometry of a small plan, from given prices: the smallest call
        dict(name="openings_small", path="openings", K=36, arcs=1, n_rows=20, n_cols=20, interdig=False),
        # pricing under the interdigitation constraint at the clinical MLC size, in mid plan
        dict(name="openings_interdig", path="openings", K=180, arcs=1, n_rows=64, n_cols=64, interdig=True),
        # dose(y), objective and their gradient for the apertures of a small plan (a tuning
        # loop's step: short kernels, many launches)
        dict(name="grad_small", path="grad", nx=40, ny=40, nz=40, K=36, arcs=1, n_rows=20, n_cols=20,
             dtype="f32", brick=True, n_ap=20),
        # the same for 60 apertures on the full-size single-arc matrix: one whole D x and one
        # whole D^T g pass over 9.7e8 nonzeros
        dict(name="grad_large", path="grad", nx=128, ny=128, nz=96, K=180, arcs=1, n_rows=64, n_cols=64,
             dtype="f32", brick=True, n_ap=60),
        # beamlet prices inside the leaf-travel windows of a half-made two-arc plan, BF16 storage
        dict(name="price_win_bf16", path="price_win", nx=128, ny=128, nz=96, K=180, arcs=2, n_rows=64, n_cols=64,
             dtype="bf16", brick=True),
        # beamlet prices of the unoccupied CPs, FP8 storage, odd grid and MLC sizes
        dict(name="price_fp8_odd", path="price", nx=101, ny=93, nz=77, K=121, arcs=1, n_rows=53, n_cols=37,
             dtype="fp8", brick=True),
        # forward dose, BF16 storage, voxel order, a mid-size plan
        dict(name="dose_bf16", path="dose", nx=112, ny=112, nz=84, K=120, arcs=1, n_rows=56, n_cols=40,
             dtype="bf16", brick=False),
        # one master problem from the user's own dose columns (zero start, default stopping rules)
        dict(name="master_mid", path="master", nx=88, ny=80, nz=60, n_ap=40),
        # a new patient's matrix: load the COO, build both orientations, the first two products
        dict(name="build_f32", path="build", nx=96, ny=96, nz=72, K=90, arcs=1, n_rows=48, n_cols=48,
             dtype="f32", brick=True),
        # whole plans, small and full size
        dict(name="plan_small", path="plan", nx=40, ny=40, nz=40, K=36, arcs=1, n_rows=20, n_cols=20,
             dtype="f32", brick=True, n_ap=20, limits=False),
        dict(name="plan_large", path="plan", nx=128, ny=128, nz=96, K=180, arcs=1, n_rows=64, n_cols=64,
             dtype="f32", brick=True, n_ap=60, limits=False),
        # four plans of uneven size advanced together (one graph launch), their first apertures with
        # converged master problems (the batch shares its CTAs out again as plans finish, so its
        # sums differ in the last bits from run to run; long plans would part after near ties)
        dict(name="batch_bf16", path="batch", n_plans=4, nx=80, ny=80, nz=60, K=45, arcs=1, n_rows=40, n_cols=32,
             dtype="bf16", brick=True, n_ap=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same paths, sizes over their whole range, odd ones among them."""
    path = rng.choice(["openings", "openings", "grad", "price_win", "price", "dose", "master", "build", "plan", "plan",
                       "batch"])
    if path == "openings":
        interdig = rng.random() < 0.4
        return dict(path=path, K=_log_int(rng, 20, 360), arcs=rng.choice([1, 1, 2]), n_rows=_log_int(rng, 12, 80),
                    n_cols=_log_int(rng, 12, 64 if interdig else 96), interdig=interdig)
    if path == "master":
        return dict(path=path, nx=_log_int(rng, 24, 112), ny=_log_int(rng, 24, 112), nz=_log_int(rng, 20, 84),
                    n_ap=_log_int(rng, 4, 72))
    big = 0.5 if path in ("batch", "build") else 1.0
    nx, ny, nz = _log_int(rng, 24, 128), _log_int(rng, 24, 128), _log_int(rng, 20, 96)
    c = dict(path=path, nx=nx, ny=ny, nz=nz, K=_log_int(rng, 24, 180 * big), arcs=rng.choice([1, 1, 2]),
             n_rows=_log_int(rng, 12, min(64, nz)), n_cols=_log_int(rng, 12, min(64, nx, ny)),
             dtype=rng.choice(["f32", "f32", "bf16", "fp8"]), brick=rng.random() < 0.75)
    if path in ("grad", "plan", "batch"):
        c["n_ap"] = min(_log_int(rng, 4, 60) if path != "batch" else rng.randint(3, 8), c["K"])
    if path == "plan":
        c["limits"] = rng.random() < 0.25
    if path == "batch":
        c["n_plans"] = rng.randint(2, 5)
    return c


# ---------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7fffffff)
    return g


def _mlc(c, K=None):
    K = c["K"] if K is None else K
    arcs = min(c["arcs"], K)
    first = np.array([a * (K // arcs) for a in range(arcs)], np.int32)
    return SimpleNamespace(K=K, n_rows=c["n_rows"], n_cols=c["n_cols"], arc_first_cp=first, travel_cols=TRAVEL,
                           interdigitation=bool(c.get("interdig", False)), machine=None)


def _machine(mlc):
    """Delivery limits whose travel window is reachable at the slowest gantry speed."""
    step = 360.0 * len(mlc.arc_first_cp) / mlc.K
    return SimpleNamespace(cp_step_deg=step, speed_min=0.5, speed_max=4.0, speed_step_max=0.5, rate_min=0.02,
                           rate_max=0.025, leaf_speed_cols=1.25 * TRAVEL * 0.5 / step)


def _angles(mlc, phase):
    first = list(mlc.arc_first_cp) + [mlc.K]
    out = []
    for a in range(len(mlc.arc_first_cp)):
        n = int(first[a + 1] - first[a])
        out += [phase + 2 * math.pi * i / n + a * math.pi / 180 for i in range(n)]
    return out


def pencil_beams(nx, ny, nz, mlc, seed):
    """COO of the pencil-beam matrix on the GPU: voxel, beamlet (int32) and value (float32),
    beamlet by beamlet, voxels ascending within a beamlet (as a dose engine writes columns)."""
    g = _gen(seed)
    V, nr, nc = nx * ny * nz, mlc.n_rows, mlc.n_cols
    phase = float(torch.rand((), generator=g, device=DEV)) * 2 * math.pi
    gain = 0.8 + 0.4 * torch.rand(mlc.K * nr * nc, generator=g, device=DEV)
    px = torch.arange(nx, device=DEV, dtype=torch.float32).repeat(ny) - (nx - 1) / 2
    py = torch.arange(ny, device=DEV, dtype=torch.float32).repeat_interleave(nx) - (ny - 1) / 2
    pz = torch.arange(nz, device=DEV, dtype=torch.float32) - (nz - 1) / 2
    # (z, MLC row) pairs within the lateral reach
    dz = pz[:, None] - (torch.arange(nr, device=DEV, dtype=torch.float32) - (nr - 1) / 2)[None, :]
    zi, ri = torch.nonzero(dz * dz / 2 <= LOGCUT, as_tuple=True)
    qz = (dz * dz / 2)[zi, ri]
    col = torch.arange(nc, device=DEV, dtype=torch.float32) - (nc - 1) / 2
    vox, blt, val = [], [], []
    for k, th in enumerate(_angles(mlc, phase)):
        ct, st = math.cos(th), math.sin(th)
        t, u = px * ct + py * st, py * ct - px * st
        # where each column's axis enters and leaves the grid box
        t0 = torch.full((nc,), -1e30, device=DEV)
        t1 = torch.full((nc,), 1e30, device=DEV)
        for o, d, h in ((-st * col, ct, nx / 2), (ct * col, st, ny / 2)):
            if abs(d) > 1e-9:
                a, b = (-h - o) / d, (h - o) / d
                t0, t1 = torch.maximum(t0, torch.minimum(a, b)), torch.minimum(t1, torch.maximum(a, b))
            else:
                t1 = torch.where(o.abs() > h, torch.full_like(t1, -1e30), t1)
        c0 = torch.round(u + (nc - 1) / 2).to(torch.int64)
        cc = c0[:, None] + torch.arange(-3, 4, device=DEV)
        ok = (cc >= 0) & (cc < nc)
        cc = cc.clamp(0, nc - 1)
        depth = t[:, None] - t0[cc]
        du = u[:, None] - col[cc]
        q = MU * depth + du * du / 2
        ok &= (depth >= 0) & (q <= LOGCUT) & (t0 < t1)[cc]
        pi_, ci = torch.nonzero(ok, as_tuple=True)
        qa, ca = q[pi_, ci], cc[pi_, ci]
        qq = qa[:, None] + qz[None, :]
        ia, ib = torch.nonzero(qq <= LOGCUT, as_tuple=True)
        b = ri[ib] * nc + ca[ia]
        key, order = torch.sort(b * V + zi[ib] * (nx * ny) + pi_[ia])
        b = torch.div(key, V, rounding_mode="floor")
        vox.append((key - b * V).to(torch.int32))
        b = (b + k * nr * nc).to(torch.int32)
        blt.append(b)
        val.append(torch.exp(-qq[ia, ib])[order] * gain[b])
    return torch.cat(vox), torch.cat(blt), torch.cat(val)


def _structures(nx, ny, nz, seed):
    """Labels and dose parameters: tissue (overdose only), OARs, targets (both sides)."""
    r = np.random.default_rng([int(seed), 7])
    n = np.array([nx, ny, nz], float)
    x = torch.arange(nx, device=DEV)[None, None, :] - (nx - 1) / 2
    y = torch.arange(ny, device=DEV)[None, :, None] - (ny - 1) / 2
    z = torch.arange(nz, device=DEV)[:, None, None] - (nz - 1) / 2
    sid = torch.zeros((nz, ny, nx), dtype=torch.uint8, device=DEV)
    T, wo, wu = [0.6], [0.05], [0.0]
    rows = [(r.uniform(-0.2, 0.2, 3) * n, r.uniform(0.05, 0.09, 3) * n, 0.5, 0.3, 0.0) for _ in range(4)]
    rows += [(r.uniform(-0.08, 0.08, 3) * n, r.uniform(0.07, 0.12, 3) * n, rx, 1.0, 1.0) for rx in (0.8, 0.9, 1.0)]
    for ctr, ax, t, o, u in rows:
        ax = np.maximum(ax, 1.5)
        sid[((x - ctr[0]) / ax[0]) ** 2 + ((y - ctr[1]) / ax[1]) ** 2 + ((z - ctr[2]) / ax[2]) ** 2 <= 1] = len(T)
        T.append(t), wo.append(o), wu.append(u)
    f = lambda a: torch.tensor(a, dtype=torch.float32, device=DEV)  # noqa: E731
    return sid.reshape(-1), f(T), f(wo), f(wu)


def _apertures(mlc, n, seed):
    """Random open apertures: CPs with repetition, every leaf row one interval."""
    r = np.random.default_rng([int(seed), 11])
    hi = min(40, mlc.n_cols)
    ln = r.integers(min(4, hi), hi + 1, size=(n, mlc.n_rows))
    st = (r.random((n, mlc.n_rows)) * (mlc.n_cols - ln + 1)).astype(np.int64)
    return (r.integers(0, mlc.K, n).astype(np.int32), np.stack([st, st + ln], -1).astype(np.int16),
            r.random(n).astype(np.float32))


def _mid_plan(mlc, seed):
    """State of a half-made plan: every third CP or so occupied, its leaves around the target's
    projection (within the leaf travel of its neighbours)."""
    r = np.random.default_rng([int(seed), 13])
    occ = (r.random(mlc.K) < 0.35).astype(np.uint8)
    rows = np.arange(mlc.n_rows)
    half = np.sqrt(np.clip(1 - ((rows - (mlc.n_rows - 1) / 2) / (0.45 * mlc.n_rows)) ** 2, 0, 1)) * 0.3 * mlc.n_cols
    mid = mlc.n_cols * (0.5 + 0.05 * r.uniform(-1, 1))
    lv = np.stack([np.round(mid - half), np.round(mid + half)], -1)[None] + r.integers(-1, 2, (mlc.K, mlc.n_rows, 2))
    lv = np.clip(np.sort(lv, -1), 0, mlc.n_cols).astype(np.int16)
    return torch.from_numpy(occ).to(DEV), torch.from_numpy(lv).to(DEV)


def _prices(mlc, seed):
    """Beamlet prices of a half-made plan: positive over the underdosed target, negative outside."""
    g = _gen(seed * 5 + 3)
    r = (torch.arange(mlc.n_rows, device=DEV) - (mlc.n_rows - 1) / 2) / (0.35 * mlc.n_rows)
    c = (torch.arange(mlc.n_cols, device=DEV) - (mlc.n_cols - 1) / 2) / (0.3 * mlc.n_cols)
    b = torch.exp(-(r[:, None] ** 2 + c[None, :] ** 2)) - 0.45
    amp = 5 + 10 * torch.rand((mlc.K, 1, 1), generator=g, device=DEV)
    return (amp * b[None] + 1.5 * torch.randn((mlc.K, mlc.n_rows, mlc.n_cols), generator=g, device=DEV)).reshape(-1)


def _vector(n, seed, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=_gen(seed), device=DEV)


def _dose_columns(nx, ny, nz, n, seed):
    """Aperture dose vectors of n beams around the patient (float32 [n, V]), zero off the beam."""
    r = np.random.default_rng([int(seed), 17])
    x = torch.arange(nx, device=DEV)[None, None, :] - (nx - 1) / 2
    y = torch.arange(ny, device=DEV)[None, :, None] - (ny - 1) / 2
    z = torch.arange(nz, device=DEV)[:, None, None] - (nz - 1) / 2
    out = torch.empty((n, nx * ny * nz), device=DEV)
    R = 0.5 * max(nx, ny)
    for i in range(n):
        th = 2 * math.pi * (i + r.uniform(0, 1)) / n
        ct, st = math.cos(th), math.sin(th)
        t, u = x * ct + y * st, y * ct - x * st - r.uniform(-0.05, 0.05) * R
        w, h = r.uniform(0.1, 0.22) * min(nx, ny), r.uniform(0.1, 0.22) * nz
        d = torch.exp(-MU * 0.5 * (t + R)) * torch.sigmoid(2 * (w - u.abs())) * torch.sigmoid(2 * (h - z.abs()))
        out[i] = torch.where(d < 1e-3, torch.zeros_like(d), d).reshape(-1)
    return out


def _plan_shapes(c):
    """The plans of a batch: the case's sizes, shrunk plan by plan."""
    out = []
    for p in range(c["n_plans"]):
        f = 1.0 - 0.12 * p
        s = dict(c, nx=max(16, int(c["nx"] * f)), ny=max(16, int(c["ny"] * f)), nz=max(16, int(c["nz"] * f)),
                 K=max(c["n_ap"], int(c["K"] * (1.0 - 0.1 * p))))
        s["n_rows"], s["n_cols"] = min(s["n_rows"], s["nz"]), min(s["n_cols"], s["nx"], s["ny"])
        out.append(s)
    return out


def _matrix(c, seed, mlc):
    """The built handle a program keeps: both orientations, SpMV configurations tuned."""
    vox, blt, val = pencil_beams(c["nx"], c["ny"], c["nz"], mlc, seed)
    V, J = c["nx"] * c["ny"] * c["nz"], mlc.K * mlc.n_rows * mlc.n_cols
    return api.Ddc(V, J, vox, blt, val, dtype=c["dtype"], autotune=True,
                   vox_grid=(c["nx"], c["ny"], c["nz"]) if c["brick"] else None)


# ---------------------------------------------------------------------------- prepare and run

def prepare(c, seed):
    s = SimpleNamespace(path=c["path"], c=c)
    path = c["path"]
    if path == "openings":
        s.mlc = _mlc(c)
        s.occ, s.leaves = _mid_plan(s.mlc, seed)
        s.pi = _prices(s.mlc, seed)
        s.cp = torch.empty(1, dtype=torch.int32, device=DEV)
        s.lv = torch.empty(2 * s.mlc.n_rows, dtype=torch.int16, device=DEV)
        s.price = torch.empty(1, dtype=torch.float64, device=DEV)
        return s
    if path == "master":
        s.DA = _dose_columns(c["nx"], c["ny"], c["nz"], c["n_ap"], seed)
        s.vox = api.VoxelParams(*_structures(c["nx"], c["ny"], c["nz"], seed))
        s.y = torch.empty(c["n_ap"], device=DEV)
        s.z = torch.empty(s.DA.shape[1], device=DEV)
        return s
    if path == "batch":
        s.plans, s.ddcs = [], []
        for p, q in enumerate(_plan_shapes(c)):
            mlc = _mlc(q)
            s.ddcs.append(_matrix(q, seed * 8 + p, mlc))
            s.plans.append((s.ddcs[-1].h, mlc, api.VoxelParams(*_structures(q["nx"], q["ny"], q["nz"], seed * 8 + p)),
                            c["n_ap"]))
        s.batch = api.Batch(s.plans, api.BBOptions(max_iter=500, rel_tol5=1e-9, step_tol=1e-9))
        s.out = [(torch.empty(c["n_ap"], dtype=torch.int32, device=DEV),
                  torch.empty(c["n_ap"] * q["n_rows"] * 2, dtype=torch.int16, device=DEV),
                  torch.empty(c["n_ap"], device=DEV), torch.empty(q["nx"] * q["ny"] * q["nz"], device=DEV))
                 for q in _plan_shapes(c)]
        return s
    s.mlc = _mlc(c)
    V, J = c["nx"] * c["ny"] * c["nz"], s.mlc.K * s.mlc.n_rows * s.mlc.n_cols
    if path == "build":
        s.coo = pencil_beams(c["nx"], c["ny"], c["nz"], s.mlc, seed)
    else:
        s.ddc = _matrix(c, seed, s.mlc)
    if path in ("price", "price_win", "build"):
        s.g = _vector(V, seed + 1, -1.0, 1.0)
        s.pi = torch.zeros(J, device=DEV)
    if path in ("dose", "build"):
        s.x = _vector(J, seed + 2, 0.0, 1.0)
        s.d = torch.empty(V, device=DEV)
    if path == "price":
        s.active = 1 - _mid_plan(s.mlc, seed)[0]
    if path == "price_win":
        s.occ, s.leaves = _mid_plan(s.mlc, seed)
    if path in ("grad", "plan"):
        s.vox = api.VoxelParams(*_structures(c["nx"], c["ny"], c["nz"], seed))
    if path == "grad":
        cps, lv, y = _apertures(s.mlc, c["n_ap"], seed)
        s.dose = autograd.ApertureDose(s.ddc, s.mlc, torch.from_numpy(cps).to(DEV), torch.from_numpy(lv).to(DEV))
        s.y = (0.1 * torch.from_numpy(y)).to(DEV)
    if path == "plan":
        if c["limits"]:
            s.mlc.machine = _machine(s.mlc)
        s.cps = torch.empty(c["n_ap"], dtype=torch.int32, device=DEV)
        s.lv = torch.empty(c["n_ap"] * s.mlc.n_rows * 2, dtype=torch.int16, device=DEV)
        s.y = torch.empty(c["n_ap"], device=DEV)
        s.d = torch.empty(V, device=DEV)
    return s


def run(s):
    path = s.path
    if path == "openings":
        api.price_apertures(s.mlc, s.pi, s.occ, s.leaves, s.cp, s.lv, s.price)
        return {"cp": s.cp, "leaves": s.lv, "price": s.price}
    if path == "grad":
        y = s.y.clone().requires_grad_(True)
        d = s.dose(y)
        F = autograd.objective(d, s.vox)
        F.backward()
        return {"F": F, "dose": d, "gy": y.grad}
    if path == "price":
        api.beamlet_price(s.ddc.h, s.g, s.pi, s.active, s.mlc.n_rows * s.mlc.n_cols)
        # entries of the occupied CPs are not written: they keep the zeros of prepare()
        return {"pi": s.pi}
    if path == "price_win":
        api.beamlet_price_windowed(s.ddc.h, s.mlc, s.occ, s.leaves, s.g, s.pi)
        return {"pi": s.pi}
    if path == "dose":
        api.dose_forward(s.ddc.h, s.x, s.d)
        return {"dose": s.d}
    if path == "master":
        s.y.zero_()
        r = api.mp_bb_solve(s.DA, s.vox, s.y, s.z)
        return {"y": s.y, "z": s.z, "F": r["F"]}
    if path == "build":
        c = s.c
        ddc = api.Ddc(s.d.numel(), s.pi.numel(), *s.coo, dtype=c["dtype"],
                      vox_grid=(c["nx"], c["ny"], c["nz"]) if c["brick"] else None)
        api.beamlet_price(ddc.h, s.g, s.pi)
        api.dose_forward(ddc.h, s.x, s.d)
        ddc.close()
        return {"pi": s.pi, "dose": s.d}
    if path == "plan":
        F, _ = api.cg_plan(s.ddc.h, s.mlc, s.vox, s.c["n_ap"], None, s.cps, s.lv, s.y, s.d)
        return {"F": F, "cps": s.cps, "leaves": s.lv, "y": s.y, "dose": s.d}
    F, _ = s.batch.run()
    for i, o in enumerate(s.out):
        s.batch.result(i, *o)
    return {"F": list(F), "plans": s.out}


# ---------------------------------------------------------------------------- work

def _nnz(c):
    """Expected nonzeros: a beamlet's depth profile over its mean path, inside the lateral reach."""
    t = min(LOGCUT / MU, 1.1 * math.sqrt(c["nx"] * c["ny"]))
    return c["K"] * c["n_rows"] * c["n_cols"] * 2 * math.pi * (LOGCUT * t - MU * t * t / 2)


# Bytes of a nonzero: the value, and one byte of index (sorted indices of a local pattern need
# no more).
def _pass(c, share=1.0):
    vb = {"f32": 4, "bf16": 2, "fp8": 1}[c["dtype"]]
    nnz = share * _nnz(c)
    dense = 4 * (c["nx"] * c["ny"] * c["nz"] + share * c["K"] * c["n_rows"] * c["n_cols"])
    return nnz * (vb + 1) + dense, 2 * nnz


def work(c):
    path = c["path"]
    if path == "openings":
        rows = c["K"] * c["n_rows"] * 0.65  # the unoccupied CPs
        n = c["n_cols"]
        return {"bytes": rows * 4 * n + 20, "flops": rows * (n * n / 2 + n) * (2 if c["interdig"] else 1)}
    if path == "master":
        # about 60 iterations; the columns once (they fit on chip between iterations), 40% nonzero
        V, n = c["nx"] * c["ny"] * c["nz"], c["n_ap"]
        return {"bytes": 4.0 * n * V + 9.0 * V, "flops": 60 * 0.4 * 4.0 * n * V}
    if path == "batch":
        w = [work(dict(q, path="plan")) for q in _plan_shapes(c)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    if path == "plan":
        # each aperture: a price pass inside the windows (about half of the rows), one CP's
        # columns, and a master problem of about 20 iterations over the reached voxels
        b, f = _pass(c, 0.53)
        V, n = c["nx"] * c["ny"] * c["nz"], c["n_ap"]
        one, fl = _pass(c)
        return {"bytes": n * (b + _nnz(c) / c["K"] * 6) + one + 0.2 * 4.0 * V * n * n / 2,
                "flops": n * f + fl + 20 * 0.2 * 4.0 * V * n * n / 2}
    b, f = _pass(c, {"price": 0.65, "price_win": 0.4}.get(path, 1.0))
    if path in ("grad", "build"):
        b, f = 2 * b, 2 * f
    if path == "build":
        b += 12 * _nnz(c) + 2 * _pass(c)[0]  # the COO in, both matrices out
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------- 64-bit results

def _scales(val, blt, J):
    """E4M3 storage: s_j, the least power of two with 448 s_j >= the largest value of beamlet j."""
    m = torch.zeros(J, device=DEV).scatter_reduce_(0, blt.long(), val.abs(), "amax").double()
    return torch.where(m > 0, torch.exp2(torch.ceil(torch.log2(m / 448))), torch.ones_like(m))


def _products(coo, V, J, dtype, x=None, g=None, chunk=1 << 26):
    """D x and D^T g of the stored values in 64 bits (BF16: rounded; FP8: E4M3 codes times s_j)."""
    vox, blt, val = coo
    d = torch.zeros(V, dtype=torch.float64, device=DEV) if x is not None else None
    pi = torch.zeros(J, dtype=torch.float64, device=DEV) if g is not None else None
    s = _scales(val, blt, J) if dtype == "fp8" else None
    for a in range(0, val.numel(), chunk):
        i, k, v = vox[a:a + chunk].long(), blt[a:a + chunk].long(), val[a:a + chunk].double()
        if dtype == "bf16":
            v = v.to(torch.bfloat16).double()
        elif dtype == "fp8":
            v = (v / s[k]).float().to(torch.float8_e4m3fn).double() * s[k]
        if d is not None:
            d.index_add_(0, i, v * x.double()[k])
        if pi is not None:
            pi.index_add_(0, k, v * g.double()[i])
    return d, pi


def _windows(mlc, occ, leaves):
    """[Lmin, Lmax, Rmin, Rmax] of every (CP, row) from the nearest occupied CP on each side of
    the arc, and which CPs are free (numpy)."""
    K, N = mlc.K, mlc.n_cols
    w = np.zeros((K, mlc.n_rows, 4), np.int64)
    w[..., 1] = w[..., 3] = N
    first = list(mlc.arc_first_cp) + [K]
    for a in range(len(mlc.arc_first_cp)):
        lo, hi = int(first[a]), int(first[a + 1])
        placed = [k for k in range(lo, hi) if occ[k]]
        for k in range(lo, hi):
            near = [max([q for q in placed if q < k], default=None), min([q for q in placed if q > k], default=None)]
            for q in near:
                if q is None:
                    continue
                m = abs(k - q) * mlc.travel_cols
                L, R = leaves[q, :, 0].astype(np.int64), leaves[q, :, 1].astype(np.int64)
                w[k, :, 0] = np.maximum(w[k, :, 0], L - m)
                w[k, :, 1] = np.minimum(w[k, :, 1], L + m)
                w[k, :, 2] = np.maximum(w[k, :, 2], R - m)
                w[k, :, 3] = np.minimum(w[k, :, 3], R + m)
    return w


def _best_price(mlc, pi, occ, w):
    """The best aperture's price in 64 bits: rows alone, or as a chain under interdigitation."""
    N, best = mlc.n_cols, -np.inf
    Lg, Rg = np.meshgrid(np.arange(N + 1), np.arange(N + 1), indexing="ij")
    for k in range(mlc.K):
        if occ[k]:
            continue
        P = np.concatenate([np.zeros((mlc.n_rows, 1)), np.cumsum(pi[k], 1)], 1)
        S = None
        tot = 0.0
        for r in range(mlc.n_rows):
            a, b, c, d = w[k, r]
            v = np.where((Lg >= a) & (Lg <= b) & (Rg >= c) & (Rg <= d) & (Lg <= Rg), P[r][None, :] - P[r][:, None], -np.inf)
            if not mlc.interdigitation:
                tot += v.max()
                continue
            if S is not None:  # the previous row's best (L', R') with L' <= R and R' >= L
                M = np.maximum.accumulate(S, 0)
                M = np.maximum.accumulate(M[:, ::-1], 1)[:, ::-1]
                v = v + M[Rg, Lg]
            S = v
        best = max(best, S.max() if mlc.interdigitation else tot)
    return best


def exact(c, seed):
    """What run() returns, from the same inputs in 64-bit torch or numpy.  A plan or a master
    problem has none: its iterates depend on every rounding before them."""
    path = c["path"]
    if path in ("plan", "batch", "master"):
        return None
    mlc = _mlc(c)
    if path == "openings":
        occ, leaves = (t.cpu().numpy() for t in _mid_plan(mlc, seed))
        pi = _prices(mlc, seed).double().cpu().numpy().reshape(mlc.K, mlc.n_rows, mlc.n_cols)
        p = _best_price(mlc, pi, occ, _windows(mlc, occ, leaves))
        return {"cp": None, "leaves": None, "price": torch.tensor([p], dtype=torch.float64)}
    V, J = c["nx"] * c["ny"] * c["nz"], mlc.K * mlc.n_rows * mlc.n_cols
    coo = pencil_beams(c["nx"], c["ny"], c["nz"], mlc, seed)
    if path == "dose":
        return {"dose": _products(coo, V, J, c["dtype"], x=_vector(J, seed + 2, 0.0, 1.0))[0]}
    if path in ("price", "price_win", "build"):
        x = _vector(J, seed + 2, 0.0, 1.0) if path == "build" else None
        d, pi = _products(coo, V, J, c["dtype"], x=x, g=_vector(V, seed + 1, -1.0, 1.0))
        if path == "build":
            return {"pi": pi, "dose": d}
        occ, leaves = _mid_plan(mlc, seed)
        if path == "price":
            pi = pi.view(mlc.K, -1) * (1 - occ.double())[:, None]
            return {"pi": pi.reshape(-1)}
        o = occ.cpu().numpy()
        w = _windows(mlc, o, leaves.cpu().numpy())
        col = np.arange(mlc.n_cols)
        keep = (col >= w[..., :1]) & (col < np.maximum(w[..., :1], w[..., 3:])) & (o == 0)[:, None, None]
        return {"pi": pi * torch.from_numpy(keep.reshape(-1)).to(DEV)}
    # grad: x = A y, d = D x, F(d), gy = A^T D^T F'(d)
    cps, lv, y = _apertures(mlc, c["n_ap"], seed)
    y = (0.1 * torch.from_numpy(y)).double().numpy()
    x = np.zeros((mlc.K, mlc.n_rows, mlc.n_cols))
    col = np.arange(mlc.n_cols)
    masks = [(col >= lv[i, :, :1]) & (col < lv[i, :, 1:]) for i in range(c["n_ap"])]
    for i, m in enumerate(masks):
        x[cps[i]] += y[i] * m
    d, _ = _products(coo, V, J, c["dtype"], x=torch.from_numpy(x.reshape(-1)).to(DEV))
    sid, T, wo, wu = _structures(c["nx"], c["ny"], c["nz"], seed)
    sid, T, wo, wu = sid.long(), T.double(), wo.double(), wu.double()
    e = d - T[sid]
    wgt = torch.where(e > 0, wo[sid], wu[sid])
    _, pi = _products(coo, V, J, c["dtype"], g=2 * wgt * e)
    pi = pi.view(mlc.K, mlc.n_rows, mlc.n_cols).cpu().numpy()
    gy = torch.tensor([float((pi[cps[i]] * m).sum()) for i, m in enumerate(masks)], dtype=torch.float64)
    return {"F": (wgt * e * e).sum(), "dose": d, "gy": gy}
