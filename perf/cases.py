"""Performance cases of the advection library: the work a user has it do,
through its public entry points, with the inputs they have in hand.

A case is a dict of plain values with a ``kind``:

  step     one field, one grid, one scheme: ``advect`` (an SL_CEC pass is a step
           of each sweep order, x,y,z then z,y,x, as a time loop alternates them)
  multi    several fields carried by one velocity: ``sl_advect_multi``
  batch    a plan of independent grids of uneven sizes: ``sl_batch_step``
  wide     Courant numbers above one: ``advect_wide``
  learned  the learned one-pass corrector: ``sl_advect_learned``
  rb       a run of the Rayleigh-Benard box: ``sl_rb_set_state/step/get_state``

``exact`` evaluates the same steps from the schemes' definitions in float64
torch, on the inputs the library gets.
"""
import math

import numpy as np
import torch

from paper_1606_06117_gb300 import _lib as sl
from paper_1606_06117_gb300 import workloads as W

DEV = "cuda"
DTYPES = {"f32": torch.float32, "f64": torch.float64, "f32_d64": torch.float32}
CODES = {"f32": sl.F32, "f64": sl.F64, "f32_d64": sl.F32_D64}


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # a scalar carried round the unit square: the smallest grid of the
        # tests and the benchmark, where a launch's latency counts
        dict(name="rot128_cec_f64", kind="step", flow="rotation", scheme="CEC", dtype="f64", nx=128, ny=128, nz=0,
             cfl=0.5),
        # the first-order scheme on the ABC workload
        dict(name="abc256_cir_f32", kind="step", flow="abc", scheme="CIR", dtype="f32", nx=256, ny=256, nz=256,
             cfl=0.8),
        # forward error correction on the same workload
        dict(name="abc256_fec_f32", kind="step", flow="abc", scheme="FEC", dtype="f32", nx=256, ny=256, nz=256,
             cfl=0.8),
        # backward error correction at the large size
        dict(name="abc512_bec_f32", kind="step", flow="abc", scheme="BEC", dtype="f32", nx=512, ny=512, nz=512,
             cfl=0.8),
        # the third-order scheme at the size the throughput is quoted for
        dict(name="abc512_cec_f32", kind="step", flow="abc", scheme="CEC", dtype="f32", nx=512, ny=512, nz=512,
             cfl=0.8),
        # an ordinary grid whose sides are no multiple of anything
        dict(name="ragged_cec_f32", kind="step", flow="abc", scheme="CEC", dtype="f32", nx=187, ny=150, nz=131,
             cfl=0.8),
        # the double-precision cross-check of a single-precision run
        dict(name="abc256_cec_f64", kind="step", flow="abc", scheme="CEC", dtype="f64", nx=256, ny=256, nz=256,
             cfl=0.8),
        # three velocity components and a scalar in the deformation flow
        dict(name="deform512_cec_x4", kind="multi", scheme="CEC", fields=4, nx=512, ny=512, nz=512, cfl=0.8),
        # 48 independent grids of 64^3 to 192^3 in one launch per step
        dict(name="batch48_cec_f32", kind="batch", count=48, grids=0),
        # steps of several cells: 22 of them in place of 100 at CFL 0.8
        dict(name="wide256_cec_f32", kind="wide", scheme="CEC", dtype="f32", nx=256, ny=256, nz=256, cfl=3.64),
        # the learned corrector at its evaluation size
        dict(name="learned256", kind="learned", nx=256, ny=256, nz=256, cfl=0.8),
        # the convection box of 50 x 50 cells, 64 steps of a run
        dict(name="rb50_cec_f64", kind="rb", scheme="CEC", dtype="f64", nx=50, nz=50, steps=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi, unit):
    return max(unit, _log(rng, lo, hi) // unit * unit)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step2d", "step64", "multi", "batch", "wide", "learned", "rb"])
    scheme = rng.choice(["CIR", "FEC", "BEC", "CEC", "CEC"])
    if kind == "step":       # single precision in three dimensions, whole tiles, whole vectors or any size
        ux, uy = rng.choice([(32, 32), (4, 1), (1, 1)])
        return dict(kind="step", flow="abc", scheme=scheme, dtype="f32", nx=max(64 if ux == 32 else 0, _side(rng, 24, 400, ux)),
                    ny=_side(rng, 24, 400, uy), nz=_side(rng, 12, 400, 1), cfl=round(rng.uniform(0.3, 0.95), 3))
    if kind == "step2d":     # planes of the rotation and shear studies
        flow = rng.choice(["rotation", "shear"])
        n = _side(rng, 48, 1024, rng.choice([32, 1]))
        return dict(kind="step", flow=flow, scheme=scheme, dtype=rng.choice(["f64", "f32"]), nx=n,
                    ny=_side(rng, 48, 1024, 1), nz=0, cfl=round(rng.uniform(0.3, 0.95), 3))
    if kind == "step64":     # double precision, and single with double differences
        return dict(kind="step", flow="abc", scheme=scheme, dtype=rng.choice(["f64", "f64", "f32_d64"]),
                    nx=_side(rng, 20, 200, rng.choice([32, 1])), ny=_side(rng, 20, 200, 1), nz=_side(rng, 8, 200, 1),
                    cfl=round(rng.uniform(0.3, 0.95), 3))
    if kind == "multi":
        ux = rng.choice([32, 4])
        return dict(kind="multi", scheme=rng.choice(["CEC", "CEC", "BEC"]), fields=rng.randint(2, 4),
                    nx=max(64, _side(rng, 48, 256, ux)), ny=_side(rng, 32, 256, ux), nz=_side(rng, 12, 256, 1),
                    cfl=round(rng.uniform(0.3, 0.95), 3))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 32), grids=rng.randint(1, 1000))
    if kind == "wide":
        return dict(kind="wide", scheme=scheme, dtype=rng.choice(["f32", "f32", "f64"]), nx=_side(rng, 32, 320, rng.choice([32, 1])),
                    ny=_side(rng, 24, 320, 1), nz=_side(rng, 12, 320, 1), cfl=round(rng.uniform(1.2, 4.2), 3))
    if kind == "learned":
        return dict(kind="learned", nx=_side(rng, 32, 256, 32), ny=_side(rng, 16, 256, 4), nz=_side(rng, 8, 256, 1),
                    cfl=round(rng.uniform(0.3, 0.95), 3))
    return dict(kind="rb", scheme=scheme, dtype=rng.choice(["f64", "f64", "f32"]), nx=_side(rng, 16, 128, 1),
                nz=_side(rng, 8, 64, 1), steps=rng.randint(4, 80))


# ------------------------------------------------------------------ their inputs
def _shape(case):
    return ((case["nz"],) if case["nz"] else ()) + (case["ny"], case["nx"])


def _field(shape, length, seed, dtype):
    modes = W.draw_modes(len(shape), 32, 8, seed=seed)
    return W.random_modes(shape, modes, length=length, device=DEV, dtype=dtype)


def _grid(case):
    """Velocity, box length, spacing (x, y, z) and dt of a grid case."""
    shape, t = _shape(case), DTYPES[case.get("dtype", "f32")]
    flow = {"multi": "deformation"}.get(case["kind"], case.get("flow", "abc"))
    make = {"abc": W.abc_velocity, "rotation": W.rotation_velocity, "shear": W.shear_patch_velocity,
            "deformation": W.deformation_velocity}[flow]
    length = W.TWO_PI if flow == "abc" else 1.0
    vel = make(shape, device=DEV, dtype=t)
    spacing = [length / n for n in shape[::-1]]
    top = max(float(vel[d].abs().max()) / spacing[d] for d in range(len(shape)))
    return vel, length, spacing, case["cfl"] / top


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("step", "wide", "multi", "learned"):
        shape, t = _shape(case), DTYPES[case.get("dtype", "f32")]
        st["vel"], length, st["spacing"], st["dt"] = _grid(case)
        if kind == "multi":   # the velocity's components and random-mode scalars
            st["in"] = [f.clone() for f in st["vel"][:case["fields"] - 1]] + [_field(shape, length, seed, t)]
            for k, f in enumerate(st["in"][:-1]):
                f.mul_(1.0 + 0.1 * math.cos(seed + k))   # the flow's phase
            st["mid"] = [torch.empty_like(f) for f in st["in"]]
            st["out"] = [torch.empty_like(f) for f in st["in"]]
            return st
        st["phi"] = _field(shape, length, seed, t)
        st["mid"], st["out"] = torch.empty_like(st["phi"]), torch.empty_like(st["phi"])
        if kind == "wide":
            need = sl.sl_advect_wide_workspace(3, shape[::-1], sl.SCHEMES[case["scheme"]], CODES[case["dtype"]])
            st["work"] = torch.empty(need + 256, dtype=torch.uint8, device=DEV) if need else None
        if kind == "learned":
            st["net"] = _Handle(sl.sl_corrector_create(seed), sl.sl_corrector_destroy)
            st["weights"] = _weights(seed)
            sl.sl_corrector_set_params(st["net"].h, st["weights"])
        return st
    if kind == "batch":
        st["grids"], recs = [], []
        for k, inst in enumerate(W.draw_batch(case["count"], seed=case["grids"])):
            inst.modes_seed = 1000 * seed + k
            a, vel = W.instance_fields(inst, device=DEV)
            b = torch.empty_like(a)
            dx = W.TWO_PI / inst.n
            dt = 0.8 * dx / float(vel.abs().max())
            st["grids"].append((a, b, vel, dx, dt))
            recs.append(sl.Instance(a.data_ptr(), b.data_ptr(), vel.data_ptr(), (inst.n,) * 3, (dx,) * 3, dt))
        st["plan"] = _Handle(sl.sl_batch_create(recs), sl.sl_batch_destroy)
        return st
    # the box: a plume under way, theta spots with noise in a circulation
    nx, nz, t = case["nx"], case["nz"], DTYPES[case["dtype"]]
    rng = np.random.default_rng(seed)
    theta = W.rb_spots(nx, nz) + 0.01 * rng.standard_normal((nz, nx))
    x, z = (np.arange(nx) + 0.5) / nx, (np.arange(nz) + 0.5) / nz
    amp = 20.0 * rng.uniform(0.5, 1.0)
    u = amp * np.outer(np.sin(2 * math.pi * z), np.sin(math.pi * x) ** 2)
    w = -amp * 0.5 * np.outer(np.sin(math.pi * z) ** 2, np.sin(2 * math.pi * x))
    st["start"] = [torch.from_numpy(f).to(device=DEV, dtype=t) for f in (u, w, theta)]
    st["out"] = [torch.empty_like(f) for f in st["start"]]
    st["dt"] = 2e-5 * min(1.0, 50.0 / max(nx, nz)) ** 2
    st["box"] = _Handle(sl.sl_rb_create(nx, nz, scheme=case["scheme"], dtype=CODES[case["dtype"]]), sl.sl_rb_destroy)
    return st


class _Handle:
    """A library object, given back with the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def _weights(seed):
    """A network of the size of a trained one: unit-gain hidden layers, a small
    output layer (the correction is a few per cent of the stencil's range)."""
    rng = np.random.default_rng(seed)
    parts = [rng.standard_normal((64, 67)) * math.sqrt(2 / 67), rng.standard_normal(64) * 0.1,
             rng.standard_normal((64, 64)) * math.sqrt(2 / 64), rng.standard_normal(64) * 0.1,
             rng.standard_normal(64) * 0.01, rng.standard_normal(1) * 0.01]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


# ----------------------------------------------------------------------- a pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        d64 = case["dtype"] == "f32_d64"
        args = (st["vel"], st["dt"], st["spacing"], case["scheme"])
        if case["scheme"] != "CEC":
            return sl.advect(st["phi"], *args, 0, out=st["out"], delta64=d64)
        sl.advect(st["phi"], *args, 0, out=st["mid"], delta64=d64)
        return sl.advect(st["mid"], *args, 1, out=st["out"], delta64=d64)
    if kind == "wide":
        args = (st["vel"], st["dt"], st["spacing"], case["scheme"])
        if case["scheme"] != "CEC":
            return sl.advect_wide(st["phi"], *args, 0, out=st["out"], workspace=st["work"])
        sl.advect_wide(st["phi"], *args, 0, out=st["mid"], workspace=st["work"])
        return sl.advect_wide(st["mid"], *args, 1, out=st["out"], workspace=st["work"])
    if kind == "multi":
        dims = list(st["in"][0].shape)[::-1]
        args = (st["vel"], 3, dims, st["spacing"], st["dt"], sl.SCHEMES[case["scheme"]], sl.F32)
        sl.sl_advect_multi(st["mid"], st["in"], *args, 0)
        sl.sl_advect_multi(st["out"], st["mid"], *args, 1)
        return st["out"]
    if kind == "batch":      # A -> B and back: the plan's own double buffer
        sl.sl_batch_step(st["plan"].h, 0)
        sl.sl_batch_step(st["plan"].h, 1)
        return [a for a, *_ in st["grids"]]
    if kind == "learned":
        dims = list(st["phi"].shape)[::-1]
        sl.sl_advect_learned(st["net"].h, st["out"], st["phi"], st["vel"], 3, dims, st["spacing"], st["dt"])
        return st["out"]
    sl.sl_rb_set_state(st["box"].h, *st["start"])
    sl.sl_rb_step(st["box"].h, st["dt"], case["steps"])
    sl.sl_rb_get_state(st["box"].h, *st["out"])
    return st["out"]


# -------------------------------------------- what a pass cannot do without
# arithmetic of one cell's step: an interpolation of 2^d corners is 2^d - 1
# lerps of 3 operations; a 1D third-order sweep is 17 operations
def _flops(scheme, ndim):
    lerps = 3 * (2 ** ndim - 1)
    return {"CIR": lerps + 2 * ndim, "FEC": 2 * lerps + 2 * ndim + 3, "BEC": 3 * lerps + 2 * ndim + 3,
            "CEC": 17 * ndim}[scheme]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        cells = sum(i.n ** 3 for i in W.draw_batch(case["count"], seed=case["grids"]))
        return {"bytes": 2 * cells * 20, "flops": 2 * cells * _flops("CEC", 3)}
    if kind == "rb":
        n = case["nx"] * case["nz"]
        es = 4 if case["dtype"] == "f32" else 8
        one = n * (3 * _flops(case["scheme"], 2) + 80 + 4 * (case["nx"] + case["nz"]))
        return {"bytes": es * n * 6, "flops": one * case["steps"]}
    shape = _shape(case)
    nd, cells = len(shape), int(np.prod(shape))
    es = 8 if case.get("dtype") == "f64" else 4
    if kind == "learned":
        return {"bytes": 20 * cells, "flops": cells * 2 * (67 * 64 + 64 * 64 + 64)}
    fields = case.get("fields", 1)
    steps = 2 if case["scheme"] == "CEC" or kind == "multi" else 1
    return {"bytes": steps * es * cells * (2 * fields + nd), "flops": steps * fields * cells * _flops(case["scheme"], nd)}


# ------------------------------------------------- the same in 64 bits, plainly
def _interp(f, C, axes):
    """Multilinear value of f at i - C on the given axes (tensor axes of f; C by
    axis), periodic."""
    n = f.shape
    idx0 = [torch.arange(n[a], device=f.device).view([-1 if b == a else 1 for b in range(f.dim())]) for a in range(f.dim())]
    low, frac = {}, {}
    for a in axes:
        fl = torch.floor(-C[a])
        frac[a] = -C[a] - fl
        low[a] = torch.remainder(idx0[a] + fl.to(torch.int64), n[a])
    out = None
    flat = f.reshape(-1)
    for c in range(2 ** len(axes)):
        at, wt = 0, 1.0
        for a in range(f.dim()):
            if a in low:
                k = axes.index(a)
                up = (c >> k) & 1
                i = torch.remainder(low[a] + 1, n[a]) if up else low[a]
                wt = wt * (frac[a] if up else 1.0 - frac[a])
            else:
                i = idx0[a]
            at = at * n[a] + i
        v = wt * flat[at.expand(n)]
        out = v if out is None else out + v
        del at, wt, v
    return out


def _shifted(f, j, axis):
    """f at the cells j along one axis (periodic)."""
    return torch.gather(f, axis, torch.remainder(j, f.shape[axis]))


def _unsplit(f, C, scheme):
    axes = list(range(f.dim()))
    L = _interp(f, C, axes)
    if scheme == "CIR":
        return L
    half = (f - _interp(L, {a: -C[a] for a in axes}, axes)) / 2
    if scheme == "FEC":
        return L + half
    return _interp(f + half, C, axes)


def _sweep(f, c, axis):
    """One 1D third-order sweep: the correction is taken at the departure cell
    (the arrival cell for |C| < 1)."""
    L = _interp(f, {axis: c}, [axis])
    delta = f - _interp(L, {axis: -c}, [axis])
    m = torch.trunc(c)
    r = c - m
    i = torch.arange(f.shape[axis], device=f.device).view([-1 if b == axis else 1 for b in range(f.dim())])
    j = i - m.to(torch.int64)
    dj = _shifted(delta, j, axis)
    du = _shifted(delta, j - torch.sign(r).to(torch.int64), axis)
    return L + dj / 2 + (1 + r.abs()) / 6 * (du - dj)


def _step(f, C, scheme, parity):
    if scheme != "CEC":
        return _unsplit(f, C, scheme)
    axes = list(range(f.dim()))[::-1]     # x first
    for a in (axes[::-1] if parity else axes):
        f = _sweep(f, C[a], a)
    return f


def _courant(vel, dt, spacing):
    """Courant numbers by tensor axis (z, y, x) of a velocity ordered x, y, z."""
    nd = vel.shape[0]
    return {nd - 1 - d: vel[d].double() * (dt / spacing[d]) for d in range(nd)}


def exact(case, seed):
    kind = case["kind"]
    st = prepare(case, seed)
    if kind in ("step", "wide"):
        C = _courant(st["vel"], st["dt"], st["spacing"])
        f = _step(st["phi"].double(), C, case["scheme"], 0)
        return _step(f, C, case["scheme"], 1) if case["scheme"] == "CEC" else f
    if kind == "multi":
        C = _courant(st["vel"], st["dt"], st["spacing"])
        return [_step(_step(f.double(), C, case["scheme"], 0), C, case["scheme"], 1) for f in st["in"]]
    if kind == "batch":
        out = []
        for a, _, vel, dx, dt in st["grids"]:
            C = _courant(vel, dt, [dx] * 3)
            out.append(_step(_step(a.double(), C, "CEC", 0), C, "CEC", 1))
        return out
    if kind == "learned":
        return _learned(st)
    return _box(case, st)


def _learned(st):
    """m + s MLP((stencil - m) / s, f - 1/2) in 64 bits, plane by plane."""
    p = torch.from_numpy(st["weights"]).to(DEV).double()
    cut = np.cumsum([0, 64 * 67, 64, 64 * 64, 64, 64, 1])
    w1, b1, w2, b2, w3, b3 = (p[a:b] for a, b in zip(cut, cut[1:]))
    phi = st["phi"].double()
    C = _courant(st["vel"], st["dt"], st["spacing"])
    nz, ny, nx = phi.shape
    flat, out = phi.reshape(-1), torch.empty_like(phi)
    y0 = torch.arange(ny, device=DEV).view(-1, 1)
    x0 = torch.arange(nx, device=DEV).view(1, -1)
    for k in range(nz):
        fl = {a: torch.clamp(torch.floor(-C[a][k]), max=0).to(torch.int64) for a in range(3)}
        fr = [-C[a][k] - fl[a] for a in range(3)]
        z, y, x = k + fl[0], y0 + fl[1], x0 + fl[2]
        v = torch.stack([flat[(torch.remainder(z + c, nz) * ny + torch.remainder(y + b, ny)) * nx + torch.remainder(x + a, nx)]
                         for c in (-1, 0, 1, 2) for b in (-1, 0, 1, 2) for a in (-1, 0, 1, 2)], -1)
        q = v.view(ny, nx, 4, 4, 4)[..., 1:3, 1:3, 1:3]
        for t in fr:        # z, then y, then x
            q = q[:, :, 0] + t.view(ny, nx, *[1] * (q.dim() - 3)) * (q[:, :, 1] - q[:, :, 0])
        m = q[..., None]
        s = (v - m).abs().amax(-1, keepdim=True).clamp(min=1e-30)
        feat = torch.cat([(v - m) / s, torch.stack(fr[::-1], -1) - 0.5], -1)
        h = torch.relu(feat @ w1.view(64, 67).T + b1)
        h = torch.relu(h @ w2.view(64, 64).T + b2)
        out[k] = (m + s * (h @ w3 + b3)[..., None])[..., 0]
    return out


def _box(case, st):
    """The Rayleigh-Benard steps: mirrored ghosts, advection, explicit forces,
    Neumann projection in the cosine eigenbasis."""
    nx, nz, dt = case["nx"], case["nz"], st["dt"]
    dx, dz, Ra, Pr, G = 2.0 / nx, 1.0 / nz, 1e5, 1.0, 3
    u, w, th = (f.double() for f in st["start"])

    def cosines(n, h):
        j = torch.arange(n, device=DEV, dtype=torch.float64)
        c = torch.cos(math.pi * j[:, None] * (j + 0.5) / n) * math.sqrt(2.0 / n)
        c[0] /= math.sqrt(2.0)
        return c, -4.0 / h ** 2 * torch.sin(math.pi * j / (2 * n)) ** 2
    (cx, lx), (cz, lz) = cosines(nx, dx), cosines(nz, dz)
    lam = lz[:, None] + lx
    lam[0, 0] = 1.0

    def padded(f, sx, sz):
        f = torch.cat([sx * f[:, :G].flip(1), f, sx * f[:, -G:].flip(1)], 1)
        return torch.cat([sz * f[:G].flip(0), f, sz * f[-G:].flip(0)], 0)

    def inner(p):
        return p[G:-G, G:-G]

    def lap(p):
        c = p[1:-1, 1:-1]
        full = (p[1:-1, 2:] - 2 * c + p[1:-1, :-2]) / dx ** 2 + (p[2:, 1:-1] - 2 * c + p[:-2, 1:-1]) / dz ** 2
        return full[G - 1:-(G - 1), G - 1:-(G - 1)]

    def faces(f, axis):
        zero = torch.zeros_like(f.narrow(axis, 0, 1))
        return torch.cat([zero, f, zero], axis)

    for k in range(case["steps"]):
        pu, pw, pt = padded(u, -1, -1), padded(w, -1, -1), padded(th, 1, -1)
        C = {0: pw * (dt / dz), 1: pu * (dt / dx)}
        au, aw, at = (inner(_step(p, C, case["scheme"], k & 1)) for p in (pu, pw, pt))
        u2 = au + dt * Pr * lap(pu)
        w2 = aw + dt * (Ra * Pr * th + Pr * lap(pw))
        th = at + dt * (w + lap(pt))
        uf, wf = faces((u2[:, :-1] + u2[:, 1:]) / 2, 1), faces((w2[:-1] + w2[1:]) / 2, 0)
        F = cz @ ((uf[:, 1:] - uf[:, :-1]) / dx + (wf[1:] - wf[:-1]) / dz) @ cx.T / lam
        F[0, 0] = 0.0
        phi = cz.T @ F @ cx
        gx, gz = faces((phi[:, 1:] - phi[:, :-1]) / dx, 1), faces((phi[1:] - phi[:-1]) / dz, 0)
        u, w = u2 - (gx[:, :-1] + gx[:, 1:]) / 2, w2 - (gz[:-1] + gz[1:]) / 2
    return [u, w, th]
