"""The work that is measured: what a user of the dose engine has it do, through
the Python binding of its C ABI, over the range of sizes it is used at.

A case is a dict of plain values.  Its "kind" says which call is made:

  dose         dc_fspb_dose: one dose of a resident plan (an optimiser's inner step)
  replan       dc_fspb_set_density + dc_fspb_dose: a new CT of the day on a resident plan,
               in the paper's lateral form, the axis-stencil form or the network form
  matrix       dc_fspb_set_density + dc_fspb_dose_and_matrix: the whole plan, with the sparse
               dose-deposition matrix (FP32 or BF16 values) an optimiser works on
  batch        dc_fspb_dose_batch: k fluence vectors at once (scenarios, apertures)
  spmm         dc_fspb_spmm: k fluence vectors through the prepared BF16 matrix
  spmm_replan  dc_fspb_set_density + dc_fspb_spmm_prepare + dc_fspb_spmm: the same after a new density
  vjp          dc_fspb_dose_vjp: the backward pass of the commissioning fit
  gamma        dc_gamma_index: 3 %-3 mm comparison of two doses
  plans        dc_fspb_batch_dose with the density steps: several uneven plans as one graph

All arrays are CUDA tensors; the seed sets the phantom, the fluences and the
weights, the case sets the grid and the beams.
"""
import math
import random

import numpy as np
import torch

from paper_1103_1164_gb300 import dc_fspb, synth

DEV = "cuda"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _plan(kind, body, n, vox, beams, field, beamlet, roi=5.0, couch=False, layout=1, **more):
    c = dict(kind=kind, body=body, nx=n[0], ny=n[1], nz=n[2], vx=vox[0], vy=vox[1], vz=vox[2], beams=beams,
             field_lo=field[0], field_hi=field[1], bx=beamlet[0], by=beamlet[1], roi=roi, couch=couch, layout=layout)
    c.update(more)
    return c


def listed():
    iso = (0.25, 0.25, 0.25)
    thorax = dict(body="thorax", n=(128, 128, 96), vox=iso, beams=9, field=(8.0, 15.0), beamlet=(0.5, 0.5))
    cases = [
        # a phantom check or a unit of a service: launches and latency are what counts
        ("dose_tiny", _plan("dose", "mixed", (20, 18, 12), (0.3, 0.3, 0.3), 3, (3.0, 3.0), (0.5, 0.5), roi=2.0)),
        # the inner step of a fluence optimiser on the nine-field thorax plan
        ("dose_thorax9", _plan("dose", **thorax)),
        # the benchmark's step: density in, dose and FP32 matrix out
        ("matrix_thorax9", _plan("matrix", **thorax, dtype="f32")),
        # head and neck in fine beamlets, voxels whose half is not the water tables' step
        ("dose_head_neck", _plan("dose", "head_neck", (149, 149, 101), (0.23, 0.23, 0.23), 7, (10.0, 12.0),
                                 (0.25, 0.25), layout=5)),
        # a clinical non-coplanar case: CT voxels, beamlets of one leaf's width, BF16 matrix
        ("matrix_noncoplanar", _plan("matrix", "head_neck", (128, 128, 72), (0.4, 0.4, 0.25), 8, (6.0, 7.0),
                                     (0.2, 0.5), couch=True, layout=3, dtype="bf16")),
        # 64 fluence vectors in FP32 in one call (robust scenarios)
        ("batch64_thorax9", _plan("batch", **thorax, k=64, precision=0)),
        # 64 fluence vectors through the prepared matrix of a one-beam slab plan
        ("spmm64_slab", _plan("spmm", "slab", (64, 64, 64), iso, 1, (10.0, 10.0), (0.5, 0.5), roi=3.0, k=64)),
        # new density, new matrix, an odd number of vectors, several beams
        ("spmm_replan", _plan("spmm_replan", "head_neck", (113, 113, 65), (0.25, 0.25, 0.25), 5, (8.0, 9.0),
                              (0.25, 0.25), layout=8, k=21)),
        # a new density in the axis-stencil lateral form, on a ragged grid
        ("replan_axis", _plan("replan", "thorax", (97, 91, 71), (0.3, 0.3, 0.3), 5, (7.0, 10.0), (0.5, 0.5),
                              layout=2, lateral="axis")),
        # one slab phantom of the commissioning fit, backward
        ("vjp_slab", _plan("vjp", "slab", (60, 60, 60), (0.5, 0.5, 0.5), 1, (10.0, 10.0), (0.5, 0.5))),
        # plan evaluation: 3-D gamma of two doses on the thorax grid
        ("gamma_thorax", dict(kind="gamma", nx=128, ny=128, nz=96, vx=0.25, vy=0.25, vz=0.25, pct=3.0, dta=0.3)),
        # several small uneven patients as one graph, density steps included
        ("plans_uneven", dict(kind="plans", plans=6, layout=4)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["dose", "replan", "matrix", "batch", "spmm", "spmm_replan", "vjp", "gamma", "plans"])
    layout = rng.randrange(10, 10000)
    if kind == "plans":
        return dict(kind="plans", plans=rng.randint(2, 6), layout=layout)
    n = int(_log(rng, 24, 150))
    nz = max(9, int(n * rng.uniform(0.45, 0.8)))
    if kind == "gamma":
        v = round(rng.uniform(0.2, 0.5), 2)
        return dict(kind="gamma", nx=n, ny=max(8, n - rng.randint(0, 9)), nz=min(nz, 96), vx=v, vy=v,
                    vz=round(rng.uniform(0.2, 0.5), 2), pct=rng.choice([2.0, 3.0]), dta=rng.choice([0.2, 0.3]))
    if kind == "vjp":
        n = rng.randint(20, 60)
        b = rng.choice([0.5, 1.0])
        return _plan("vjp", rng.choice(["slab", "mixed"]), (n, n, n), (0.5, 0.5, 0.5), rng.randint(1, 2), (4.0, 10.0),
                     (b, b), roi=rng.uniform(2.0, 5.0), layout=layout)
    # voxels of 0.25 cm put the water tables on the plan's depth grid; others do not
    vox = round(_log(rng, 24.0, 34.0) / n, 3) if n > 70 else rng.choice([0.25, 0.3])
    body = rng.choice(["thorax", "head_neck", "mixed"])
    fine = rng.random() < 0.3
    beamlet = rng.choice([(0.25, 0.25), (0.2, 0.5)]) if fine else (0.5, 0.5)
    most = min(14.0, 0.45 * n * vox)
    hi = max(2.0, rng.uniform(0.5, 1.0) * most)
    beams = rng.randint(1, 9)
    roi = rng.choice([2.0, 3.0, 5.0])
    more = {}
    if kind in ("dose", "batch"):
        more["precision"] = 1 if rng.random() < 0.25 else 0
    if kind == "replan":
        more["lateral"] = rng.choice(["iso", "axis", "network"])
    if kind == "matrix":
        more["dtype"] = rng.choice(["f32", "bf16"])
        hi = min(hi, 7.0 if fine else 12.0)
    if kind in ("batch", "spmm", "spmm_replan"):
        more["k"] = rng.choice([rng.randint(2, 16), rng.randint(17, 64)])
        hi = min(hi, 6.0 if fine else 12.0)
    if kind == "replan" and more["lateral"] != "iso":
        beams = min(beams, 5)
    shape = (n, max(8, n - rng.randint(0, 7)), nz)
    return _plan(kind, body, shape, (vox, vox, round(vox * rng.choice([1.0, 1.0, 0.8]), 3)), beams,
                 (max(1.0, 0.6 * hi), hi), beamlet, roi=roi, couch=rng.random() < 0.3, layout=layout, **more)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _grid(c):
    return synth.centred_grid(c["nx"], c["ny"], c["nz"], c["vx"], c["vy"], c["vz"])


def _beams(c):
    """Evenly spread gantry angles (0, 90, 180 and 270 degrees among them for
    some counts) with square-ish fields in whole beamlets; non-coplanar cases
    turn couch and collimator of every other beam."""
    r = random.Random(c["layout"])
    start = 0.0 if c["layout"] == 1 else r.uniform(0.0, 360.0 / c["beams"])
    out = []
    for b in range(c["beams"]):
        f = [max(1, round(r.uniform(c["field_lo"], c["field_hi"]) / w)) * w for w in (c["bx"], c["by"])]
        couch = coll = 0.0
        if c["couch"] and b % 2 == 1:
            couch, coll = r.choice([-1.0, 1.0]) * r.uniform(15.0, 45.0), r.uniform(-15.0, 15.0)
        out.append(synth.Beam(start + 360.0 * b / c["beams"], 100.0, (0.0, 0.0, 0.0), f[0], f[1], couch, coll))
    return out


def _phantom(c, seed):
    """float32 [nz, ny, nx] density: the bodies of the repository's synthetic
    phantoms with the seed's own positions, radii and densities."""
    r = random.Random(seed * 1000003 + 17)
    g = _grid(c)
    ax = [torch.arange(k, device=DEV, dtype=torch.float32) * d + o
          for k, d, o in ((g.nx, g.dx, g.ox), (g.ny, g.dy, g.oy), (g.nz, g.dz, g.oz))]
    Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    ex, ey, ez = g.nx * g.dx, g.ny * g.dy, g.nz * g.dz
    if c["body"] == "slab":        # water with one slab across the beam of gantry 0
        d0, rho = r.uniform(0.15, 0.35) * ey, torch.ones_like(X)
        depth = Y - (g.oy - 0.5 * g.dy)
        rho[(depth >= d0) & (depth < d0 + r.uniform(0.2, 0.5) * ey)] = r.uniform(0.1, 1.9)
        return rho
    if c["body"] == "mixed":       # water with slabs and spheres
        rho = torch.ones_like(X)
        for _ in range(r.randint(1, 4)):
            at = [r.uniform(-0.35, 0.35) * e for e in (ex, ey, ez)]
            rad = r.uniform(0.1, 0.3) * min(ex, ey, ez)
            inside = (X - at[0]) ** 2 + (Y - at[1]) ** 2 + (Z - at[2]) ** 2 <= rad * rad
            if r.random() < 0.5:
                inside = ((X, Y, Z)[r.randrange(3)] - at[0]).abs() <= rad
            rho[inside] = r.uniform(0.05, 2.0)
        return rho
    rho = torch.full_like(X, 0.001)
    if c["body"] == "thorax":      # ellipse with two lungs, a spine and noise
        a, b = r.uniform(0.41, 0.45) * ex, r.uniform(0.29, 0.33) * ey
        body = (X / a) ** 2 + (Y / b) ** 2 <= 1.0
        rho[body] = 1.0
        for sx in (-1.0, 1.0):
            lung = ((X - 0.46 * a * sx) / (0.32 * a)) ** 2 + ((Y + 0.05 * b) / (0.6 * b)) ** 2 + (Z / (0.4 * ez)) ** 2 <= 1.0
            rho[lung] = r.uniform(0.20, 0.35)
        rho[X ** 2 + (Y - 0.65 * b) ** 2 <= (0.1 * a) ** 2] = r.uniform(1.5, 1.8)
        gen = torch.Generator(device=DEV).manual_seed(seed + 1)
        noise = 0.02 * torch.randn(rho.shape, device=DEV, generator=gen)
        return torch.where(body, rho + noise, rho).clamp_(min=0.001)
    rad = r.uniform(0.38, 0.42) * min(ex, ey)   # head and neck: cylinder, air, bone, a lung base
    body = X ** 2 + Y ** 2 <= rad ** 2
    zlo = g.oz - 0.5 * g.dz
    rho[body] = 1.0
    rho[body & (Z < zlo + 0.25 * ez)] = r.uniform(0.20, 0.35)
    for _ in range(r.randint(2, 4)):
        at = [r.uniform(-0.5, 0.5) * e for e in (rad, rad, 0.5 * ez)]
        s = r.uniform(0.8, 2.0)
        rho[(X - at[0]) ** 2 + (Y - at[1]) ** 2 + (Z - at[2]) ** 2 <= s * s] = 0.001
    bone, bx = r.uniform(1.0, 2.0), r.uniform(-0.3, 0.3) * rad
    rho[((X - bx) ** 2 + (Y - 0.6 * rad) ** 2 <= bone ** 2) & body] = r.uniform(1.6, 1.9)
    rho[body & (X ** 2 + Y ** 2 >= (rad - 0.6) ** 2) & (Z > zlo + 0.25 * ez)] = r.uniform(1.6, 1.9)
    return rho


def _comm(c):
    """The commissioned beam model (the machine's: the same for every plan)."""
    return synth.make_commissioning(roi_radius=c["roi"])


def _n_beamlets(c):
    return sum(round(b.field_x / c["bx"]) * round(b.field_y / c["by"]) for b in _beams(c))


def _uniform(shape, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed + 77)
    return torch.rand(shape, device=DEV, generator=gen)


def _network(seed):
    """Parameters of the lateral network: fan-in weights, a small last layer."""
    r = np.random.default_rng(seed + 5)
    parts = []
    for fi, fo, s in ((48, 64, 1.0), (64, 64, 1.0), (64, 3, 0.1)):
        lim = s * math.sqrt(3.0 / fi)
        parts += [r.uniform(-lim, lim, (fi, fo)).ravel(), r.uniform(-0.05, 0.05, fo)]
    return np.concatenate(parts).astype(np.float32)


NETWORK_RANGE = (0.05, 2.0)


def _doses(c, seed):
    """Two doses on a grid as a plan evaluation compares them: crossing beams
    with penumbra and build-up, the second slightly shifted, rescaled and with
    a smooth local difference."""
    r = random.Random(seed * 1000003 + 29)
    g = _grid(c)
    z, y, x = (torch.arange(k, device=DEV, dtype=torch.float32) * d + o
               for k, d, o in ((g.nz, g.dz, g.oz), (g.ny, g.dy, g.oy), (g.nx, g.dx, g.ox)))
    Z, Y, X = torch.meshgrid(z, y, x, indexing="ij")
    ext = min(g.nx * g.dx, g.ny * g.dy)

    def dose(dx, scale):
        D = torch.zeros_like(X)
        for q in range(5):
            t = math.radians(72.0 * q + turn)
            u, w = (X - dx) * math.cos(t) + Y * math.sin(t), -(X - dx) * math.sin(t) + Y * math.cos(t)
            depth = w + 0.5 * ext
            lat = torch.sigmoid((0.15 * ext - u.abs()) / 0.25) * torch.sigmoid((0.15 * ext - Z.abs()) / 0.25)
            D += lat * torch.where(depth > 0, (1 - torch.exp(-2.0 * depth)) * torch.exp(-0.05 * depth), 0 * depth)
        return scale * D

    turn = r.uniform(0.0, 72.0)
    ref = dose(0.0, 1.0)
    at = [r.uniform(-0.2, 0.2) * ext for _ in range(3)]
    bump = torch.exp(-((X - at[0]) ** 2 + (Y - at[1]) ** 2 + (Z - at[2]) ** 2) / (0.02 * ext * ext))
    ev = dose(r.uniform(-0.2, 0.2), r.uniform(0.98, 1.02)) * (1.0 + r.uniform(0.03, 0.08) * bump)
    return ref.contiguous(), ev.contiguous()


def _members(c):
    """The plans of a batch: small and middling head-and-neck and thorax plans."""
    r = random.Random(c["layout"])
    out = []
    for j in range(c["plans"]):
        n = int(_log(r, 32, 104))
        out.append(_plan("replan", r.choice(["thorax", "head_neck"]), (n, n - r.randint(0, 5), int(0.65 * n)),
                         (0.3, 0.3, 0.3) if r.random() < 0.5 else (0.25, 0.25, 0.25), r.randint(3, 6), (4.0, 7.0), (0.5, 0.5),
                         layout=c["layout"] + j + 2, lateral="iso"))
    return out


def _make_plan(c, rho, lateral=None, seed=0):
    mode = dc_fspb.DC_LATERAL_AXIS if lateral == "axis" else dc_fspb.DC_LATERAL_ISO
    p = dc_fspb.dc_fspb_create(rho, _grid(c), _beams(c), c["bx"], c["by"], _comm(c), lateral_mode=mode)
    if lateral == "network":
        dc_fspb.dc_fspb_set_surrogate(p, _network(seed), *NETWORK_RANGE)
        dc_fspb.dc_fspb_set_lateral_mode(p, dc_fspb.DC_LATERAL_MLP)
    return p


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind == "gamma":
        s["ref"], s["ev"] = _doses(c, seed)
        s["gamma"], s["grid"] = torch.empty_like(s["ref"]), _grid(c)
        return s
    if kind == "plans":
        members = _members(c)
        rho = [_phantom(m, seed + 31 * j) for j, m in enumerate(members)]
        s["plans"] = [_make_plan(m, x) for m, x in zip(members, rho)]
        s["fluences"] = [_uniform((p.n_beamlets,), seed + j) for j, p in enumerate(s["plans"])]
        s["doses"] = [torch.empty(p.shape, device=DEV) for p in s["plans"]]
        s["batch"] = dc_fspb.dc_fspb_batch_create(s["plans"])
        return s
    rho = _phantom(c, seed)
    p = s["plan"] = _make_plan(c, rho, c.get("lateral"), seed)
    if kind in ("replan", "matrix", "spmm_replan"):
        s["rho"] = rho
    if c.get("precision"):
        dc_fspb.dc_fspb_set_precision(p, dc_fspb.DC_PRECISION_BF16)
    if kind in ("spmm", "spmm_replan"):
        s["F"] = _uniform((p.n_beamlets, c["k"]), seed)
        s["Y"] = torch.empty((p.n_voxels, c["k"]), device=DEV)
        if kind == "spmm":
            dc_fspb.dc_fspb_spmm_prepare(p)
        return s
    if kind == "batch":
        s["fluence"] = _uniform((c["k"], p.n_beamlets), seed)
        s["dose"] = torch.empty((c["k"],) + p.shape, device=DEV)
        return s
    s["fluence"] = _uniform((p.n_beamlets,), seed)
    if kind == "vjp":
        s["weights"] = _uniform((p.n_voxels,), seed + 3) - 0.3
        m = _comm(c)
        s["tables"] = (m.water.shape[1], m.dens.shape[1])
        s["out"] = tuple(torch.empty(n, device=DEV) for n in ((4, m.water.shape[1]), (4, m.dens.shape[1]), (2,)))
        return s
    s["dose"] = torch.empty(p.shape, device=DEV)
    if kind == "matrix":
        # buffers with room for the pairs of any density on this grid, as a
        # program that recalculates a plan keeps them; zero past the pattern
        room = int(2 * _pairs(c)) + 1024
        if dc_fspb.dc_fspb_pair_count(p) > room:
            raise ValueError("the matrix is larger than its buffers")
        s["rowptr"] = torch.empty(p.n_voxels + 1, dtype=torch.int64, device=DEV)
        s["cols"] = torch.zeros(room, dtype=torch.int32, device=DEV)
        s["vals"] = torch.zeros(room, dtype=torch.float32 if c["dtype"] == "f32" else torch.bfloat16, device=DEV)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "gamma":
        g, stats = dc_fspb.dc_gamma_index(s["ref"], s["ev"], s["grid"], c["pct"], c["dta"], gamma=s["gamma"])
        return {"gamma": g, "stats": stats}
    if kind == "plans":
        return dc_fspb.dc_fspb_batch_dose(s["batch"], s["fluences"], s["doses"], density=True)
    p = s["plan"]
    if kind in ("replan", "matrix", "spmm_replan"):
        dc_fspb.dc_fspb_set_density(p, s["rho"])
    if kind in ("dose", "replan"):
        return dc_fspb.dc_fspb_dose(p, s["fluence"], s["dose"])
    if kind == "matrix":
        dt = dc_fspb.DC_F32 if c["dtype"] == "f32" else dc_fspb.DC_BF16
        d, rp, cols, vals = dc_fspb.dc_fspb_dose_and_matrix(p, s["fluence"], s["dose"], dt, s["rowptr"], s["cols"], s["vals"])
        return {"dose": d, "rowptr": rp, "cols": cols, "vals": vals}
    if kind == "batch":
        return dc_fspb.dc_fspb_dose_batch(p, s["fluence"], s["dose"])
    if kind == "spmm":
        return dc_fspb.dc_fspb_spmm(p, s["F"], s["Y"])
    if kind == "spmm_replan":
        dc_fspb.dc_fspb_spmm_prepare(p)
        return dc_fspb.dc_fspb_spmm(p, s["F"], s["Y"])
    if kind == "vjp":
        return dc_fspb.dc_fspb_dose_vjp(p, s["fluence"], s["weights"], *s["tables"], out=s["out"])
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

# FP32 operations of one (voxel, beamlet) evaluation of eqs. (2)-(4): 8
# exponentials, a reciprocal and the arithmetic of the definition.
PAIR_OPS = 74


def _pairs(c):
    """About how many (voxel, beamlet) pairs the plan has: each beamlet's
    cylinder of the ROI radius along its mean path in the body."""
    ex, ey = c["nx"] * c["vx"], c["ny"] * c["vy"]
    path = {"thorax": 1.6 * math.sqrt(0.43 * ex * 0.31 * ey), "head_neck": 1.6 * 0.4 * min(ex, ey)}.get(c["body"], min(ex, ey))
    area = min(math.pi * c["roi"] ** 2, ex * c["nz"] * c["vz"])
    return _n_beamlets(c) * area * path / (c["vx"] * c["vy"] * c["vz"])


def work(case):
    c, kind = case, case["kind"]
    if kind == "plans":
        w = [work(m) for m in _members(c)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    V = c["nx"] * c["ny"] * c["nz"]
    if kind == "gamma":
        # the two doses in, gamma out; the ball of the distance criterion per voxel
        ball = 4.19 * c["dta"] ** 3 / (c["vx"] * c["vy"] * c["vz"])
        return {"bytes": 12.0 * V, "flops": 4.0 * V * max(1.0, ball)}
    B, pairs = _n_beamlets(c), _pairs(c)
    k = c.get("k", 1)
    flops = pairs * (PAIR_OPS + 2 * k)
    nbytes = 4.0 * (V + B * k + V * k)          # density, fluences, doses
    if kind == "matrix":
        nbytes += 8.0 * V + pairs * (8 if c["dtype"] == "f32" else 6)
    if kind == "spmm":
        flops, nbytes = 2.0 * k * pairs, 2.0 * pairs + 4.0 * k * (B + V)
    if kind == "vjp":
        flops = 2.0 * pairs * PAIR_OPS
        nbytes = 4.0 * (2 * V + B)
    if kind == "replan" and c["lateral"] != "iso":
        # every axis stencil: 3 x 16 trilinear taps (or the network) per (voxel, beam) near a field
        flops += V * c["beams"] * 0.5 * (48 * 14 if c["lateral"] == "axis" else 2 * 7360)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _f(x):
    """The value that reaches the library: its interface takes 32-bit floats."""
    return float(np.float32(x))


def _lut(f, x0, h, x):
    """Linear interpolation in a table of equal steps, clamped to its domain."""
    n = f.shape[-1]
    s = ((x - x0) / h).clamp(0.0, n - 1.0)
    j = s.detach().floor().clamp(max=n - 2).long()
    w = s - j
    return (1.0 - w) * f[j] + w * f[j + 1]


def _smooth(rho, dims, sigma):
    """Separable Gaussian truncated at ceil(3 sigma / step), edges repeated."""
    out = rho
    for axis, step in enumerate((dims[2], dims[1], dims[0])):
        r = math.ceil(3.0 * sigma / step) if sigma > 0 else 0
        w = [math.exp(-(q * step) ** 2 / (2.0 * sigma * sigma)) if sigma > 0 else 1.0 for q in range(-r, r + 1)]
        n = out.shape[axis]
        at = torch.arange(n, device=out.device)
        out = sum(wq / sum(w) * out.index_select(axis, (at + q).clamp(0, n - 1)) for q, wq in zip(range(-r, r + 1), w))
    return out


class _Model:
    """The dose model of one plan in 64 bits: geometry, ray integrals and the
    pair evaluation, beam by beam."""

    def __init__(self, c, rho, lateral="iso", network=None):
        g, m = _grid(c), _comm(c)
        self.c, self.lateral, self.network = c, lateral, network
        t64 = dict(device=DEV, dtype=torch.float64)
        self.dim, self.step, self.org = (g.nx, g.ny, g.nz), [_f(v) for v in (g.dx, g.dy, g.dz)], [_f(v) for v in (g.ox, g.oy, g.oz)]
        self.d = 0.5 * min(self.step)
        self.rho = rho.double()
        self.A, self.water, self.dens = (torch.tensor(a, **t64) for a in (m.A, m.water, m.dens))
        self.a_dt, self.a_dth, self.w_dt, self.r0, self.dr = (_f(v) for v in (m.a_dt, m.a_dtheta, m.w_dt, m.f_rho0, m.f_drho))
        self.roi, self.sigma, self.surf = _f(m.roi_radius), _f(m.smooth_sigma), _f(m.rho_surface)
        self.bx, self.by = _f(c["bx"]), _f(c["by"])
        self.scale = torch.ones(2, **t64)     # of omega_1^corr and omega_2^corr
        self.rhos = _smooth(self.rho, self.step, self.sigma).reshape(-1)
        self.flat = self.rho.reshape(-1)
        v = torch.arange(self.flat.numel(), device=DEV)
        ijk = torch.stack((v % g.nx, v // g.nx % g.ny, v // (g.nx * g.ny)), 1).double()
        self.r = ijk * torch.tensor(self.step, **t64) + torch.tensor(self.org, **t64)
        self.beams, first = [], 0
        for b in _beams(c):
            self.beams.append(self._beam(b, first))
            first += self.beams[-1]["n"].shape[0]

    def _beam(self, b, first):
        def turn(axis, deg, v):
            q, (i, j) = math.radians(_f(deg)), ((0, 1) if axis == "z" else (2, 0))
            w = list(v)
            w[i], w[j] = math.cos(q) * v[i] - math.sin(q) * v[j], math.sin(q) * v[i] + math.cos(q) * v[j]
            return w
        ex, ey, ez = (turn("y", b.couch_deg, turn("z", b.gantry_deg, v)) for v in ([1.0, 0, 0], [0, 0, 1.0], [0, 1.0, 0]))
        t64 = dict(device=DEV, dtype=torch.float64)
        ex, ey, ez = (torch.tensor(v, **t64) for v in (ex, ey, ez))
        q = math.radians(_f(b.coll_deg))
        ex, ey = math.cos(q) * ex + math.sin(q) * ey, -math.sin(q) * ex + math.cos(q) * ey
        sad, fx, fy = _f(b.sad), _f(b.field_x), _f(b.field_y)
        M, N = round(fx / self.bx), round(fy / self.by)
        a = (-0.5 * fx + (torch.arange(M, **t64) + 0.5) * self.bx).repeat(N)
        cc = (-0.5 * fy + (torch.arange(N, **t64) + 0.5) * self.by).repeat_interleave(M)
        n = a[:, None] * ex + cc[:, None] * ey + sad * ez
        n = n / n.norm(dim=1, keepdim=True)
        lx = ex - (n @ ex)[:, None] * n
        lx = lx / lx.norm(dim=1, keepdim=True)
        src = torch.tensor([_f(v) for v in b.iso], **t64) - sad * ez
        out = dict(src=src, ex=ex, ey=ey, ez=ez, sad=sad, hx=0.5 * fx, hy=0.5 * fy, n=n, lx=lx, ly=torch.linalg.cross(lx, n),
                   theta=torch.atan2(torch.sqrt(a * a + cc * cc), torch.tensor(sad, **t64)), first=first)
        out.update(self._trace(src, n))
        r = (out["theta"] / self.a_dth).clamp(0.0, self.A.shape[0] - 1.0)
        l = r.floor().clamp(max=self.A.shape[0] - 2).long()
        w = (r - l)[:, None]
        out["A"] = (1 - w) * self.A[l] + w * self.A[l + 1]
        return out

    def _trace(self, src, n):
        """Body entry and exit and the integrals of rho, b_1, b_2 at the depths k d."""
        inf = float("inf")
        nb = n.shape[0]
        lo, hi = torch.zeros(nb, device=DEV, dtype=torch.float64), torch.full((nb,), inf, device=DEV, dtype=torch.float64)
        cuts, miss = [], torch.zeros(nb, dtype=torch.bool, device=DEV)
        for a in range(3):
            planes = self.org[a] + (torch.arange(self.dim[a] + 1, device=DEV, dtype=torch.float64) - 0.5) * self.step[a]
            par = n[:, a].abs() < 1e-15
            miss |= par & ((src[a] <= planes[0]) | (src[a] >= planes[-1]))
            x = (planes[None] - src[a]) / torch.where(par, torch.ones_like(n[:, a]), n[:, a])[:, None]
            e0, e1 = torch.minimum(x[:, 0], x[:, -1]), torch.maximum(x[:, 0], x[:, -1])
            lo, hi = torch.maximum(lo, torch.where(par, lo, e0)), torch.minimum(hi, torch.where(par, hi, e1))
            cuts.append(torch.where(par[:, None], torch.full_like(x, -inf), x))
        miss |= ~(lo < hi)
        lo, hi = torch.where(miss, torch.zeros_like(lo), lo), torch.where(miss, torch.zeros_like(hi), hi)
        al = torch.cat(cuts + [lo[:, None], hi[:, None]], 1)
        al = torch.minimum(torch.maximum(al, lo[:, None]), hi[:, None]).sort(1).values
        mid = 0.5 * (al[:, 1:] + al[:, :-1])
        at = []
        for a in range(3):
            p = src[a] + mid * n[:, a:a + 1]
            at.append(((p - (self.org[a] - 0.5 * self.step[a])) / self.step[a]).floor().long().clamp(0, self.dim[a] - 1))
        rho = self.flat[(at[2] * self.dim[1] + at[1]) * self.dim[0] + at[0]]
        ln = al[:, 1:] - al[:, :-1]
        dense = (rho > self.surf) & (ln > 0) & ~miss[:, None]
        hit = dense.any(1)
        l_in = torch.where(dense, al[:, :-1], torch.full_like(ln, inf)).min(1).values
        l_out = torch.where(dense, al[:, 1:], torch.full_like(ln, -inf)).max(1).values
        l_in, l_out = torch.where(hit, l_in, torch.zeros_like(l_in)), torch.where(hit, l_out, torch.full_like(l_out, -1.0))
        K = int(((l_out - l_in).max() / self.d).ceil()) + 2
        pos = torch.minimum(l_in[:, None] + torch.arange(max(K, 2), device=DEV) * self.d, hi[:, None])
        tabs = []
        for f in (rho, _lut(self.dens[4], self.r0, self.dr, rho), _lut(self.dens[5], self.r0, self.dr, rho)):
            cum = torch.cat((torch.zeros_like(lo)[:, None], (f * ln).cumsum(1)), 1)

            def upto(x):
                j = (torch.searchsorted(al, x.contiguous(), right=True) - 1).clamp(0, ln.shape[1] - 1)
                return cum.gather(1, j) + f.gather(1, j) * (x - al.gather(1, j))
            tabs.append(upto(pos) - upto(l_in[:, None]))
        return dict(l_in=l_in, l_out=l_out, tabs=torch.stack(tabs, 2))

    def near(self, b):
        """The voxels whose projection lies within the ROI radius of the field."""
        w = self.r - b["src"]
        z = w @ b["ez"]
        s = b["sad"] / z
        reach = 1.05 * self.roi * s + 1e-3
        return (((w @ b["ex"]) * s).abs() <= b["hx"] + reach).logical_and_(((w @ b["ey"]) * s).abs() <= b["hy"] + reach).nonzero()[:, 0]

    def factors(self, vox, b):
        """f_u1, f_u2 along x and y, f_omega1, f_omega2 of the voxels for the beam."""
        f = lambda q, r: _lut(self.dens[q], self.r0, self.dr, r)  # noqa: E731
        own = self.flat[vox]
        if self.lateral == "iso":
            ux = uy = om = self.rhos[vox]
        else:
            om, ux, uy = self._stencil(vox, b)
        return torch.stack((f(0, own), f(1, ux), f(1, uy), f(2, om), f(3, om)), 1)

    def _points(self, vox, b):
        s = (torch.arange(16, device=DEV, dtype=torch.float64) - 7.5) * self.d
        e = torch.stack((b["ex"], b["ey"], b["ez"]))
        p = self.r[vox][:, None, None, :] + s[None, None, :, None] * e[None, :, None, :]
        return (p - torch.tensor(self.org, device=DEV, dtype=torch.float64)) / torch.tensor(self.step, device=DEV, dtype=torch.float64), s

    def _stencil(self, vox, b):
        out = []
        for part in vox.split(200_000):
            u, s = self._points(part, b)
            dim = torch.tensor(self.dim, device=DEV)
            g = torch.exp(-s * s / (2.0 * self.sigma ** 2))
            v = u.clamp(min=torch.zeros(3, device=DEV, dtype=torch.float64), max=(dim - 1).double())
            i0 = torch.minimum(v.floor().long(), (dim - 2).clamp(min=0))
            w = v - i0
            val = 0.0
            for q in range(8):
                at = [torch.minimum(i0[..., a] + (q >> a & 1), dim[a] - 1) for a in range(3)]
                wt = 1.0
                for a in range(3):
                    wt = wt * (w[..., a] if q >> a & 1 else 1.0 - w[..., a])
                val = val + wt * self.flat[(at[2] * self.dim[1] + at[1]) * self.dim[0] + at[0]]
            avg = (val * g).sum(2) / g.sum()
            eff = torch.stack((avg.mean(1), avg[:, 0], avg[:, 1]), 1)
            if self.lateral == "network":
                near = [(u[..., a] + 0.5).floor().long().clamp(0, self.dim[a] - 1) for a in range(3)]
                taps = self.flat[(near[2] * self.dim[1] + near[1]) * self.dim[0] + near[0]].reshape(len(part), 48)
                th, o, x = torch.tensor(self.network, device=DEV).double(), 0, taps - 1.0
                for k, (fi, fo) in enumerate(((48, 64), (64, 64), (64, 3))):
                    x = x @ th[o:o + fi * fo].view(fi, fo) + th[o + fi * fo:o + fi * fo + fo]
                    x = x * torch.sigmoid(x) if k < 2 else x
                    o += fi * fo + fo
                ok = ((taps >= _f(NETWORK_RANGE[0])) & (taps <= _f(NETWORK_RANGE[1]))).all(1, keepdim=True)
                eff = torch.where(ok, 1.0 + x, eff)
            out.append(eff)
        return torch.cat(out).unbind(1)

    def pairs(self, vox, fac, b):
        """(row in vox, beamlet of the beam, D) of every pair, voxel by voxel."""
        w = self.r[vox] - b["src"]
        L = w @ b["n"].T
        x, y = w @ b["lx"].T, w @ b["ly"].T
        vi, bi = ((x * x + y * y <= self.roi ** 2) & (L >= b["l_in"]) & (L <= b["l_out"])).nonzero(as_tuple=True)
        L, x, y = L[vi, bi], x[vi, bi], y[vi, bi]
        t, s = L - b["l_in"][bi], b["sad"] / L
        q = t / self.d
        k = q.floor().long().clamp(0, b["tabs"].shape[1] - 2)
        fr = (q - k)[:, None]
        teq, c1, c2 = ((1 - fr) * b["tabs"][bi, k] + fr * b["tabs"][bi, k + 1]).unbind(1)
        j = (teq / self.a_dt).clamp(0.0, self.A.shape[1] - 1.0)
        j0 = j.floor().clamp(max=self.A.shape[1] - 2).long()
        Av = (1 - (j - j0)) * b["A"][bi, j0] + (j - j0) * b["A"][bi, j0 + 1]
        u1, u2, o1, o2 = (_lut(self.water[r], 0.0, self.w_dt, t) for r in range(4))
        f = fac[vi]
        ax, ay, x0, y0 = (x * s).abs(), (y * s).abs(), 0.5 * self.bx, 0.5 * self.by

        def p(a, u, a0):
            e1, e2 = torch.exp(-u * (a - a0).abs()), torch.exp(-u * (a + a0))
            return torch.where(a <= a0, 1.0 - 0.5 * (e1 + e2), 0.5 * (e1 - e2))
        u1, ux, uy = f[:, 0] * u1, f[:, 1] * u2, f[:, 2] * u2
        w1, w2 = (f[:, 3] * (o1 + self.scale[0] * c1)).clamp(min=0.0), (f[:, 4] * (o2 + self.scale[1] * c2)).clamp(min=0.0)
        F = w1 * p(ax, u1, x0) * p(ay, u1, y0) + w2 * p(ax, ux, x0) * p(ay, uy, y0)
        return vi, bi, F * Av * s * s

    def chunks(self):
        """(beam, voxels, their factors) in pieces that fit in memory."""
        for b in self.beams:
            for vox in self.near(b).split(max(1, 20_000_000 // b["n"].shape[0])):
                yield b, vox

    def dose(self, F):
        """F [k, B] -> dose [k, V]."""
        F = F.double()
        out = torch.zeros((self.flat.numel(), F.shape[0]), device=DEV, dtype=torch.float64)
        for b, vox in self.chunks():
            vi, bi, D = self.pairs(vox, self.factors(vox, b), b)
            f = F[:, b["first"]:b["first"] + b["n"].shape[0]]
            if F.shape[0] == 1:
                out[:, 0].index_add_(0, vox[vi], D * f[0, bi])
            else:
                M = torch.zeros((len(vox), f.shape[1]), device=DEV, dtype=torch.float64)
                M[vi, bi] = D
                out[vox] += M @ f.T
        return out.T

    def backward(self, fluence, weights):
        for t in (self.water, self.dens, self.scale):
            t.requires_grad_(True)
        for b, vox in self.chunks():
            for part in vox.split(max(1, len(vox) // 4)):
                vi, bi, D = self.pairs(part, self.factors(part, b), b)
                (weights.double()[part][vi] * fluence.double()[b["first"] + bi] * D).sum().backward()
        return self.water.grad, self.dens.grad[:4], self.scale.grad


def _gamma64(c, ref, ev):
    g = _grid(c)
    d, dta, pct = [_f(v) for v in (g.dx, g.dy, g.dz)], _f(c["dta"]), _f(c["pct"])
    search = _f(5.0 * c["dta"])
    ref, ev = ref.double(), ev.double()
    inv = 1.0 / (pct / 100.0 * ref.max()) ** 2
    best = torch.full_like(ref, (search / dta) ** 2)
    reach = [int(search / v + 1e-9) for v in d]
    n = (g.nx, g.ny, g.nz)
    cut = lambda k, o: (slice(max(0, -o), k - max(0, o)), slice(max(0, o), k - max(0, -o)))  # noqa: E731
    for k in range(-reach[2], reach[2] + 1):
        for j in range(-reach[1], reach[1] + 1):
            for i in range(-reach[0], reach[0] + 1):
                r2 = (i * d[0]) ** 2 + (j * d[1]) ** 2 + (k * d[2]) ** 2
                if r2 > search ** 2 * (1 + 1e-12) or abs(i) >= n[0] or abs(j) >= n[1] or abs(k) >= n[2]:
                    continue
                (a, p), (b, q), (e, s) = cut(n[2], k), cut(n[1], j), cut(n[0], i)
                near = (ev[p, q, s] - ref[a, b, e]) ** 2 * inv + r2 / (dta * dta)
                best[a, b, e] = torch.minimum(best[a, b, e], near)
    gam = best.sqrt()
    in50 = ref >= 0.5 * ref.max()
    g50 = gam[in50]
    return gam, dict(gamma_max=float(gam.max()), gamma_avg50=float(g50.mean()), pass50_pct=100.0 * float((g50 < 1).double().mean()),
                     n50=None, dose_max=float(ref.max()))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "gamma":
        gam, stats = _gamma64(c, *_doses(c, seed))
        return {"gamma": gam, "stats": stats}
    if kind == "plans":
        out = []
        for j, m in enumerate(_members(c)):
            rho = _phantom(m, seed + 31 * j)
            out.append(_Model(m, rho).dose(_uniform((1, _n_beamlets(m)), seed + j))[0].view(rho.shape))
        return out
    rho = _phantom(c, seed)
    B = _n_beamlets(c)
    m = _Model(c, rho, c.get("lateral", "iso"), _network(seed))
    if kind == "vjp":
        return m.backward(_uniform((B,), seed), _uniform((m.flat.numel(),), seed + 3) - 0.3)
    if kind in ("spmm", "spmm_replan"):
        return m.dose(_uniform((B, c["k"]), seed).T).T.contiguous()
    if kind == "batch":
        return m.dose(_uniform((c["k"], B), seed)).reshape((c["k"],) + rho.shape)
    dose = m.dose(_uniform((1, B), seed))[0].view(rho.shape)
    # which pairs lie inside the ROI is decided in 32 bits, so the stored
    # pattern has no 64-bit counterpart entry by entry; the dose of the same
    # call sums every stored value
    return {"dose": dose, "rowptr": None, "cols": None, "vals": None} if kind == "matrix" else dose
