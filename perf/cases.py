"""Timed cases of the electrode-charge library: what its users have it do, through the binding.

Every case is one call, or one short chain of calls, of the two kinds of program that use the
library: an MD driver, which needs the potential of the electrolyte on the electrode, the
charges and the forces every step for one frame, and an analysis or training program, which
takes many frames of one electrode, or many electrodes, at once.

Geometries are the package's own workloads: two graphene sheets in a slab cell, padded
along z (512 atoms is the small cell, 12,800 atoms the precision cell), and six stacked
sheets with pinholes (here 45 x 26 cells a sheet, about 26,700 atoms, instead of 90 x 52: the
same shape of work at a size whose inputs are made in a second).  Sizes in between, odd ones
among them, come from ``draw``.

``exact`` gives the same results from plain 64-bit torch arithmetic: direct Ewald sums, dense
solves, a plain network.
"""
import math

import numpy as np
import torch

from paper_2111_06704_gb300 import cpm
from paper_2111_06704_gb300 import workloads as wl
from paper_2111_06704_gb300.guess import LearnedGuess

F64 = torch.float64
DEV = "cuda"
EPS = 1e-8  # k-space truncation, the library's default

PRECISIONS = {"fp64": cpm.CPM_PREC_FP64, "fp32": cpm.CPM_PREC_FP32,
              "bf16x6": cpm.CPM_PREC_BF16X6}


def listed():
    return [
        # the smallest whole call: one MD step of the 512-atom cell with 200 ions in FP64
        # (potential, solve from the last step's charges, neutral charges, forces)
        {"name": "md_step_512_fp64", "kind": "md_step", "nx": 8, "ny": 8, "ions": 200,
         "precision": "fp64"},
        # the potential every MD step of the small cell starts with, default precision
        {"name": "potential_512", "kind": "potential", "cell": "sheets", "nx": 8, "ny": 8,
         "ions": 200, "frames": 1, "precision": "bf16x6"},
        # post-processing of a trajectory: 256 dense frames of the small cell in one call ...
        {"name": "potential_512_256_frames", "kind": "potential", "cell": "sheets", "nx": 8,
         "ny": 8, "ions": 2000, "frames": 256, "precision": "bf16x6"},
        # ... and their charges in one block solve
        {"name": "solve_512_256_frames", "kind": "solve", "cell": "sheets", "nx": 8, "ny": 8,
         "frames": 256, "guess": False, "precision": "bf16x6"},
        # one MD step of the 12,800-atom precision cell, call by call: the potential ...
        {"name": "potential_12800", "kind": "potential", "cell": "sheets", "nx": 40, "ny": 40,
         "ions": 2000, "frames": 1, "precision": "bf16x6"},
        # ... the charges from the last step's (one right-hand side, bound by reading E) ...
        {"name": "solve_12800", "kind": "solve", "cell": "sheets", "nx": 40, "ny": 40,
         "frames": 1, "guess": True, "precision": "bf16x6"},
        # ... and the forces of the charges on the ions
        {"name": "forces_12800", "kind": "forces", "nx": 40, "ny": 40, "ions": 2000,
         "frames": 1, "precision": "bf16x6"},
        # the build for a new geometry of that cell: E, the preconditioner, d
        {"name": "build_12800", "kind": "build", "nx": 40, "ny": 40, "precision": "bf16x6"},
        # the large stacked electrode, 16 frames a step, with the operand streamed as the
        # 106,568-atom electrode has it: the potential ...
        {"name": "potential_stacked_16_frames", "kind": "potential", "cell": "stacked",
         "nx": 45, "ny": 26, "ions": 5000, "frames": 16, "precision": "bf16x6"},
        # ... and the 16 right-hand sides of its solve
        {"name": "solve_stacked_16_frames", "kind": "solve", "cell": "stacked", "nx": 45,
         "ny": 26, "frames": 16, "guess": False, "precision": "bf16x6"},
        # a screening study: eight electrodes of uneven size, one solve over all of them
        {"name": "ragged_8_systems", "kind": "ragged", "count": 8, "n_lo": 500, "n_hi": 8000},
        # training and using the initial guess on the stacked electrode's 16 frames: the
        # features, one training step on them, the network's prediction
        {"name": "learn_stacked_16_frames", "kind": "learn", "nx": 45, "ny": 26, "frames": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sheet_cells(rng, lo, hi):
    """Cells (nx, ny) of a sheet with 8 nx ny atoms in about [lo, hi], sides within a factor
    of two; both edges exceed twice the preconditioner's 8 A cutoff."""
    cells = math.exp(rng.uniform(math.log(lo / 8), math.log(hi / 8)))
    nx = max(7, round(math.sqrt(cells * 1.73 * math.exp(rng.uniform(-0.3, 0.3)))))
    return nx, max(4, round(cells / nx))


def draw(rng):
    kind = rng.choice(["md_step", "potential", "potential", "potential_stacked", "solve",
                       "solve_frames", "solve_stacked", "forces", "build", "ragged", "learn"])
    nx, ny = _sheet_cells(rng, 300, 10000)
    n = 8 * nx * ny
    if kind == "md_step":
        nx, ny = _sheet_cells(rng, 300, 2000)
        return {"kind": kind, "nx": nx, "ny": ny, "ions": 2 * _log_int(rng, 10, 300),
                "precision": "fp64"}
    if kind == "potential":
        frames = min(256, max(1, _log_int(rng, 1, 1e5 / n)))
        return {"kind": kind, "cell": "sheets", "nx": nx, "ny": ny,
                "ions": 2 * _log_int(rng, 50, 1000), "frames": frames,
                "precision": rng.choice(["bf16x6", "bf16x6", "fp32", "fp64"])
                if n < 2500 and frames < 20 else "bf16x6"}
    if kind == "solve":
        return {"kind": kind, "cell": "sheets", "nx": nx, "ny": ny, "frames": 1,
                "guess": rng.random() < 0.7, "precision": rng.choice(["bf16x6", "fp32", "fp64"])
                if n < 2500 else "bf16x6"}
    if kind == "solve_frames":
        return {"kind": "solve", "cell": "sheets", "nx": nx, "ny": ny,
                "frames": min(256, max(2, _log_int(rng, 2, 1e5 / n))), "guess": False,
                "precision": "bf16x6"}
    if kind == "forces":
        return {"kind": kind, "nx": nx, "ny": ny, "ions": 2 * _log_int(rng, 50, 1000),
                "frames": max(1, _log_int(rng, 1, 1e4 / n)), "precision": "bf16x6"}
    if kind == "build":
        return {"kind": kind, "nx": nx, "ny": ny,
                "precision": rng.choice(["bf16x6", "fp32"]) if n < 2500 else "bf16x6"}
    if kind == "ragged":
        return {"kind": kind, "count": rng.randint(2, 8), "n_lo": 500,
                "n_hi": _log_int(rng, 1000, 8000)}
    sx = rng.randint(20, 44)
    sy = max(12, round(sx * 0.577 * rng.uniform(0.9, 1.1)))
    c = {"nx": sx, "ny": min(sy, 26), "frames": rng.randint(2, 16)}
    if kind == "learn":
        return {"kind": kind, **c}
    if kind == "potential_stacked":
        return {"kind": "potential", "cell": "stacked", **c, "ions": 10 * rng.randint(50, 500),
                "precision": "bf16x6"}
    return {"kind": "solve", "cell": "stacked", **c, "guess": False, "precision": "bf16x6"}


# ---- inputs ------------------------------------------------------------------------------

STACKED = {"g_ewald": 0.15, "rcut_real": 24.0}  # as the package's scale point


def _is_stacked(case):
    return case.get("cell") == "stacked" or case["kind"] == "learn"


def _strained(el, seed):
    """The electrode strained by up to 0.2% in x and y, as the cells of one study differ."""
    s = 1.0 + 0.002 * np.random.default_rng(2000 + seed).uniform(-1, 1)
    box = (el.box[0] * s, el.box[1] * s, el.box[2])
    return wl.Electrode(xyz=el.xyz * np.array([s, s, 1.0]), alpha=el.alpha, chi=el.chi, box=box)


def _electrode(case, seed):
    if _is_stacked(case):
        rng = np.random.default_rng(1000 + 100 * case["nx"] + case["ny"])
        el = wl.stacked_electrode(rng, nx=case["nx"], ny=case["ny"])
    else:
        el = wl.two_sheet_electrode(case["nx"], case["ny"])
    return _strained(el, seed)


def _params(case):
    """The Ewald parameters (g, r_c) and the context's keyword arguments."""
    kw = {"precision": PRECISIONS[case.get("precision", "bf16x6")]}
    if _is_stacked(case):
        return STACKED["g_ewald"], STACKED["rcut_real"], {**kw, **STACKED, "stream_operand": 1}
    return wl.G_EWALD, wl.RCUT_REAL, kw


def _ions(case, el, seed):
    """(xyz [F, I, 3], q [F, I]): consecutive or independent frames of the electrolyte."""
    rng = np.random.default_rng(3000 + seed)
    frames, n_ion = case["frames"], case["ions"]
    if _is_stacked(case):
        per, xyz, q = n_ion // 5, [], []
        for k in range(5):
            p, qq = wl.random_ions(rng, per // 2, per - per // 2, el.box, zlo=7.0 * k + 2.0,
                                   zhi=7.0 * k + 5.0, min_sep=None)
            xyz.append(p)
            q.append(qq)
        base, q = np.concatenate(xyz), np.concatenate(q)
        f = base + rng.normal(0.0, 0.5, size=(frames,) + base.shape)
        f[..., :2] %= el.box[:2]
        lo = 7.0 * np.floor(base[:, 2] / 7.0) + 2.0
        f[..., 2] = lo + 3.0 - np.abs((f[..., 2] - lo) % 6.0 - 3.0)  # reflected into its band
        xyz = f
    else:
        # a 2.5 A separation where the slit has room for it
        room = el.box[0] * el.box[1] * 24.0 / n_ion > 60.0
        base, q = wl.random_ions(rng, n_ion // 2, n_ion - n_ion // 2, el.box,
                                 min_sep=2.5 if room else None)
        xyz = base[None] if frames == 1 else wl.perturb_frames(rng, base, frames, 0.5, el.box)
    return xyz, np.broadcast_to(q, (frames, q.shape[0])).copy()


def _rough_potential(el, case, seed, frames):
    """Right-hand sides b [frames, n] of the solve cases (V): chi minus the potential of
    random ions, screened (erfc(r / 5 A) / r, nearest image), in plain torch."""
    gen = torch.Generator(device=DEV).manual_seed(4000 + seed)
    r = torch.tensor(el.xyz, device=DEV)
    box = torch.tensor(el.box, device=DEV, dtype=F64)
    m = min(400, max(20, el.n // 4 // 2 * 2))
    hi = 35.0 if _is_stacked(case) else 30.0
    b = torch.empty((frames, el.n), dtype=F64, device=DEV)
    q = torch.ones(m, dtype=F64, device=DEV)
    q[m // 2:] = -1.0
    for f in range(frames):
        p = torch.rand((m, 3), generator=gen, dtype=F64, device=DEV)
        p = torch.cat([p[:, :2] * box[:2], p[:, 2:] * hi], dim=1)
        d = r[:, None, :2] - p[None, :, :2]
        d -= box[:2] * torch.round(d / box[:2])
        r2 = (d * d).sum(-1) + (r[:, None, 2] - p[None, :, 2]) ** 2
        rr = torch.sqrt(r2 + 1.0)
        b[f] = torch.tensor(el.chi, device=DEV) - cpm.KE * (torch.special.erfc(rr / 5.0) / rr) @ q
    return b


def _charges_like(el, seed, frames):
    """Charges (e) of the magnitude the solves give, neutral, a smooth pattern plus noise."""
    gen = torch.Generator(device=DEV).manual_seed(5000 + seed)
    q = 0.01 * torch.randn((frames, el.n), generator=gen, dtype=F64, device=DEV)
    q += 0.02 * torch.sign(torch.tensor(el.chi, device=DEV))
    return q - q.mean(dim=1, keepdim=True)


def _built(case, el):
    _, _, kw = _params(case)
    ctx = cpm.Context(el.box, **kw)
    ctx.cpm_build_E(el.xyz, el.alpha)
    return ctx


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


def _network(case, seed, n, frames):
    """A network in mid-training and a batch for it: parameters [10,497], Adam's moments, the
    normalisation [64], targets [frames * n]."""
    gen = torch.Generator(device=DEV).manual_seed(6000 + seed)
    w = []
    for i, o in ((32, 64), (64, 64), (64, 64), (64, 1)):
        w.append(torch.randn(o * i, generator=gen, device=DEV) / math.sqrt(i))
        w.append(0.05 * torch.randn(o, generator=gen, device=DEV))
    p = torch.cat(w)
    m = 1e-3 * torch.randn(p.numel(), generator=gen, device=DEV)
    v = 1e-5 * (0.1 + torch.rand(p.numel(), generator=gen, device=DEV))
    mean, inv = torch.zeros(32), torch.zeros(32)
    inv[:9], inv[9:18], inv[18], inv[19], inv[20] = 2.0, 0.7, 2.0, 1.0, 20.0
    target = torch.randn(frames * n, generator=gen, device=DEV)
    return p, m, v, torch.cat([mean, inv]).to(DEV), target


def _learn_inputs(case, seed):
    el = _electrode(case, seed)
    b_prev = _rough_potential(el, case, seed, case["frames"])
    gen = torch.Generator(device=DEV).manual_seed(7000 + seed)
    b = b_prev + 0.3 * torch.randn(b_prev.shape, generator=gen, dtype=F64, device=DEV)
    return el, b, b_prev, _network(case, seed, el.n, case["frames"])


LEARN_STEP, LEARN_RATE = 100, 2e-3


def _ragged_systems(case, seed):
    works = wl.ragged_systems(case["count"], case["n_lo"], case["n_hi"], seed=case["n_hi"])
    return [_strained(w.electrode, seed + 31 * k) for k, w in enumerate(works)]


def _forces_inputs(case, seed):
    el = _electrode(case, seed)
    xyz, qi = _ions(case, el, seed)
    return el, xyz, qi, _charges_like(el, seed, case["frames"])


def prepare(case, seed):
    case = {"frames": 1, **case}
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "ragged":
        els = _ragged_systems(case, seed)
        s["ctx"] = [_built({"kind": "build"}, el) for el in els]
        for c in s["ctx"]:
            c.cpm_release_workspace()
        s["batch"] = cpm.Batch(s["ctx"])
        s["b"] = torch.cat([_rough_potential(el, case, seed + 31 * k, 1)[0]
                            for k, el in enumerate(els)])
        s["q"] = torch.zeros_like(s["b"])
        return s
    if kind == "learn":
        el, s["b"], s["b_prev"], (p, m, v, norm, s["target"]) = _learn_inputs(case, seed)
        s["ctx"] = _built(case, el)
        s["ctx"].cpm_release_workspace()
        s["chi"] = _dev(el.chi)
        g = s["net"] = LearnedGuess(s["ctx"])
        g.params.copy_(p)
        g.m.copy_(m)
        g.v.copy_(v)
        g.norm.copy_(norm)
        g.step = LEARN_STEP - 1
        return s
    if kind == "forces":
        el, xyz, qi, s["q"] = _forces_inputs(case, seed)
        s["ctx"] = _built(case, el)
        s["ctx"].cpm_release_workspace()
        s["xyz"], s["qi"] = _dev(xyz), _dev(qi)
        s["f"] = torch.empty_like(s["xyz"])
        return s
    el = _electrode(case, seed)
    if kind == "build":
        _, _, kw = _params(case)
        s["ctx"] = cpm.Context(el.box, **kw)
        s["el"] = (_dev(el.xyz), _dev(el.alpha))
        s["p"] = _charges_like(el, seed, 4)
        s["e"] = torch.empty_like(s["p"])
        return s
    s["ctx"] = _built(case, el)
    s["ctx"].cpm_release_workspace()
    s["chi"] = _dev(el.chi)
    if kind == "solve":
        s["b"] = _rough_potential(el, case, seed, case["frames"])
        s["q"] = torch.zeros_like(s["b"])
        s["q0"] = None
        if case["guess"]:  # the last step's charges: those of a nearby right-hand side
            s["q0"] = torch.zeros_like(s["b"])
            gen = torch.Generator(device=DEV).manual_seed(9000 + seed)
            near = s["b"] + 0.05 * torch.randn(s["b"].shape, generator=gen, dtype=F64, device=DEV)
            s["ctx"].cpm_solve(near, s["q0"])
        return s
    xyz, qi = _ions(case, el, seed)
    s["xyz"], s["qi"] = _dev(xyz), _dev(qi)
    s["b"] = torch.empty((case["frames"], el.n), dtype=F64, device=DEV)
    s["qsol"] = torch.empty(case["frames"], dtype=F64, device=DEV)
    if kind == "md_step":  # the last step's charges
        s["q"], s["f"] = torch.empty_like(s["b"]), torch.empty_like(s["xyz"])
        s["q0"] = _charges_like(el, seed, 1)
    return s


# ---- one pass ----------------------------------------------------------------------------

def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "potential":
        ctx.cpm_potential(s["xyz"], s["qi"], s["chi"], s["b"], s["qsol"])
        return {"b": s["b"], "qsol": s["qsol"]}
    if kind == "solve":
        if s["q0"] is not None:
            s["q"].copy_(s["q0"])
        ctx.cpm_solve(s["b"], s["q"], use_guess=s["q0"] is not None)
        ctx.cpm_neutralize(s["q"])
        return {"q": s["q"]}
    if kind == "md_step":
        ctx.cpm_potential(s["xyz"], s["qi"], s["chi"], s["b"], s["qsol"])
        s["q"].copy_(s["q0"])
        ctx.cpm_solve(s["b"], s["q"], use_guess=True, tol=1e-8)
        ctx.cpm_neutralize(s["q"], s["qsol"])
        ctx.cpm_ion_forces(s["xyz"], s["qi"], s["q"], s["f"])
        return {"b": s["b"], "q": s["q"], "f": s["f"]}
    if kind == "forces":
        return {"f": ctx.cpm_ion_forces(s["xyz"], s["qi"], s["q"], s["f"])}
    if kind == "build":
        ctx.cpm_build_E(*s["el"])
        ctx.cpm_apply_E(s["p"], s["e"])
        return {"d": ctx.cpm_get_d(), "e": s["e"]}
    if kind == "ragged":
        s["batch"].solve(s["b"], s["q"])
        s["batch"].neutralize(s["q"])
        return {"q": s["q"]}
    g = s["net"]
    feat = g.features(s["b"], s["b_prev"], s["chi"])
    loss = g.train_step(feat, s["target"], LEARN_RATE)
    y = g.forward(feat)
    return {"feat": feat, "loss": loss, "params": g.params, "m": g.m, "v": g.v, "y": y}


# ---- what a pass cannot do without -----------------------------------------------------------

def _atoms(case):
    if _is_stacked(case):
        return round(0.947 * 24 * case["nx"] * case["ny"])
    return 8 * case["nx"] * case["ny"]


def _kvectors_count(case):
    g, _, _ = _params(case)
    a, b = case["nx"] * wl.CELL_A, case["ny"] * wl.CELL_B
    lz = 105.0 if _is_stacked(case) else 90.0
    kc = 2.0 * g * math.sqrt(-math.log(EPS))
    return a * b * lz * kc ** 3 / (12.0 * math.pi ** 2)


def work(case):
    kind = case["kind"]
    if kind == "ragged":
        n2 = case["count"] * ((case["n_lo"] + case["n_hi"]) / 2.0) ** 2
        return {"bytes": 4.0 * n2, "flops": 2.0 * n2}
    n = _atoms(case)
    f = case.get("frames", 1)
    esz = 8.0 if case.get("precision") == "fp64" else 4.0
    if kind == "build":  # E written; its k-space products over half the matrix
        return {"bytes": esz * n * n, "flops": 2.0 * n * n * _kvectors_count(case)}
    if kind == "solve":  # E read once, the vectors
        return {"bytes": esz * n * n + 16.0 * n * f, "flops": 2.0 * n * n * f}
    if kind == "learn":  # potentials and targets in, features and predictions out; 6 and 2
        s = float(n * f)  # multiply-adds a parameter and sample, gradient and prediction
        return {"bytes": s * (16.0 + 4.0 + 128.0 + 4.0), "flops": 8.0 * 10497 * s}
    ions = case["ions"]
    m = _kvectors_count(case)
    # one multiply-add each for the cos and sin part of every k-vector, for ions and atoms
    flops = 4.0 * m * f * (n + ions)
    io = 8.0 * f * (4 * ions + n) + 8.0 * n
    if kind == "md_step":
        return {"bytes": io + esz * n * n + 24.0 * ions, "flops": 2.0 * flops + 2.0 * n * n}
    if kind == "forces":
        return {"bytes": io + 24.0 * f * ions, "flops": flops}
    return {"bytes": io, "flops": flops}


# ---- the same results in 64 bits ---------------------------------------------------------------

def _kspace(box, g):
    """Half of the k-vectors within the cutoff: K [m, 3] and the weights W [m]."""
    kc = 2.0 * g * math.sqrt(-math.log(EPS))
    top = [int(kc * l / (2.0 * math.pi)) + 1 for l in box]
    h, k, l = torch.meshgrid(*(torch.arange(-t, t + 1, device=DEV) for t in top), indexing="ij")
    h, k, l = h.flatten(), k.flatten(), l.flatten()
    half = (h > 0) | ((h == 0) & (k > 0)) | ((h == 0) & (k == 0) & (l > 0))
    hkl = torch.stack([h, k, l], dim=1)[half].to(F64)
    kv = 2.0 * math.pi * hkl / torch.tensor(box, dtype=F64, device=DEV)
    k2 = (kv * kv).sum(1)
    keep = k2 <= kc * kc
    kv, k2 = kv[keep], k2[keep]
    w = 2.0 * (4.0 * math.pi / (box[0] * box[1] * box[2])) * torch.exp(-k2 / (4 * g * g)) / k2
    return kv, w


def _images(box, rc):
    """Whole-box shifts that bring a nearest image within r_c."""
    top = [0 if 2 * rc < l else int((rc + 0.5 * l) / l) for l in box]
    g = torch.meshgrid(*(torch.arange(-t, t + 1, device=DEV) for t in top), indexing="ij")
    return torch.stack([x.flatten() for x in g], 1).to(F64) * torch.tensor(box, dtype=F64, device=DEV)


def _pair_blocks(ra, rb, box, rc, rows=None):
    """(a, b, r_a - r_b of one image, r) of every image within r_c, block by block."""
    lx = torch.tensor(box, dtype=F64, device=DEV)
    rows = rows or max(1, 20_000_000 // max(1, rb.shape[0]))
    shifts = _images(box, rc)
    for a0 in range(0, ra.shape[0], rows):
        d = ra[a0:a0 + rows, None] - rb[None]
        d -= lx * torch.round(d / lx)
        for s in shifts:
            r2 = (d[..., 0] + s[0]) ** 2 + (d[..., 1] + s[1]) ** 2 + (d[..., 2] + s[2]) ** 2
            ia, ib = torch.nonzero((r2 < rc * rc) & (r2 > 0.0), as_tuple=True)
            yield ia + a0, ib, d[ia, ib] + s, torch.sqrt(r2[ia, ib])


def _exact_potential(el, xyz, q, g, rc):
    r, alpha = _dev(el.xyz), _dev(el.alpha)
    xyz, q = _dev(xyz), _dev(q)
    frames, n = q.shape[0], r.shape[0]
    kv, w = _kspace(el.box, g)
    bs = torch.zeros((frames, n), dtype=F64, device=DEV)
    step = max(1, 60_000_000 // max(n, xyz.shape[1]))
    for k0 in range(0, kv.shape[0], step):
        k, wk = kv[k0:k0 + step], w[k0:k0 + step]
        re = torch.empty((frames, k.shape[0]), dtype=F64, device=DEV)
        im = torch.empty_like(re)
        for f in range(frames):
            ph = xyz[f] @ k.T
            re[f], im[f] = q[f] @ torch.cos(ph), q[f] @ torch.sin(ph)
        ph = r @ k.T
        bs += (wk * re) @ torch.cos(ph).T + (wk * im) @ torch.sin(ph).T
    for f in range(frames):
        for ia, ib, _, d in _pair_blocks(r, xyz[f], el.box, rc):
            v = q[f][ib] * (torch.special.erfc(g * d) - torch.special.erfc(alpha[ia] * d)) / d
            bs[f].index_add_(0, ia, v)
    vol = el.box[0] * el.box[1] * el.box[2]
    bs += (4.0 * math.pi / vol) * r[:, 2] * (q * xyz[..., 2]).sum(1, keepdim=True)
    return _dev(el.chi) - cpm.KE * bs, q.sum(1)


def _exact_matrix(el, g, rc):
    """E in the neutral-equivalent form the library stores."""
    r, alpha = _dev(el.xyz), _dev(el.alpha)
    n = r.shape[0]
    e = torch.zeros((n, n), dtype=F64, device=DEV)
    kv, w = _kspace(el.box, g)
    step = max(1, 100_000_000 // n)
    for k0 in range(0, kv.shape[0], step):
        ph = r @ kv[k0:k0 + step].T
        sw = torch.sqrt(w[k0:k0 + step])
        c = sw * torch.cos(ph)
        e += c @ c.T
        c = sw * torch.sin(ph)
        e += c @ c.T
    for ia, ib, _, d in _pair_blocks(r, r, el.box, rc):
        a = 1.0 / torch.sqrt(alpha[ia] ** -2 + alpha[ib] ** -2)
        e.index_put_((ia, ib), (torch.special.erfc(g * d) - torch.special.erfc(a * d)) / d,
                     accumulate=True)
    e.diagonal().add_(math.sqrt(2.0 / math.pi) * alpha - 2.0 * g / math.sqrt(math.pi))
    vol = el.box[0] * el.box[1] * el.box[2]
    return e + (4.0 * math.pi / vol) * r[:, 2:] * r[:, 2]


def _exact_charges(e, b, qsol):
    """Neutral charges of b [F, n] (V) with total -qsol [F], and d."""
    n = e.shape[0]
    rhs = torch.cat([b / cpm.KE, torch.ones((1, n), dtype=F64, device=DEV)])
    x = torch.cholesky_solve(rhs.T, torch.linalg.cholesky(e)).T
    d = x[-1] / x[-1].sum()
    return x[:-1] - (x[:-1].sum(1, keepdim=True) + qsol[:, None]) * d, d


def _exact_forces(el, xyz, qi, qe, g, rc):
    r, alpha, xyz, qi = _dev(el.xyz), _dev(el.alpha), _dev(xyz), _dev(qi)
    kv, w = _kspace(el.box, g)
    vol = el.box[0] * el.box[1] * el.box[2]
    grad = torch.zeros_like(xyz)  # of sum_i q_i e_iI over the ion's position
    step = max(1, 60_000_000 // max(r.shape[0], xyz.shape[1]))
    for k0 in range(0, kv.shape[0], step):
        k, wk = kv[k0:k0 + step], w[k0:k0 + step]
        ph = r @ k.T
        c, s = qe @ torch.cos(ph), qe @ torch.sin(ph)
        for f in range(xyz.shape[0]):
            ph = xyz[f] @ k.T
            grad[f] += (wk * (s[f] * torch.cos(ph) - c[f] * torch.sin(ph))) @ k
    a2 = 2.0 / math.sqrt(math.pi)
    for f in range(xyz.shape[0]):
        for ia, ib, d, x in _pair_blocks(r, xyz[f], el.box, rc):
            al = alpha[ia]
            num = a2 * (al * torch.exp(-(al * x) ** 2) - g * torch.exp(-(g * x) ** 2))
            fp = num / x - (torch.special.erfc(g * x) - torch.special.erfc(al * x)) / (x * x)
            grad[f].index_add_(0, ib, -(qe[f][ia] * fp / x)[:, None] * d)
    z = (qe * r[:, 2]).sum(1)[:, None] - qe.sum(1)[:, None] * xyz[..., 2]
    grad[..., 2] += (4.0 * math.pi / vol) * z
    return -qi[..., None] * grad


def _exact_features(el, b, b_prev):
    """The network's 32 features of every atom, [F, n, 32]."""
    r = _dev(el.xyz)
    n, frames = r.shape[0], b.shape[0]
    rc, g = wl.RCUT_DC, wl.G_DC
    rows, cols, dist = [], [], []
    for ia, ib, _, d in _pair_blocks(r, r, el.box, rc + 1e-9):
        keep = d <= rc
        rows.append(ia[keep])
        cols.append(ib[keep])
        dist.append(d[keep])
    rows, cols, dist = torch.cat(rows), torch.cat(cols), torch.cat(dist)
    db = b - b_prev
    out = torch.zeros((frames, n, 32), dtype=F64, device=DEV)
    out[..., 0], out[..., 9], out[..., 18] = db, b, _dev(el.chi)
    out[..., 19] = torch.where(r[:, 2] > r[:, 2].mean(), 1.0, -1.0)
    shell = torch.floor(dist + 0.5).long()
    for k in range(1, 9):
        i, j = rows[shell == k], cols[shell == k]
        count = torch.bincount(i, minlength=n).clamp(min=1)
        for f in range(frames):
            zero = torch.zeros(n, dtype=F64, device=DEV)
            out[f, :, k] = zero.index_add(0, i, db[f][j]) / count
            out[f, :, 9 + k] = zero.index_add(0, i, b[f][j]) / count
    # (P Delta b) / k_e: column tau of P is column tau of the inverse of the local matrix of
    # tau's neighbours (itself first here)
    order = torch.argsort(rows, stable=True)
    rows, cols = rows[order], cols[order]
    count = torch.bincount(rows, minlength=n)
    m = int(count.max()) + 1
    nb = torch.full((n, m), -1, dtype=torch.long, device=DEV)
    nb[:, 0] = torch.arange(n, device=DEV)
    first = torch.cumsum(count, 0) - count  # each atom's first pair
    nb[rows, 1 + torch.arange(rows.shape[0], device=DEV) - first[rows]] = cols
    lx = torch.tensor(el.box, dtype=F64, device=DEV)
    cut = math.erfc(g * rc)
    diag = math.sqrt(2.0 / math.pi) * _dev(el.alpha)
    pdb = torch.zeros((frames, n), dtype=F64, device=DEV)
    eye = torch.eye(m, dtype=torch.bool, device=DEV)
    for t0 in range(0, n, 2048):
        at = nb[t0:t0 + 2048]
        live = at >= 0
        x = r[at.clamp(min=0)]
        d = x[:, :, None] - x[:, None]
        d -= lx * torch.round(d / lx)
        d = torch.sqrt((d * d).sum(-1))
        mat = torch.where((d < rc) & (d > 0), (torch.special.erfc(g * d) - cut) / d, 0.0)
        mat *= live[:, :, None] & live[:, None]
        mat = torch.where(eye, torch.where(live, diag[at.clamp(min=0)], 1.0)[:, :, None], mat)
        rhs = torch.zeros((at.shape[0], m, 1), dtype=F64, device=DEV)
        rhs[:, 0] = 1.0
        p = torch.linalg.solve(mat, rhs)[..., 0] * live
        v = p[None] * db[:, t0:t0 + 2048, None]
        pdb.index_add_(1, at.clamp(min=0).flatten(), v.flatten(1))
    out[..., 20] = pdb / cpm.KE
    return out


def _unpack(p):
    at, got = 0, []
    for i, o in ((32, 64), (64, 64), (64, 64), (64, 1)):
        got.append((p[at:at + i * o].reshape(o, i), p[at + i * o:at + i * o + o]))
        at += i * o + o
    return got


def _exact_net(p, norm, feat):
    """The network on features [S, 32]: weights and biases rounded to bf16 where used."""
    h = (feat - norm[:32]) * norm[32:]
    layers = _unpack(p)
    for k, (w, c) in enumerate(layers):
        h = h @ w.T + c
        if k < 3:
            h = h * torch.sigmoid(h)
    return h[:, 0]


def _exact_learn(case, seed):
    el, b, b_prev, (p, m, v, norm, target) = _learn_inputs(case, seed)
    feat = _exact_features(el, b, b_prev)
    flat, norm = feat.reshape(-1, 32), norm.to(F64)
    used = p.to(torch.bfloat16).to(F64).requires_grad_(True)
    loss = 0.0
    for s0 in range(0, flat.shape[0], 65536):
        y = _exact_net(used, norm, flat[s0:s0 + 65536])
        part = ((y - target[s0:s0 + 65536].to(F64)) ** 2).sum() / flat.shape[0]
        part.backward()
        loss += float(part)
    grad = used.grad
    m = 0.9 * m.to(F64) + 0.1 * grad
    v = 0.999 * v.to(F64) + 0.001 * grad * grad
    step = (m / (1.0 - 0.9 ** LEARN_STEP)) / (torch.sqrt(v / (1.0 - 0.999 ** LEARN_STEP)) + 1e-8)
    # a weight next to the middle of two bf16 values may round to either after the step, so
    # the prediction that follows it has no one value
    return {"feat": feat, "loss": loss, "params": p.to(F64) - LEARN_RATE * step, "m": m, "v": v,
            "y": None}


def exact(case, seed):
    kind = case["kind"]
    case = {"frames": 1, **case}
    g, rc, _ = _params(case)
    if kind == "learn":
        return _exact_learn(case, seed)
    if kind == "forces":
        el, xyz, qi, qe = _forces_inputs(case, seed)
        return {"f": _exact_forces(el, xyz, qi, qe, g, rc)}
    if kind == "potential":
        el = _electrode(case, seed)
        b, qsol = _exact_potential(el, *_ions(case, el, seed), g, rc)
        return {"b": b, "qsol": qsol}
    if kind == "ragged":
        els = _ragged_systems(case, seed)
        if sum(el.n ** 3 for el in els) > 3.5e10:  # over twenty seconds
            return None
        q = []
        for k, el in enumerate(els):
            b = _rough_potential(el, case, seed + 31 * k, 1)
            zero = torch.zeros(1, dtype=F64, device=DEV)
            q.append(_exact_charges(_exact_matrix(el, g, rc), b, zero)[0][0])
        return {"q": torch.cat(q)}
    el = _electrode(case, seed)
    if el.n > (8000 if _is_stacked(case) else 3000):  # over twenty seconds
        return None
    e = _exact_matrix(el, g, rc)
    if kind == "build":
        p = _charges_like(el, seed, 4)
        _, d = _exact_charges(e, p, torch.zeros(4, dtype=F64, device=DEV))
        return {"d": d, "e": p @ e}
    if kind == "solve":
        b = _rough_potential(el, case, seed, case["frames"])
        zero = torch.zeros(case["frames"], dtype=F64, device=DEV)
        return {"q": _exact_charges(e, b, zero)[0]}
    xyz, qi = _ions(case, el, seed)
    b, qsol = _exact_potential(el, xyz, qi, g, rc)
    q, _ = _exact_charges(e, b, qsol)
    return {"b": b, "q": q, "f": _exact_forces(el, xyz, qi, q, g, rc)}
