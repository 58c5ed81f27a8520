"""What the speed of this framework is measured on: the calls that its users make, over the range they make them in.

A case is one structure (or a batch of them) and one way of using it:

  step     macro steps of a field on a context whose kernels are built (fdirw_step): the steady state
  job      create a context, build its kernels, take the macro steps, read the mass, destroy it: one structure's whole run
  batch    the same for several structures in one context, each source with its own window radius
  flow     the same with a steady face-velocity field (convection)
  coupled  create a coarse-mesh context with a far field, build P and P_BC, take coupled macro steps
  train    one Adam step of the learned kernel on FD kernels of a structure

Geometries are this repository's seeded sphere packings; the recipes (porosity, contrast, radius, substeps at
the stability limit, initial field) are those of its workloads, at sizes that a pass of at most about a second allows.
"""
import math

import numpy as np
import torch

from paper_2408_11376_gb300 import FDiRW, FDiRWBatch, FDiRWCoarse, fdirw, surrogate, synth

DEV = "cuda"


def listed():
    return [
        # The smallest call: one macro step of the 32^3 workload from a program's time loop (launches count).
        dict(name="step 32 r3", kind="step", nx=32, ny=32, nz=32, R=3, n_sub=50, prec="fp32", accum="ff", steps=1, mode="two_phase"),
        # The steady state of a large structure with the default precision and accumulation.
        dict(name="step 112 r8 fp32 ff", kind="step", nx=112, ny=112, nz=112, R=8, n_sub=200, prec="fp32", accum="ff", steps=5, mode="two_phase"),
        # The steady state as the benchmark runs it: BF16 kernels, FP32 sums, mass restored every step.
        dict(name="step 112 r8 bf16 fp32", kind="step", nx=112, ny=112, nz=112, R=8, n_sub=200, prec="bf16", accum="fp32", steps=10, mode="two_phase"),
        # The 32^3 workload from create to destroy, default precision: a parameter study over small structures.
        dict(name="job 32 r3", kind="job", nx=32, ny=32, nz=32, R=3, n_sub=50, prec="fp32", accum="ff", steps=2, mode="two_phase"),
        # A ragged box (no axis a multiple of a vector), float-float sums over BF16 kernels, a rough diffusivity.
        dict(name="job ragged r5", kind="job", nx=53, ny=47, nz=61, R=5, n_sub=100, prec="bf16", accum="ff", steps=10, mode="per_sphere"),
        # The 96^3 workload (radius 6, per-sphere contrast), ten steps.
        dict(name="job 96 r6", kind="job", nx=96, ny=96, nz=96, R=6, n_sub=120, prec="bf16", accum="fp32", steps=10, mode="per_sphere"),
        # The benchmark's recipe (radius 8, 200 substeps, 20 steps) on the largest cube of the range.
        dict(name="job 112 r8", kind="job", nx=112, ny=112, nz=112, R=8, n_sub=200, prec="bf16", accum="fp32", steps=20, mode="two_phase"),
        # The plain FP64 path: the accuracy reference that a user checks a cheaper precision against.
        dict(name="job 36 r6 fp64", kind="job", nx=36, ny=36, nz=36, R=6, n_sub=120, prec="fp64", accum="ff", steps=4, mode="two_phase"),
        # Four structures of the batched workload, radii 3 to 10 by the radius rule.
        dict(name="batch 4 r3to10", kind="batch", n=4, side=32, side_step=16, R=10, R_min=3, n_sub=75, prec="bf16", accum="fp32", steps=10, mode="per_sphere"),
        # Convection through the pore space at radius 8 (the substeps raised by a tenth), default precision.
        dict(name="flow 48 r8", kind="flow", nx=48, ny=48, nz=48, R=8, n_sub=220, prec="fp32", accum="ff", steps=4, mode="two_phase"),
        # The paper's production path: coarse mesh, far field, interface exchange and slow solid march.
        dict(name="coupled 96 b5", kind="coupled", nx=96, ny=96, nz=96, R=8, B=5, n_sub=200, n_sub_solid=1, steps=20, mode="two_phase"),
        # Training of the learned kernel: forward, backward and Adam on a batch of 256 kernels.
        dict(name="train 256", kind="train", nx=48, ny=48, nz=48, R=8, n_sub=200, samples=256, mode="per_sphere"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any of the kinds, box sides over their whole range (odd ones and unequal ones among them),
    every radius of the kind, every storage precision and accumulation that it takes."""
    kind = rng.choice(["step", "step", "job", "job", "job", "fp64", "batch", "flow", "coupled", "train"])
    mode = rng.choice(["two_phase", "per_sphere"])
    if kind == "train":
        return dict(kind="train", nx=_log_int(rng, 24, 48), ny=_log_int(rng, 24, 48), nz=_log_int(rng, 24, 48), R=8,
                    n_sub=200, samples=_log_int(rng, 64, 512), mode="per_sphere")
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(2, 5), side=rng.randint(17, 40), side_step=rng.randint(3, 10), R=10,
                    R_min=3, n_sub=rng.randint(50, 75), prec=rng.choice(["fp32", "fp16", "bf16"]),
                    accum=rng.choice(["ff", "fp32"]), steps=rng.randint(1, 10), mode="per_sphere")
    if kind == "coupled":
        B = rng.choice([3, 5])
        return dict(kind="coupled", nx=_log_int(rng, 24, 96), ny=_log_int(rng, 24, 96), nz=_log_int(rng, 24, 96),
                    R=rng.randint(4, 10 - (B - 1) // 2), B=B, n_sub=rng.randint(50, 200), n_sub_solid=rng.randint(1, 4),
                    steps=rng.randint(2, 20), mode="two_phase")
    if kind == "flow":
        return dict(kind="flow", nx=_log_int(rng, 16, 48), ny=_log_int(rng, 16, 48), nz=_log_int(rng, 16, 48),
                    R=rng.randint(3, 10), n_sub=rng.randint(50, 220), prec=rng.choice(["fp32", "bf16"]),
                    accum=rng.choice(["ff", "fp32"]), steps=rng.randint(1, 10), mode="two_phase")
    if kind == "fp64":
        return dict(kind="job", nx=_log_int(rng, 16, 36), ny=_log_int(rng, 16, 36), nz=_log_int(rng, 16, 36),
                    R=rng.randint(3, 8), n_sub=rng.randint(50, 120), prec="fp64", accum="ff", steps=rng.randint(1, 8), mode=mode)
    n = [_log_int(rng, 20, 96) for _ in range(3)]
    if rng.random() < 0.5:
        n[0] = (n[0] + 7) // 8 * 8                    # half of the boxes with aligned rows, as cubes of 32, 48, ... have
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], R=rng.randint(3, 8), n_sub=rng.randint(50, 200),
                prec=rng.choice(["fp32", "fp16", "bf16", "bf16"]), accum=rng.choice(["ff", "fp32"]),
                steps=rng.randint(1, 20), mode=mode)


# ------------------------------------------------------------------------------------------ inputs

def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _packing(shape, mode, seed):
    p = synth.sphere_packing(shape, 0.35 if mode == "per_sphere" else 0.40, seed, r_range=(2.0, min(5.0, min(shape) / 4 + 1)))
    D = synth.diffusivity_per_sphere(p) if mode == "per_sphere" else synth.diffusivity_two_phase(p, 1.0, 1e-6)
    return p, D


def _batch_shapes(case):
    return [(case["side"] + i // 2 * case["side_step"] * (1 + i % 2),) * 3 for i in range(case["n"])]


def _geometries(case, seed):
    shapes = _batch_shapes(case) if case["kind"] == "batch" else [_shape(case)]
    return [(s, *_packing(s, case["mode"], 1000 * seed + 7 + i)) for i, s in enumerate(shapes)]


def _field(packing, seed):
    """1 in solid and 0 in pore, as the workloads start, times a smooth seeded variation of the loading."""
    rng = np.random.default_rng(seed)
    return packing.solid * (1.0 + 0.25 * np.cos(np.arange(packing.solid.size) * 0.01 + rng.uniform(0, 6.28)))


def _velocity(case, packing, seed):
    return synth.face_velocity(_shape(case), seed + 40, (0.03, 0.0, 0.0), 0.03, packing.solid)


def _params(seed):
    return surrogate.init_params(seed)


def _sources(case, seed):
    return np.random.default_rng(seed).integers(0, case["nx"] * case["ny"] * case["nz"], case["samples"])


# The coupled step's kinetics in lattice units: no face moves more than a percent of its liquid cell in a step.
KINETICS = dict(k=1e-7, cS_eq=1.0, cL_eq=1e-5)
LIQUID0, SOLID0 = 2.12e-3, 1e-6
LR = 1e-4


def prepare(case, seed):
    kind = case["kind"]
    geo = _geometries(case, seed)
    st = {"case": case, "shapes": [g[0] for g in geo], "D": [torch.from_numpy(g[2]).to(DEV) for g in geo]}
    shape, D = st["shapes"][0], st["D"][0]
    st["dt"] = min(fdirw.fdirw_stable_dt(s, d) for s, d in zip(st["shapes"], st["D"]))
    if kind == "flow":                                # a tenth more substeps leaves room for the outflow
        st["dt"] *= 10.0 / 11.0
        st["w"] = torch.from_numpy(_velocity(case, geo[0][1], seed).reshape(-1)).to(DEV)
    if kind == "train":
        # Targets: the FD kernels of the batch's sources, as the training set holds them.
        src = _sources(case, seed)
        f = FDiRW(shape, D, case["n_sub"] * st["dt"], 8, case["n_sub"], "fp32")
        f.kernels()
        st.update(ctx=f, net=fdirw.Net(_params(seed)), src=src,
                  targets=torch.from_numpy(f.read_kernels(src).reshape(len(src), -1)).to(DEV))
        return st
    if kind == "coupled":
        liquid = ~geo[0][1].solid
        st["liquid"] = torch.from_numpy(liquid.astype(np.uint8)).to(DEV)
        st["c0"] = torch.from_numpy(np.where(liquid, LIQUID0, SOLID0)).to(DEV)
        st["V_far"] = float(liquid.sum())
    else:
        st["c0"] = torch.from_numpy(np.concatenate([_field(g[1], seed + i) for i, g in enumerate(geo)])).to(DEV)
    if kind == "step":
        st["ctx"] = FDiRW(shape, D, case["n_sub"] * st["dt"], case["R"], case["n_sub"], case["prec"], accum=case["accum"])
        st["ctx"].kernels()
        st["out"] = torch.empty_like(st["c0"])
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "step":
        st["ctx"].step(st["c0"], st["out"], c["steps"])
        return st["out"]
    if kind == "train":
        loss = st["net"].train_step(st["ctx"].ctx, st["src"], st["targets"], LR)
        return {"loss": loss, "params": st["net"].params()}
    dt = c["n_sub"] * st["dt"]
    if kind == "coupled":
        field = st["c0"].clone()
        with FDiRWCoarse(st["shapes"][0], st["D"][0], st["liquid"], c["B"], dt, c["R"], c["n_sub"]) as f:
            f.far_field(st["V_far"], LIQUID0)
            f.kernels()
            QL, QS, c_far = f.coupled_step(field, c["steps"], dt=dt, n_sub_solid=c["n_sub_solid"], **KINETICS)
            pbc = f.read_pbc()
        return {"field": field, "QL": QL, "QS": QS, "c_far": c_far, "pbc": pbc}
    out = torch.empty_like(st["c0"])
    if kind == "batch":
        f = FDiRWBatch(st["shapes"], st["D"], dt, c["R_min"], c["R"], c["n_sub"], c["prec"], accum=c["accum"])
    else:
        f = FDiRW(st["shapes"][0], st["D"][0], dt, c["R"], c["n_sub"], c["prec"], accum=c["accum"])
    with f:
        if kind == "flow":
            f.set_velocity(st["w"])
        f.kernels()
        mass = f.step(st["c0"], out, c["steps"], want_mass=True)
    return {"field": out, "mass": mass}


# ------------------------------------------------------------------------------------------ necessary work

STORE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}


def _window_cells(shape, R):
    """Cells of all clipped windows of a box."""
    total = 1.0
    for n in shape:
        total *= sum(min(x + R, n - 1) - max(x - R, 0) + 1 for x in range(n))
    return total


def work(case):
    """13 flop per cell and substep of a march, 2 per kernel value and macro step; each cell's diffusivity read
    once, its field read and written once, the kernels written once and read once per macro step."""
    kind = case["kind"]
    if kind == "train":
        # four 3^3 convolutions of 16 to 16 channels on 17^3 voxels (the head has one output), forward and twice backward
        mac = 17 ** 3 * 27 * (16 * 16 * 3 + 16)
        return {"bytes": case["samples"] * 17 ** 3 * 10 + 12 * fdirw.NET_NPARAM, "flops": 2 * mac * (2 + 1) * case["samples"]}
    if kind == "batch":
        # a pore share of 0.35 has the largest radius, the solid the smallest one
        shapes = _batch_shapes(case)
        cells = sum(s[0] * s[1] * s[2] for s in shapes)
        win = sum(0.35 * _window_cells(s, case["R"]) + 0.65 * _window_cells(s, case["R_min"]) for s in shapes)
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
        win = _window_cells(_shape(case), case["R"])
    if kind == "coupled":
        B, R = case["B"], case["R"]
        nodes = math.prod(-(-n // B) for n in _shape(case))
        steps = case["steps"]
        # the solid march needs each cell's three face coefficients and its value in and out, per substep
        return {"bytes": cells * (9 + steps * 16 * (2 + case["n_sub_solid"])),
                "flops": 13 * case["n_sub"] * (nodes * (B + 2 * R) ** 3 + cells) + steps * cells * (30 + 13 * case["n_sub_solid"])}
    kernels = win * STORE[case["prec"]]
    if kind == "step":
        return {"bytes": case["steps"] * kernels + 24 * cells, "flops": 2 * win * case["steps"]}
    return {"bytes": (1 + case["steps"]) * kernels + (24 + (24 if kind == "flow" else 0)) * cells,
            "flops": 13 * case["n_sub"] * win + 2 * win * case["steps"]}


# ------------------------------------------------------------------------------------------ the same in 64 bits

def _conductances(D, shape):
    """Harmonic-mean conductance of the +x, +y, +z face of every cell, [3, nz, ny, nx] (0 on the last plane)."""
    nx, ny, nz = shape
    D = D.view(nz, ny, nx)
    g = torch.zeros(3, nz, ny, nx, dtype=torch.float64, device=D.device)
    for a, ax in enumerate((2, 1, 0)):
        n = D.shape[ax] - 1
        lo, hi = D.narrow(ax, 0, n), D.narrow(ax, 1, n)
        s = lo + hi
        g[a].narrow(ax, 0, n).copy_(torch.where(s > 0, 2 * lo * hi / s, torch.zeros_like(s)))
    return g


def _face_sum(g):
    total = g.sum(0)
    for a, ax in enumerate((2, 1, 0)):
        n = g.shape[ax + 1]
        total.narrow(ax, 1, n - 1).add_(g[a].narrow(ax, 0, n - 1))
    return total


def _march(A, B, loss, centres, u, R, n_sub):
    """n_sub substeps of u [S, W, W, W] on the windows of radius R around centres [S, 3] (z, y, x); A and B: what
    crosses each +face upwards and downwards, [3, nz, ny, nx]; loss: what each cell loses outwards, or None."""
    W = 2 * R + 1
    pad = lambda t: torch.nn.functional.pad(t, (R,) * 6)  # noqa: E731
    nz, ny, nx = A.shape[1:]
    o = torch.arange(W, device=A.device)
    off = (o[:, None, None] * (ny + 2 * R) + o[None, :, None]) * (nx + 2 * R) + o[None, None, :]
    at = ((centres[:, 0] * (ny + 2 * R) + centres[:, 1]) * (nx + 2 * R) + centres[:, 2])[:, None, None, None] + off
    take = lambda t: pad(t).reshape(-1)[at]  # noqa: E731
    a = [take(A[i]).narrow(3 - i, 0, W - 1).contiguous() for i in range(3)]
    b = a if B is A else [take(B[i]).narrow(3 - i, 0, W - 1).contiguous() for i in range(3)]
    l = None if loss is None else take(loss)
    for _ in range(n_sub):
        lo = [u.narrow(3 - i, 0, W - 1) for i in range(3)]
        hi = [u.narrow(3 - i, 1, W - 1) for i in range(3)]
        if b is a:
            F = [(lo[i] - hi[i]).mul_(a[i]) for i in range(3)]
        else:
            F = [(lo[i] * a[i]).sub_(hi[i] * b[i]) for i in range(3)]
        if l is not None:
            u = u - l * u
        for i in range(3):
            u.narrow(3 - i, 0, W - 1).sub_(F[i])
            u.narrow(3 - i, 1, W - 1).add_(F[i])
    return u


def _superpose(shape, A, B, R, n_sub, which, fields):
    """Adds what the sources `which` (flat indices) of radius R spread to each field: a list of (field in, padded out)."""
    nx, ny, nz = shape
    W = 2 * R + 1
    o = torch.arange(W, device=A.device)
    off = (o[:, None, None] * (ny + 2 * R) + o[None, :, None]) * (nx + 2 * R) + o[None, None, :]
    for s in which.split(max(1, int(4e7) // W ** 3)):
        zyx = torch.stack((s // (nx * ny), s // nx % ny, s % nx), 1)
        u = torch.zeros(len(s), W, W, W, dtype=torch.float64, device=A.device)
        u[:, R, R, R] = 1
        u = _march(A, B, None, zyx, u, R, n_sub)
        at = ((zyx[:, 0] * (ny + 2 * R) + zyx[:, 1]) * (nx + 2 * R) + zyx[:, 2])[:, None, None, None] + off
        yield s, at, u


def _steps(shape, A, B, radius, n_sub, c, steps):
    """`steps` macro steps of c: every source spreads over its own window (radius: {R: flat indices})."""
    nx, ny, nz = shape
    keep = {R: list(_superpose(shape, A, B, R, n_sub, which, None)) for R, which in radius.items()}
    for _ in range(steps):
        new = torch.zeros(nz, ny, nx, dtype=torch.float64, device=A.device)
        for R, parts in keep.items():
            out = torch.zeros((nz + 2 * R) * (ny + 2 * R) * (nx + 2 * R), dtype=torch.float64, device=A.device)
            for s, at, u in parts:
                out.index_add_(0, at.reshape(-1), (u * c[s][:, None, None, None]).reshape(-1))
            new += out.view(nz + 2 * R, ny + 2 * R, nx + 2 * R)[R:R + nz, R:R + ny, R:R + nx]
        c = new.reshape(-1)
    return c


def exact(case, seed):
    kind = case["kind"]
    shapes = _batch_shapes(case) if kind == "batch" else [_shape(case)]
    if kind in ("step", "job", "flow"):
        cost = _window_cells(shapes[0], case["R"])
        if cost * case["n_sub"] > 2.2e11 or cost > 2e9:
            return None                               # minutes of FP64 marches, or more kernels than fit
    geo = _geometries(case, seed)
    D = [torch.from_numpy(g[2]).to(DEV) for g in geo]
    g = [_conductances(d, s) for d, s in zip(D, shapes)]
    dt = min(1.0 / float(_face_sum(x).max()) for x in g)
    if kind == "train":
        return _exact_train(case, seed, D[0], dt * g[0])
    if kind == "coupled":
        return _exact_coupled(case, geo[0][1], D[0], g[0], dt)
    fields = []
    for i, (s, p, _) in enumerate(geo):
        N = s[0] * s[1] * s[2]
        every = torch.arange(N, device=DEV)
        c = torch.from_numpy(_field(p, seed + i)).to(DEV)
        A = B = dt * g[i]
        if kind == "flow":
            lam = dt * 10.0 / 11.0
            w = torch.from_numpy(_velocity(case, p, seed)).to(DEV).view(3, *g[i].shape[1:])
            inside = torch.zeros_like(w)              # faces of the box carry no flow
            inside[0, :, :, :-1] = inside[1, :, :-1] = inside[2, :-1] = 1
            A, B = lam * g[i] + lam * inside * w.clamp(min=0), lam * g[i] + lam * inside * (-w).clamp(min=0)
        if kind == "batch":
            r = torch.ceil(2 * torch.sqrt(2 * D[i] * (case["n_sub"] * dt))).clamp(case["R_min"], case["R"]).long()
            radius = {int(v): every[r == v] for v in r.unique()}
        else:
            radius = {case["R"]: every}
        fields.append(_steps(s, A, B, radius, case["n_sub"], c, case["steps"]))
    out = torch.cat(fields)
    if kind == "step":
        return out
    return {"field": out, "mass": float(out.sum())}


def _exact_coupled(case, packing, D, g, dt):
    nx, ny, nz = _shape(case)
    B, R, n_sub = case["B"], case["R"], case["n_sub"]
    Rw, Rc = R + (B - 1) // 2, (R + B - 1) // B
    liquid = torch.from_numpy(~packing.solid).to(DEV).view(nz, ny, nx)
    D = D.view(nz, ny, nx)
    both = torch.zeros_like(g)                        # faces between two liquid cells, between two solid ones
    solid = torch.zeros_like(g)
    for a, ax in enumerate((2, 1, 0)):
        n = liquid.shape[ax] - 1
        lo, hi = liquid.narrow(ax, 0, n), liquid.narrow(ax, 1, n)
        both[a].narrow(ax, 0, n).copy_(lo & hi)
        solid[a].narrow(ax, 0, n).copy_(~lo & ~hi)
    A = dt * g * both
    faces = torch.zeros_like(D)
    for ax in range(3):
        faces.narrow(ax, 0, 1).add_(1)
        faces.narrow(ax, faces.shape[ax] - 1, 1).add_(1)
    loss = dt * D * faces * liquid
    # blocks: their liquid counts, each cell's block, the march from the liquid of every block
    nc = [-(-n // B) for n in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*(torch.arange(n, device=DEV) for n in (nz, ny, nx)), indexing="ij")
    block = ((z // B) * nc[1] + y // B) * nc[2] + x // B
    count = torch.zeros(math.prod(nc), dtype=torch.float64, device=DEV).index_add_(0, block[liquid], torch.ones_like(D[liquid]))
    nodes = torch.nonzero(count > 0).flatten()
    W, bh = 2 * Rw + 1, (B - 1) // 2
    pad = lambda t: torch.nn.functional.pad(t, (Rw,  Rw + B) * 3)  # noqa: E731
    lq = pad(liquid.double())
    o = torch.arange(W, device=DEV)
    off = (o[:, None, None] * lq.shape[1] + o[None, :, None]) * lq.shape[2] + o[None, None, :]
    near = ((o - Rw).abs() <= bh).double()
    near = near[:, None, None] * near[None, :, None] * near[None, None, :]
    blk = pad(block + 1).long() - 1                   # the padding belongs to no block
    rows, cols, vals = [], [], []
    grow = lambda t: torch.nn.functional.pad(t, (0, B) * 3)  # noqa: E731  (a clipped block's centre may lie past the box)
    Ap, lp = torch.stack([grow(t) for t in A]), grow(loss)
    for J in nodes.split(max(1, int(4e7) // W ** 3)):
        c = torch.stack((J // (nc[1] * nc[2]), J // nc[2] % nc[1], J % nc[2]), 1) * B + bh
        at = ((c[:, 0] * lq.shape[1] + c[:, 1]) * lq.shape[2] + c[:, 2])[:, None, None, None] + off
        u = _march(Ap, Ap, lp, c, lq.reshape(-1)[at] * near, Rw, n_sub)
        I = blk.reshape(-1)[at].reshape(-1)
        Jx = J[:, None, None, None].expand_as(u).reshape(-1)
        ok = (u.reshape(-1) != 0) & (I >= 0)
        key, inv = torch.unique(I[ok] * len(count) + Jx[ok], return_inverse=True)
        v = torch.zeros(len(key), dtype=torch.float64, device=DEV).index_add_(0, inv, u.reshape(-1)[ok])
        rows.append(key // len(count)), cols.append(key % len(count)), vals.append(v)
    rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    vals = vals / count[rows]

    def flux(u, a):                                   # what the faces a bring each cell
        d = torch.zeros_like(u)
        for i, ax in enumerate((2, 1, 0)):
            n = u.shape[ax] - 1
            F = a[i].narrow(ax, 0, n) * (u.narrow(ax, 0, n) - u.narrow(ax, 1, n))
            d.narrow(ax, 0, n).sub_(F)
            d.narrow(ax, 1, n).add_(F)
        return d

    u = torch.zeros_like(D)
    for _ in range(n_sub):
        u = u + flux(u, A) + loss * (1 - u)
    to_blocks = lambda f: torch.where(count > 0, torch.zeros_like(count).index_add_(0, block[liquid], f[liquid]) / count.clamp(min=1), torch.zeros_like(count))  # noqa: E731
    pbc = to_blocks(u)
    c = torch.where(liquid, LIQUID0, SOLID0).double()
    V, cf, T = float(liquid.sum()), LIQUID0, case["n_sub"] * dt
    k, cS, cL = KINETICS["k"], KINETICS["cS_eq"], KINETICS["cL_eq"]
    QL, QS = [], []
    for _ in range(case["steps"]):
        d = torch.zeros_like(c)
        for ax in (2, 1, 0):
            n = c.shape[ax] - 1
            for l, s in ((0, 1), (1, 0)):
                ok = liquid.narrow(ax, l, n) & ~liquid.narrow(ax, s, n)
                m = ok * k * ((c.narrow(ax, l, n) - cL) / cL).clamp(min=0) * ((cS - c.narrow(ax, s, n)) / cS).clamp(min=0) * T
                d.narrow(ax, l, n).sub_(m)
                d.narrow(ax, s, n).add_(m)
        c = c + d
        for _ in range(case["n_sub_solid"]):
            c = c + T / case["n_sub_solid"] * flux(c, g * solid)
        m0 = c.sum()
        C = to_blocks(c)
        Cn = torch.zeros_like(C).index_add_(0, rows, vals * C[cols]) + pbc * cf
        c = torch.where(liquid, Cn[block], c)
        cf = float((m0 + V * cf - c.sum()) / V)
        QL.append(float(c[liquid].sum())), QS.append(float(c[~liquid].sum()))
    return {"field": c.reshape(-1), "QL": np.array(QL), "QS": np.array(QS), "c_far": cf, "pbc": pbc}


def _exact_train(case, seed, D, A):
    """The loss and the updated parameters of a first Adam step, with no rounding of weights or activations."""
    nx, ny, nz = _shape(case)
    src = torch.from_numpy(_sources(case, seed)).to(DEV)
    n, W = len(src), 17
    zyx = torch.stack((src // (nx * ny), src // nx % ny, src % nx), 1)
    k = torch.zeros(n, W, W, W, dtype=torch.float64, device=DEV)
    k[:, 8, 8, 8] = 1
    k = _march(A, A, None, zyx, k, 8, case["n_sub"])
    o = torch.arange(W, device=DEV) - 8
    p = zyx[:, :, None] + o
    ok = (p >= 0) & (p < torch.tensor([nz, ny, nx], device=DEV)[None, :, None])
    inside = ok[:, 0, :, None, None] & ok[:, 1, None, :, None] & ok[:, 2, None, None, :]
    q = p.clamp(min=0)
    q = torch.minimum(q, torch.tensor([nz - 1, ny - 1, nx - 1], device=DEV)[None, :, None])
    d = D.view(nz, ny, nx)[q[:, 0, :, None, None], q[:, 1, None, :, None], q[:, 2, None, None, :]]
    f = torch.zeros(n, 16, W, W, W, dtype=torch.float64, device=DEV)
    f[:, 0] = torch.where(inside, (torch.log10(d) / 8 + 1).clamp(-0.5, 1.5), torch.zeros_like(d))
    f[:, 1] = inside.double()
    f[:, 2, 8, 8, 8] = 1
    f[:, 3], f[:, 4], f[:, 5] = (o / 8.0)[None, None, :], (o / 8.0)[None, :, None], (o / 8.0)[:, None, None]
    f[:, 6] = (o[:, None, None] ** 2 + o[None, :, None] ** 2 + o[None, None, :] ** 2) / 256.0
    params = torch.from_numpy(_params(seed)).double().to(DEV).requires_grad_()
    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    for b in torch.arange(n, device=DEV).split(32):
        wts, bias = params[:-64].view(4, 27, 16, 16), params[-64:].view(4, 16)
        a = torch.nn.functional.pad(f[b], (1,) * 6)
        for l in range(4):
            z = bias[l][None, :, None, None, None].expand(len(b), 16, W, W, W)
            for t in range(27):                       # tap t = (dx + 1) + 3 (dy + 1) + 9 (dz + 1)
                dx, dy, dz = t % 3, t // 3 % 3, t // 9
                z = z + torch.einsum("ncxyz,oc->noxyz", a[:, :, dz:dz + W, dy:dy + W, dx:dx + W], wts[l, t])
            a = torch.nn.functional.pad(z.relu(), (1,) * 6)
        z, kb = z[:, 0], k[b]
        part = ((z.exp() - kb * z + torch.xlogy(kb, kb) - kb) * inside[b]).sum() / n
        part.backward()
        loss += part.detach()
    grad = params.grad
    frozen = torch.zeros_like(grad, dtype=torch.bool)  # the head has one output: the other 15 stay as they are
    frozen[:-64].view(4, 27, 16, 16)[3, :, 1:] = True
    frozen[-64:].view(4, 16)[3, 1:] = True
    new = torch.where(frozen, params, params - LR * grad / (grad.abs() + 1e-8))
    return {"loss": float(loss), "params": new.detach()}
