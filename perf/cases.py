"""Workloads of the metadynamics bias path, each through its public entry points.

``listed()`` holds the workloads, ``draw(rng)`` gives others of the same
ranges, ``prepare`` makes what a program holds before the call (positions on
the GPU, or page-locked for the host-buffer step; contexts with their hills
loaded), ``run`` is one pass, ``work`` the bytes and operations it cannot do
without, and ``exact`` the same outputs in 64 bits from plain torch.

Positions: half of the box B4 wurtzite GaN with N(0, 0.1 A) disorder, the
other half the same lattice with large random displacements (up to 0.4 A) and
the few vacancies that make the atom count exact, in random caller order.
Frame f of a stretch adds a per-atom random walk and N(0, 0.05 A) thermal
noise.  Hill centres lie within 10 sigma of the CVs, as a run that has filled
its basin leaves them.

A pass returns what the program keeps of it.  Forces are float32, as the
entry points write them.  Contexts with float32 pair arithmetic have their
CVs, bias and box gradient kept as float32 (the digits of a trajectory log);
FP64 contexts and the free-energy passes return float64.
"""
import math

import numpy as np
import torch

from paper_2510_06873_gb300 import autograd, metad

DEV = "cuda" if torch.cuda.is_available() else "cpu"
RC, R0, KB, TEMP, GAMMA = 3.5, 2.5, 0.0083144626, 300.0, 10.0
SIGMA = (0.05, 0.02)       # coordination number, averaged Q6
SIGMA_L = 0.1              # box lengths, Angstrom
CENTRE = (3.13, 0.239)     # CVs of these structures (they vary by a sigma or so with size and seed)
GRID_N, GRID_HALF = 200, 16.0  # bias grid: nodes per axis, half width in sigmas
WURTZITE = (3.19, math.sqrt(3.0) * 3.19, 5.19)

_stream = None


def listed():
    return [
        # one alanine-dipeptide-sized walker, two periodic torsions, a long hill list: the smallest call
        dict(name="torsion_walker", kind="torsion", walkers=1, hills=10000, n_cv=2, fp64=False),
        # 256 such walkers stepped as one batch (multiple-walker metadynamics)
        dict(name="torsion_walkers", kind="torsion", walkers=256, hills=10000, n_cv=2, fp64=False),
        # 32 rutile slab + water systems, the nearest-hydrogen CV, one batch
        dict(name="nearest_walkers", kind="nearest", walkers=32, waters=111, hills=1500, beta=0.0),
        # 1,000 atoms, coordination number, FP64 throughout, CVs and bias read back every step
        dict(name="step_1k_fp64", kind="step", n=1000, n_cv=1, fp64=True, hills=200, grid=False, graph=False,
             frames=1, walk=0.0, read=True),
        # the paper's smallest GaN run, replayed from a captured graph
        dict(name="step_27k_graph", kind="step", n=27648, n_cv=2, fp64=False, hills=1000, grid=False, graph=True,
             frames=4, walk=0.01, read=False),
        # 100,000 atoms, a stretch of trajectory long enough for its list rebuild
        dict(name="step_100k", kind="step", n=100000, n_cv=2, fp64=False, hills=5000, grid=False, graph=False,
             frames=8, walk=0.035, read=False),
        # 1,000,000 atoms, 200 x 200 bias grid and 20,000 live hills, with rebuilds: the largest
        dict(name="step_1m_grid", kind="step", n=1000000, n_cv=2, fp64=False, hills=20000, grid=True, graph=False,
             frames=8, walk=0.035, read=False),
        # 16 walkers of very different sizes in one batched step, CVs and biases read back
        dict(name="walkers_mixed", kind="batch", walkers=16, n_lo=2000, n_hi=100000, hills=1000),
        # NPT: a new box every step, the box lengths as CVs too, box gradient for the barostat
        dict(name="npt_250k", kind="npt", n=250001, hills=5000, strain=1e-3),
        # the MD engine's buffers live in page-locked host memory
        dict(name="host_500k", kind="host", n=500000, hills=5000),
        # the bias as a differentiable torch function, forward and backward
        dict(name="autograd_65537", kind="autograd", n=65537, hills=2000),
        # analysis of a run: sum-of-hills surface and the reweighted one
        dict(name="free_energy", kind="fes", bins0=101, bins1=96, hills=5000, samples=20001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["torsion", "nearest", "step", "step", "step", "batch", "npt", "host", "autograd", "fes"])
    if kind == "torsion":
        return dict(kind=kind, walkers=_log(rng, 1, 256), hills=_log(rng, 100, 10000), n_cv=rng.choice([1, 2]),
                    fp64=rng.random() < 0.25)
    if kind == "nearest":
        return dict(kind=kind, walkers=_log(rng, 1, 32), waters=_log(rng, 30, 400), hills=_log(rng, 100, 3000),
                    beta=rng.choice([0.0, 20.0]))
    if kind == "step":
        n = _log(rng, 1000, 900000)
        n_cv = rng.choice([1, 2])
        return dict(kind=kind, n=n, n_cv=n_cv, fp64=n < 30000 and rng.random() < 0.4, hills=_log(rng, 100, 20000),
                    grid=n_cv == 2 and rng.random() < 0.3, graph=rng.random() < 0.3, frames=rng.choice([1, 4, 8]),
                    walk=0.035, read=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, walkers=_log(rng, 2, 24), n_lo=_log(rng, 1000, 4000), n_hi=_log(rng, 20000, 120000),
                    hills=_log(rng, 100, 5000))
    if kind == "npt":
        return dict(kind=kind, n=_log(rng, 5000, 500000), hills=_log(rng, 100, 10000), strain=rng.choice([3e-4, 1e-3]))
    if kind == "host":
        return dict(kind=kind, n=_log(rng, 5000, 800000), hills=_log(rng, 100, 10000))
    if kind == "autograd":
        return dict(kind=kind, n=_log(rng, 1000, 200000), hills=_log(rng, 100, 5000))
    return dict(kind=kind, bins0=_log(rng, 40, 160), bins1=_log(rng, 40, 160), hills=_log(rng, 300, 8000),
                samples=_log(rng, 1000, 40000))


# ----------------------------------------------------------------- inputs
def _gen(seed, *key):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(np.random.SeedSequence([int(seed), *key]).generate_state(1, dtype=np.uint64)[0] >> 2))
    return g


def _np_rng(seed, *key):
    return np.random.default_rng(np.random.SeedSequence([int(seed), *key]))


def _normal(g, n):
    return torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64)


def _cells_for(n):
    """Wurtzite cells per axis, near cubic, with at least n and few more sites."""
    L = (n * WURTZITE[0] * WURTZITE[1] * WURTZITE[2] / 8.0) ** (1.0 / 3.0)
    best = None
    for ny in range(max(2, round(L / WURTZITE[1]) - 2), max(2, round(L / WURTZITE[1]) + 2) + 1):
        for nz in range(max(2, round(L / WURTZITE[2]) - 2), max(2, round(L / WURTZITE[2]) + 2) + 1):
            nx = max(3, -(-n // (8 * ny * nz)))
            edges = [c * w for c, w in zip((nx, ny, nz), WURTZITE)]
            score = (8 * nx * ny * nz - n) / n + 0.3 * math.log(max(edges) / min(edges))
            if best is None or score < best[0]:
                best = (score, nx, ny, nz)
    return best[1:]


def _structure(n, seed, key):
    """Base positions float64 [n, 3], species float32 [n] and the box."""
    nx, ny, nz = _cells_for(n)
    box = np.array([nx * WURTZITE[0], ny * WURTZITE[1], nz * WURTZITE[2]])
    fa = np.array([[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 1.0 / 6.0, 0.5], [0.0, 2.0 / 3.0, 0.5]])
    frac = torch.tensor(np.concatenate([fa, fa + [0.0, 0.0, 0.375]]) % 1.0, device=DEV)
    ijk = torch.cartesian_prod(*[torch.arange(k, device=DEV) for k in (nx, ny, nz)]).double()
    xyz = ((ijk[:, None, :] + frac[None]) * torch.tensor(WURTZITE, device=DEV, dtype=torch.float64)).reshape(-1, 3)
    species = torch.tensor([0.0] * 4 + [1.0] * 4, device=DEV).repeat(ijk.shape[0])
    g = _gen(seed, key, 1)
    order = torch.randperm(xyz.shape[0], generator=g, device=DEV)
    molten = xyz[order, 0] > 0.5 * box[0]
    extra = xyz.shape[0] - n
    # vacancies: the first `extra` molten sites of the random order
    drop = molten & (torch.cumsum(molten.long(), 0) <= extra)
    order, molten = order[~drop][:n], molten[~drop][:n]
    xyz, species = xyz[order], species[order]
    big = 0.22 * _normal(g, n)
    big *= torch.clamp(0.4 / big.norm(dim=1, keepdim=True).clamp_min(1e-9), max=1.0)
    return xyz + torch.where(molten[:, None], big, 0.1 * _normal(g, n)), species, box


def _wrap(xyz, species, box):
    L = torch.tensor(box, device=DEV, dtype=torch.float64)
    w = (xyz - L * torch.floor(xyz / L)).float()
    w = torch.where(w.double() >= L, torch.zeros_like(w), w)
    return torch.cat([w, species[:, None]], dim=1).contiguous()


def _frames(n, count, walk, seed, key, strain=None):
    """count frames float32 [n, 4] on the GPU and their boxes."""
    xyz, species, box = _structure(n, seed, key)
    g = _gen(seed, key, 2)
    out, boxes = [], []
    for f in range(count):
        if f:
            xyz = xyz + walk * _normal(g, n)
        scale = np.ones(3)
        if strain:
            phase = _np_rng(seed, key, 3).uniform(0.0, 2.0 * math.pi, 3)
            scale = 1.0 + strain * np.sin(2.0 * math.pi * f / 40.0 + phase)
        b = box * scale
        moved = xyz * torch.tensor(scale, device=DEV) + 0.05 * _normal(g, n)
        out.append(_wrap(moved, species, b))
        boxes.append(b)
    return out, boxes


def _hills(count, centre, sigma, seed, key):
    r = _np_rng(seed, key, 4)
    c = np.asarray(centre) + np.asarray(sigma) * r.uniform(-10.0, 10.0, (count, len(centre)))
    return c, r.uniform(0.05, 1.0, count)


def _torsion_inputs(case, seed):
    """Chain molecules of 22 atoms in a 24 A box: float32 [walkers, 22, 4]."""
    W, r = case["walkers"], _np_rng(seed, 11)
    unit = lambda v: v / np.linalg.norm(v, axis=-1, keepdims=True)  # noqa: E731
    xyz = np.zeros((W, 22, 3))
    bond = unit(r.normal(size=(W, 3)))
    for k in range(1, 9):  # backbone: bonds of 1.52 A at 105 to 120 degrees, any torsion
        if k > 1:
            a = np.radians(180.0 - r.uniform(105.0, 120.0, (W, 1)))
            side = unit(np.cross(bond, unit(r.normal(size=(W, 3)))))
            bond = np.cos(a) * bond + np.sin(a) * side
        xyz[:, k] = xyz[:, k - 1] + 1.52 * bond
    for k in range(9, 22):
        host = r.integers(0, 9, W)
        xyz[:, k] = xyz[np.arange(W), host] + r.uniform(1.0, 1.1, (W, 1)) * unit(r.normal(size=(W, 3)))
    xyz = (xyz + r.uniform(0.0, 24.0, (W, 1, 3))) % 24.0
    pos = np.zeros((W, 22, 4), dtype=np.float32)
    pos[..., :3] = np.where(xyz.astype(np.float32) >= 24.0, 0.0, xyz)
    pos[:, 9:, 3] = 2.0
    hills = [(r.uniform(-math.pi, math.pi, (case["hills"], case["n_cv"])), np.full(case["hills"], 1.2))
             for _ in range(W)]
    return pos, hills, [2, 3, 4, 5, 3, 4, 5, 6][: 4 * case["n_cv"]]


def _nearest_inputs(case, seed):
    """A TiO2 slab of 384 atoms under water molecules, one of them near the
    reference oxygen: float32 [walkers, N, 4], box, reference + hydrogens."""
    W, m, r = case["walkers"], case["waters"], _np_rng(seed, 12)
    ijk = np.stack(np.meshgrid(np.arange(4), np.arange(4), np.arange(4), indexing="ij"), -1).reshape(-1, 3)
    u = 0.305
    basis = np.array([[0, 0, 0], [0.5, 0.5, 0.5], [u, u, 0], [1 - u, 1 - u, 0], [0.5 + u, 0.5 - u, 0.5],
                      [0.5 - u, 0.5 + u, 0.5]])
    cell = np.array([2.959, 4.594, 4.594])
    slab = ((ijk[:, None] + basis[None][..., [2, 0, 1]]) * cell).reshape(-1, 3)
    spec = np.tile([0, 0, 1, 1, 1, 1], 64)
    side = cell * 4
    layers = max(1, -(-m // 16))
    box = np.array([side[0], side[1], side[2] + 3.1 * layers + 14.0])
    top = int(np.argmax(np.where(spec == 1, slab[:, 2], -1.0)))
    grid = np.stack(np.meshgrid(np.arange(layers), np.arange(4), np.arange(4), indexing="ij"), -1).reshape(-1, 3)[:m]
    n = 384 + 3 * m
    pos = np.zeros((W, n, 4), dtype=np.float32)
    for w in range(W):
        o = np.stack([(grid[:, 1] + 0.5) * side[0] / 4, (grid[:, 2] + 0.5) * side[1] / 4,
                      side[2] + 4.5 + 3.1 * grid[:, 0]], 1) + r.uniform(-0.15, 0.15, (m, 3))
        d1 = r.normal(size=(m, 3))
        d1 /= np.linalg.norm(d1, axis=1, keepdims=True)
        p = np.cross(d1, r.normal(size=(m, 3)))
        p /= np.linalg.norm(p, axis=1, keepdims=True)
        a = math.radians(104.5)
        h1, h2 = o + 0.96 * d1, o + 0.96 * (math.cos(a) * d1 + math.sin(a) * p)
        shift = slab[top] + [0.0, 0.0, r.uniform(0.9, 3.6)] - h1[0]
        for x in (o, h1, h2):
            x[0] += shift
        xyz = np.concatenate([slab, np.stack([o, h1, h2], 1).reshape(-1, 3)]) + r.normal(0.0, 0.05, (n, 3))
        xyz = (xyz % box).astype(np.float32)
        pos[w, :, :3] = np.where(xyz >= box, 0.0, xyz)
    pos[:, :384, 3] = spec
    pos[:, 384:, 3] = np.tile([1, 2, 2], m)
    hyd = [384 + 3 * k + h for k in range(m) for h in (1, 2)]
    hills = [(r.uniform(0.9, 3.6, (case["hills"], 1)), r.uniform(0.05, 1.0, case["hills"])) for _ in range(W)]
    return pos, box, [top] + hyd, hills


def _inputs(case, seed):
    """Everything random of a case, shared by prepare and exact."""
    k = case["kind"]
    if k == "torsion":
        return _torsion_inputs(case, seed)
    if k == "nearest":
        return _nearest_inputs(case, seed)
    if k == "batch":
        W = case["walkers"]
        sizes = [int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** (w / max(1, W - 1)))) for w in range(W)]
        return [(_frames(n, 1, 0.0, seed, 20 + w), _hills(case["hills"], CENTRE, SIGMA, seed, 20 + w))
                for w, n in enumerate(sizes)]
    if k == "fes":
        r = _np_rng(seed, 13)
        c, w = _hills(case["hills"], CENTRE, SIGMA, seed, 13)
        samples = np.asarray(CENTRE) + np.asarray(SIGMA) * r.normal(0.0, 4.0, (case["samples"], 2))
        return c, w, samples, r.uniform(0.0, 30.0, case["samples"])
    if k == "npt":
        frames, boxes = _frames(case["n"], 2, 0.01, seed, 1, case["strain"])
        centre = (*CENTRE, *_structure_box(case["n"]))
        return frames, boxes, _hills(case["hills"], centre, (*SIGMA, 0.06, 0.06, 0.06), seed, 1)
    n_cv = case.get("n_cv", 2)
    frames, boxes = _frames(case["n"], case.get("frames", 1), case.get("walk", 0.0), seed, 1)
    hills = _hills(case["hills"], CENTRE[:n_cv], SIGMA[:n_cv], seed, 1)
    folded = _hills(20000, CENTRE, SIGMA, seed, 2) if case.get("grid") else None
    return frames, boxes, hills, folded


def _structure_box(n):
    return np.array(_cells_for(n)) * np.array(WURTZITE)


def _grid_range():
    return ([c - GRID_HALF * s for c, s in zip(CENTRE, SIGMA)], [c + GRID_HALF * s for c, s in zip(CENTRE, SIGMA)])


def _fes_range():
    return ([c - 12.0 * s for c, s in zip(CENTRE, SIGMA)], [c + 12.0 * s for c, s in zip(CENTRE, SIGMA)])


# ----------------------------------------------------------------- prepare
def _params(n, box, hills, **kw):
    return metad.params_for(n, box, hill_capacity=max(1, hills) + 64, stream=_stream.cuda_stream, **kw)


def prepare(case, seed):
    global _stream
    if _stream is None:  # torch's work and the contexts' kernels in one stream order
        _stream = torch.cuda.Stream()
    torch.cuda.set_stream(_stream)
    k, inp = case["kind"], _inputs(case, seed)
    st = dict(case=case)
    if k in ("torsion", "nearest"):
        if k == "torsion":
            pos, hills, atoms = inp
            kw = dict(n_cv=case["n_cv"], sigma=(0.35,) * case["n_cv"], w0=1.2, biasfactor=math.inf,
                      cv_kind="torsion", fp64=case["fp64"])
            box = (24.0, 24.0, 24.0)
        else:
            pos, box, atoms, hills = inp
            kw = dict(n_cv=1, sigma=(0.1,), cv_kind="nearest", softmin_beta=case["beta"])
        ctxs = []
        for c, w in hills:
            ctx = metad.Metad(_params(pos.shape[1], box, case["hills"], **kw))
            ctx.set_cv_atoms(atoms)
            ctx.load_hills(c, w)
            ctxs.append(ctx)
        st.update(ctxs=ctxs, pos=[torch.from_numpy(p).to(DEV) for p in pos])
    elif k == "batch":
        st.update(ctxs=[], pos=[])
        for (frames, boxes), (c, w) in inp:
            ctx = metad.Metad(_params(frames[0].shape[0], boxes[0], case["hills"], sigma=SIGMA))
            ctx.load_hills(c, w)
            st["ctxs"].append(ctx)
            st["pos"].append(frames[0])
    elif k == "fes":
        c, w, samples, V = inp
        ctx = metad.Metad(_params(1000, (25.0, 25.0, 25.0), case["hills"], sigma=SIGMA))
        ctx.load_hills(c, w)
        st.update(ctx=ctx, samples=samples, V=V)
    else:
        if k == "npt":
            frames, boxes, hills = inp
            folded = None
            kw = dict(sigma=SIGMA, lattice_cvs=True, sigma_lattice=(SIGMA_L,) * 3)
        else:
            frames, boxes, hills, folded = inp
            n_cv = case.get("n_cv", 2)
            kw = dict(n_cv=n_cv, sigma=SIGMA[:n_cv], fp64=case.get("fp64", False), step_graph=case.get("graph", False))
            if folded:
                kw["grid"] = ((GRID_N, GRID_N), *_grid_range())
        p = _params(case["n"], _structure_box(case["n"]), max(case["hills"], 20000 if folded else 0), **kw)
        ctx = autograd.BiasContext(p) if k == "autograd" else metad.Metad(p)
        if folded:
            ctx.load_hills(*folded)
            ctx.fold_hills()
        ctx.load_hills(*hills)
        st.update(ctx=ctx, pos=frames, boxes=boxes)
        if k == "host":
            st["pos"] = frames[0].cpu().pin_memory().numpy()
            st["forces"] = torch.zeros((case["n"], 3), dtype=torch.float32).pin_memory().numpy()
        elif k == "autograd":
            st["pos"] = frames[0].requires_grad_(True)
        else:
            st["forces"] = torch.zeros((len(frames), case["n"], 3), dtype=torch.float32, device=DEV)
    if "ctxs" in st:
        # one buffer for all walkers' forces, each walker writing its own rows
        st["all_forces"] = torch.zeros((sum(p.shape[0] for p in st["pos"]), 3), dtype=torch.float32, device=DEV)
        st["forces"] = list(torch.split(st["all_forces"], [p.shape[0] for p in st["pos"]]))
        if len(st["ctxs"]) > 1:
            st["batch"] = metad.Batch(st["ctxs"])
    torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    k = case["kind"]
    if k in ("torsion", "nearest", "batch"):
        if "batch" not in state:
            state["ctxs"][0].step(state["pos"][0], state["forces"][0])
            return {"forces": state["all_forces"]}
        state["batch"].step(state["pos"], state["forces"])
        cv, V = state["batch"].read()
        if not case.get("fp64", k == "nearest"):
            cv, V = cv.astype(np.float32), V.astype(np.float32)
        return {"cv": cv, "bias": V, "forces": state["all_forces"]}
    if k == "step":
        ctx, F = state["ctx"], state["forces"]
        rows = []
        for f, pos in enumerate(state["pos"]):
            ctx.step(pos, F[f])
            if case["read"]:
                cv, V, dV = ctx.read_results()
                rows.append(np.concatenate([cv, [V], dV]))
        out = {"forces": F}
        if rows:
            out["results"] = np.array(rows, dtype=np.float64 if case["fp64"] else np.float32)
        return out
    if k == "npt":
        ctx, F, grads = state["ctx"], state["forces"], []
        for f, pos in enumerate(state["pos"]):
            ctx.set_box(state["boxes"][f])
            ctx.step(pos, F[f])
            grads.append(ctx.box_gradient())
        return {"forces": F, "box_gradient": np.array(grads, dtype=np.float32)}
    if k == "host":
        cv, V = state["ctx"].step_host(state["pos"], state["forces"])
        return {"forces": state["forces"], "cv": cv.astype(np.float32), "bias": np.float32(V)}
    if k == "autograd":
        V = autograd.bias(state["pos"], state["ctx"])
        (g,) = torch.autograd.grad(V, state["pos"])
        return {"bias": V.detach().float(), "grad": g}
    ctx, n = state["ctx"], (case["bins0"], case["bins1"])
    lo, hi = _fes_range()
    return {"sum": ctx.fes_grid(lo, hi, n), "reweighted": ctx.fes_reweight(state["samples"], state["V"], lo, hi, n)}


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: positions in, forces out, hills in, once a step.  Operations:
    a hill ~40, a pair ~500 (two CVs) or ~80 (coordination number alone),
    8.5 pairs an atom, ~800 an atom for the averaged Q6."""
    k = case["kind"]
    if k == "torsion":
        W, K, D = case["walkers"], case["hills"], case["n_cv"]
        return dict(bytes=W * (22 * 28 + 8 * (D + 1) * K), flops=W * (40.0 * K + 500 * D))
    if k == "nearest":
        W, K, n = case["walkers"], case["hills"], 384 + 3 * case["waters"]
        return dict(bytes=W * (n * 28 + 16 * K), flops=W * (25.0 * K + 20 * case["waters"]))
    if k == "fes":
        B, K, T = case["bins0"] * case["bins1"], case["hills"], case["samples"]
        # the Gaussians of a regular grid are products of per-axis ones
        return dict(bytes=24 * (K + T) + 16 * B, flops=2.0 * B * K + 25.0 * K * (case["bins0"] + case["bins1"]) + 40.0 * T)
    if k == "batch":
        W = case["walkers"]
        atoms = sum(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** (w / max(1, W - 1))) for w in range(W))
        return dict(bytes=28 * atoms + 24 * case["hills"] * W, flops=5050.0 * atoms + 40.0 * case["hills"] * W)
    steps = case.get("frames", 2 if k == "npt" else 1)
    per_atom = 5050.0 if case.get("n_cv", 2) == 2 else 700.0
    return dict(bytes=steps * (28 * case["n"] + 24 * case["hills"]), flops=steps * (per_atom * case["n"] + 40.0 * case["hills"]))


# ------------------------------------------------------------------- exact
def _pairs(x, box):
    """Unordered pairs (i < j) with minimum-image r^2 < RC^2, in 64 bits."""
    n = x.shape[0]
    L = torch.tensor(box, device=x.device, dtype=torch.float64)

    def near(i, j):
        d = x[j] - x[i]
        d = d - L * torch.round(d / L)
        return (d * d).sum(1) < RC * RC

    nc = torch.floor(L / (RC * 1.0001)).long()
    ids = torch.arange(n, device=x.device)
    if int(nc.min()) < 3:
        i, j = [t.reshape(-1) for t in torch.meshgrid(ids, ids, indexing="ij")]
        keep = (i < j) & near(i, j)
        return i[keep], j[keep]
    c3 = torch.minimum((x / L * nc).long(), nc - 1)
    lin = lambda c: (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]  # noqa: E731
    cell = lin(c3)
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=int(nc.prod()))
    start = torch.cumsum(count, 0) - count
    got = []
    for o in torch.cartesian_prod(*[torch.tensor([-1, 0, 1], device=x.device)] * 3):
        other = lin((c3 + o) % nc)
        for s in range(int(count.max())):
            i = ids[s < count[other]]
            j = order[start[other[i]] + s]
            keep = i < j
            i, j = i[keep], j[keep]
            keep = near(i, j)
            got.append(torch.stack([i[keep], j[keep]]))
    return torch.cat(got, 1)


def _cvs(x, species, box, strain, n_cv):
    """The CVs of positions x (a leaf) in a box strained by 1 + strain."""
    i, j = _pairs(x.detach(), box)
    L = torch.tensor(box, device=x.device, dtype=torch.float64)
    d = x[j] - x[i]
    d = (d - L * torch.round(d.detach() / L)) * (1.0 + strain)
    r = torch.sqrt((d * d).sum(1))
    sc = 1.0 / (1.0 + (RC / R0) ** 6)
    w = (1.0 / (1.0 + (r / R0) ** 6) - sc) / (1.0 - sc)
    n = x.shape[0]
    s = [2.0 * (w * (species[i] != species[j])).sum() / n]
    if n_cv == 2:
        u = d / r[:, None]
        p6 = np.polynomial.Polynomial(np.polynomial.legendre.leg2poly([0] * 6 + [1]))
        Y, K, cs = [], [], (torch.ones_like(r), torch.zeros_like(r))
        for m in range(7):  # d^m P6 / dz^m times the real and imaginary part of (x + iy)^m
            pm = sum(float(a) * u[:, 2] ** k for k, a in enumerate((p6.deriv(m) if m else p6).coef))
            k2 = (2.0 if m else 1.0) * math.factorial(6 - m) / math.factorial(6 + m)
            for part in (cs if m else cs[:1]):
                Y.append(pm * part)
                K.append(k2)
            cs = (u[:, 0] * cs[0] - u[:, 1] * cs[1], u[:, 0] * cs[1] + u[:, 1] * cs[0])
        wy = w[:, None] * torch.stack(Y, 1)
        zero = torch.zeros((n, 13), device=x.device, dtype=torch.float64)
        W = zero[:, 0].index_add(0, i, w).index_add(0, j, w)
        q = zero.index_add(0, i, wy).index_add(0, j, wy) / torch.where(W > 0, W, torch.ones_like(W))[:, None]
        qa = (q + zero.index_add(0, i, w[:, None] * q[j]).index_add(0, j, w[:, None] * q[i])) / (1.0 + W)[:, None]
        s.append(torch.sqrt((qa * qa * torch.tensor(K, device=x.device, dtype=torch.float64)).sum(1)).mean())
    return s


def _gauss(s, hills, sigma, period=None):
    c, w = (torch.as_tensor(a, device=s.device) for a in hills)
    d = s - c
    if period:
        d = d - period * torch.round(d.detach() / period)
    return (w * torch.exp(-(d * d / (2.0 * torch.tensor(sigma, device=s.device, dtype=torch.float64) ** 2)).sum(-1))).sum()


def _grid_bias(s, hills):
    """Bicubic Hermite patch of the folded hills' exact node values."""
    lo, hi = _grid_range()
    V, cell, t, h = 0.0, [], [], []
    for a in range(2):
        h.append((hi[a] - lo[a]) / (GRID_N - 1))
        k = min(max(int(math.floor((float(s[a]) - lo[a]) / h[a])), 0), GRID_N - 2)
        if not lo[a] <= float(s[a]) <= hi[a]:
            return 0.0 * s.sum()
        cell.append(k)
        t.append((s[a] - (lo[a] + k * h[a])) / h[a])
    A = [(2 * u**3 - 3 * u**2 + 1, 3 * u**2 - 2 * u**3) for u in t]
    B = [(u**3 - 2 * u**2 + u, u**3 - u**2) for u in t]
    c, w = hills
    for a in range(2):
        for b in range(2):
            x = np.array([lo[0] + (cell[0] + a) * h[0], lo[1] + (cell[1] + b) * h[1]])
            d = x - c
            g = w * np.exp(-(d * d / (2.0 * np.square(SIGMA))).sum(1))
            e = d / np.square(SIGMA)
            f, f0, f1, f01 = g.sum(), -(g * e[:, 0]).sum(), -(g * e[:, 1]).sum(), (g * e[:, 0] * e[:, 1]).sum()
            V = V + (A[0][a] * A[1][b] * f + B[0][a] * A[1][b] * h[0] * f0 + A[0][a] * B[1][b] * h[1] * f1
                     + B[0][a] * B[1][b] * h[0] * h[1] * f01)
    return V


def _bias_step(frame, box, hills, n_cv=2, folded=None, lattice=False):
    """(s, V, dV/ds, forces, dV/dL) of one frame, in 64 bits."""
    x = frame[:, :3].detach().double().requires_grad_(True)
    strain = torch.zeros(3, device=x.device, dtype=torch.float64, requires_grad=True)
    s = _cvs(x, frame[:, 3].detach(), box, strain, n_cv)
    sigma = SIGMA[:n_cv]
    if lattice:
        s += list(torch.tensor(box, device=x.device, dtype=torch.float64) * (1.0 + strain))
        sigma = (*SIGMA, SIGMA_L, SIGMA_L, SIGMA_L)
    s = torch.stack(s)
    V = _gauss(s, hills, sigma)
    if folded:
        V = V + _grid_bias(s, folded)
    gs, gx, ge = torch.autograd.grad(V, [s, x, strain])
    return s.detach(), V.detach(), gs, -gx, ge / torch.tensor(box, device=x.device, dtype=torch.float64)


def _torsions(x, atoms, L):
    out = []
    for k in range(0, len(atoms), 4):
        b = [x[atoms[k + m + 1]] - x[atoms[k + m]] for m in range(3)]
        b = [v - L * torch.round(v.detach() / L) for v in b]
        n1, n2 = torch.linalg.cross(b[0], b[1]), torch.linalg.cross(b[1], b[2])
        out.append(torch.atan2(torch.linalg.norm(b[1]) * (b[0] * n2).sum(), (n1 * n2).sum()))
    return torch.stack(out)


def exact(case, seed):
    k, inp = case["kind"], _inputs(case, seed)
    num = lambda t: t.cpu().numpy()  # noqa: E731
    if k in ("torsion", "nearest"):
        if k == "torsion":
            pos, hills, atoms = inp
        else:
            pos, box, atoms, hills = inp
        cvs, Vs, Fs = [], [], []
        for p, h in zip(pos, hills):
            x = torch.tensor(p[:, :3], dtype=torch.float64, requires_grad=True)
            if k == "torsion":
                s = _torsions(x, atoms, 24.0)
                V = _gauss(s, h, (0.35,) * case["n_cv"], 2.0 * math.pi)
            else:
                d = x[atoms[1:]] - x[atoms[0]]
                L = torch.tensor(box)
                r = torch.sqrt(((d - L * torch.round(d.detach() / L)) ** 2).sum(1))
                lowest = r.min()
                if case["beta"] > 0:
                    lowest = -torch.logsumexp(-case["beta"] * (r - lowest.detach()), 0) / case["beta"] + lowest.detach()
                s = lowest[None]
                V = _gauss(s, h, (0.1,))
            (g,) = torch.autograd.grad(V, x)
            cvs.append(np.pad(num(s.detach()), (0, 2 - s.numel())))
            Vs.append(float(V))
            Fs.append(-g)
        out = {} if len(pos) == 1 else {"cv": np.array(cvs), "bias": np.array(Vs)}
        return {**out, "forces": torch.cat(Fs)}
    if k == "batch":
        got = [_bias_step(fr[0], bx[0], h) for (fr, bx), h in inp]
        return {"cv": np.stack([num(g[0]) for g in got]), "bias": np.array([float(g[1]) for g in got]),
                "forces": torch.cat([g[3] for g in got])}
    if k == "step":
        frames, boxes, hills, folded = inp
        got = [_bias_step(f, b, hills, case["n_cv"], folded) for f, b in zip(frames, boxes)]
        out = {"forces": torch.stack([g[3] for g in got])}
        if case["read"]:
            out["results"] = np.stack([np.concatenate([num(g[0]), [float(g[1])], num(g[2])]) for g in got])
        return out
    if k == "npt":
        frames, boxes, hills = inp
        got = [_bias_step(f, b, hills, lattice=True) for f, b in zip(frames, boxes)]
        return {"forces": torch.stack([g[3] for g in got]), "box_gradient": np.stack([num(g[4]) for g in got])}
    if k in ("host", "autograd"):
        frames, boxes, hills, _ = inp
        s, V, _, F, _ = _bias_step(frames[0], boxes[0], hills)
        if k == "host":
            return {"forces": num(F), "cv": num(s), "bias": np.float64(float(V))}
        return {"bias": V, "grad": torch.cat([-F, torch.zeros_like(F[:, :1])], 1)}
    c, w, samples, V = inp
    lo, hi, n = *_fes_range(), (case["bins0"], case["bins1"])
    axes = [lo[d] + (np.arange(n[d]) + 0.5) * ((hi[d] - lo[d]) / n[d]) for d in range(2)]
    ex = [np.exp(-np.square(axes[d][:, None] - c[None, :, d]) / (2.0 * SIGMA[d] ** 2)) for d in range(2)]
    F = -(GAMMA / (GAMMA - 1.0)) * ((ex[0] * w) @ ex[1].T)
    idx = [np.floor((samples[:, d] - lo[d]) / ((hi[d] - lo[d]) / n[d])).astype(int) for d in range(2)]
    inside = np.all([(samples[:, d] >= lo[d]) & (samples[:, d] < hi[d]) & (idx[d] < n[d]) for d in range(2)], axis=0)
    beta = 1.0 / (KB * TEMP)
    acc = np.bincount(idx[0][inside] * n[1] + idx[1][inside], np.exp(beta * (V[inside] - V.max())), n[0] * n[1])
    with np.errstate(divide="ignore"):
        R = -np.log(acc / acc.sum()) / beta
    return {"sum": F - F.min(), "reweighted": (R - R.min()).reshape(n)}
