"""Performance cases: what a user of the library has it do, call by call.

Each case goes through the public Python binding (``paper_1609_09833_gb300.abp``,
one function per C entry point) with inputs made from a seed. Every grid that
a program could have resumed starts from a smooth bias of a few kJ/mol
(``abp_grid_restore``), as a run does that continues from a checkpoint, so
that every look-up and force is non-zero from the first step.

Kinds:
  engine   a host MD engine's step: abp_step on this step's coordinates, then
           abp_forces adds the bias force to the engine's force array
  md       abp_md_run: closed-loop MD steps of walkers on their own grids
  md64     the same in FP64 (one long walker on a double well)
  replay   abp_run over recorded frames (COM distance + dihedral; reweighting
           or seeding a bias from an existing trajectory)
  rmsd     abp_run over frames of the paper's setup: two RMSD CVs, mABP with a
           compact hill every step on a 480 x 480 grid over [0, 12] nm
  pocket   abp_run over frames of ligand / pocket walkers with coordination
           numbers, grids of one to three CVs in one batch
  shared   abp_md_run of walkers that share one 3D grid, a coordination number
           over thousands of environment atoms each
  serve    the step server: a backlog of single-step requests from host memory
  fes      a chunk of recorded frames, then every walker's bias grid read back
           to the host (the free-energy estimate written at a checkpoint)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1609_09833_gb300 import abp, synth

OVER, ACC = abp.ABP_FORCES_OVERWRITE, abp.ABP_FORCES_ACCUMULATE
DEV = "cuda"
FRAMES_ENGINE = 8  # the frames an engine's calls cycle through


def listed():
    return [
        # the smallest call: one simulation of an MD engine, one bias step
        {"name": "engine_1", "kind": "engine", "walkers": 1, "cvs": "sweep"},
        # a small ensemble of ligand / pocket simulations, one bias step
        {"name": "engine_pocket_16", "kind": "engine", "walkers": 16, "cvs": "pocket", "ligand": 40, "pocket": 400},
        # one closed-loop MD step of 64 walkers per call (coupled to a host loop)
        {"name": "md_64x1", "kind": "md", "walkers": 64, "steps": 1, "side": 256},
        # the production run: 64 walkers, 1000 closed-loop steps per call
        {"name": "md_64x1000", "kind": "md", "walkers": 64, "steps": 1000, "side": 256},
        # one FP64 walker on the double well (the reference-quality run)
        {"name": "md_fp64_1x1000", "kind": "md64", "walkers": 1, "steps": 1000, "nodes": 512},
        # recorded trajectories of 64 walkers
        {"name": "replay_64x1000", "kind": "replay", "walkers": 64, "steps": 1000, "side": 256, "fp64": False},
        # the paper's ligand setup
        {"name": "rmsd_mabp_64x1000", "kind": "rmsd", "walkers": 64, "steps": 1000, "side": 480},
        # the uneven batch of ligand / pocket walkers
        {"name": "pocket_1000x25", "kind": "pocket", "walkers": 1000, "steps": 25, "ligand": 40, "pocket": 400},
        # a few walkers with a larger ligand and odd sizes
        {"name": "pocket_3x101_odd", "kind": "pocket", "walkers": 3, "steps": 101, "ligand": 53, "pocket": 307},
        # multiple walkers on one shared 256^3 grid
        {"name": "shared_32x10", "kind": "shared", "walkers": 32, "steps": 10, "side": 256, "ligand": 200,
         "env": 10000},
        # a served backlog, eight steps of 512 simulations
        {"name": "serve_512x8", "kind": "serve", "sims": 512, "depth": 8},
        # a checkpoint: 50 steps, then 16 bias grids to the host
        {"name": "fes_16x50", "kind": "fes", "walkers": 16, "steps": 50, "side": 256},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["engine", "engine", "md", "md", "md64", "replay", "rmsd", "pocket", "pocket", "shared",
                       "serve", "fes"])
    if kind == "engine":
        if rng.random() < 0.5:
            return {"kind": kind, "walkers": _log(rng, 1, 128), "cvs": "sweep"}
        return {"kind": kind, "walkers": _log(rng, 1, 128), "cvs": "pocket", "ligand": rng.randint(5, 60),
                "pocket": rng.randint(50, 440)}
    if kind == "md":
        return {"kind": kind, "walkers": _log(rng, 1, 128), "steps": _log(rng, 1, 400), "side": rng.randint(64, 300)}
    if kind == "md64":
        return {"kind": kind, "walkers": _log(rng, 1, 8), "steps": _log(rng, 1, 1000), "nodes": rng.randint(200, 1024)}
    if kind == "replay":
        return {"kind": kind, "walkers": _log(rng, 1, 96), "steps": _log(rng, 1, 600), "side": rng.randint(64, 300),
                "fp64": rng.random() < 0.25}
    if kind == "rmsd":
        return {"kind": kind, "walkers": _log(rng, 1, 64), "steps": _log(rng, 1, 1000), "side": rng.randint(240, 480)}
    if kind == "pocket":
        n = _log(rng, 1, 1000)
        return {"kind": kind, "walkers": n, "steps": _log(rng, 1, max(1, min(100, 25000 // n))),
                "ligand": rng.randint(5, 40 if n > 100 else 60), "pocket": rng.randint(50, 400)}
    if kind == "shared":
        return {"kind": kind, "walkers": _log(rng, 2, 32), "steps": rng.randint(1, 10), "side": rng.randint(48, 256),
                "ligand": rng.randint(16, 200), "env": _log(rng, 500, 10000)}
    if kind == "serve":
        return {"kind": kind, "sims": _log(rng, 16, 512), "depth": rng.randint(1, 8)}
    return {"kind": kind, "walkers": _log(rng, 1, 16), "steps": _log(rng, 1, 100), "side": rng.randint(64, 256)}


# ---------------------------------------------------------------- the workloads' walkers and inputs


def _pocket_specs(case, seed):
    """Ligand / pocket walkers: 40 % one CV (coordination number, 1024
    nodes), 50 % two (COM distance, CN; 128^2 to 512^2), 10 % three (COM
    distance, ligand dihedral, CN; 64^3); the CN axis scaled with the pairs."""
    nl, npk = case["ligand"], case["pocket"]
    f = nl * npk / 16000.0
    r = np.random.default_rng(seed + 5)
    lo, hi = synth.CN_RANGE_UNEVEN[0] * f, synth.CN_RANGE_UNEVEN[1] * f
    lig, poc = np.arange(nl), np.arange(nl, nl + npk)
    cn = {"type": "coord", "a": lig, "b": poc, "r0": 0.4, "n": 6, "m": 12}
    dist = {"type": "com_dist", "a": lig, "b": poc}
    dih = {"type": "dihedral", "a": np.arange(0, 4)}
    specs = []
    for i in range(case["walkers"]):
        q = (i * 7) % 10  # the kinds in fixed proportions, interleaved
        if q < 4:
            g, cvs = synth.grid((lo,), (hi,), (1024,), (False,)), [cn]
        elif q < 9:
            side = int(r.choice((128, 256, 512)))
            g, cvs = synth.grid((0.0, lo), (2.0, hi), (side, side), (False, False)), [dist, cn]
        else:
            g = synth.grid((0.0, -math.pi, lo), (2.0, math.pi, hi), (64,) * 3, (False, True, False))
            cvs = [dist, dih, cn]
        sig = [synth.bins(g, k, 2.0) for k in range(len(cvs))]
        specs.append({"natoms": nl + npk, "cvs": cvs, "grid": g, "hill": synth.hill(0.5, sig, 50, 15.0)})
    return specs


def _specs(case, seed):
    kind = case["kind"]
    if kind == "engine":
        return synth.mb64_specs(nw=case["walkers"]) if case["cvs"] == "sweep" else _pocket_specs(case, seed)
    if kind in ("md", "replay", "fes"):
        # a hill of about the same nodes on every grid size
        n = case["side"]
        sig = (0.04 * 256 / n, 0.1 * 256 / n)
        return synth.mb64_specs(nw=case["walkers"], n=(n, n), sigma=sig)
    if kind == "md64":
        return [synth.double_well_com_spec(n=case["nodes"]) for _ in range(case["walkers"])]
    if kind == "rmsd":
        return synth.paper_rmsd_specs(nw=case["walkers"], n=case["side"], seed=seed + 11)
    if kind == "pocket":
        return _pocket_specs(case, seed)
    if kind == "shared":
        f = case["ligand"] * case["env"] / 2.0e6
        lo, hi = synth.CN_RANGE_SHARED
        return synth.shared256_specs(nw=case["walkers"], n=case["side"], n_lig=case["ligand"], n_env=case["env"],
                                     cn_range=(lo * f, hi * f))
    return synth.serve_specs(61, nsim=case["sims"])  # the same simulations, other coordinates


def _jitter(templates, T, seed):
    """[T, atoms, 4] float32 records on the GPU: templates + N(0, 0.02^2)."""
    t = torch.as_tensor(np.concatenate(templates), dtype=torch.float32, device=DEV)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    rec = torch.zeros(T, t.shape[0], 4, device=DEV)
    for k in range(T):
        rec[k, :, :3] = t + 0.02 * torch.randn(t.shape, generator=g, device=DEV)
    return rec


def _frames(case, seed, specs):
    """The case's coordinate records on the GPU ([T, atoms, 4])."""
    kind, nw = case["kind"], case.get("walkers")
    if kind == "engine" and case["cvs"] == "sweep":
        fr = synth.SweepFrames(nw, seed=seed + 3).frames(0, FRAMES_ENGINE)
    elif kind == "md":
        fr = synth.SweepFrames(nw, seed=seed + 3).frames(0, 1)
    elif kind in ("replay", "fes"):
        fr = synth.SweepFrames(nw, seed=seed + 3).frames(0, case["steps"])
        if case.get("fp64"):
            fr = fr.astype(np.float64)
    elif kind == "md64":
        fr = np.concatenate([synth.double_well_com_coords(seed * 131 + i) for i in range(nw)])[None]
    elif kind == "rmsd":
        fr = synth.RmsdFrames(specs, seed=seed + 41).frames(0, case["steps"])
    elif kind == "shared":
        tm = synth.shared256_templates(seed + 41, nw=nw, n_lig=case["ligand"], n_env=case["env"])
        return _jitter(tm, 1, seed + 42)
    else:  # pocket walkers
        tm = synth.uneven1000_templates(seed + 31, nw=nw, n_lig=case["ligand"], n_pocket=case["pocket"])
        return _jitter(tm, FRAMES_ENGINE if kind == "engine" else case["steps"], seed + 32)
    rec = torch.zeros(fr.shape[:2] + (4,), dtype=torch.as_tensor(fr).dtype, device=DEV)
    rec[..., :3] = torch.as_tensor(fr, device=DEV)
    return rec


def _start_bias(spec, i, seed):
    """Amplitude and per-axis phases of walker i's starting bias
    A (1 + prod_k cos(2 pi j_k / n_k + phi_k)), j the node index."""
    r = np.random.default_rng((seed * 1_000_003 + i * 17 + 1) & 0x7FFFFFFF)
    A = 2000.0 * (0.5 + r.random()) if spec["hill"].get("method") == "mabp" else 4.0 * (0.5 + r.random())
    return A, r.uniform(0, 2 * math.pi, size=len(spec["grid"]["n"]))


def _spacing(g):
    return [(g["hi"][k] - g["lo"][k]) / (g["n"][k] if g["periodic"][k] else g["n"][k] - 1) for k in range(len(g["n"]))]


def _start_field(spec, i, seed):
    """The starting bias on the grid: list of 1 + d float64 fields [nodes], axis 0 fastest."""
    g = spec["grid"]
    d, D = len(g["n"]), _spacing(g)
    A, phi = _start_bias(spec, i, seed)
    c, s = [], []
    for k in range(d):
        th = 2 * math.pi * torch.arange(g["n"][k], dtype=torch.float64, device=DEV) / g["n"][k] + float(phi[k])
        c.append(torch.cos(th))
        s.append(-torch.sin(th) * (2 * math.pi / (g["n"][k] * D[k])))

    def outer(v):
        out = v[d - 1]
        for k in range(d - 2, -1, -1):
            out = (out[..., None] * v[k]).contiguous()
        return out.reshape(-1)

    fields = [A * (1.0 + outer(c))]
    for k in range(d):
        fields.append(A * outer([s[q] if q == k else c[q] for q in range(d)]))
    return fields


def _records(fields, fp64):
    """Node records as abp_grid_save stores them (device tensor)."""
    d, n = len(fields) - 1, fields[0].shape[0]
    w = 2 if d == 1 else 4
    f = torch.zeros(n, w, dtype=torch.float64, device=DEV)
    for q in range(1 + d):
        f[:, q] = fields[q]
    if fp64:
        return f
    hi = f.to(torch.float32)
    return torch.cat([hi, (f - hi.double()).to(torch.float32)], dim=1)


def _restore(ctx, walkers, specs, seed, fp64=False):
    done = set()
    for i, (w, sp) in enumerate(zip(walkers, specs)):
        if w.grid in done:
            continue
        done.add(w.grid)
        fields = _start_field(sp, i, seed)
        rec = _records(fields, fp64)
        if sp.get("shared"):  # the FP64 accumulator follows the records
            sh = torch.zeros(fields[0].shape[0], 4, dtype=torch.float64, device=DEV)
            for q in range(len(fields)):
                sh[:, q] = fields[q]
            rec = torch.cat([rec.reshape(-1).view(torch.uint8), sh.reshape(-1).view(torch.uint8)])
        torch.cuda.current_stream().synchronize()
        abp._check(abp.load().abp_grid_restore(ctx.handle, w.grid, rec.data_ptr(), 1))


class State:
    """What the program holds: context, walkers, buffers, the MD step."""

    def __init__(self, case):
        self.case, self.step, self.srv = case, 0, None
        self.ctx = abp.Context(torch.cuda.current_device(), budget=0)

    def __del__(self):
        try:
            if self.srv:
                abp.abp_server_destroy(self.srv)
            torch.cuda.synchronize()
            self.ctx.close()
        except Exception:
            pass


def _md(case, seed):
    if case["kind"] == "md":
        return synth.md_muller_brown(seed=seed + 2024)
    if case["kind"] == "md64":
        return synth.md_double_well(seed=seed + 7)
    return synth.md_params(seed=seed + 43, mu=0.05)


def prepare(case, seed):
    st = State(case)
    kind = case["kind"]
    specs = _specs(case, seed)
    if kind == "serve":
        st.srv = abp.abp_server_create(st.ctx.handle, max_batch=4096, max_atoms=256, nstreams=2)
        sims = []
        for sp in specs:
            desc, keep = abp.walker_desc(sp)
            sims.append(abp.abp_server_admit(st.srv, abp.grid_desc(sp["grid"]), desc))
            del keep
        st.coords, st.order = _serve_inputs(case, seed, specs)
        st.sims = np.array([sims[i] for i in st.order], dtype=np.int64)
        st.steps = np.repeat(np.arange(case["depth"], dtype=np.int64), case["sims"])
        st.forces = np.zeros_like(st.coords)
        return st
    fp64 = kind == "md64" or bool(case.get("fp64"))
    prec = abp.ABP_PREC_FP64 if fp64 else abp.ABP_PREC_FP32_COMP
    st.dtype = abp.ABP_F64 if fp64 else abp.ABP_F32
    st.walkers = st.ctx.make_walkers(specs, precision=prec)
    _restore(st.ctx, st.walkers, specs, seed, fp64)
    st.wa = abp.walker_array(st.walkers)
    st.offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device=DEV)
    x = _frames(case, seed, specs)
    st.atoms = x.shape[1]
    if kind in ("md", "md64", "shared"):
        st.x = x[0].contiguous()
        st.md = abp.md_desc(_md(case, seed))
        st.streams = np.arange(case["walkers"], dtype=np.uint32)
    elif kind == "engine":
        st.frames = x
        st.forces = _engine_forces(case, seed, st.atoms)
    else:
        st.frames = x
        st.forces = torch.zeros_like(x)
    return st


def _engine_forces(case, seed, atoms):
    """The engine's own MD forces of the step, which the bias force is added to."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 77)
    F = torch.zeros(atoms, 4, device=DEV)
    F[:, :3] = 10.0 * torch.randn(atoms, 3, generator=g, device=DEV)
    return F


def _serve_inputs(case, seed, specs):
    """Packed request coordinates (step by step, every simulation once per
    step) and the simulation index of each request."""
    r = np.random.default_rng(seed + 62)
    tmpl = synth.serve_templates(seed, specs)
    t = np.concatenate(tmpl).astype(np.float32)
    x = np.zeros((case["depth"], t.shape[0], 4), dtype=np.float32)
    x[..., :3] = t[None] + 0.02 * r.standard_normal((case["depth"],) + t.shape, dtype=np.float32)
    return np.ascontiguousarray(x.reshape(-1, 4)), np.tile(np.arange(case["sims"]), case["depth"])


def run(st):
    case, ctx = st.case, st.ctx
    kind = case["kind"]
    if kind == "engine":
        x = st.frames[st.step % FRAMES_ENGINE]
        abp.abp_step(ctx.handle, st.wa, x, abp.ABP_F32, st.offs, st.step)
        abp.abp_forces(ctx.handle, st.wa, st.forces, abp.ABP_F32, st.offs, ACC)
        st.step += 1
        return st.forces
    if kind in ("md", "md64", "shared"):
        abp.abp_md_run(ctx.handle, st.wa, st.x, st.dtype, st.offs, st.md, st.streams, step0=st.step,
                       nsteps=case["steps"])
        st.step += case["steps"]
        return st.x
    if kind == "serve":
        n = len(st.sims)
        abp.abp_server_submit_many(st.srv, st.sims, st.steps, st.coords, st.forces)
        got = 0
        while got < n:
            got += len(abp.abp_server_poll(st.srv, n, wait_ms=50))
        st.steps += case["depth"]
        return st.forces
    abp.abp_run(ctx.handle, st.wa, st.frames, st.dtype, st.offs, st.atoms, st.forces, st.offs, st.atoms, OVER,
                st.step, case["steps"])
    st.step += case["steps"]
    if kind == "fes":
        return [st.forces] + [ctx.bias(w, abp.ABP_F32) for w in st.walkers]
    return st.forces


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    kind = case["kind"]
    specs = _specs(case, 1)
    steps = {"engine": 1, "serve": case.get("depth")}.get(kind, case.get("steps"))
    nbytes = flops = 0.0
    for sp in specs:
        g, h = sp["grid"], sp["hill"]
        d, D = len(g["n"]), _spacing(g)
        rsz = 32 if kind == "md64" or case.get("fp64") else 16
        node = (1 + d) * 8
        width = h["a"] if h.get("method") == "mabp" else [h["cutoff"] * s for s in h["sigma"]]
        box = 1.0
        for k in range(d):
            box *= 2 * math.ceil(width[k] / D[k]) + 1
        closed = kind in ("md", "md64", "shared")
        nbytes += sp["natoms"] * rsz * 2.0 * (1 if closed else steps)
        nbytes += steps * (1 if h.get("method") == "mabp" else 2 ** d) * node + steps / h["stride"] * box * node * 2
        flops += steps * (60.0 * d + sp["natoms"] * 30.0) + steps / h["stride"] * box * (1 + d) * 8
        for cv in sp["cvs"]:
            if cv["type"] == "coord":
                flops += steps * float(len(cv["a"])) * len(cv["b"]) * (35.0 if cv.get("pbc") else 29.0)
        if kind == "fes":
            nbytes += float(np.prod(g["n"])) * (1 + d) * 16
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits


def _min_image(v, cv):
    if not cv.get("pbc"):
        return v
    L = torch.tensor(cv["box"], dtype=v.dtype, device=v.device)
    return v - L * torch.floor(v / L + 0.5)


def _cv(cv, x):
    """One CV of x [B, atoms, 3]: values [B], gradient [B, atoms, 3]."""
    B = x.shape[0]
    grad = torch.zeros_like(x)
    ia = torch.as_tensor(np.asarray(cv["a"]), device=x.device, dtype=torch.long)
    if cv["type"] == "rmsd":
        diff = x[:, ia] - torch.as_tensor(np.asarray(cv["ref"], dtype=np.float64), device=x.device)
        s = torch.sqrt((diff ** 2).sum((1, 2)) / len(ia) + 0.01)
        grad[:, ia] = diff / (len(ia) * s)[:, None, None]
        return s, grad
    if cv["type"] == "dihedral":
        p = x[:, ia]
        b1, b2, b3 = (_min_image(p[:, q + 1] - p[:, q], cv) for q in range(3))
        m, n = torch.cross(b1, b2, dim=1), torch.cross(b2, b3, dim=1)
        l2 = b2.norm(dim=1)
        s = torch.atan2(l2 * (b1 * n).sum(1), (m * n).sum(1))
        g1 = -(l2 / (m * m).sum(1))[:, None] * m
        g4 = (l2 / (n * n).sum(1))[:, None] * n
        u, r = ((v * b2).sum(1) / l2 ** 2 for v in (b1, b3))
        u, r = u[:, None], r[:, None]
        grad[:, ia[0]], grad[:, ia[3]] = g1, g4
        grad[:, ia[1]] = -(1 + u) * g1 + r * g4
        grad[:, ia[2]] = -(1 + r) * g4 + u * g1
        return s, grad
    ib = torch.as_tensor(np.asarray(cv["b"]), device=x.device, dtype=torch.long)
    if cv["type"] == "com_dist":
        v = _min_image(x[:, ib].mean(1) - x[:, ia].mean(1), cv)
        s = v.norm(dim=1)
        e = v / s[:, None]
        grad[:, ia] -= e[:, None] / len(ia)
        grad[:, ib] += e[:, None] / len(ib)
        return s, grad
    s = torch.empty(B, dtype=x.dtype, device=x.device)
    chunk = max(1, 20_000_000 // (len(ia) * len(ib)))
    for b in range(0, B, chunk):
        v = _min_image(x[b:b + chunk, ia][:, :, None] - x[b:b + chunk, ib][:, None], cv)
        q = (v * v).sum(3) / cv["r0"] ** 2
        f = 1 / (1 + q ** 3)
        s[b:b + chunk] = f.sum((1, 2))
        pair = (-6 * q * q * f * f / cv["r0"] ** 2)[..., None] * v
        grad[b:b + chunk, ia] += pair.sum(2)
        grad[b:b + chunk, ib] -= pair.sum(1)
    return s, grad


class Grids64:
    """G bias grids of one dimension in FP64: the starting bias in closed form
    plus the hills deposited since (evaluated at the nodes that are read)."""

    def __init__(self, specs, amps, dev):
        def t(v):
            return torch.tensor(np.array(v, dtype=np.float64), device=dev)
        g, h = [s["grid"] for s in specs], [s["hill"] for s in specs]
        self.dev, self.d = dev, len(g[0]["n"])
        self.n, self.lo, self.D = t([v["n"] for v in g]), t([v["lo"] for v in g]), t([_spacing(v) for v in g])
        self.per = t([v["periodic"] for v in g]) > 0
        self.mabp = h[0].get("method") == "mabp"
        wid = [v["a"] if self.mabp else v["sigma"] for v in h]
        self.wid = t(wid)
        self.R = torch.floor(self.wid / self.D) if self.mabp else \
            torch.ceil(t([[v["cutoff"]] for v in h]) * self.wid / self.D)
        self.h, self.w = h[0], t([v["w"] for v in h])
        self.idT = None if self.mabp else 1 / ((t([v["gamma"] for v in h]) - 1) * t([v["kT"] for v in h]))
        self.stride = np.array([v["stride"] for v in h])
        self.A = None if amps is None else t([a for a, _ in amps])
        self.phi = None if amps is None else t([p for _, p in amps])
        self.hills = []  # (time, centre node [G, d], centre u [G, d], height [G])

    def u(self, s):  # [G, M, d]
        return (s - self.lo[:, None]) / self.D[:, None]

    def at(self, j, time):
        """Fields (1 + d) at nodes j [G, M, d] as of times [M] (hills up to and including them)."""
        n, D, d = self.n[:, None], self.D[:, None], self.d
        out = torch.zeros(1 + d, *j.shape[:2], dtype=torch.float64, device=self.dev)
        if self.A is not None:
            th = 2 * math.pi * j / n + self.phi[:, None]
            c, s = torch.cos(th), -torch.sin(th) * 2 * math.pi / (n * D)
            out[0] = self.A[:, None] * (1 + c.prod(2))
            for k in range(d):
                f = s[..., k].clone()
                for q in range(d):
                    f = f * c[..., q] if q != k else f
                out[1 + k] = self.A[:, None] * f
        lo = float(time.min())
        for th, cen, u, h in self.hills:
            if th > float(time.max()):
                continue
            rel = j - cen[:, None]
            rel = torch.where(self.per[:, None], rel - n * torch.floor(rel / n + 0.5), rel)
            ok = (rel.abs() <= self.R[:, None]).all(2)
            if th > lo:
                ok = ok & (time >= th)[None]
            dist = (rel + (cen - u)[:, None]) * D
            if self.mabp:
                x = dist / self.wid[:, None]
                om = (1 - x * x).clamp_min(1e-300)
                ok = ok & (x.abs() < 1).all(2)
                p = float(self.h["p"])
                val = torch.exp(-(p * x * x / om).sum(2))
                fac = -2 * p * dist / (self.wid[:, None] * om) ** 2
            else:
                val = torch.exp(-(dist ** 2 / (2 * self.wid[:, None] ** 2)).sum(2))
                fac = -dist / self.wid[:, None] ** 2
            val = torch.where(ok, val * h[:, None], torch.zeros_like(val))
            out[0] += val
            for k in range(d):
                out[1 + k] += torch.where(ok, val * fac[..., k], torch.zeros_like(val))
        return out

    def centre(self, u):
        c = torch.floor(u + 0.5)
        if self.mabp:
            c = torch.where(self.per, c - self.n * torch.floor(c / self.n), torch.minimum(c.clamp_min(0), self.n - 1))
        return c

    def look(self, s, time):
        """V and dV/ds at s [G, M, d], times [M]."""
        u, d, n = self.u(s), self.d, self.n[:, None]
        if self.mabp:
            c = torch.floor(u + 0.5)
            lim = ~self.per[:, None] & ((c < 0) | (c > n - 1))
            c = torch.where(self.per[:, None], c - n * torch.floor(c / n), torch.minimum(c.clamp_min(0), n - 1))
            f = self.at(c, time)
            b, cc, kT = self.h["b"], self.h["c"], self.h["kT"]
            den = 1 + cc * (1 - b) * f[0]
            dv = torch.stack([cc * b * kT * f[1 + k] / den for k in range(d)], 2)
            return kT * b / (1 - b) * torch.log(den), torch.where(lim, torch.zeros_like(dv), dv)
        per = self.per[:, None]
        clamped = ~per & ((u < 0) | (u > n - 1))
        u = torch.where(per, u - n * torch.floor(u / n), torch.minimum(u.clamp_min(0), n - 1))
        i0 = torch.floor(u)
        i0 = torch.where(per, i0, torch.minimum(i0, n - 2))
        f = u - i0
        V, dv = 0, 0
        for c in range(2 ** d):
            bit = torch.tensor([(c >> k) & 1 for k in range(d)], dtype=torch.float64, device=self.dev)
            j = i0 + bit
            j = torch.where(per, j - n * torch.floor(j / n), j)
            w = torch.where(bit > 0, f, 1 - f).prod(2)
            v = self.at(j, time)
            V = V + w * v[0]
            dv = dv + torch.stack([w * v[1 + k] for k in range(d)], 2)
        return V, torch.where(clamped, torch.zeros_like(dv), dv)

    def deposit(self, s, t, step, who=None):
        """The hills of MD step `step` at s [G, d] (time index t), heights from before."""
        dep = (step % self.stride) == 0
        if not dep.any():
            return
        u = self.u(s[:, None])[:, 0]
        if self.mabp:
            h = self.w.clone()
        else:
            V = self.look(s[:, None], torch.tensor([t - 0.5], device=self.dev))[0][:, 0]
            h = self.w * torch.exp(-V * self.idT)
        h = h * torch.tensor(dep.astype(np.float64), device=self.dev)
        c = self.centre(u)
        self.hills.append((t, c, c if self.mabp else u, h))


def _exact_frames(specs, x, amps, step0):
    """Forces [T, G, atoms, 3] of walkers with alike CVs over frames x [T, G, atoms, 3], and their grids."""
    T, G, na = x.shape[:3]
    d = len(specs[0]["grid"]["n"])
    grid = Grids64(specs, amps, x.device)
    s, J = [], []
    for k in range(d):
        if specs[0]["cvs"][k]["type"] == "rmsd":  # a reference of its own per walker
            both = [_cv(sp["cvs"][k], x[:, i]) for i, sp in enumerate(specs)]
            s.append(torch.stack([v[0] for v in both], 1))
            J.append(torch.stack([v[1] for v in both], 1))
        else:
            v, g = _cv(specs[0]["cvs"][k], x.reshape(T * G, na, 3))
            s.append(v.reshape(T, G))
            J.append(g.reshape(T, G, na, 3))
    s = torch.stack(s, 2).transpose(0, 1)  # [G, T, d]
    for t in range(T):
        grid.deposit(s[:, t], t, step0 + t)
    _, dv = grid.look(s, torch.arange(T, dtype=torch.float64, device=x.device))
    F = torch.zeros_like(x)
    for k in range(d):
        F -= dv[..., k].T[:, :, None, None] * J[k]
    return F, grid


def _exact_run(specs, x, seed, start=True):
    """Forces [T, atoms, 4] of abp_run over records x [T, atoms, 4], and the grids after it."""
    offs = synth.offsets_of(specs)
    out = torch.zeros(x.shape, dtype=torch.float64, device=x.device)
    x = x.double()
    groups, grids = {}, []
    for i, sp in enumerate(specs):
        key = (sp["natoms"],) + tuple(c["type"] for c in sp["cvs"])
        groups.setdefault(key, []).append(i)
    for idx in groups.values():
        for b in range(0, len(idx), 64):
            part = idx[b:b + 64]
            sp = [specs[i] for i in part]
            na = sp[0]["natoms"]
            xx = torch.stack([x[:, offs[i]:offs[i] + na, :3] for i in part], 1)
            amps = [_start_bias(specs[i], i, seed) for i in part] if start else None
            F, grid = _exact_frames(sp, xx, amps, 0)
            for q, i in enumerate(part):
                out[:, offs[i]:offs[i] + na, :3] = F[:, q]
            grids.append(grid)
    return out, grids


def _philox(ctr, key):
    """Philox-4x32-10 (Salmon et al., SC'11) of counters [4][N] (uint64 arrays of 32-bit words)."""
    c, (k0, k1), m32 = [v.copy() for v in ctr], key, np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _normals(seed, nw, na, step):
    """[nw, na, 3] standard normals of MD step `step`, walker w on stream w."""
    atom = np.tile(np.arange(na, dtype=np.uint64), nw)
    w = np.repeat(np.arange(nw, dtype=np.uint64), na)
    one = np.ones_like(atom)
    c = _philox([atom, one * np.uint64(step & 0xFFFFFFFF), one * np.uint64(step >> 32), w],
                (seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF))
    u = [((v >> np.uint64(8)).astype(np.float64) + 0.5) * 2.0 ** -24 for v in c]
    r0, r2 = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
    z = np.stack([r0 * np.cos(2 * np.pi * u[1]), r0 * np.sin(2 * np.pi * u[1]), r2 * np.cos(2 * np.pi * u[3])], 1)
    return z.reshape(nw, na, 3)


def _potential_grad(md, s):
    """dU/ds [G, d] of the closed loop's CV potential at s [G, d]."""
    g = torch.zeros_like(s)
    if md["potential"] == "double_well":
        A, B = md["dw"]
        g[:, 0] = 4 * A * s[:, 0] * (s[:, 0] ** 2 - B * B)
    elif md["potential"] == "muller_brown":
        mb = md["mb"]
        mx, cx, my, cy = mb["map"]
        X, Y = mx * s[:, 0] + cx, my * s[:, 1] + cy
        for i in range(4):
            dx, dy = X - mb["x0"][i], Y - mb["y0"][i]
            a, b, c = mb["a"][i], mb["b"][i], mb["c"][i]
            e = mb["scale"] * mb["A"][i] * torch.exp(a * dx * dx + b * dx * dy + c * dy * dy)
            g[:, 0] += e * (2 * a * dx + b * dy) * mx
            g[:, 1] += e * (b * dx + 2 * c * dy) * my
    return g


def _exact_md(case, seed, specs, x):
    """Coordinates [atoms, 4] after the closed-loop steps, nothing rounded to 32 bits on the way."""
    nw, na, md = len(specs), specs[0]["natoms"], _md(case, seed)
    shared = bool(specs[0].get("shared"))
    dev = x.device
    pos = x[:, :3].double().reshape(nw, na, 3)
    amps = [_start_bias(sp, i, seed) for i, sp in enumerate(specs)]
    grid = Grids64(specs[:1], amps[:1], dev) if shared else Grids64(specs, amps, dev)
    c1, c2 = md["dt"] * md["mu"], math.sqrt(2 * md["mu"] * md["kT"] * md["dt"])
    d = len(specs[0]["grid"]["n"])
    for t in range(case["steps"]):
        both = [_cv(cv, pos) for cv in specs[0]["cvs"][:d]]
        s = torch.stack([v[0] for v in both], 1)
        if shared:  # heights of every walker before any deposit of the step
            before = list(grid.hills)
            added = []
            for w in range(nw):
                grid.hills = list(before)
                grid.deposit(s[w:w + 1], t, t)
                added += grid.hills[len(before):]
            grid.hills = before + added
            dv = grid.look(s[None], torch.full((nw,), float(t), dtype=torch.float64, device=dev))[1][0]
        else:
            grid.deposit(s, t, t)
            dv = grid.look(s[:, None], torch.tensor([float(t)], dtype=torch.float64, device=dev))[1][:, 0]
        dv = dv + _potential_grad(md, s)
        F = 0
        for k in range(d):
            F = F - dv[:, k, None, None] * both[k][1]
        pos = pos + c1 * F + c2 * torch.as_tensor(_normals(md["seed"], nw, na, t), device=dev)
    out = torch.zeros(nw * na, 4, dtype=torch.float64, device=dev)
    out[:, :3] = pos.reshape(-1, 3)
    return out


def exact(case, seed):
    kind = case["kind"]
    specs = _specs(case, seed)
    if kind == "serve":
        coords, _ = _serve_inputs(case, seed, specs)
        x = torch.as_tensor(coords, device=DEV).reshape(case["depth"], -1, 4)
        out = np.zeros(x.shape)
        offs = synth.offsets_of(specs)
        for i, sp in enumerate(specs):
            xi = x[:, offs[i]:offs[i] + sp["natoms"], None, :3].transpose(1, 2).double().cpu()
            out[:, offs[i]:offs[i] + sp["natoms"], :3] = _exact_frames([sp], xi, None, 0)[0][:, 0].numpy()
        return out.reshape(-1, 4)
    x = _frames(case, seed, specs)
    if kind in ("md", "md64", "shared"):
        # an FP32 closed loop amplifies its roundings step by step: beyond a
        # few steps its trajectory has no 64-bit counterpart
        if kind == "md" and case["steps"] > 8:
            return None
        return _exact_md(case, seed, specs, x[0].cpu() if kind == "md64" else x[0])
    if kind == "engine":
        return _engine_forces(case, seed, x.shape[1]).double() + _exact_run(specs, x[:1], seed)[0][0]
    F, grids = _exact_run(specs, x, seed)
    if kind != "fes":
        return F
    n, grid = case["side"], grids[0]  # at most 64 alike walkers: one group
    j = torch.stack(torch.meshgrid(torch.arange(n), torch.arange(n), indexing="ij")[::-1], -1).reshape(1, -1, 2)
    j = j.to(DEV, torch.float64).expand(len(specs), -1, -1)
    fields = grid.at(j, torch.tensor([float(case["steps"])], dtype=torch.float64, device=DEV))
    return [F] + [fields[:, i].T for i in range(len(specs))]
