"""Performance cases: what users of the library have it compute, at the sizes they use.

A case is one call sequence through the public entry points of
``paper_2102_06248_gb300.fempic`` on a synthetic workload (the recipes of
``workloads.py``: thermal plasma cube, Larmor orbit, plasma ball, electron
beam, batched runs).  ``listed()`` names the cases, ``draw()`` gives more of
the same ranges, ``prepare()`` builds the inputs and handles of a case,
``run()`` makes one pass, ``work()`` says what a pass cannot do without, and
``exact()`` computes a pass's results in FP64 with plain torch, element by
element from the definitions, without the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2102_06248_gb300 import fempic as F
from paper_2102_06248_gb300 import workloads as W

# leapfrog-stable step in units of h / c (tests/golden/dt_cfl.json)
KAPPA_CUBE, KAPPA_BOX, KAPPA_JITTER = 0.2341540837709529, 0.23045965185323428, 0.19447878340721006
LE = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))          # local edges (i, j), i < j
LF = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))              # local face opposite vertex k


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest self-consistent run (smoke test, parity tests): launches and latency are all of it
        dict(name="cube", do="step", load="cube", nx=6, ny=6, nz=6, n=10_000, precision="plain", form="we"),
        # one electron gyrating (single-particle study, 10,000 steps): the field solve at a large time step
        dict(name="orbit", do="step", load="orbit", nx=20, ny=20, nz=20, n=1, precision="plain", form="mfem"),
        # the headline workload at full size, mixed precision
        dict(name="ball", do="step", load="ball", nx=64, ny=64, nz=64, n=16_777_216, precision="mixed", form="we"),
        # a plasma ball in FP64 throughout, where FP64 state is wanted
        dict(name="ball_plain", do="step", load="ball", nx=40, ny=40, nz=40, n=2_000_000, precision="plain", form="we"),
        # a beam source: electrons injected from host arrays before every step, losses at the far wall
        dict(name="beam", do="beam", load="beam", nx=32, ny=32, nz=128, n=2_000_000, precision="mixed", form="we"),
        # expansion into vacuum: absorbing walls, Maxwell-solver form, few particles per cell
        dict(name="expansion", do="step", load="expansion", nx=48, ny=48, nz=48, n=200_000, precision="mixed",
             form="mfem"),
        # Adams-Bashforth 4 along the curved path, backward-difference fields
        dict(name="adams", do="step", load="adams", nx=16, ny=16, nz=16, n=100_000, precision="plain", form="bd"),
        # many small uneven runs (a parameter scan) stepped together, one six-step graph per pass
        dict(name="batch", do="batch", load="cube", runs=16, lo=8, hi=24, n_lo=10_000, n_hi=500_000,
             precision="mixed", form="we"),
        # particles in frozen fields (test-particle study), many per cell, odd sizes
        dict(name="push", do="push", load="cube", nx=23, ny=25, nz=21, n=4_000_003, precision="mixed", form="we"),
        # an electrostatic solve without allocation, for hosts that own the memory
        dict(name="poisson", do="poisson", nx=48, ny=48, nz=48, jitter=0.2, tol=1e-12),
        # a step whose Newmark solve uses the learned preconditioner (inference)
        dict(name="learned", do="learned", load="ball", nx=32, ny=32, nz=32, n=500_000, precision="mixed", form="we"),
        # one training evaluation of that preconditioner: loss and gradients (forward and backward)
        dict(name="train", do="train", load="ball", nx=32, ny=32, nz=32, n=10_000, precision="mixed", form="we"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: any kind, sizes spread over their logarithm, boxes that are not cubes."""
    kind = rng.choice(("cube", "orbit", "ball", "ball", "beam", "expansion", "adams", "batch", "push", "push",
                       "poisson", "learned", "train"))

    def box(lo, hi):
        return {"nx": _log(rng, lo, hi), "ny": _log(rng, lo, hi), "nz": _log(rng, lo, hi)}

    precision = rng.choice(("plain", "mixed"))
    if kind == "cube":
        return dict(do="step", load="cube", n=_log(rng, 1_000, 1_000_000), precision=precision,
                    form=rng.choice(("we", "mfem", "bd")), **box(4, 24))
    if kind == "orbit":
        c = _log(rng, 8, 24)
        return dict(do="step", load="orbit", nx=c, ny=c, nz=c, n=1, precision=precision, form="mfem")
    if kind == "ball":
        return dict(do="step", load="ball", n=_log(rng, 50_000, 8_000_000), precision=precision,
                    form=rng.choice(("we", "we", "mfem")), **box(12, 60))
    if kind == "beam":
        c = _log(rng, 6, 30)
        return dict(do="beam", load="beam", nx=c, ny=c, nz=_log(rng, 24, 120), n=_log(rng, 20_000, 2_000_000),
                    precision=precision, form="we")
    if kind == "expansion":
        return dict(do="step", load="expansion", n=_log(rng, 20_000, 400_000), precision=precision, form="mfem",
                    **box(14, 46))
    if kind == "adams":
        return dict(do="step", load="adams", n=_log(rng, 2_000, 300_000), precision="plain",
                    form=rng.choice(("we", "mfem", "bd")), **box(5, 22))
    if kind == "batch":
        return dict(do="batch", load="cube", runs=rng.randint(2, 20), lo=rng.randint(5, 9), hi=rng.randint(12, 22),
                    n_lo=_log(rng, 2_000, 20_000), n_hi=_log(rng, 50_000, 400_000), precision=precision, form="we")
    if kind == "push":
        return dict(do="push", load=rng.choice(("cube", "ball")), n=_log(rng, 20_000, 6_000_000), precision=precision,
                    form="we", **box(8, 44))
    if kind == "poisson":
        return dict(do="poisson", jitter=rng.choice((0.0, 0.2)), tol=rng.choice((1e-10, 1e-12, 1e-14)), **box(8, 60))
    if kind == "learned":
        return dict(do="learned", load="ball", n=_log(rng, 20_000, 800_000), precision=precision, form="we",
                    **box(12, 34))
    return dict(do="train", load="ball", n=10_000, precision="mixed", form="we", **box(12, 34))


# ---------------------------------------------------------------------------
# workloads on the GPU (the recipes of workloads.py, drawn with torch so that
# tens of millions of particles take milliseconds)
# ---------------------------------------------------------------------------
_MESHES = {}


def _recipe(case):
    """Box, time step, fields and species of a case: plain numbers only."""
    load = case.get("load", "ball")
    cells = (case["nx"], case["ny"], case["nz"])
    r = dict(cells=cells, jitter=case.get("jitter", 0.0), b0=(0.0, 0.0, 0.0), rho_bg=0.0, absorb=False, pusher="boris",
             curved=False, load=load)
    n = case.get("n", 0)
    if load in ("cube", "adams"):
        c = max(cells)
        h = 1.0 / c
        vol = h ** 3 * cells[0] * cells[1] * cells[2]
        density = 1.0e11 * (c / 6.0) ** 2                     # lambda_D about one cell
        r.update(h=h, dt=2.0 * KAPPA_CUBE * h / W.C0, rho_bg=-W.Q_E * density, vth=(0.01 * W.C0,),
                 species=[(W.Q_E, W.M_E, density * vol / max(n, 1), n)])
        if load == "cube":
            r["b0"] = (0.0, 0.0, 0.1)
        else:
            r.update(pusher="ab4", curved=True)
    elif load == "orbit":
        wc = abs(W.Q_E) * 0.05 / W.M_E
        r_l = 0.05 * W.C0 / wc
        r.update(h=10.0 * r_l / cells[0], dt=2.0 * math.pi / wc / 64.0, b0=(0.0, 0.0, 0.05), r_l=r_l,
                 vth=(0.05 * W.C0,), species=[(W.Q_E, W.M_E, 1.0, 1)])
    elif load in ("ball", "expansion"):
        te, ti, debye, frac, mass = ((10.0, 0.1, 2.0, 0.15, W.MASS_RATIO_P) if load == "ball"
                                     else (1000.0, 10.0, 0.35, 0.1, 100.0))
        h = 1.0e-4
        sigma = [frac * h * c for c in cells]
        peak = W.EPS0 * te * W.EV / ((debye * h) ** 2 * W.Q_E ** 2)
        w = peak * (2.0 * math.pi) ** 1.5 * sigma[0] * sigma[1] * sigma[2] / max(n, 1)
        dt = 4.0 * KAPPA_JITTER * h / W.C0
        if load == "expansion":
            dt = 0.2 * debye * h / math.sqrt(te * W.EV / W.M_E)
        r.update(h=h, jitter=0.2, dt=dt, sigma=sigma, absorb=load == "expansion",
                 vth=(math.sqrt(te * W.EV / W.M_E), math.sqrt(ti * W.EV / (mass * W.M_E))),
                 species=[(W.Q_E, W.M_E, w, n), (-W.Q_E, mass * W.M_E, w, n)])
    elif load == "beam":
        h, vz = 1.25e-3, 0.1 * W.C0
        lz = cells[2] * h
        dt = 4.0 * KAPPA_BOX * h / W.C0
        r.update(h=h, dt=dt, vz=vz, inject=max(1, int(round(n * vz * dt / lz))), vth=(0.01 * vz,),
                 species=[(W.Q_E, W.M_E, 0.25 * lz / (vz * abs(W.Q_E) * n), n)])
    return r


def _box(r):
    return W.kuhn_box(r["cells"], tuple(c * r["h"] for c in r["cells"]), jitter=r["jitter"], seed=1004)


def _mesh(r):
    """The library's mesh and the torch copy of its arrays (a program keeps one mesh for all its runs on it)."""
    key = (r["cells"], r["h"], r["jitter"], r["absorb"])
    if key not in _MESHES:
        box = _box(r)
        bc = W.box_wall_bc(box) if r["absorb"] else None
        _MESHES[key] = (F.Mesh(box.xyz, box.tets, wall_bc=bc), torch.from_numpy(box.xyz).cuda(),
                        torch.from_numpy(box.tets).cuda().long())
    return _MESHES[key]


_KUHN_ID = [0, 0, 1, 2, 0, 3, 4, 5]        # permutation number by 3 * (first axis) + (second axis)


def _place(r, xyz, tets, ref):
    """Physical points and tets of points given in unjittered box coordinates (workloads.place_in_box)."""
    cells = torch.tensor(r["cells"], device=ref.device)
    s = torch.minimum((ref / r["h"]).clamp_min(1e-9), cells - 1e-9)
    c = torch.minimum(s.floor().long(), cells - 1)
    fs, order = torch.sort(s - c, dim=1, descending=True, stable=True)
    perm = torch.tensor(_KUHN_ID, device=ref.device)[3 * order[:, 0] + order[:, 1]]
    tet = 6 * (c[:, 0] + cells[0] * (c[:, 1] + cells[1] * c[:, 2])) + perm
    lam = (1.0 - fs[:, 0], fs[:, 0] - fs[:, 1], fs[:, 1] - fs[:, 2], fs[:, 2])
    x = torch.zeros_like(ref)
    for k in range(4):
        x += lam[k][:, None] * xyz[tets[tet, k]]
    return x, tet.int()


def _particles(r, xyz, tets, seed):
    """Per species: positions [n, 3], velocities [n, 3] (FP64) and tets on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    size = torch.tensor([c * r["h"] for c in r["cells"]], dtype=torch.float64, device="cuda")
    out = []
    for s, (q, m, w, n) in enumerate(r["species"]):
        if r["load"] == "orbit":
            a = 2.0 * math.pi * torch.rand(1, generator=g, device="cuda", dtype=torch.float64).item()
            off = [r["r_l"] * math.cos(a), r["r_l"] * math.sin(a) + 0.137 * r["h"], 0.291 * r["h"]]
            ref = (0.5 * size + torch.tensor(off, dtype=torch.float64, device="cuda"))[None]
            v = torch.tensor([[-math.sin(a) * r["vth"][0], math.cos(a) * r["vth"][0], 0.0]], dtype=torch.float64,
                             device="cuda")
        else:
            v = r["vth"][s] * torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
            if r["load"] in ("ball", "expansion"):
                sigma = torch.tensor(r["sigma"], dtype=torch.float64, device="cuda")
                ref = 0.5 * size + sigma * torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
                ref = torch.minimum(torch.maximum(ref, 0.01 * size), 0.99 * size)
            elif r["load"] == "beam":
                ref, v = _beam(r, g, n, 0.0, float(size[2]), v)
            else:
                ref = size * torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
        x, tet = _place(r, xyz, tets, ref)
        out.append((q, m, w, x, v, tet))
    return out


def _beam(r, g, n, z0, z1, v):
    """Reference points of beam electrons with z in (z0, z1); v gets the axial speed."""
    side = r["cells"][0] * r["h"]
    ref = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64) * (0.1 * side)
    ref = 0.5 * side + ref.clamp(-0.45 * side, 0.45 * side)
    ref[:, 2] = z0 + (z1 - z0) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    v[:, 2] += r["vz"]
    return ref, v


def _slabs(r, xyz, tets, seed, count):
    """Host arrays of the electrons that enter before each of `count` steps."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    out = []
    for _ in range(count):
        n = r["inject"]
        v = r["vth"][0] * torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
        ref, v = _beam(r, g, n, 0.0, r["vz"] * r["dt"], v)
        x, tet = _place(r, xyz, tets, ref)
        out.append((x.cpu().numpy(), v.cpu().numpy(), tet.cpu().numpy()))
    return out


def _sim(case, r, seed, preconditioner="jacobi"):
    mesh, xyz, tets = _mesh(r)
    sim = F.Sim(mesh, r["dt"], form=case["form"], pusher=r["pusher"], precision=case["precision"], b0=r["b0"],
                rho_background=r["rho_bg"], preconditioner=preconditioner, curved_path=r["curved"])
    for k, (q, m, w, x, v, tet) in enumerate(_particles(r, xyz, tets, seed)):
        sim.particles_load(k, q, m, w, x, v, tet)
    sim.init()
    return sim


def _batch_members(case):
    """Cells and particle counts of a batch's runs: log-uniform over the ranges, in a fixed uneven order."""
    out = []
    for k in range(case["runs"]):
        a, b = (0.5 + 0.6180339887498949 * k) % 1.0, (0.25 + 0.7548776662466927 * k) % 1.0
        c = int(math.exp(math.log(case["lo"]) + a * math.log((case["hi"] + 0.999) / case["lo"])))
        n = int(round(math.exp(math.log(case["n_lo"]) + b * math.log(case["n_hi"] / case["n_lo"]))))
        out.append(dict(case, nx=c, ny=c, nz=c, n=n))
    return out


def _weights(seed):
    """Network weights of the size that training reaches (uniform by fan-in, a small output layer)."""
    g = np.random.RandomState(int(seed) % (1 << 31))
    w = np.empty(F.GNN_PARAMS, dtype=np.float32)
    n_in, n_layers = 96, 3 * (2 * 32 * 32 + 32)
    w[:n_in] = g.uniform(-1, 1, n_in) * math.sqrt(3.0 / 2)
    w[n_in:n_in + n_layers] = g.uniform(-1, 1, n_layers) * math.sqrt(3.0 / 64)
    w[n_in + n_layers:] = g.uniform(-1, 1, F.GNN_PARAMS - n_in - n_layers) * 0.1
    return w


def _residual(mesh_edges, seed):
    """A residual on the edges as a solve leaves it: all scales present, no preferred direction."""
    g = np.random.RandomState(int(seed) % (1 << 31) ^ 0x5EED)
    return g.standard_normal(mesh_edges) * 1.0e-15


def _charge(r, xyz, seed):
    """Node charges: two Gaussian clouds of opposite sign, a little apart, with noise."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    size = torch.tensor([c * r["h"] for c in r["cells"]], dtype=torch.float64, device="cuda")
    off = 0.05 * size * torch.randn(2, 3, generator=g, device="cuda", dtype=torch.float64)
    rho = torch.zeros(xyz.shape[0], dtype=torch.float64, device="cuda")
    for k, sign in enumerate((1.0, -1.0)):
        rho += sign * torch.exp(-(((xyz - 0.5 * size - off[k]) / (0.15 * size)) ** 2).sum(1) / 2.0)
    rho *= 1.0 + 0.05 * torch.randn(rho.shape, generator=g, device="cuda", dtype=torch.float64)
    return rho * 1.0e-17


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
STEP_FIELDS = ("E", "B", "G", "RHO")


def _buffers(sim, names):
    return {f: torch.zeros(sim.field_len(f), dtype=torch.float64, device="cuda") for f in names}


def prepare(case, seed):
    do = case["do"]
    if do == "batch":
        sims = [_sim(c, _recipe(c), seed + 1000 * k) for k, c in enumerate(_batch_members(case))]
        return dict(do=do, sims=sims, batch=F.Batch(sims), out=[_buffers(s, ("E", "G", "RHO")) for s in sims])
    r = _recipe(dict(case, load=case.get("load", "none")))
    if do == "poisson":
        r.update(h=1.0e-4, dt=4.0 * KAPPA_JITTER * 1.0e-4 / W.C0)
        mesh, xyz, _ = _mesh(r)
        owner = F.Sim(mesh, r["dt"])                     # puts the mesh on the GPU
        rho = _charge(r, xyz, seed)
        return dict(do=do, mesh=mesh, owner=owner, rho=rho, phi=torch.zeros_like(rho), tol=case["tol"])
    if do == "learned":
        sim = _sim(case, r, seed, preconditioner="gnn")
        sim.step()
        sim.gnn_train(steps=60, samples=6)
        return dict(do="step", sim=sim, out=_buffers(sim, STEP_FIELDS))
    if do == "train":
        sim = _sim(case, r, seed, preconditioner="gnn")
        sim.gnn_set_weights(_weights(seed))
        return dict(do=do, sim=sim, r=_residual(sim.mesh.n_edges, seed))
    sim = _sim(case, r, seed)
    if do == "push":
        return dict(do=do, sim=sim, out=_buffers(sim, ("DG", "RHO", "WALL")))
    if do == "beam":
        mesh, xyz, tets = _mesh(r)
        return dict(do=do, sim=sim, slabs=_slabs(r, xyz, tets, seed, 8), next=0,
                    out=_buffers(sim, STEP_FIELDS + ("WALL",)))
    return dict(do="step", sim=sim, out=_buffers(sim, STEP_FIELDS))


def run(state):
    do = state["do"]
    if do == "poisson":
        return F.electrostatic_solve_noalloc(state["mesh"], state["rho"], state["phi"], state["tol"])
    if do == "batch":
        state["batch"].step(6)
        return [{f: s.field(f, out=b) for f, b in o.items()} for s, o in zip(state["sims"], state["out"])]
    sim = state["sim"]
    if do == "train":
        loss, grad = sim.gnn_loss_grad(state["r"])
        return {"loss": loss, "grad": grad}
    if do == "push":
        sim.particle_phase()
    elif do == "beam":
        x, v, tet = state["slabs"][state["next"] % len(state["slabs"])]
        state["next"] += 1
        sim.particles_inject(0, x, v, tet)
        sim.step()
    else:
        sim.step()
    return {f: sim.field(f, out=b) for f, b in state["out"].items()}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: the particles' state read and written once, the mesh (coordinates, tets) read once, the fields a step
    reads and those it writes once each.  Flops: the push, walk and deposit of each particle and the iterations'
    sparse products of the solves (fifty of the field system, a dozen of the node system, for a step)."""
    if case["do"] == "batch":
        each = [work(dict(c, do="step")) for c in _batch_members(case)]
        return {k: 6.0 * sum(w[k] for w in each) for k in ("bytes", "flops")}
    cells = case["nx"] * case["ny"] * case["nz"]
    nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    edges, faces, tets = 7.0 * cells, 12.0 * cells, 6.0 * cells
    mesh = 24.0 * nodes + 16.0 * tets
    if case["do"] == "poisson":
        its = 3.0 * max(case["nx"], case["ny"], case["nz"])
        return {"bytes": mesh + 16.0 * nodes, "flops": its * nodes * (2 * 15 + 12)}
    if case["do"] == "train":
        return {"bytes": mesh + 16.0 * edges, "flops": 3.0 * 3.0 * edges * (2 * 16 * 32 + 2 * 64 * 32)}
    species = 2 if case["load"] in ("ball", "expansion") else 1
    real = 8.0 if case["precision"] == "plain" else 4.0
    n = float(case["n"] * species)
    particles = n * 2.0 * (6 * real + 8.0)
    if case["do"] == "push":
        return {"bytes": mesh + particles + 8.0 * (2 * edges + faces + 2 * nodes), "flops": 250.0 * n}
    fields = 8.0 * (2 * edges + 2 * edges + faces + 2 * edges + faces + 2 * nodes)
    flops = 250.0 * n + 50.0 * edges * (2 * 16 + 12) + 12.0 * nodes * (2 * 15 + 12)
    if case["do"] == "learned":
        flops += 12.0 * 3.0 * edges * (2 * 16 * 32 + 2 * 64 * 32)
    return {"bytes": mesh + particles + fields, "flops": flops}


# ---------------------------------------------------------------------------
# exact: the same pass in FP64 with plain torch, from the definitions
# ---------------------------------------------------------------------------
class _Space:
    """Whitney forms of a box mesh: entities, geometry and the element matrices, in the canonical numbering
    (edges and faces sorted by their node ids, pointing from the lower to the higher one)."""

    def __init__(self, box, absorb):
        xyz = torch.from_numpy(box.xyz).cuda()
        t = torch.from_numpy(box.tets).cuda().long().sort(dim=1).values
        nn, nt = xyz.shape[0], t.shape[0]
        self.xyz, self.t, self.nn, self.nt = xyz, t, nn, nt
        key, inv = torch.unique(torch.stack([t[:, i] * nn + t[:, j] for i, j in LE], 1), return_inverse=True)
        self.te, self.ne = inv.view(nt, 6), key.numel()
        self.edge = torch.stack([key // nn, key % nn], 1)
        fkey, finv = torch.unique(torch.stack([(t[:, a] * nn + t[:, b]) * nn + t[:, c] for a, b, c in LF], 1),
                                  return_inverse=True)
        self.tf, self.nf = finv.view(nt, 4), fkey.numel()
        fn = torch.stack([fkey // (nn * nn), (fkey // nn) % nn, fkey % nn], 1)
        find = lambda a, b: torch.searchsorted(key, a * nn + b)  # noqa: E731
        self.fe = torch.stack([find(fn[:, 0], fn[:, 1]), find(fn[:, 1], fn[:, 2]), find(fn[:, 0], fn[:, 2])], 1)
        # neighbours across faces, wall faces, wall nodes, edges held at zero
        order = torch.argsort(self.tf.reshape(-1), stable=True)
        count = torch.bincount(self.tf.reshape(-1), minlength=self.nf)
        first = torch.cumsum(count, 0) - count
        self.nbr = torch.full((nt * 4,), -1, dtype=torch.long, device=t.device)
        two = (count == 2).nonzero()[:, 0]
        a, b = order[first[two]], order[first[two] + 1]
        self.nbr[a], self.nbr[b] = b // 4, a // 4
        self.nbr = self.nbr.view(nt, 4)
        wall = count == 1
        self.wall_node = torch.zeros(nn, dtype=torch.bool, device=t.device)
        self.wall_node[fn[wall].reshape(-1)] = True
        self.fixed = torch.zeros(self.ne, dtype=torch.bool, device=t.device)
        if not absorb:
            self.fixed[self.fe[wall].reshape(-1)] = True
        # barycentric gradients, volumes, signs
        x = xyz[t]
        d = x[:, 1:] - x[:, :1]
        det = (d[:, 0] * torch.linalg.cross(d[:, 1], d[:, 2])).sum(1)
        g = torch.stack([torch.linalg.cross(d[:, 1], d[:, 2]), torch.linalg.cross(d[:, 2], d[:, 0]),
                         torch.linalg.cross(d[:, 0], d[:, 1])], 1) / det[:, None, None]
        self.g = torch.cat([-g.sum(1, keepdim=True), g], 1)
        self.x0, self.vol, sign = x[:, 0], det.abs() / 6.0, torch.sign(det)
        self.D = sign[:, None] * torch.tensor([1.0, -1.0, 1.0, -1.0], dtype=torch.float64, device=t.device)
        gg = self.g @ self.g.transpose(1, 2)
        self.M = self._mass(gg, W.EPS0 * self.vol / 20.0)
        cr = torch.stack([torch.linalg.cross(self.g[:, i], self.g[:, j]) for i, j in LE], 1)
        self.K = (4.0 / W.MU0) * self.vol[:, None, None] * (cr @ cr.transpose(1, 2))
        self.L = W.EPS0 * self.vol[:, None, None] * gg
        cen = x.mean(1)
        dk = cen[:, None] - x
        spread = ((x - cen[:, None]) ** 2).sum((1, 2))
        self.H = (self.vol[:, None, None] * (dk @ dk.transpose(1, 2)) + (self.vol * spread / 20.0)[:, None, None]) \
            * self.D[:, :, None] * self.D[:, None, :] / (9.0 * self.vol[:, None, None] ** 2 * W.MU0)
        self.I = None
        if absorb:                                        # surface impedance of every wall face
            self.I = torch.zeros_like(self.M)
            tk = wall[self.tf]
            for k in range(4):
                at = tk[:, k].nonzero()[:, 0]
                gk = self.g[at, k]
                gn = gk.norm(dim=1)
                nrm = gk / gn[:, None]
                gs = self.g[at] - (self.g[at] * nrm[:, None]).sum(2, keepdim=True) * nrm[:, None]
                m = self._mass(gs @ gs.transpose(1, 2), 3.0 * self.vol[at] * gn / (12.0 * W.MU0))
                on = torch.tensor([k not in e for e in LE], device=t.device)
                self.I[at] += m * (on[:, None] & on[None, :])

    @staticmethod
    def _mass(gg, scale):
        rows = []
        for i, j in LE:
            rows.append(torch.stack([(1.0 + (i == p)) * gg[:, j, q] - (1.0 + (i == q)) * gg[:, j, p]
                                     - (1.0 + (j == p)) * gg[:, i, q] + (1.0 + (j == q)) * gg[:, i, p]
                                     for p, q in LE], 1))
        return torch.stack(rows, 1) * scale[:, None, None]

    def apply(self, local, ids, n, x):
        y = torch.einsum("tij,tj...->ti...", local, x[ids])
        return torch.zeros((n,) + tuple(x.shape[1:]), dtype=x.dtype, device=x.device).index_add(
            0, ids.reshape(-1), y.reshape((-1,) + tuple(x.shape[1:])))

    def diag(self, local, ids, n):
        d = torch.diagonal(local, dim1=1, dim2=2)
        return torch.zeros(n, dtype=torch.float64, device=d.device).index_add(0, ids.reshape(-1), d.reshape(-1))

    def solve(self, local, ids, n, hold, b, x, tol):
        """Jacobi-PCG to ||r|| <= tol ||b|| with the entries `hold` kept at zero."""
        keep = (~hold).double()
        dinv = keep / torch.where(hold, torch.ones_like(b), self.diag(local, ids, n))
        b = b * keep
        x = x * keep
        r = b - keep * self.apply(local, ids, n, x)
        bb = float(b @ b)
        if bb == 0.0:
            return torch.zeros_like(b)
        z = dinv * r
        p, rz = z.clone(), r @ z
        best, since = float("inf"), 0
        for it in range(20000):
            q = keep * self.apply(local, ids, n, p)
            a = rz / (p @ q)
            x = x + a * p
            r = r - a * q
            z = dinv * r
            rn = r @ z
            p = z + (rn / rz) * p
            rz = rn
            if it % 10 == 9:
                rr = float(r @ r)
                since = 0 if rr < 0.25 * best else since + 1
                best = min(best, rr)
                if rr <= tol * tol * bb or since > 40:
                    break
        return x


class _Run:
    """One simulation: electrostatic start, then steps (Boris; the first step of Adams-Bashforth)."""

    def __init__(self, sp, r, form, particles):
        self.sp, self.r, self.form, self.dt = sp, r, form, r["dt"]
        self.parts = [[q, m, w, x.clone(), v.clone(), tet.long().clone()] for q, m, w, x, v, tet in particles]
        z = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")  # noqa: E731
        self.b = self.bp = z(sp.nf)
        self.g, self.gp, self.wall = z(sp.ne), z(sp.ne), z(sp.nn)
        rho = z(sp.nn)
        for q, m, w, x, v, tet in self.parts:
            for c in torch.arange(x.shape[0], device="cuda").split(4_000_000):
                lam = self._bary(x[c], tet[c])
                rho.index_add_(0, sp.t[tet[c]].reshape(-1), (q * w * lam).reshape(-1))
        bg = torch.zeros_like(rho).index_add(0, sp.t.reshape(-1), (r["rho_bg"] * sp.vol / 4.0).repeat_interleave(4))
        phi = sp.solve(sp.L, sp.t, sp.nn, sp.wall_node, rho + bg, z(sp.nn), 1e-15)
        self.e = (phi[sp.edge[:, 0]] - phi[sp.edge[:, 1]]) * (~sp.fixed)
        self.ep = self.e
        self.rho = rho

    def _bary(self, x, tet):
        sp = self.sp
        lam = torch.einsum("nki,ni->nk", sp.g[tet], x - sp.x0[tet])
        lam[:, 0] += 1.0
        return lam

    def inject(self, x, v, tet):
        sp, p = self.sp, self.parts[0]
        x, v, tet = (torch.from_numpy(a).cuda() for a in (x, v, tet))
        c = (p[0] * p[2] * self._bary(x, tet.long())).reshape(-1)
        self.wall = self.wall.index_add(0, sp.t[tet.long()].reshape(-1), -c)
        p[3], p[4], p[5] = torch.cat([p[3], x]), torch.cat([p[4], v]), torch.cat([p[5], tet.long()])

    def _push(self, q, m, x, v, tet, boris):
        sp, dt = self.sp, self.dt
        lam, g = self._bary(x, tet), sp.g[tet]
        ev = self.e[sp.te[tet]]
        E = torch.zeros_like(x)
        for k, (i, j) in enumerate(LE):
            E += ev[:, k, None] * (lam[:, i, None] * g[:, j] - lam[:, j, None] * g[:, i])
        db = sp.D[tet] * self.b[sp.tf[tet]] / (3.0 * sp.vol[tet])[:, None]
        B = torch.tensor(self.r["b0"], dtype=torch.float64, device=x.device).expand_as(x).clone()
        for k in range(4):
            B += db[:, k, None] * (x - sp.xyz[sp.t[tet, k]])
        if not boris:
            return x + dt * v, v + dt * (q / m) * (E + torch.linalg.cross(v, B))
        h = 0.5 * q / m * dt
        vm, tv = v + h * E, h * B
        vp = vm + torch.linalg.cross(vm, tv)
        vn = vm + torch.linalg.cross(vp, 2.0 * tv / (1.0 + (tv * tv).sum(1, keepdim=True))) + h * E
        return x + dt * vn, vn

    def _walk(self, x, xe, tet, dg, rho, wall, qw):
        """Deposits the straight paths x -> xe; returns the end tets (-1: absorbed)."""
        sp = self.sp
        end = tet.clone()
        at = torch.arange(x.shape[0], device=x.device)
        T, lS, xe = tet, self._bary(x, tet), xe
        entry = torch.full_like(T, -1)
        four = torch.arange(4, device=x.device)
        while at.numel():
            lE = self._bary(xe, T)
            out = (lE < 0) & (four[None] != entry[:, None])
            s = torch.where(out, (lS / (lS - lE)).clamp_min(0.0), torch.full_like(lE, 2.0))
            smin, kmin = s.min(1)
            kmin = torch.argmax((s == smin[:, None]).int(), 1)
            stop = ~out.any(1)
            lX = lS + smin[:, None] * (lE - lS)
            lX.scatter_(1, kmin[:, None], 0.0)
            lX = torch.where(stop[:, None], lE, lX)
            cur = torch.stack([lS[:, i] * lX[:, j] - lX[:, i] * lS[:, j] for i, j in LE], 1)
            dg.index_add_(0, sp.te[T].reshape(-1), (qw * cur).reshape(-1))
            rho.index_add_(0, sp.t[T[stop]].reshape(-1), (qw * lE[stop]).reshape(-1))
            end[at[stop]] = T[stop]
            go = ~stop
            nb = sp.nbr[T].gather(1, kmin[:, None])[:, 0]
            hit = go & (nb < 0)
            wall.index_add_(0, sp.t[T[hit]].reshape(-1), (qw * lX[hit]).reshape(-1))
            end[at[hit]] = -1
            go &= nb >= 0
            same = sp.t[nb[go]][:, :, None] == sp.t[T[go]][:, None, :]
            lS = torch.where(same, lX[go][:, None, :], torch.zeros_like(lX[go][:, None, :])).sum(2)
            entry = torch.argmax((~same.any(2)).int(), 1)
            at, T, xe = at[go], nb[go], xe[go]
        return end

    def particle_phase(self):
        sp = self.sp
        dg, rho, wall = torch.zeros_like(self.g), torch.zeros_like(self.rho), self.wall.clone()
        for p in self.parts:
            q, m, w, x, v, tet = p
            xe, ve, end = torch.empty_like(x), torch.empty_like(v), torch.empty_like(tet)
            for c in torch.arange(x.shape[0], device="cuda").split(4_000_000):
                xe[c], ve[c] = self._push(q, m, x[c], v[c], tet[c], self.r["pusher"] == "boris")
                end[c] = self._walk(x[c], xe[c], tet[c], dg, rho, wall, q * w)
            live = end >= 0
            p[3], p[4], p[5] = xe[live], ve[live], end[live]
        self.dg, self.rho, self.wall = dg, rho, wall

    def step(self):
        sp, dt, form = self.sp, self.dt, self.form
        self.particle_phase()
        gn = self.g + self.dg
        c4 = (1.0 if form == "bd" else 0.25) * dt * dt
        ci = (1.0 if form == "bd" else 0.5) * dt / W.C0
        A = sp.M + c4 * sp.K + (ci * sp.I if sp.I is not None else 0.0)
        mul = lambda loc, x: sp.apply(loc, sp.te, sp.ne, x)  # noqa: E731
        e, ep = self.e, self.ep
        if form == "we":
            rhs = mul(sp.M, 2 * e - ep) - c4 * mul(sp.K, 2 * e + ep) - (gn - 2 * self.g + self.gp)
            if sp.I is not None:
                rhs = rhs + ci * mul(sp.I, ep)
        else:
            hb = sp.apply(sp.H, sp.tf, sp.nf, self.b + (self.bp if form == "mfem" else 0.0))
            ct = torch.zeros_like(e)
            for k, s in enumerate((1.0, 1.0, -1.0)):
                ct = ct.index_add(0, sp.fe[:, k], s * hb)
            if form == "mfem":
                rhs = mul(sp.M, ep) - c4 * mul(sp.K, 2 * e + ep) + dt * ct - (gn - self.gp)
                if sp.I is not None:
                    rhs = rhs - dt / W.C0 * mul(sp.I, e + 0.5 * ep)
            else:
                rhs = mul(sp.M, e) + dt * ct - (gn - self.g)
        x = sp.solve(A, sp.te, sp.ne, sp.fixed, rhs, 2 * e - ep, 1e-15)
        curl = lambda u: u[sp.fe[:, 0]] + u[sp.fe[:, 1]] - u[sp.fe[:, 2]]  # noqa: E731
        if form == "bd":
            bn = self.b - dt * curl(x)
        elif form == "we":
            bn = self.b - 0.5 * dt * curl(x + e)
        else:
            bn = self.bp - 2.0 * dt * curl(0.25 * x + 0.5 * e + 0.25 * ep)
        self.e, self.ep, self.b, self.bp, self.g, self.gp = x, e, bn, self.b, gn, self.g

    def fields(self, names):
        have = {"E": self.e, "B": self.b, "G": self.g, "RHO": self.rho, "WALL": self.wall}
        have["DG"] = getattr(self, "dg", None)
        return {f: have[f] for f in names}


def _loss_grad(sp, A, r, weights):
    """Loss and gradients of the learned preconditioner at the bfloat16 roundings of `weights`."""
    keep = ~sp.fixed
    ids = (torch.cumsum(keep, 0) - 1)[sp.te]
    n = int(keep.sum())
    ids = torch.where(keep[sp.te], ids, torch.full_like(ids, n))                # held edges: one spare row
    A = A * keep[sp.te][:, :, None] * keep[sp.te][:, None, :]
    r = torch.from_numpy(r).cuda()[keep]
    d = sp.diag(A, ids, n + 1)[:n]
    isd = 1.0 / torch.sqrt(d)
    pad = lambda v: torch.cat([v, torch.zeros((1,) + tuple(v.shape[1:]), dtype=v.dtype, device=v.device)])  # noqa: E731
    mul = lambda x: sp.apply(A, ids, n + 1, pad(x))[:n]  # noqa: E731
    th = torch.from_numpy(weights).cuda().bfloat16().double().requires_grad_(True)
    rho2 = (r * r / d).mean()
    rho = torch.sqrt(rho2)
    a = torch.log(d) - torch.log(d).mean()
    h = torch.relu((r * isd / rho)[:, None] * th[0:32] + a[:, None] * th[32:64] + th[64:96])
    off = 96
    for _ in range(3):
        Wl, Q, b = th[off:off + 1024].view(32, 32), th[off + 1024:off + 2048].view(32, 32), th[off + 2048:off + 2080]
        agg = isd[:, None] * mul(isd[:, None] * h)
        h = torch.relu(h @ Wl.T + agg @ Q.T + b)
        off += 2080
    z = r / d + rho * (h @ th[off:off + 32] + th[off + 32]) * isd
    loss = ((z * mul(z)).sum() - 2.0 * (z * r).sum()) / (n * rho2)
    loss.backward()
    return {"loss": float(loss.detach()), "grad": th.grad}


def exact(case, seed):
    do = case["do"]
    if do == "batch":
        out = []
        for k, c in enumerate(_batch_members(case)):
            r = _recipe(c)
            mesh, xyz, tets = _mesh(r)
            one = _Run(_Space(_box(r), False), r, c["form"], _particles(r, xyz, tets, seed + 1000 * k))
            for _ in range(6):
                one.step()
            out.append(one.fields(("E", "G", "RHO")))
        return out
    r = _recipe(dict(case, load=case.get("load", "none")))
    if do == "poisson":
        r["h"] = 1.0e-4
        sp = _Space(_box(r), False)
        rho = _charge(r, sp.xyz, seed)
        return sp.solve(sp.L, sp.t, sp.nn, sp.wall_node, rho, torch.zeros_like(rho), 1e-15)
    sp = _Space(_box(r), r["absorb"])
    if do == "train":
        return _loss_grad(sp, sp.M + 0.25 * r["dt"] ** 2 * sp.K, _residual(sp.ne, seed), _weights(seed))
    tets = torch.from_numpy(_box(r).tets).cuda().long()
    one = _Run(sp, r, case["form"], _particles(r, sp.xyz, tets, seed))
    if do == "push":
        one.particle_phase()
        return one.fields(("DG", "RHO", "WALL"))
    if do == "learned":
        one.step()
    if do == "beam":
        one.inject(*_slabs(r, sp.xyz, tets, seed, 8)[0])
    one.step()
    return one.fields(STEP_FIELDS + (("WALL",) if do == "beam" else ()))
