"""Performance cases of the NEP3 library: what its users run, through its public entry points.

A case is a dict of plain values. ``kind`` selects the entry point:

  compute     nep_compute: one evaluation of a structure (energy, forces, per-atom virials)
  md          md_init, md_run (or md_run_ex with the heat current), md_get_state: a short run
              from a fresh state, list builds and the step graph's capture included
  fire        md_init, fire_run, md_get_state: a relaxation of a fixed number of steps
  batch       nep_compute_batch: many small structures (a training set) in one call
  population  nep_eval_population: the loss of a population of candidates on a structure set
  serve       nep.Server: a burst of mixed jobs submitted, awaited and read back

Results are returned in single precision, the precision in which the library computes them
(site energies, forces and virials are FP32 values widened to FP64 on output; a program that
keeps results, trajectory frames or thermo rows keeps them like that). ``exact`` gives the same
quantities in 64 bits from the definitions of the method (descriptors, network and automatic
differentiation in plain torch), so totals and trajectories are held to the true values too.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2205_10046_gb300 import nep, workloads as W

# Published hyper-parameters of the three-species alloy model (n_max = N_bas = 12/8, 50
# neurons): a shape that takes its sizes at run time.
MGALCU_MODEL = dict(n_types=3, rc_radial=6.0, rc_angular=3.5, n_max_radial=12, n_max_angular=8, basis_radial=12,
                    basis_angular=8, l_max_3b=4, l_max_4b=2, l_max_5b=1, n_neuron=50)
# Hyper-parameters, masses and weight seed (the seeds of the repository's workloads: a program
# keeps its model, its structures change).
MODELS = {
    "si": (W.SI_MODEL, [W.MASS_SI], 0),
    "pbte": (W.PBTE_MODEL, [W.MASS_PB, W.MASS_TE], 1),
    "mixed": (W.MIXED_MODEL, [W.MASS_SI, W.MASS_GE, W.MASS_C], 0),
    "mgalcu": (MGALCU_MODEL, [24.305, 26.982, 63.546], 7),
}
# Crystals of the molecular-dynamics workloads: lattice, constant (A), jitter (A), time step (fs), skin (A).
CRYSTALS = {"si": ("diamond", 5.43, 0.05, 1.0, 0.3), "pbte": ("rocksalt", 6.46, 0.1, 2.0, 0.4)}
FIRE_DT = 1.0
FIRE_FMAX = 1e-9  # below any force met here: every step of the relaxation is taken
BATCH_SKIN = 0.4
SERVE_SKIN = 0.4
LAMBDAS = (1.0, 1.0, 0.5, 1e-3, 2e-3)


def listed():
    return [
        # One small structure at a time: an outer program (a relaxer, a sampler) calls the
        # potential on the 216-atom silicon cell. Latency and launches count.
        dict(name="compute_si_216", kind="compute", model="si", n=216, precision=0),
        # A ragged, sheared three-species cell of ordinary size: one single-point evaluation.
        dict(name="compute_mixed_4999", kind="compute", model="mixed", n=4999, precision=0),
        # A published alloy model without a compiled instantiation: the run-time-shape kernels.
        dict(name="compute_mgalcu_20000", kind="compute", model="mgalcu", n=20000, precision=0),
        # The small configuration as stated: 216 silicon atoms, 100 NVE steps, thermo rows.
        dict(name="md_si_216", kind="md", model="si", n=216, precision=0, steps=100, every=10, heat=False),
        # An ordinary simulation cell that does not fill the GPU.
        dict(name="md_si_13824", kind="md", model="si", n=13824, precision=0, steps=50, every=10, heat=False),
        # The lead telluride cell of the thermal-transport runs, with the heat current.
        dict(name="md_pbte_262144", kind="md", model="pbte", n=262144, precision=0, steps=20, every=5, heat=True),
        # Half a million silicon atoms with the split-BF16 tensor-core network.
        dict(name="md_si_512000_split", kind="md", model="si", n=512000, precision=2, steps=20, every=10, heat=False),
        # The largest: 8,000,000 silicon atoms, FP32 network.
        dict(name="md_si_8000000", kind="md", model="si", n=8000000, precision=0, steps=8, every=4, heat=False),
        # The first steps of the relaxation of a distorted alloy cell.
        dict(name="fire_mixed_1001", kind="fire", model="mixed", n=1001, precision=0, steps=20),
        # A training set: structures of 8 to 512 atoms, energies, forces and virials of all.
        dict(name="batch_4096", kind="batch", model="mixed", structures=4096, precision=0),
        # One generation of the evolutionary training: candidates on a subset of the set.
        dict(name="population_32x256", kind="population", model="mixed", structures=256, members=32, precision=0),
        # A burst of mixed requests to the server (single points, relaxations, NVE runs).
        dict(name="serve_48", kind="serve", model="mixed", jobs=48, n_max=4000, precision=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compute", "compute", "md", "md", "md", "fire", "batch", "population", "serve"])
    prec = rng.choice([0, 0, 0, 2])
    if kind == "compute":
        model = rng.choice(["si", "pbte", "mixed", "mgalcu"])
        n = _log(rng, 64, 60000 if model == "mgalcu" else 400000)
        return dict(kind=kind, model=model, n=n, precision=0 if model == "mgalcu" else prec)
    if kind == "md":
        model = rng.choice(["si", "pbte"])
        n = _log(rng, 150, 2000000)
        steps = max(6, min(100, 4 * 10**6 // n))
        return dict(kind=kind, model=model, n=n, precision=prec, steps=steps, every=max(1, steps // 4),
                    heat=rng.random() < 0.3)
    if kind == "fire":
        return dict(kind=kind, model="mixed", n=_log(rng, 40, 20000), precision=0, steps=rng.randint(10, 20))
    if kind == "batch":
        return dict(kind=kind, model="mixed", structures=_log(rng, 4, 4096), precision=prec)
    if kind == "population":
        return dict(kind=kind, model="mixed", structures=_log(rng, 16, 512), members=rng.randint(3, 40), precision=prec)
    return dict(kind=kind, model="mixed", jobs=rng.randint(8, 64), n_max=_log(rng, 200, 4000), precision=0)


# ------------------------------------------------------------------------------- inputs
def _model(case):
    hyper, mass, seed = MODELS[case["model"]]
    return W.random_model(hyper, seed, mass)


def _supercell(n_cells):
    """Near-cubic (nx, ny, nz) with at least n_cells cells."""
    nx = max(1, int(round(n_cells ** (1.0 / 3.0))))
    while nx > 1 and nx ** 3 > n_cells:
        nx -= 1
    ny = max(nx, int(math.ceil(math.sqrt(n_cells / nx) - 1e-9)))
    return nx, ny, int(math.ceil(n_cells / (nx * ny)))


def _crystal(model, n, seed, mass):
    """n atoms of the crystal (vacancies where n is no full supercell), jitter, velocities at
    300 K; positions and velocities [n, 3] FP64 and types [n] int32 on the GPU, the box on the host."""
    kind, a, sigma, _, _ = CRYSTALS[model]
    g = torch.Generator(device="cuda").manual_seed(seed)
    fcc = [[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]]
    other = [[x + .25 for x in r] for r in fcc] if kind == "diamond" else [[(r[0] + .5) % 1.0, r[1], r[2]] for r in fcc]
    frac = torch.tensor(fcc + other, dtype=torch.float64, device="cuda")
    reps = _supercell(-(-n // 8))
    ax = [torch.arange(m, device="cuda", dtype=torch.float64) for m in reps]
    cells = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 1, 3)
    pos = ((cells + frac) * a).reshape(-1, 3)
    types = torch.zeros(pos.shape[0], dtype=torch.int32, device="cuda")
    if kind == "rocksalt":
        types.view(-1, 8)[:, 4:] = 1
    if pos.shape[0] > n:
        keep = torch.randperm(pos.shape[0], generator=g, device="cuda")[:n].sort().values
        pos, types = pos[keep], types[keep]
    pos = pos + sigma * torch.randn(pos.shape, generator=g, dtype=torch.float64, device="cuda")
    m = torch.tensor(mass, dtype=torch.float64, device="cuda")[types.long()][:, None]
    vel = torch.randn(pos.shape, generator=g, dtype=torch.float64, device="cuda") * (
        W.KB_EV * 300.0 / (m * W.AMU_A2_PER_FS2_IN_EV)).sqrt()
    vel -= (m * vel).sum(0) / m.sum()
    return pos.contiguous(), types.contiguous(), vel.contiguous(), np.diag([r * a for r in reps]).astype(np.float64)


def _structure(case, seed, mass):
    if case["model"] in CRYSTALS:
        return _crystal(case["model"], case["n"], seed, mass)
    pos, types, box = W.random_structure(seed, case["n"])
    return torch.tensor(pos, device="cuda"), torch.tensor(types, device="cuda"), None, box


def _jobs(case, seed, mass):
    """Requests of the serving workload: half single points, the rest relaxations and NVE runs."""
    rng = np.random.default_rng(case["jobs"])  # sizes and lengths belong to the case
    jobs = []
    for k in range(case["jobs"]):
        n = int(np.exp(rng.uniform(np.log(32), np.log(case["n_max"]))))
        pos, types, box = W.random_structure(seed * 1009 + k, n)
        kind = (nep.JOB_SINGLE, nep.JOB_FIRE, nep.JOB_SINGLE, nep.JOB_NVE)[k % 4]
        vel = W.maxwell_boltzmann(np.asarray(mass)[types], 300.0, seed * 1013 + k) if kind == nep.JOB_NVE else None
        steps = {nep.JOB_SINGLE: 0, nep.JOB_FIRE: 30, nep.JOB_NVE: int(rng.integers(10, 61))}[kind]
        jobs.append(dict(kind=kind, pos=pos, types=types, box=box, vel=vel, n_steps=steps, dt_fs=1.0, fmax=FIRE_FMAX))
    return jobs


def _structures(case, seed):
    """A structure set of 8 to 512 atoms each (the sizes belong to the case)."""
    sizes = np.random.default_rng(3).integers(8, 513, case["structures"])
    return W.concat_structures([W.random_structure(1000003 * seed + k, int(n)) for k, n in enumerate(sizes)])


def _targets(case, b, seed):
    """Reference labels of a structure set: energy per atom, forces, six virial components per atom."""
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    r = lambda *s: torch.randn(*s, generator=g, dtype=torch.float64, device="cuda")  # noqa: E731
    return 0.1 * r(b.n_struct), 0.05 * r(b.n_atoms, 3), 0.1 * r(b.n_struct, 6)


def _candidates(case, model, seed):
    z0 = model.to_vector()
    rng = np.random.default_rng(seed + 9)
    return np.stack([z0 * (1.0 + 0.1 * rng.standard_normal(z0.shape[0])) for _ in range(case["members"])])


class _Outputs:
    """One FP64 buffer with a view for every output array; kept in single precision in one go."""

    def __init__(self, **shapes):
        sizes = {k: int(np.prod(s)) for k, s in shapes.items()}
        self.flat = torch.zeros(sum(sizes.values()), dtype=torch.float64, device="cuda")
        self.shapes, self.at, o = shapes, {}, 0
        for k, s in shapes.items():
            self.at[k] = (o, o + sizes[k])
            o += sizes[k]
        self.v = {k: self.flat[a:e].view(shapes[k]) for k, (a, e) in self.at.items()}

    def single(self):
        f = self.flat.float()
        return {k: f[a:e].view(self.shapes[k]) for k, (a, e) in self.at.items()}


def prepare(case, seed):
    model = _model(case)
    s = dict(case=case, model=model)
    kind = case["kind"]
    if kind == "serve":
        s["jobs"] = _jobs(case, seed, model.mass)
        s["server"] = nep.Server(model, memory_budget=8 << 30, workers=256, precision=case["precision"],
                                 skin=SERVE_SKIN, compact_every=8, min_chunk=4)
        return s
    skin = CRYSTALS[case["model"]][4] if kind == "md" else BATCH_SKIN if kind in ("batch", "population") else 1.0
    s["nep"] = nep.NEP(model, skin=skin, precision=case["precision"])
    if kind in ("batch", "population"):
        b = _structures(case, seed)
        s["batch"] = b
        s["pos"], s["types"] = torch.tensor(b.pos, device="cuda"), torch.tensor(b.types, device="cuda")
        if kind == "batch":
            s["out"] = _Outputs(E=(b.n_struct,), F=(b.n_atoms, 3), W_struct=(b.n_struct, 9), U=(b.n_atoms,),
                                W=(b.n_atoms, 9))
        else:
            s["z"] = torch.tensor(_candidates(case, model, seed), device="cuda")
            s["targets"] = _targets(case, b, seed)
            s["out"] = _Outputs(loss=(case["members"], 6))
        return s
    s["pos"], s["types"], s["vel"], s["box"] = _structure(case, seed, model.mass)
    n = case["n"]
    if kind == "compute":
        s["out"] = _Outputs(U=(n,), E=(1,), F=(n, 3), W=(n, 9), W_total=(9,))
    elif kind == "md":
        rows = case["steps"] // case["every"]
        more = dict(heat=(rows, 3)) if case["heat"] else {}
        s["out"] = _Outputs(pos=(n, 3), vel=(n, 3), F=(n, 3), thermo=(rows, 4), **more)
    else:
        s["out"] = _Outputs(pos=(n, 3), vel=(n, 3), F=(n, 3), thermo=(case["steps"], 4))
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        return _serve(state["server"], state["jobs"])
    h, o = state["nep"].h, state["out"].v
    if kind == "compute":
        nep.nep_compute(h, state["pos"], state["types"], state["box"], o["U"], o["E"], o["F"], o["W"], o["W_total"])
    elif kind == "md":
        dt = CRYSTALS[case["model"]][3]
        nep.md_init(h, state["pos"], state["types"], state["box"], state["vel"])
        if case["heat"]:
            nep.md_run_ex(h, case["steps"], dt, case["every"], o["thermo"], o["heat"])
        else:
            nep.md_run(h, case["steps"], dt, case["every"], o["thermo"])
        nep.md_get_state(h, o["pos"], o["vel"], o["F"])
    elif kind == "fire":
        nep.md_init(h, state["pos"], state["types"], state["box"])
        nep.fire_run(h, case["steps"], FIRE_DT, FIRE_FMAX, o["thermo"])
        nep.md_get_state(h, o["pos"], o["vel"], o["F"])
    elif kind == "batch":
        b = state["batch"]
        nep.nep_compute_batch(h, b.offsets, state["pos"], state["types"], b.boxes, o["U"], o["E"], o["F"], o["W"],
                              o["W_struct"])
    else:
        b, (e, f, w) = state["batch"], state["targets"]
        nep.nep_eval_population(h, state["z"], b.offsets, state["pos"], state["types"], b.boxes, e, f, w, LAMBDAS,
                                o["loss"])
    return state["out"].single()


def _serve(server, jobs):
    ids = [server.submit(**j) for j in jobs]
    done = {}
    while len(done) < len(jobs):
        r = server.wait(60.0)
        if r is None or r["status"] != 0:
            raise RuntimeError("a served job failed: %s" % (r and r["message"]))
        done[r["id"]] = (r["energy"], r["virial"], *server.arrays(r["id"]))
    got = [done[i] for i in ids]
    out = dict(energy=np.array([g[0] for g in got]), virial=np.stack([g[1] for g in got]),
               pos=np.concatenate([g[2] for g in got]), F=np.concatenate([g[3] for g in got]),
               vel=np.concatenate([g[4] for g in got]))
    return {k: v.astype(np.float32) for k, v in out.items()}


# --------------------------------------------------------------------------------- work
def _density(case):
    """Atoms per cubic Angstrom (random structures: the mean of the three lattices)."""
    if case["model"] in CRYSTALS:
        return 8.0 / CRYSTALS[case["model"]][1] ** 3
    return (4 / 4.05 ** 3 + 2 / 3.30 ** 3 + 8 / 5.43 ** 3) / 3


def _flops_per_evaluation(case):
    """Arithmetic of one atom's evaluation: radial pairs (basis, sums, both force terms),
    angular pairs (basis, g_n, S_nk, both contractions with dU/dS_nk, the polynomials and
    their gradients), the invariants and the network forward and backward."""
    h = MODELS[case["model"]][0]
    nr, na = (_density(case) * 4 / 3 * math.pi * h[k] ** 3 for k in ("rc_radial", "rc_angular"))
    n1, k1, kr = h["n_max_angular"] + 1, h["basis_angular"] + 1, h["basis_radial"]
    des = h["n_max_radial"] + 1 + 6 * n1
    return nr * (13 * kr + 60) + na * (6 * n1 * k1 + 6 * 24 * n1 + 250) + 240 * n1 + h["n_neuron"] * (4 * des + 10)


def work(case):
    """Per pass: every input read once and every result written once; in a run of several steps
    also the state (position, velocity, force) of each step read and written."""
    f = _flops_per_evaluation(case)
    kind = case["kind"]
    if kind == "compute":
        n = case["n"]
        return {"bytes": n * (24 + 4 + 8 + 24 + 72) + 80, "flops": n * f}
    if kind in ("md", "fire"):
        n, k = case["n"], case["steps"]
        return {"bytes": n * (24 + 24 + 4 + 72) + k * n * 2 * 72, "flops": n * f * (k + 1)}
    if kind == "batch":
        n = 260 * case["structures"]
        return {"bytes": n * (24 + 4 + 8 + 24 + 72) + case["structures"] * 160, "flops": n * f}
    if kind == "population":
        n = 260 * case["structures"]
        return {"bytes": n * (24 + 4 + 24) + case["structures"] * 130, "flops": n * f * case["members"]}
    n = case["jobs"] * (case["n_max"] - 32) / math.log(case["n_max"] / 32)
    return {"bytes": n * (24 + 4 + 24 + 72), "flops": n * f * (1 + 0.25 * 30 + 0.25 * 35)}


# -------------------------------------------------------------------------------- exact
# The method in 64 bits from its definitions, in plain torch.
C3B = [3, 3, 3, 5 / 4, 15, 15, 15 / 4, 15 / 4, 7 / 4, 21 / 8, 21 / 8, 105 / 4, 105 / 4, 35 / 8, 35 / 8, 9 / 64,
       45 / 8, 45 / 8, 45 / 16, 45 / 16, 315 / 8, 315 / 8, 315 / 64, 315 / 64]
Y20, Y21, Y22 = (0.25 * math.sqrt(5 / math.pi), 0.5 * math.sqrt(7.5 / math.pi), 0.25 * math.sqrt(7.5 / math.pi))
C4B = [-math.sqrt(2 / 35) * Y20 ** 3, -6 * math.sqrt(1 / 70) * Y20 * Y21 ** 2, 6 * math.sqrt(2 / 35) * Y20 * Y22 ** 2,
       6 * math.sqrt(3 / 35) * Y21 ** 2 * Y22, -12 * math.sqrt(3 / 35) * Y21 ** 2 * Y22]
C5B = [21 / (80 * math.pi ** 2), 21 / (40 * math.pi ** 2), 21 / (80 * math.pi ** 2)]


def _harmonics(u):
    x, y, z = u.unbind(1)
    z2, c2, s2 = z * z, x * x - y * y, 2 * x * y
    c3, s3 = (x * x - 3 * y * y) * x, (3 * x * x - y * y) * y
    return torch.stack([
        z, x, y, 3 * z2 - 1, x * z, y * z, c2, s2, (5 * z2 - 3) * z, (5 * z2 - 1) * x, (5 * z2 - 1) * y, c2 * z, s2 * z,
        c3, s3, (35 * z2 - 30) * z2 + 3, (7 * z2 - 3) * x * z, (7 * z2 - 3) * y * z, (7 * z2 - 1) * c2,
        (7 * z2 - 1) * s2, c3 * z, s3 * z, c2 * c2 - s2 * s2, 2 * c2 * s2], 1)


def _basis(r, rc, k_max):
    x = 2 * (r / rc - 1) ** 2 - 1
    t = [torch.ones_like(x), x]
    while len(t) <= k_max:
        t.append(2 * x * t[-1] - t[-2])
    fc = 0.5 * (1 + torch.cos(math.pi * r / rc))
    return 0.5 * (torch.stack(t[:k_max + 1], 1) + 1) * fc[:, None]


def _find_pairs(pos, box, rc):
    """(i, j, d) of every ordered pair, all images, |d| < rc; sorted by i."""
    H = torch.tensor(np.asarray(box), dtype=torch.float64, device=pos.device)
    Hi = torch.linalg.inv(H)
    s = pos @ Hi
    s = s - s.floor()
    thick = (1.0 / Hi.norm(dim=0)).tolist()
    x = s @ H
    n = pos.shape[0]
    nc = [int(t / rc) for t in thick]
    if n <= 4096 or min(nc) < 3:
        R = [int(math.ceil(rc / t)) for t in thick]
        sh = torch.stack(torch.meshgrid(*[torch.arange(-r, r + 1, device=pos.device) for r in R], indexing="ij"), -1)
        sh = sh.reshape(-1, 3).double() @ H
        out = []
        step = max(1, int(6e7 // (n * sh.shape[0])))
        for a in range(0, n, step):
            d = x[None, :, None, :] - x[a:a + step, None, None, :] + sh
            r2 = (d * d).sum(-1)
            i, j, m = torch.nonzero((r2 < rc * rc) & (r2 > 1e-12), as_tuple=True)
            out.append((i + a, j, d[i, j, m]))
        return [torch.cat(v) for v in zip(*out)]
    ncs = torch.tensor(nc, device=pos.device)
    c = torch.minimum((s * ncs).long(), ncs - 1)
    cid = (c[:, 0] * nc[1] + c[:, 1]) * nc[2] + c[:, 2]
    order = cid.argsort()
    cnt = torch.bincount(cid, minlength=nc[0] * nc[1] * nc[2])
    start = cnt.cumsum(0) - cnt
    width = int(cnt.max())
    table = torch.full((cnt.shape[0], width), -1, dtype=torch.long, device=pos.device)
    table[cid[order], torch.arange(n, device=pos.device) - start[cid[order]]] = order
    out = []
    for ox in (-1, 0, 1):
        for oy in (-1, 0, 1):
            for oz in (-1, 0, 1):
                nb = c + torch.tensor([ox, oy, oz], device=pos.device)
                k = torch.div(nb, ncs, rounding_mode="floor")
                nb = nb - k * ncs
                shift = k.double() @ H
                rows = table[(nb[:, 0] * nc[1] + nb[:, 1]) * nc[2] + nb[:, 2]]
                for w in range(width):
                    j = rows[:, w]
                    i = torch.nonzero(j >= 0).squeeze(1)
                    j = j[i]
                    d = x[j] - x[i] + shift[i]
                    r2 = (d * d).sum(1)
                    ok = (r2 < rc * rc) & (r2 > 1e-12)
                    out.append((i[ok], j[ok], d[ok]))
    i, j, d = [torch.cat(v) for v in zip(*out)]
    o = i.argsort()
    return [i[o], j[o], d[o]]


class _Exact:
    """Site energies, forces and per-atom virials of one model from the pairs of a structure."""

    def __init__(self, model):
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        self.m = model
        self.cR, self.cA, self.w0, self.b0, self.w1 = map(t, (model.c_radial, model.c_angular, model.w0, model.b0, model.w1))
        self.b1 = float(model.b1)
        self.c3 = t(C3B) / (4 * math.pi)

    def sites(self, types, i, j, d, n):
        """U_i of n atoms whose pairs are (i, j, d); types of all atoms, i counted from 0."""
        m, T = self.m, self.m.n_types
        ti, tj = types[0][i].long(), types[1][j].long()
        r = d.norm(dim=1)
        k = torch.nonzero(r < m.rc_radial).squeeze(1)
        f = _basis(r[k], m.rc_radial, m.basis_radial)
        A = torch.zeros(n * T, f.shape[1], dtype=f.dtype, device=f.device).index_add(0, i[k] * T + tj[k], f)
        qr = torch.einsum("itk,itnk->in", A.view(n, T, -1), self.cR[types[0].long()])
        k = torch.nonzero(r < m.rc_angular).squeeze(1)
        f = _basis(r[k], m.rc_angular, m.basis_angular)
        g = f @ self.cA[0, 0].T if T == 1 else torch.einsum("pk,pnk->pn", f, self.cA[ti[k], tj[k]])
        b = _harmonics(d[k] / r[k, None])
        n1 = g.shape[1]
        S = torch.zeros(n, n1 * 24, dtype=f.dtype, device=f.device)
        S = S.index_add(0, i[k], (g[:, :, None] * b[:, None, :]).reshape(-1, n1 * 24)).view(n, n1, 24)
        q3 = S * S * self.c3
        q = [qr] + [q3[:, :, a:e].sum(2) for a, e in ((0, 3), (3, 8), (8, 15), (15, 24))[:m.l_max_3b]]
        if m.l_max_4b >= 2:
            s3, s4, s5, s6, s7 = S[:, :, 3:8].unbind(2)
            q.append(C4B[0] * s3 ** 3 + C4B[1] * s3 * (s4 ** 2 + s5 ** 2) + C4B[2] * s3 * (s6 ** 2 + s7 ** 2)
                     + C4B[3] * s6 * (s5 ** 2 - s4 ** 2) + C4B[4] * s4 * s5 * s7)
        if m.l_max_5b >= 1:
            s0, s12 = S[:, :, 0], S[:, :, 1] ** 2 + S[:, :, 2] ** 2
            q.append(C5B[0] * s0 ** 4 + C5B[1] * s0 ** 2 * s12 + C5B[2] * s12 ** 2)
        return torch.tanh(torch.cat(q, 1) @ self.w0.T - self.b0) @ self.w1 - self.b1

    def evaluate(self, types, pairs, n, virial=True, chunk=65536):
        i, j, d = pairs
        U, P = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty_like(d)
        bounds = torch.searchsorted(i, torch.arange(0, n + chunk, chunk, device="cuda").clamp(max=n)).tolist()
        for c, a in enumerate(range(0, n, chunk)):
            e, p0, p1 = min(n, a + chunk), bounds[c], bounds[c + 1]
            dd = d[p0:p1].detach().requires_grad_(True)
            u = self.sites((types[a:e], types), i[p0:p1] - a, j[p0:p1], dd, e - a)
            P[p0:p1] = torch.autograd.grad(u.sum(), dd)[0]
            U[a:e] = u.detach()
        F = torch.zeros(n, 3, dtype=torch.float64, device="cuda").index_add(0, i, P).index_add(0, j, -P)
        if not virial:
            return U, F, None
        # W_j = sum over its neighbours i of (r_i - r_j) (x) dU_i/dr_ij, dU_i/dr_ij the pair's gradient
        Wm = torch.zeros(n, 9, dtype=torch.float64, device="cuda")
        Wm.index_add_(0, j, (-d[:, :, None] * P[:, None, :]).reshape(-1, 9))
        return U, F, Wm[:, [0, 4, 8, 1, 2, 5, 3, 6, 7]]

    def single(self, pos, types, box, virial=True):
        rc = self.m.rc_radial
        return self.evaluate(types, _find_pairs(pos, box, rc), pos.shape[0], virial)


class _Track:
    """Forces along a trajectory: the pairs are searched with a margin and kept while they hold."""

    def __init__(self, ex, types, box):
        self.ex, self.types, self.box, self.ref = ex, types, box, None

    def __call__(self, x, virial=False):
        if self.ref is None or float((x - self.ref).norm(dim=1).max()) > 0.45:
            self.i, self.j, d = _find_pairs(x, self.box, self.ex.m.rc_radial + 1.0)
            self.shift, self.ref = d - (x[self.j] - x[self.i]), x.clone()
        d = x[self.j] - x[self.i] + self.shift
        k = torch.nonzero((d * d).sum(1) < self.ex.m.rc_radial ** 2).squeeze(1)
        return self.ex.evaluate(self.types, (self.i[k], self.j[k], d[k]), x.shape[0], virial)


def _wrap(x, box):
    H = torch.tensor(np.asarray(box), dtype=torch.float64, device=x.device)
    s = x @ torch.linalg.inv(H)
    return (s - s.floor()) @ H


def _thermo(U, Wm, v, m, box):
    ke = 0.5 * float((m * v * v).sum())
    n = v.shape[0]
    vol = abs(float(np.linalg.det(np.asarray(box))))
    p = (2 * ke + float(Wm[:, :3].sum())) / (3 * vol) * 160.21766208
    return [float(U.sum()), ke, 2 * ke / ((3 * n - 3) * W.KB_EV), p]


def _trajectory(ex, x, v, types, box, steps, dt, every, fire=False):
    """Velocity Verlet, or FIRE (Bitzek et al. 2006), with thermo rows and heat currents."""
    m = torch.tensor(ex.m.mass, device="cuda")[types.long()][:, None] * W.AMU_A2_PER_FS2_IN_EV
    force = _Track(ex, types, box)
    U, F, _ = force(x)
    rows, heat = [], []
    alpha, n_pos, dt_max = 0.1, 0, 10 * dt
    for s in range(1, steps + 1):
        v = v + 0.5 * dt * F / m
        x = x + dt * v
        row = every and s % every == 0
        U, F, Wm = force(x, virial=bool(row))
        v = v + 0.5 * dt * F / m
        if row:
            rows.append(_thermo(U, Wm, v, m, box))
            a = Wm[:, [0, 3, 4, 6, 1, 5, 7, 8, 2]].view(-1, 3, 3)
            heat.append(torch.einsum("iab,ib->a", a, v))
        if fire:
            p = float((F * v).sum())
            if p > 0:
                v = (1 - alpha) * v + alpha * v.norm() / F.norm() * F
                if n_pos > 5:
                    dt, alpha = min(1.1 * dt, dt_max), 0.99 * alpha
                n_pos += 1
            else:
                v, dt, alpha, n_pos = torch.zeros_like(v), 0.5 * dt, 0.1, 0
    return _wrap(x, box), v, U, F, rows, heat


def exact(case, seed):
    kind = case["kind"]
    model = _model(case)
    ex = _Exact(model)
    if kind == "compute":
        if case["n"] > 400000:
            return None
        pos, types, _, box = _structure(case, seed, model.mass)
        U, F, Wm = ex.single(pos, types, box)
        return dict(U=U, E=U.sum().view(1), F=F, W=Wm, W_total=Wm.sum(0))
    if kind in ("md", "fire"):
        if case["n"] * case["steps"] > 11e6:  # more than about 20 seconds
            return None
        pos, types, vel, box = _structure(case, seed, model.mass)
        fire = kind == "fire"
        dt, every = (FIRE_DT, 1) if fire else (CRYSTALS[case["model"]][3], case["every"])
        x, v, _, F, rows, heat = _trajectory(ex, pos, torch.zeros_like(pos) if fire else vel, types, box, case["steps"],
                                             dt, every, fire)
        out = dict(pos=x, vel=v, F=F, thermo=torch.tensor(rows, dtype=torch.float64))
        if fire:
            # a row holds the kinetic energy and temperature before the step's velocity mixing
            return out
        if case["heat"]:
            out["heat"] = torch.stack(heat)
        return out
    if kind in ("batch", "population"):
        b = _structures(case, seed)
        pos, types = torch.tensor(b.pos, device="cuda"), torch.tensor(b.types, device="cuda")
        parts = []
        for s in range(b.n_struct):
            a, e = int(b.offsets[s]), int(b.offsets[s + 1])
            i, j, d = _find_pairs(pos[a:e], b.boxes[s], model.rc_radial)
            parts.append((i + a, j + a, d))
        pairs = [torch.cat(v) for v in zip(*parts)]
        sid = torch.repeat_interleave(torch.arange(b.n_struct, device="cuda"),
                                      torch.tensor(np.diff(b.offsets), device="cuda").long())
        per = lambda v: torch.zeros((b.n_struct,) + v.shape[1:], dtype=v.dtype, device="cuda").index_add(0, sid, v)  # noqa: E731
        if kind == "batch":
            U, F, Wm = ex.evaluate(types, pairs, b.n_atoms)
            return dict(E=per(U), F=F, W_struct=per(Wm), U=U, W=Wm)
        e_tar, f_tar, w_tar = _targets(case, b, seed)
        cnt = torch.tensor(np.diff(b.offsets), device="cuda").double()
        rms = lambda v: float(v.square().mean().sqrt())  # noqa: E731
        rows = []
        for z in _candidates(case, model, seed):
            U, F, Wm = _Exact(model.with_vector(z)).evaluate(types, pairs, b.n_atoms)
            w = per(Wm) / cnt[:, None]
            w6 = torch.stack([w[:, 0], w[:, 1], w[:, 2], (w[:, 3] + w[:, 6]) / 2, (w[:, 5] + w[:, 8]) / 2,
                              (w[:, 4] + w[:, 7]) / 2], 1)
            t = [rms(per(U) / cnt - e_tar), rms(F - f_tar), rms(w6 - w_tar), float(np.abs(z).mean()),
                 float(np.sqrt(np.square(z).mean()))]
            rows.append([sum(a * b_ for a, b_ in zip(LAMBDAS, t))] + t)
        return dict(loss=torch.tensor(rows, dtype=torch.float64))
    got = []
    for j in _jobs(case, seed, model.mass):
        pos, types = torch.tensor(j["pos"], device="cuda"), torch.tensor(j["types"], device="cuda")
        v = torch.zeros_like(pos) if j["vel"] is None else torch.tensor(j["vel"], device="cuda")
        x, v, _, _, _, _ = _trajectory(ex, pos, v, types, j["box"], j["n_steps"], j["dt_fs"], 0,
                                       j["kind"] == nep.JOB_FIRE)
        U, F, Wm = ex.single(x, types, j["box"])
        if j["kind"] == nep.JOB_FIRE:  # a relaxed structure is handed back at rest
            v = torch.zeros_like(v)
        got.append((float(U.sum()), Wm.sum(0), x, F, v))
    return dict(energy=torch.tensor([g[0] for g in got], dtype=torch.float64), virial=torch.stack([g[1] for g in got]),
                pos=torch.cat([g[2] for g in got]), F=torch.cat([g[3] for g in got]), vel=torch.cat([g[4] for g in got]))
