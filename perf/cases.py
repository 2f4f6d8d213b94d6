"""The work this framework is used for, as cases of one timed pass each, through its public entry points.

Kinds of work (see `listed` for what each listed case stands for):
  eval    energies, forces, virial and charges of successive frames of one structure (an external driver, a sampler)
  energy  the autograd energy of a batch of configurations, forward and backward (a fitting or learning program)
  md      molecular dynamics: some steps, then the state read back; one system or an ensemble of replicas, NVE or NVT
  grad    the force-matching loss and its gradient with respect to the 144 potential parameters, at two parameter sets
  screen  the removal energies of every surface Si of a slab
  relax   FIRE iterations of a slab from its unrelaxed positions
  rings   the primitive C rings of an ensemble

Results of the FP64 policy are taken as float64, those of the mixed policy (FP32 terms) as float32, the type a program
that holds them beside its own single-precision tensors gives them.

`exact` restates the model in plain torch in 64 bits: pair lists by testing every pair of atoms, energies as sums over
pairs and triplets, forces by automatic differentiation, charges by conjugate gradients on the sparse Hessian.
"""
import functools
import math

import numpy as np
import torch

from paper_1802_07871_gb300 import autograd, ctbop, desorption, rings
from paper_1802_07871_gb300 import structures as st

DT = 0.5          # fs
TAU = 100.0       # fs, thermostat
EXACT_ATOMS = 30_000


# ---------------------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest calls: a sampler or an external MD driver on a 64-atom cell, everything in FP64
        {"name": "eval 64 atoms fp64", "kind": "eval", "precision": "fp64", "cells": 2, "cells_z": 2, "frames": 2},
        # the small crystal of the plain FP64 method: NVE at 300 K, read every ten steps
        {"name": "md 512 atoms fp64", "kind": "md", "precision": "fp64", "shape": "bulk", "cells": 4, "T": 300.0,
         "nvt": False, "steps": 10},
        # a learning program's minibatch of fitting configurations: energies forward, forces backward
        {"name": "energy 32 configs mixed", "kind": "energy", "precision": "mixed", "configs": 32, "frames": 2},
        # a production run of the paper's size (a growth cell of about 12,000 atoms, NVT at 2500 K)
        {"name": "md 12k nvt mixed", "kind": "md", "precision": "mixed", "shape": "slab", "nx": 24, "ny": 14, "nb": 10,
         "T": 2500.0, "nvt": True, "steps": 20},
        # the stepped slab of about 20,000 atoms at 2000 K on the FP64 path (reference trajectories)
        {"name": "md 20k fp64", "kind": "md", "precision": "fp64", "shape": "slab", "nx": 24, "ny": 14, "nb": 16,
         "T": 2000.0, "nvt": False, "steps": 4},
        # the headline: the stepped slab of about a million atoms at 2500 K, mixed precision
        {"name": "md 1m mixed", "kind": "md", "precision": "mixed", "shape": "slab", "nx": 96, "ny": 48, "nb": 56,
         "T": 2500.0, "nvt": False, "steps": 4},
        # the annealing ensemble: uneven replicas (defected slabs, amorphous C, graphene on SiC), each with its thermostat
        {"name": "md ensemble 96 nvt mixed", "kind": "md", "precision": "mixed", "shape": "ensemble", "replicas": 96,
         "n_max": 3000, "nvt": True, "steps": 10},
        # one epoch's gradient of a parameter fit, mixed precision
        {"name": "grad 192 configs mixed", "kind": "grad", "precision": "mixed", "configs": 192},
        # the same in FP64 on a small batch (checks, the last steps of a fit)
        {"name": "grad 24 configs fp64", "kind": "grad", "precision": "fp64", "configs": 24},
        # desorption screening between MD intervals: every surface Si, each a full evaluation without it
        {"name": "screen 4k slab mixed", "kind": "screen", "precision": "mixed", "nx": 16, "ny": 8, "nb": 10},
        # relaxing a generated slab before it is used
        {"name": "relax 20k mixed", "kind": "relax", "precision": "mixed", "nx": 24, "ny": 14, "nb": 16, "iters": 25},
        # analysis of saved frames: the ring statistics of an ensemble
        {"name": "rings 96 replicas mixed", "kind": "rings", "precision": "mixed", "replicas": 96, "n_max": 3000},
    ]


def _slab_size(rng, lo, hi):
    """Cells and bilayers of a slab of about lo..hi atoms (log-uniform), odd ones among them."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nb = min(max(5, int(round((n / 16.0) ** (1.0 / 3.0) * rng.uniform(0.8, 1.4)))), 56)
    per = max(12.0, n / (4.0 * nb))
    ny = max(3, int(round(math.sqrt(per / math.sqrt(3.0)))))
    return {"nx": max(4, int(round(per / ny))), "ny": ny, "nb": nb}


def draw(rng):
    kind = rng.choice(("eval", "energy", "md", "md", "md", "grad", "screen", "relax", "rings"))
    prec = rng.choice(("mixed", "mixed", "fp64"))
    logint = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    if kind == "eval":
        return {"kind": kind, "precision": prec, "cells": rng.randint(2, 9), "cells_z": rng.randint(2, 9),
                "frames": rng.randint(1, 3)}
    if kind == "energy":
        return {"kind": kind, "precision": prec, "configs": logint(3, 128 if prec == "mixed" else 32), "frames": 2}
    if kind == "md":
        shape = rng.choice(("bulk", "slab", "slab", "ensemble"))
        case = {"kind": kind, "precision": prec, "shape": shape, "nvt": rng.random() < 0.5, "steps": rng.randint(3, 12)}
        if shape == "bulk":
            return {**case, "cells": rng.randint(2, 12 if prec == "mixed" else 8), "T": round(rng.uniform(200, 1500), 1)}
        if shape == "slab":
            return {**case, **_slab_size(rng, 500, 300_000 if prec == "mixed" else 20_000),
                    "T": round(rng.uniform(1500, 3000), 1)}
        return {**case, "replicas": logint(3, 96 if prec == "mixed" else 16), "n_max": rng.randint(400, 3000)}
    if kind == "grad":
        return {"kind": kind, "precision": prec, "configs": logint(3, 192 if prec == "mixed" else 24)}
    if kind == "screen":
        return {"kind": kind, "precision": "mixed", **_slab_size(rng, 600, 3_500)}
    if kind == "relax":
        return {"kind": kind, "precision": prec, "iters": rng.randint(8, 25),
                **_slab_size(rng, 500, 20_000 if prec == "mixed" else 5_000)}
    return {"kind": "rings", "precision": prec, "replicas": logint(2, 96), "n_max": rng.randint(400, 3000)}


# --------------------------------------------------------------------------------------------------------- the inputs
@functools.lru_cache(maxsize=4)
def _slab_base(nx, ny, nb, adatoms=True):
    s = st.sic_4h_slab(nx, ny, nb, step="staircase")
    n = s.n
    return (st.add_adatoms(s, max(1, int(round(0.05 * s.meta["atoms_per_bilayer"])))) if adatoms else s), n


_batch = functools.lru_cache(maxsize=4)(lambda configs: st.differentiation_batch(configs))
_ensemble = functools.lru_cache(maxsize=2)(lambda replicas, n_max: st.annealing_ensemble(replicas, n_max=n_max))


def _moved(s, seed, sigma, n=None):
    """The structure with its first n atoms (all of them by default), unless frozen, displaced by a clipped noise."""
    n = s.n if n is None else n
    x = s.x.copy()
    d = np.clip(np.random.default_rng(seed).normal(0.0, sigma, (n, 3)), -2.5 * sigma, 2.5 * sigma)
    d[s.frozen[:n]] = 0.0
    x[:n] += d
    return st.Structure(s.name, x, s.types, s.box, s.pbc, s.frozen)


def _structures(case, seed):
    """The case's structures and, for MD, their temperatures: the seed moves the atoms, the sizes are the case's."""
    kind = case["kind"]
    if kind in ("energy", "grad"):
        return [_moved(s, seed + r, 0.01) for r, s in enumerate(_batch(case["configs"]))], None
    if kind == "eval":
        return [st.sic_3c((case["cells"], case["cells"], case["cells_z"]), 4.36, 0.05, seed)], None
    if kind in ("screen", "relax"):
        s, n = _slab_base(case["nx"], case["ny"], case["nb"], kind == "relax")
        return [_moved(s, seed, 0.03, n)], None
    if kind == "rings" or case["shape"] == "ensemble":
        structs, temps = _ensemble(case["replicas"], case["n_max"])
        return [_moved(s, seed + r, 0.01) for r, s in enumerate(structs)], temps
    if case["shape"] == "bulk":
        return [st.sic_3c(case["cells"], 4.36, 0.05, seed)], [case["T"]]
    s, n = _slab_base(case["nx"], case["ny"], case["nb"])
    return [_moved(s, seed, 0.1 * math.sqrt(case["T"] / 2500.0), n)], [case["T"]]   # the adatoms stay where they are


def _velocities(structs, temps, seed):
    return np.concatenate([st.maxwell_boltzmann(s.types, T, seed=seed + 1 + r, frozen=s.frozen)
                           for r, (s, T) in enumerate(zip(structs, temps))])


def _frames(case, structs, seed):
    """Positions of successive frames: the structures with another small displacement each."""
    rng = np.random.default_rng(seed + 77)
    x = np.concatenate([s.x for s in structs])
    return [x + rng.uniform(-0.02, 0.02, x.shape) for _ in range(case["frames"])]


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _thetas(params, seed, dtype):
    """Two points of a fit: the parameter set with each constant moved by a per mille or so."""
    rng = np.random.default_rng(seed + 5)
    v = ctbop.params_vector(ctbop.params_struct(params))
    out = []
    for _ in range(2):
        w = ctbop.params_from_vector(v)
        for name in ("A", "B", "kappa"):
            f = rng.uniform(0.999, 1.001, 3)
            a = getattr(w, name)
            a[0], a[1], a[2], a[3] = a[0] * f[0], a[1] * f[1], a[2] * f[1], a[3] * f[2]
        for t in range(2):
            w.chi[t] *= rng.uniform(0.999, 1.001)
            w.J[t] *= rng.uniform(0.999, 1.001)
        out.append(torch.tensor(ctbop.params_vector(w), dtype=dtype))
    return out


def _targets(structs, seed):
    """Fitting targets and weights: energies and forces of another level of theory, as noise about plausible values."""
    rng = np.random.default_rng(seed + 9)
    n = np.array([s.n for s in structs], dtype=np.float64)
    return dict(w_E=1.0 / n ** 2, E_ref=-6.3 * n + rng.normal(0.0, 0.1, len(n)) * n, w_F=1.0 / (3.0 * n),
                F_ref=rng.normal(0.0, 1.0, (int(n.sum()), 3)))


def prepare(case, seed):
    P = st.load_params("p1")
    structs, temps = _structures(case, seed)
    kind, dtype = case["kind"], _dtype(case)
    sysm = ctbop.System(P, precision=case["precision"])
    if len(structs) == 1:
        sysm.load(structs[0])
    else:
        sysm.load_replicas(structs)
    n, r = sysm.n, sysm.R
    state = {"case": case, "sys": sysm, "dtype": dtype}
    size = {"energy": (r,), "virial": (r, 3, 3), "thermostat": (r, 4), "charges": (n,)}
    names = {"eval": ("energy", "forces", "virial", "charges"), "relax": ("positions", "energy"),
             "md": ("positions", "velocities", "forces", "charges", "energy")}.get(kind, ())
    if case.get("nvt"):
        names += ("thermostat",)
    state["out"] = {k: torch.empty(size.get(k, (n, 3)), dtype=torch.float64, device="cuda") for k in names}
    if kind == "md":
        sysm.set_velocities(torch.tensor(_velocities(structs, temps, seed), device="cuda"))
        if case["nvt"]:
            sysm.set_thermostat(np.array(temps), TAU)
    elif kind == "eval":
        state["frames"] = [torch.tensor(x, device="cuda") for x in _frames(case, structs, seed)]
    elif kind == "energy":
        state["frames"] = [torch.tensor(x, dtype=dtype, device="cuda").requires_grad_(True)
                           for x in _frames(case, structs, seed)]
    elif kind == "grad":
        state["theta"] = [t.requires_grad_(True) for t in _thetas(P, seed, dtype)]
        state["targets"] = _targets(structs, seed)
    elif kind == "relax":
        state["x0"] = torch.tensor(structs[0].x, device="cuda")
    elif kind == "screen":
        state["types"], state["frozen"] = structs[0].types, structs[0].frozen
    sysm.compute()
    return state


# ------------------------------------------------------------------------------------------------------------ one pass
def _read(state):
    out = {}
    for name, buf in state["out"].items():
        state["sys"].get(name, out=buf)
        out[name] = buf.to(state["dtype"], copy=True)
    return out


def run(state):
    case, sysm = state["case"], state["sys"]
    kind = case["kind"]
    if kind == "eval":
        outs = []
        for x in state["frames"]:
            sysm.set_positions(x)
            sysm.compute()
            outs.append(_read(state))
        return outs
    if kind == "energy":
        outs = []
        for x in state["frames"]:
            E = autograd.Energy.apply(x, sysm)
            (g,) = torch.autograd.grad(E.sum(), x)
            outs.append({"E": E.detach(), "dE_dx": g})
        return outs
    if kind == "md":
        sysm.step(case["steps"], DT)
        return _read(state)
    if kind == "grad":
        outs = []
        for theta in state["theta"]:
            loss = autograd.ForceMatchingLoss.apply(theta, sysm, *(state["targets"][k] for k in ("w_E", "E_ref", "w_F",
                                                                                               "F_ref")))
            (g,) = torch.autograd.grad(loss, theta)
            outs.append({"loss": loss.detach(), "dtheta": g})
        return outs
    if kind == "screen":
        cand, _ = desorption.surface_si(sysm, state["types"], state["frozen"])
        dE = sysm.removal_energies(cand)
        return {"candidates": cand, "dE": dE.astype(np.float32)}
    if kind == "relax":
        sysm.set_positions(state["x0"])
        iters, fmax = sysm.minimize(max_iter=case["iters"], fmax=1e-3)
        return {"iters": iters, "fmax": fmax.astype(np.float64 if state["dtype"] is torch.float64 else np.float32),
                **_read(state)}
    rec = sysm.rings()
    return {"counts": rings.counts(rec, sysm.R), "orientation": rings.orientation_histogram(rec)}


# ------------------------------------------------------------------------------------------------------------- the work
# per atom and evaluation: 195 neighbours inside the charge cutoff (each pair once: kernel and derivative), four bonds,
# twelve triplets, and a charge solve of a dozen matrix products over the same neighbours
FLOPS_PAIR, FLOPS_BOND, FLOPS_SOLVE = 195 / 2 * 45.0, 4 * 50.0 + 12 * 130.0, 12 * 195 * 2.0
FLOPS_EVAL = FLOPS_PAIR + FLOPS_BOND + FLOPS_SOLVE


def _atoms(case):
    kind = case["kind"]
    if kind in ("energy", "grad"):
        return 288.0 * case["configs"]
    if kind == "eval":
        return 8.0 * case["cells"] ** 2 * case["cells_z"]
    if kind == "rings" or case.get("shape") == "ensemble":
        return case["replicas"] * (200 + case["n_max"]) / 2.0
    if case.get("shape") == "bulk":
        return 8.0 * case["cells"] ** 3
    return 4.0 * case["nx"] * case["ny"] * (case["nb"] - 1.5)


def work(case):
    n, kind = _atoms(case), case["kind"]
    w = 8.0 if case["precision"] == "fp64" else 4.0
    if kind == "eval":
        return {"bytes": case["frames"] * n * (24 + 4 * w), "flops": case["frames"] * n * FLOPS_EVAL}
    if kind == "energy":
        return {"bytes": case["frames"] * n * 6 * w, "flops": case["frames"] * n * FLOPS_EVAL}
    if kind == "md":
        return {"bytes": n * (2 * 48 + 4 * w), "flops": case["steps"] * n * FLOPS_EVAL}
    if kind == "grad":      # two parameter sets; an evaluation, an adjoint solve and the derivatives of every term
        return {"bytes": n * 52.0, "flops": 2 * n * (2 * FLOPS_EVAL + 2 * (FLOPS_PAIR + 3 * FLOPS_BOND))}
    if kind == "screen":    # every surface Si: about one bilayer's worth of candidates
        cand = 2.0 * case["nx"] * case["ny"]
        return {"bytes": n * 40 + cand * 8, "flops": cand * n * (FLOPS_EVAL - FLOPS_BOND / 2)}
    if kind == "relax":
        return {"bytes": n * (24 + 3 * w), "flops": case["iters"] * n * FLOPS_EVAL}
    return {"bytes": n * 30.0, "flops": n * 3000.0}


# ------------------------------------------------------------------------------------------- the same in plain 64 bits
_ACC, _KB = 9.648533212e-3, 8.617333262e-5


def _tables(theta):
    """Named tables of a parameter vector (the 144 doubles of the parameter struct)."""
    t, at = {}, 0
    for name, shape in ([(k, (2, 2)) for k in ("A", "B", "l1", "l2", "R", "S", "kappa", "sigma", "p")]
                        + [(k, (2, 2, 2)) for k in ("g", "n")]
                        + [(k, (2, 2, 2, 2)) for k in ("gam", "c", "d", "h", "alpha")]
                        + [(k, (2,)) for k in ("E0", "chi", "J", "gc", "mass")] + [("rc", ()), ("ke", ())]):
        m = int(np.prod(shape)) if shape else 1
        t[name] = theta[at:at + m].reshape(shape)
        at += m
    return t


def _pairs(x, box, pbc, rc):
    """Every directed pair (i, j, shift) closer than rc, over all periodic images, by testing all of them."""
    n = len(x)
    spans = [range(-int(math.ceil(rc / L)), int(math.ceil(rc / L)) + 1) if p else (0,) for L, p in zip(box, pbc)]
    out, step = [], max(1, 40_000_000 // max(n, 1))
    lo, hi = x.amin(0), x.amax(0)
    for a in spans[0]:
        for b in spans[1]:
            for c in spans[2]:
                s = torch.tensor([a * box[0], b * box[1], c * box[2]], dtype=x.dtype, device=x.device)
                J = torch.nonzero(((x + s > lo - rc) & (x + s < hi + rc)).all(1)).flatten()
                I = torch.nonzero(((x > lo + s - rc) & (x < hi + s + rc)).all(1)).flatten()
                if not len(I) or not len(J):
                    continue
                for k in range(0, len(I), step):
                    i = I[k:k + step]
                    r2 = sum((x[J, d][None] + s[d] - x[i, d][:, None]) ** 2 for d in range(3))
                    u, v = torch.nonzero((r2 < rc * rc) & (r2 > 0), as_tuple=True)
                    out.append((i[u], J[v], s.expand(len(u), 3)))
    return tuple(torch.cat(v) for v in zip(*out))


class _Model:
    """The potential on a batch of structures, energies and their derivatives by automatic differentiation."""

    def __init__(self, structs, theta, margin=0.0):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.structs, self.margin = structs, margin
        self.theta = torch.as_tensor(np.asarray(theta, dtype=np.float64), device=self.dev)
        self.type = torch.tensor(np.concatenate([s.types for s in structs]), dtype=torch.long, device=self.dev)
        self.rep = torch.tensor(np.repeat(np.arange(len(structs)), [s.n for s in structs]), device=self.dev)
        self.n, self.R = len(self.type), len(structs)
        self.x_list = None
        self.sol = None

    def lists(self, x):
        """Pairs and triplets for positions within half the margin of these."""
        if self.x_list is not None and float((x - self.x_list).norm(dim=1).max()) < self.margin / 2:
            return
        t = _tables(self.theta)
        rc, smax = float(t["rc"]) + self.margin, float(t["S"].max()) + self.margin
        parts, at = [], 0
        for s in self.structs:
            i, j, sh = _pairs(x[at:at + s.n], s.box, s.pbc, rc)
            parts.append((i + at, j + at, sh))
            at += s.n
        i, j, sh = (torch.cat(v) for v in zip(*parts))
        order = torch.argsort(i, stable=True)
        self.ci, self.cj, self.cs = i[order], j[order], sh[order]
        r = (x[self.cj] + self.cs - x[self.ci]).norm(dim=1)
        b = r < smax
        self.bi, self.bj, self.bs = self.ci[b], self.cj[b], self.cs[b]
        cnt = torch.bincount(self.bi, minlength=self.n)
        first = torch.cumsum(cnt, 0) - cnt
        m = cnt[self.bi]
        self.ta = torch.repeat_interleave(torch.arange(len(self.bi), device=self.dev), m)
        off = torch.arange(len(self.ta), device=self.dev) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
        self.tb = first[self.bi[self.ta]] + off
        keep = self.ta != self.tb
        self.ta, self.tb = self.ta[keep], self.tb[keep]
        self.x_list = x.detach().clone()

    def terms(self, x, t):
        """Bond terms (f_c f_R, f_c f_A b, kappa) and the charge kernel of every pair."""
        ty = self.type
        u = x[self.bj] + self.bs - x[self.bi]
        r = u.norm(dim=1)
        p = (ty[self.bi], ty[self.bj])
        R, S = t["R"][p], t["S"][p]
        y = (r - R) / (S - R)
        fc = torch.where(r < R, torch.ones_like(r),
                         torch.where(r < S, 0.5 * (1 + torch.cos(math.pi * y)), torch.zeros_like(r)))
        a, b = self.ta, self.tb
        ct = (u[a] * u[b]).sum(1) / (r[a] * r[b])
        q = (ty[self.bi[a]], ty[self.bj[a]], ty[self.bj[b]])
        live = fc[b].detach() > 0
        zs = []
        for l in range(2):
            g, c2, d2 = t["gam"][q][:, l], t["c"][q][:, l] ** 2, t["d"][q][:, l] ** 2
            ang = g * (1 + c2 / d2 - c2 / (d2 + (t["h"][q][:, l] - ct) ** 2))
            z = fc[b] * ang * torch.exp(t["alpha"][q][:, l] * (r[a] - r[b]))
            zs.append(torch.zeros_like(r).index_add(0, a, torch.where(live, z, torch.zeros_like(z))))
        hat = []
        for l in range(2):
            pos = zs[l] > 0
            zn = torch.where(pos, torch.where(pos, zs[l], torch.ones_like(r)) ** t["n"][p][:, l], torch.zeros_like(r))
            hat.append(t["g"][p][:, l] + zn)
        pp, sg = t["p"][p], t["sigma"][p]
        G = (t["g"][p][:, 0] ** -pp + t["g"][p][:, 1] ** -pp) ** (-1 / (2 * sg * pp))
        bij = G * (hat[0] ** -pp + hat[1] ** -pp) ** (1 / (2 * sg * pp))
        rep = fc * t["A"][p] * torch.exp(-t["l1"][p] * r)
        att = fc * t["B"][p] * torch.exp(-t["l2"][p] * r) * bij
        rc = (x[self.cj] + self.cs - x[self.ci]).norm(dim=1)
        y = rc / t["rc"]
        T = torch.where(y < 1, 1 + y ** 4 * (-35 + y * (84 + y * (-70 + 20 * y))), torch.zeros_like(y))
        gij = torch.sqrt(t["gc"][ty[self.ci]] * t["gc"][ty[self.cj]])
        K = t["ke"] * T * (rc ** 3 + gij ** -3) ** (-1.0 / 3.0)
        return rep, att, t["kappa"][p], K

    def energy(self, terms, q, t):
        """Energy of each replica."""
        rep, att, kap, K = terms
        dq = q[self.bi] - q[self.bj]
        eb = 0.5 * (rep - (1 - kap * dq * dq) * att)
        es = t["E0"][self.type] + t["chi"][self.type] * q + t["J"][self.type] * q * q
        ec = 0.5 * q[self.ci] * q[self.cj] * K
        e = torch.zeros(self.R, dtype=q.dtype, device=self.dev)
        return e.index_add(0, self.rep, es).index_add(0, self.rep[self.bi], eb).index_add(0, self.rep[self.ci], ec)

    def hessian(self, terms, t, drop=None):
        """The charge Hessian as (sparse off-diagonal part, diagonal); `drop`: without that atom's terms."""
        _, att, kap, K = (v.detach() for v in terms)
        w = kap * att
        if drop is not None:
            w = torch.where((self.bi == drop) | (self.bj == drop), torch.zeros_like(w), w)
            K = torch.where((self.ci == drop) | (self.cj == drop), torch.zeros_like(K), K)
        i = torch.cat([self.ci, self.bi, self.bj])
        j = torch.cat([self.cj, self.bj, self.bi])
        A = torch.sparse_coo_tensor(torch.stack([i, j]), torch.cat([K, -w, -w]), (self.n, self.n)).coalesce()
        D = 2 * t["J"][self.type]
        D = D.index_add(0, self.bi, w).index_add(0, self.bj, w)
        return A.to_sparse_csr(), D

    def solve(self, A, D, rhs, x0=None, tol=1e-14):
        """H s = rhs by conjugate gradients, one column of rhs beside the other."""
        s = torch.zeros_like(rhs) if x0 is None else x0.clone()
        H = lambda v: A @ v + D[:, None] * v  # noqa: E731
        r = rhs - H(s)
        z = r / D[:, None]
        p, rz = z.clone(), (r * z).sum(0)
        stop = tol * rhs.abs().amax(0)
        for _ in range(2000):
            if bool((r.abs().amax(0) <= stop).all()):
                break
            Hp = H(p)
            pHp = (p * Hp).sum(0)
            a = torch.where(pHp > 0, rz / torch.where(pHp > 0, pHp, torch.ones_like(pHp)), torch.zeros_like(pHp))
            s, r = s + a * p, r - a * Hp
            z = r / D[:, None]
            new = (r * z).sum(0)
            p, rz = z + torch.where(rz > 0, new / torch.where(rz > 0, rz, torch.ones_like(rz)), torch.zeros_like(rz)) * p, new
        return s

    def constrained(self, A, D, b, keep=True, mask=None):
        """q with H q = b + mu 1 and no total charge in any replica."""
        one = torch.ones_like(b) if mask is None else mask
        s = self.solve(A, D, torch.stack([b, one], 1), self.sol if keep else None)
        if keep:
            self.sol = s
        tot = torch.zeros((self.R, 2), dtype=b.dtype, device=self.dev).index_add(0, self.rep, s)
        return s[:, 0] - (tot[:, 0] / tot[:, 1])[self.rep] * s[:, 1]

    def evaluate(self, x, virial=False):
        """Energies, forces (and virial) and charges at the charge minimiser."""
        self.lists(x)
        t = _tables(self.theta)
        x = x.detach().clone().requires_grad_(True)
        eps = torch.zeros((self.R, 3, 3), dtype=x.dtype, device=self.dev, requires_grad=virial)
        if virial:      # positions and shifts under a homogeneous strain of each replica
            m = torch.eye(3, dtype=x.dtype, device=self.dev) + eps
            xs = torch.einsum("nab,nb->na", m[self.rep], x)
            keep = self.cs, self.bs
            self.cs = torch.einsum("nab,nb->na", m[self.rep[self.ci]], keep[0])
            self.bs = torch.einsum("nab,nb->na", m[self.rep[self.bi]], keep[1])
        else:
            xs = x
        terms = self.terms(xs, t)
        A, D = self.hessian(terms, t)
        q = self.constrained(A, D, -t["chi"][self.type])
        E = self.energy(terms, q, t)
        g = torch.autograd.grad(E.sum(), [x, eps] if virial else [x])
        if virial:
            self.cs, self.bs = keep
            return E.detach(), -g[0], q, -g[1].transpose(1, 2)
        return E.detach(), -g[0], q

    def gradient(self, x, tg):
        """The force-matching loss and its gradient in the parameters, the charges following their minimiser."""
        self.lists(x)
        dev = lambda a: torch.tensor(np.asarray(a), device=self.dev)  # noqa: E731
        th = self.theta.clone().requires_grad_(True)
        t = _tables(th)
        x = x.detach().clone().requires_grad_(True)
        terms = self.terms(x, t)
        A, D = self.hessian(terms, t)
        q = self.constrained(A, D, -t["chi"][self.type].detach(), keep=False).requires_grad_(True)
        E = self.energy(terms, q, t)
        gx, gq = torch.autograd.grad(E.sum(), [x, q], create_graph=True)
        wE, wF = dev(tg["w_E"]), dev(tg["w_F"])[self.rep][:, None]
        dE, dF = E.detach() - dev(tg["E_ref"]), -gx.detach() - dev(tg["F_ref"])
        loss = (wE * dE * dE).sum() + (wF * dF * dF).sum()
        a, g = 2 * wE * dE, 2 * wF * dF
        gF = -(g * gx).sum()
        (v,) = torch.autograd.grad(gF, q, retain_graph=True)
        lam = self.constrained(A, D, v, keep=False)
        (out,) = torch.autograd.grad((a * E).sum() + gF - (lam * gq).sum(), th)
        return loss, out


def _exact_md(case, seed, structs, temps, m):
    dev = m.dev
    x = torch.tensor(np.concatenate([s.x for s in structs]), device=dev)
    v = torch.tensor(_velocities(structs, temps, seed), device=dev)
    mob = torch.tensor(~np.concatenate([s.frozen for s in structs]), device=dev)[:, None]
    mass = _tables(m.theta)["mass"][m.type][:, None]
    nvt = case["nvt"]
    free = [3.0 * int((~s.frozen).sum()) - (0 if s.frozen.any() else 3) for s in structs]
    gkT = torch.tensor([g * _KB * T for g, T in zip(free, temps)], dtype=torch.float64, device=dev)
    Qm = gkT * TAU * TAU
    xi, eta = torch.zeros_like(gkT), torch.zeros_like(gkT)
    box = torch.tensor(np.stack([s.box for s in structs]), device=dev)[m.rep]
    pbc = torch.tensor(np.stack([s.pbc for s in structs]), device=dev)[m.rep]
    kin = lambda v: torch.zeros_like(gkT).index_add(0, m.rep, 0.5 * (mass * v * v).sum(1) / _ACC)  # noqa: E731
    E, F, q = m.evaluate(x)
    for _ in range(case["steps"]):
        if nvt:
            xi = xi + 0.5 * DT * (2 * kin(v) - gkT) / Qm
            eta = eta + DT * xi
            v = v * torch.exp(-0.5 * DT * xi)[m.rep][:, None]
        v = torch.where(mob, v + 0.5 * DT * _ACC * F / mass, torch.zeros_like(v))
        x = torch.where(mob, x + DT * v, x)
        E, F, q = m.evaluate(x)
        v = torch.where(mob, v + 0.5 * DT * _ACC * F / mass, torch.zeros_like(v))
        if nvt:
            v = v * torch.exp(-0.5 * DT * xi)[m.rep][:, None]
            xi = xi + 0.5 * DT * (2 * kin(v) - gkT) / Qm
    out = {"positions": None, "velocities": v, "forces": F, "charges": q, "energy": E}   # (positions: wrapped or not)
    if nvt:
        out["thermostat"] = torch.stack([xi, eta, Qm, gkT], 1)
    return out


def _exact_relax(case, structs, m):
    s = structs[0]
    x = torch.tensor(s.x, device=m.dev)
    mob = torch.tensor(~s.frozen, device=m.dev)
    mass = _tables(m.theta)["mass"][m.type][:, None]
    v = torch.zeros_like(x)
    dt, alpha, npos = 1.0, 0.1, 0
    E, F, _ = m.evaluate(x)
    for _ in range(case["iters"]):
        f, w = F[mob], v[mob]
        if float((f * w).sum()) >= 0:
            npos += 1
            if npos > 5:
                dt, alpha = min(1.1 * dt, 5.0), 0.99 * alpha
            v = (1 - alpha) * v + alpha * (w.norm() / f.norm()) * F
        else:
            npos, dt, alpha, v = 0, 0.5 * dt, 0.1, torch.zeros_like(v)
        v = torch.where(mob[:, None], v + dt * _ACC * F / mass, torch.zeros_like(v))
        x = x + dt * v
        E, F, _ = m.evaluate(x)
    return {"iters": None, "fmax": F[mob].norm(dim=1).max()[None], "positions": None, "energy": E}


def _exact_screen(structs, m):
    s = structs[0]
    x = torch.tensor(s.x, device=m.dev)
    E, _, _ = m.evaluate(x)
    t = _tables(m.theta)
    r = (x[m.bj] + m.bs - x[m.bi]).norm(dim=1)
    near = (r < t["S"][m.type[m.bi], m.type[m.bj]]).long()
    coord = torch.zeros(m.n, dtype=torch.long, device=m.dev).index_add(0, m.bi, near).cpu().numpy()
    cand = np.nonzero((s.types == 0) & (coord < 4) & ~s.frozen)[0]
    full = m.bi, m.bj, m.bs, m.ta, m.tb
    dE = []
    for c in cand:
        # bonds and triplets without the atom; its charge is held at zero by a row of its own
        kb = (full[0] != int(c)) & (full[1] != int(c))
        new = torch.cumsum(kb.long(), 0) - 1
        kt = kb[full[3]] & kb[full[4]]
        m.bi, m.bj, m.bs = (v[kb] for v in full[:3])
        m.ta, m.tb = new[full[3][kt]], new[full[4][kt]]
        with torch.no_grad():
            terms = m.terms(x, t)
            A, D = m.hessian(terms, t, drop=int(c))
            one = torch.ones(m.n, dtype=torch.float64, device=m.dev)
            one[int(c)] = 0.0
            q = m.constrained(A, D, -t["chi"][m.type] * one, mask=one)
            dE.append(m.energy(terms, q, t)[0] - E[0])    # (its E0 stays in the sum: it leaves as a neutral atom)
        m.bi, m.bj, m.bs, m.ta, m.tb = full
    return {"candidates": None, "dE": torch.stack(dE)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "rings" or _atoms(case) > EXACT_ATOMS:
        return None
    P = st.load_params("p1")
    structs, temps = _structures(case, seed)
    theta = ctbop.params_vector(ctbop.params_struct(P))
    m = _Model(structs, theta, margin=0.8 if kind in ("md", "relax") else 0.0)
    if kind == "md":
        return _exact_md(case, seed, structs, temps, m)
    if kind == "relax":
        return _exact_relax(case, structs, m)
    if kind == "screen":
        return _exact_screen(structs, m)
    if kind == "grad":
        outs, x = [], torch.tensor(np.concatenate([s.x for s in structs]), device=m.dev)
        tg = _targets(structs, seed)
        for th in _thetas(P, seed, _dtype(case)):
            loss, g = _Model(structs, th.double().numpy()).gradient(x, tg)
            outs.append({"loss": loss, "dtheta": g})
        return outs
    outs = []
    for f in _frames(case, structs, seed):
        x = torch.tensor(f, dtype=_dtype(case) if kind == "energy" else torch.float64).double().to(m.dev)
        if kind == "energy":
            E, F, _ = m.evaluate(x)
            outs.append({"E": E, "dE_dx": -F})
        else:
            E, F, q, W = m.evaluate(x, virial=True)
            outs.append({"energy": E, "forces": F, "virial": W, "charges": q})
        m.x_list = None
    return outs
