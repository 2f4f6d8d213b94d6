#!/usr/bin/env python
"""Benchmark: MD steps of the charge-transfer bond-order potential on GB300.

Default workload: the ~1.005M-atom stepped 4H-SiC(0001) slab with 5% C
adatoms at 2500 K, dt = 0.5 fs, mixed precision (FP32 bond-order/charge-kernel
arithmetic, FP64 reductions and CG vectors). A step is one velocity-Verlet
step: neighbour-list check/rebuild, bond orders, charge assembly, the
per-step charge CG, forces, virial and both half kicks.

Prints one JSON line (rank 0). Multi-GPU: replicas only (the single system is
not partitioned); each rank steps its own copy, value = all atoms x steps /
max-over-ranks time. `--impl reference` times the FP64 CPU oracle on a
bounded sample of the same workload (there is no other reference
implementation: the paper ships no code).
"""
import os

# The CPU baseline (the oracle) runs single-threaded, so that its reported
# core count is what it used: pin the BLAS/OpenMP pools before numpy loads.
for _v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

import argparse
import json
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "atom-steps/s at 1M atoms, mixed vs FP64 on one GB300 at force rel err ≤1e-4"
UNIT = "atom-steps/s"
DT = 0.5
T_K = 2500.0


def args_():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="1m", choices=["1m", "250k", "20k", "512"])
    ap.add_argument("--no-fp64", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-ensemble", action="store_true")
    ap.add_argument("--no-grad", action="store_true")
    ap.add_argument("--no-screen", action="store_true")
    ap.add_argument("--no-relax", action="store_true")
    ap.add_argument("--no-rings", action="store_true")
    ap.add_argument("--no-drift", action="store_true")
    ap.add_argument("--no-nvt", action="store_true")
    ap.add_argument("--no-sustained", action="store_true")
    ap.add_argument("--profile-steps", type=int, default=3)
    ap.add_argument("--e2e-steps", type=int, default=0, help="0: as many as --steps")
    return ap.parse_args()


WORKLOADS = {
    "1m": "stepped 4H-SiC(0001) slab 96x48 cells x 56 bilayers, 3 steps, + 5% C adatoms",
    "250k": "stepped 4H-SiC(0001) slab 48x24 cells x 56 bilayers, 3 steps, + 5% C adatoms",
    "20k": "stepped 4H-SiC(0001) slab 24x14 cells x 15 bilayers, 2 step edges",
    "512": "3C-SiC 4x4x4 cells",
}


def workload(name):
    from paper_1802_07871_gb300 import structures as st
    s = {"1m": st.stepped_slab_1m, "250k": st.stepped_slab_250k, "20k": st.stepped_slab_20k,
         "512": st.bulk_3c_512}[name]()
    v = st.maxwell_boltzmann(s.types, T_K, seed=103, frozen=s.frozen)
    return s, v, WORKLOADS[name]


class Clocks:
    """nvidia-smi samples during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, dev):
        self.dev = dev
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.dev}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.fh.close()
        rows = []
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) >= 9:
                rows.append(f)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# DRAM traffic of one k_cg_mv launch from one `ncu --set full` capture on
# the 251,366-atom stepped slab (dram__bytes_read.sum + dram__bytes_write.sum)
# and the stored matrix entries of that launch. Traffic grows with the entries
# (1.05 x the algorithmic bytes there, atoms stored along a Morton curve), so
# a full launch is scaled by its entry count. Reset to None when the kernel
# changes.
MV_TRAFFIC_CAPTURE = {"bytes": 416.962816e6 + 4.241920e6, "entries": 251366 * 193.9466117135969}


def cg_matvec_bytes(n_atoms, entries, rs):
    """Algorithmic bytes of one CG matrix pass: per list entry the neighbour
    index and the stored coefficient; per atom the gathered y (once), its own
    y, d, v, r and D, the written w, the entry count and the replica id."""
    return entries * (4 + rs) + n_atoms * (7 * rs + 8)


# Algorithmic work of each phase of a step, per unit the method must
# process (skin entries, padding and recomputation excluded). Flops count a
# fused multiply-add as 2; special-function operations (exp2, log2,
# reciprocal, reciprocal root, sin/cos) are counted apart ("mufu"), because
# they issue on their own pipe. Counted from the formulas of the model card:
#   bond pass (Eq. 2, 7), per directed bond r < S: bond length and cutoff
#     (12 flops, 2 mufu), Eq. 7 with its two derivatives (19 flops, 13 mufu);
#     per triplet (i, j, k), k != j both bonds of i: the cosine (8 flops,
#     1 mufu), per channel l the angular function, the bond-length factor
#     and the accumulation (12 flops, 2 mufu);
#   covalent force pass, per bond: both pair exponentials, the cutoff
#     derivative, the covalent-ionic factor, energy, radial derivative, the
#     two dE/dzeta_l and the slot (41 flops, 4 mufu); per triplet: the
#     cosine's gradient for both legs (18 flops) and per channel the
#     derivatives of the triplet term and their chain rule into both legs
#     (37 flops) (forward values reused, not recomputed);
#   charge-force gather, per pair inside Rc: relative vector and length
#     (15 flops, 1 mufu), K(r) and K'(r)/r with the taper (35 flops, 2 mufu),
#     force, energy and virial sums (34 flops).
# Bytes count one DRAM read or write of every array element the phase must
# touch: per list entry the (index, image code) pair (8 B); per stored
# matrix entry the (index, coefficient) pair (8 B); per atom its own vectors.
UNIT_COST = {
    "bond": {"per_bond": (31, 15), "per_triplet": (8 + 2 * 12, 1 + 2 * 2)},
    "cov_force": {"per_bond": (41, 4), "per_triplet": (18 + 2 * 37, 0)},
    "coul_gather": {"per_pair": (15 + 35 + 34, 3)},
}


def phase_work(n, entries_all, entries_mat, n_cov_entries, bonds, triplets, rs=4):
    """Algorithmic (flops, mufu ops, DRAM bytes) of each phase for a system of
    n atoms, per step (per launch for the CG phases, which launch once per
    iteration): entries_all list entries (charge
    cutoff + skin), entries_mat stored matrix entries (inside Rc),
    n_cov_entries covalent list entries, bonds directed bonds inside S,
    triplets ordered (j, k) pairs of bonds of one atom. rs = bytes of a
    working-precision scalar."""
    b, t = UNIT_COST["bond"], UNIT_COST["cov_force"]
    out = {}
    out["bond"] = dict(flops=bonds * b["per_bond"][0] + triplets * b["per_triplet"][0],
                       mufu=bonds * b["per_bond"][1] + triplets * b["per_triplet"][1],
                       bytes=n_cov_entries * 8 + n * 16 + bonds * 16)
    out["cov_force"] = dict(flops=bonds * t["per_bond"][0] + triplets * t["per_triplet"][0],
                            mufu=bonds * t["per_bond"][1],
                            bytes=n_cov_entries * (8 + 16 + 16) + n * (16 + 8 + 8))
    cg = UNIT_COST["coul_gather"]["per_pair"]
    # list, own position/charge/velocity/force/energy, and the two slots and
    # the reverse index of every covalent entry
    out["coul_gather_kick"] = dict(flops=entries_mat * cg[0], mufu=entries_mat * cg[1],
                                   bytes=entries_all * 8 + n_cov_entries * (16 + 16 + 4) + n * (16 + 4 + 24 + 48 + 16 + 1))
    # assembly: list read, matrix written, the bond orders of both bond
    # directions, diagonal and preconditioner vectors
    out["assemble"] = dict(flops=entries_mat * 35, mufu=entries_mat * 2,
                           bytes=entries_all * 8 + entries_mat * 8 + n_cov_entries * 2 * 16 + n * (16 + 4 + 3 * rs))
    out["cg_matvec"] = dict(flops=entries_mat * 2, mufu=0, bytes=cg_matvec_bytes(n, entries_mat, rs), per="launch")
    # element-wise update: y, d, p, w, s, r, dq read; p, s, dq, r, y written;
    # the 32 x 32 block inverse (32 entries per atom) read
    out["cg_update"] = dict(flops=n * (2 * 6 + 64), mufu=0, bytes=n * (7 * rs + 5 * rs + 32 * rs + 4), per="launch")
    out["kick_drift"] = dict(flops=n * 12, mufu=0, bytes=n * (24 * 3 + 24 * 2 + 16 + 1 + 4))
    return out


def roofline_table(ph, steps, work, peaks_meas, hbm_gbs):
    """Per phase: time per launch, algorithmic rate against each bound, the
    binding bound (largest fraction), and the time-weighted step fraction.
    ph: {phase: (ms summed, launches)} from profile_steps over `steps` steps."""
    table = {}
    num = den = 0.0
    for name, (ms_sum, launches) in ph.items():
        if name not in work or launches == 0:
            continue
        w = work[name]
        units = launches if w.get("per") == "launch" else steps
        per_launch = ms_sum / units / 1e3      # s per unit (launch or step) of the phase
        fr = {"hbm": w["bytes"] / per_launch / 1e9 / hbm_gbs}
        if peaks_meas:
            fr["fp32"] = w["flops"] / per_launch / 1e12 / peaks_meas["fp32_tflops"]
            fr["mufu"] = w["mufu"] / per_launch / 1e12 / max(peaks_meas["mufu_ex2_tops"], peaks_meas["mufu_rsq_tops"])
        bound = max(fr, key=fr.get)
        table[name] = {"ms_per_" + w.get("per", "step"): per_launch * 1e3, "bound": bound, "frac": fr[bound],
                       "frac_by_bound": {k: round(v, 4) for k, v in fr.items()},
                       "gflop": w["flops"] / 1e9, "gmufu": w["mufu"] / 1e9,
                       "gbytes": w["bytes"] / 1e9, "per": w.get("per", "step")}
        num += ms_sum * fr[bound]
        den += ms_sum
    total = sum(t for t, _ in ph.values())
    return table, {"frac": num / den if den else None, "covered_share": den / total if total else None}


class nvtx_range:
    """An NVTX push/pop range around a timed region, so that a profiler can
    select one leg's launches (e.g. ncu --nvtx --nvtx-include "param_grad_mixed/")."""

    def __init__(self, name):
        self.name = name

    def __enter__(self):
        import torch
        torch.cuda.nvtx.range_push(self.name)
        return self

    def __exit__(self, *exc):
        import torch
        torch.cuda.nvtx.range_pop()
        return False


def max_over_ranks(x, device, world):
    """Max of a per-rank float over all ranks (identity at world 1)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate_value(n_atoms, steps, world, ms):
    """Whole-job atom-steps/s: every rank steps its own n_atoms-atom replica,
    timed by the slowest rank's ms."""
    return n_atoms * steps * world / (ms / 1e3)


def tuned_shapes(d):
    """The autotuned shapes of a system's passes and the timings they were
    picked from (ms per launch, in the order of the candidates listed)."""
    r = lambda xs: [round(x, 4) for x in xs]
    return {"cg_matvec_depth": d["cg_mv_batch"], "cg_matvec_ms_by_depth_4_8_16": r(d["cg_mv_ms"]),
            "assembly_depth": d["asm_batch"], "assembly_ms_by_depth_4_8_16": r(d["asm_ms"]),
            "gather_depth": d["gather_batch"], "gather_ms_by_depth_4_6_8": r(d["gather_ms"]),
            "covalent_lanes": d["cov_lanes"], "covalent_ms_by_lanes_4_8_16": r(d["cov_ms"]),
            "list_build_shape": [d["build_warps"], d["build_batch"]],
            "list_build_ms_by_shape_2x64_2x128_4x64_4x128_8x64_8x128": r(d["build_ms"])}


def run_ensemble(dev, stream, steps=20, warmup=3):
    """Secondary measurement: the 256-replica annealing ensemble (uneven
    200-3000-atom SiC slabs with Si vacancies, amorphous C clusters and
    graphene-on-SiC flakes, 1500-3000 K), all replicas stepped together in
    one launch per kernel per step, mixed precision."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st
    structs, temps = st.annealing_ensemble(256, seed=4)
    v = np.concatenate([st.maxwell_boltzmann(s.types, T, seed=500 + r, frozen=s.frozen)
                        for r, (s, T) in enumerate(zip(structs, temps))])
    n = sum(s.n for s in structs)
    sysm = ctbop.System(st.load_params("p1"), precision="mixed", device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load_replicas(structs)
    sysm.set_velocities(v)
    sysm.compute()
    sysm.step(warmup, DT)
    st0 = sysm.status()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    sysm.step(steps, DT)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    st1 = sysm.status()
    sysm.close()
    return {"workload": "annealing ensemble: 256 replicas of 200-3000 atoms (SiC slabs with 0-30% Si vacancies, "
                        "amorphous C clusters 1.8-2.3 g/cc, defected graphene flakes on SiC), 1500-3000 K",
            "n_replicas": len(structs), "n_atoms": n, "steps": steps, "warmup": warmup,
            "value": n * steps / (ms / 1e3), "unit": UNIT, "ms_per_step": ms / steps,
            "cg_iters_per_step": (st1["cg_iters_total"] - st0["cg_iters_total"]) / steps,
            "precision": "mixed", "tuned": tuned_shapes(st1)}


def run_param_grad(dev, stream, precision="mixed", calls=3, warmup=1):
    """Secondary measurement: the force-matching gradient on the 1024-config
    differentiation batch (64-512 atoms each: strained 3C-SiC, periodic
    graphene with Stone-Wales defects, random Si/C clusters). Targets E_ref,
    F_ref are the library's own FP64 energies and forces under a perturbed
    parameter set, made before the timed region (workload input, not a
    parity value). One call = loss + dL/dtheta for all 144 parameters over
    the whole batch: evaluation with the charge solve, the forward-mode pass
    along dL/dF, the adjoint solve and the forward-mode pass along the
    adjoint charges, in the given precision policy. Timed on the host clock,
    since the call synchronises with its stream."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st
    P1 = st.load_params("p1")
    structs = st.differentiation_batch(1024, seed=5)
    n = sum(s.n for s in structs)
    R = len(structs)
    ref = ctbop.System(st.perturbed_params(P1, 55), precision="fp64", device=dev.index or 0)
    ref.set_stream(stream.cuda_stream)
    ref.load_replicas(structs)
    ref.compute()
    E_ref, F_ref = ref.get("energy"), ref.get("forces")
    ref.close()
    sysm = ctbop.System(P1, precision=precision, device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load_replicas(structs)
    nr = np.array([s.n for s in structs], dtype=np.float64)
    loss = dict(w_E=1.0 / nr ** 2, E_ref=E_ref, w_F=1.0 / (3.0 * nr), F_ref=F_ref)
    for _ in range(warmup):
        sysm.param_grad(**loss)
    it0 = sysm.status()["cg_iters_total"]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with nvtx_range(f"param_grad_{precision}"):
        for _ in range(calls):
            L, _ = sysm.param_grad(**loss)
        torch.cuda.synchronize()
    sec = (time.perf_counter() - t0) / calls
    it1 = sysm.status()["cg_iters_total"]
    sysm.close()
    return {"workload": "differentiation batch: 1024 configurations of 64-512 atoms (3C-SiC under random "
                        "+-5% diagonal strain, periodic graphene with 1-3 Stone-Wales defects, random Si/C "
                        "clusters at 0.05-0.10 per A^3), force-matching loss on E and F",
            "n_configs": R, "n_atoms": n, "calls": calls, "warmup": warmup, "precision": precision,
            "ms_per_call": sec * 1e3, "value": n / sec, "unit": "atom-gradients/s",
            "configs_per_s": R / sec, "cg_iters_per_call": (it1 - it0) / calls, "loss": L}


def run_screen(dev, stream, calls=3, warmup=1):
    """Secondary measurement: one Si desorption screening of the
    19,488-atom stepped slab (Sec. 3.3): the removal energy of every surface
    Si (mobile, coordination < 4), each a full evaluation with the charge
    solve of the slab without that atom, run as batched leave-one-out
    replicas. Timed on the host clock (the call synchronises)."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import desorption as D
    from paper_1802_07871_gb300 import structures as st
    s = st.stepped_slab_20k()
    sysm = ctbop.System(st.load_params("p1"), precision="mixed", device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load(s)
    sysm.compute()
    cand, _ = D.surface_si(sysm, s.types, s.frozen)
    for _ in range(warmup):
        sysm.removal_energies(cand)
    it0 = sysm.status()["cg_iters_total"]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with nvtx_range("desorption_screen"):
        for _ in range(calls):
            dE = sysm.removal_energies(cand)
        torch.cuda.synchronize()
    sec = (time.perf_counter() - t0) / calls
    sysm.close()
    return {"workload": "Si desorption screening of the 19,488-atom stepped 4H-SiC slab: removal energy of every "
                        "surface Si, each a full evaluation (charge solve) of the slab without it",
            "n_atoms": s.n, "candidates": int(len(cand)), "calls": calls, "warmup": warmup, "precision": "mixed",
            "ms_per_screening": sec * 1e3, "value": len(cand) / sec, "unit": "candidates/s",
            "atoms_evaluated_per_s": len(cand) * (s.n - 1) / sec,
            "removal_energy_eV_min_median_max": [float(dE.min()), float(np.median(dE)), float(dE.max())]}


def run_relax(dev, stream, max_iter=500, fmax=0.05):
    """Secondary measurement: FIRE relaxation (charges re-minimised at every
    force evaluation) of the 19,488-atom stepped slab, at most max_iter
    iterations to max |F| < fmax (eV/A). Timed on the host clock (the call
    synchronises)."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st
    s = st.stepped_slab_20k()
    sysm = ctbop.System(st.load_params("p1"), precision="mixed", device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load(s)
    sysm.compute()
    E0 = float(sysm.get("energy")[0])
    st0 = sysm.status()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with nvtx_range("relax"):
        it, fm = sysm.minimize(max_iter=max_iter, fmax=fmax, dt0=1.0, dt_max=5.0)
        torch.cuda.synchronize()
    sec = time.perf_counter() - t0
    st1 = sysm.status()
    E1 = float(sysm.get("energy")[0])
    sysm.close()
    n_it = int(it[0]) if it[0] >= 0 else max_iter
    return {"workload": "FIRE relaxation of the 19,488-atom stepped 4H-SiC slab (bottom two bilayers frozen), "
                        f"max |F| < {fmax} eV/A or {max_iter} iterations",
            "n_atoms": s.n, "iterations": int(it[0]), "converged": bool(it[0] >= 0), "final_fmax": float(fm[0]),
            "energy_drop_eV": E0 - E1, "seconds": sec, "ms_per_iteration": sec * 1e3 / max(n_it, 1),
            "value": s.n * n_it / sec, "unit": "atom-iterations/s",
            "cg_iters_per_iteration": (st1["cg_iters_total"] - st0["cg_iters_total"]) / max(n_it, 1),
            "precision": "mixed"}


def run_rings(dev, stream, calls=3, warmup=1):
    """Secondary measurement: ring statistics (primitive C rings up to 8
    atoms, 6-ring orientations) of the 256-replica annealing ensemble. Timed
    on the host clock (the call synchronises and copies the records out)."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import rings as RG
    from paper_1802_07871_gb300 import structures as st
    structs, _ = st.annealing_ensemble(256, seed=4)
    n = sum(s.n for s in structs)
    n_c = int(sum(int(np.sum(s.types == 1)) for s in structs))
    sysm = ctbop.System(st.load_params("p1"), precision="mixed", device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load_replicas(structs)
    sysm.compute()
    for _ in range(warmup):
        sysm.rings()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with nvtx_range("rings"):
        for _ in range(calls):
            rec = sysm.rings()
        torch.cuda.synchronize()
    sec = (time.perf_counter() - t0) / calls
    sysm.close()
    c = RG.counts(rec, len(structs)).sum(axis=0)
    return {"workload": "primitive C rings (3-8 atoms) and 6-ring orientations of the 256-replica annealing ensemble",
            "n_atoms": n, "c_atoms": n_c, "rings": int(len(rec)), "rings_by_size_3_to_8": [int(v) for v in c],
            "ms_per_call": sec * 1e3, "value": n_c / sec, "unit": "C atoms/s", "precision": "mixed"}


def run_nvt(dev, stream, s, v, steps=30, warmup=3):
    """Secondary measurement: the same slab under the Nose-Hoover thermostat
    the paper's runs use (NVT at 2500 K, tau = 100 fs), atom-steps/s."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st
    sysm = ctbop.System(st.load_params("p1"), precision="mixed", device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load(s, velocities=v)
    sysm.set_thermostat(T_K, 100.0)
    sysm.compute()
    sysm.step(warmup, DT)
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    sysm.step(steps, DT)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    sysm.close()
    return {"workload": "the timed slab, Nose-Hoover NVT at 2500 K (tau 100 fs)", "steps": steps,
            "warmup": warmup, "ms_per_step": ms / steps, "value": s.n * steps / (ms / 1e3), "unit": UNIT}


def run_sustained(dev, stream, s, v, steps=500):
    """The metric over the whole run the workload defines: a fresh system
    from the same inputs, one step to capture the graphs (not timed), then
    `steps` steps timed as one region with CUDA events, the clocks sampled
    meanwhile. Reports atom-steps/s with the CG iterations per step and the
    list rebuilds of that window."""
    import torch
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st
    sysm = ctbop.System(st.load_params("p1"), precision="mixed", device=dev.index or 0)
    sysm.set_stream(stream.cuda_stream)
    sysm.load(s, velocities=v)
    sysm.compute()
    sysm.step(1, DT)
    st0 = sysm.status()
    torch.cuda.synchronize()
    clocks = Clocks(dev.index or 0)
    clocks.start()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    sysm.step(steps, DT)
    e1.record(stream)
    torch.cuda.synchronize()
    ck = clocks.stop()
    ms = e0.elapsed_time(e1)
    st1 = sysm.status()
    ke = float(sysm.get("kinetic")[0])
    sysm.close()
    return {"workload": "the timed slab, steps 2 to %d of a fresh run (step 1 captures the graphs)" % (steps + 1),
            "steps": steps, "ms_per_step": ms / steps, "value": s.n * steps / (ms / 1e3), "unit": UNIT,
            "cg_iters_per_step": (st1["cg_iters_total"] - st0["cg_iters_total"]) / steps,
            "rebuilds": st1["rebuilds"] - st0["rebuilds"], "kinetic_eV_per_atom_at_end": ke / s.n,
            "clocks": ck}


def run_nve_drift(dev, stream, steps=1000, every=10):
    """Energy conservation of the NVE integrator, reported as the drift of
    E_pot + E_kin in eV/atom/ns (slope of a straight-line fit over the run):
    the 512-atom 3C-SiC cell (FP64, 300 K) and the 19,488-atom stepped slab
    (mixed, 2000 K, bottom frozen), dt = 0.5 fs."""
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st
    P1 = st.load_params("p1")
    out = {}
    for name, s, T, prec, seed in (("3C-SiC 512 atoms, FP64, 300 K", st.bulk_3c_512(), 300.0, "fp64", 101),
                                   ("stepped slab 19,488 atoms, mixed, 2000 K", st.stepped_slab_20k(), 2000.0,
                                    "mixed", 102)):
        v = st.maxwell_boltzmann(s.types, T, seed=seed, frozen=s.frozen)
        sysm = ctbop.System(P1, precision=prec, device=dev.index or 0)
        sysm.set_stream(stream.cuda_stream)
        sysm.load(s, velocities=v)
        sysm.compute()
        t, e = [], []
        for k in range(0, steps + 1, every):
            if k:
                sysm.step(every, DT)
            t.append(k * DT)
            e.append(float(sysm.get("energy")[0] + sysm.get("kinetic")[0]))
        sysm.close()
        slope = np.polyfit(np.array(t), np.array(e), 1)[0]   # eV/fs
        out[name] = {"drift_eV_per_atom_per_ns": slope * 1e6 / s.n, "steps": steps,
                     "max_excursion_eV_per_atom": (max(e) - min(e)) / s.n}
    return out


def run_ours(a):
    import torch
    import torch.distributed as dist
    from paper_1802_07871_gb300 import ctbop
    from paper_1802_07871_gb300 import structures as st

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    s, v, desc = workload(a.workload)
    P1 = st.load_params("p1")
    stream = torch.cuda.Stream(device=dev)

    sysm = ctbop.System(P1, precision="mixed", device=local)
    sysm.set_stream(stream.cuda_stream)
    sysm.load(s, velocities=v)
    sysm.compute()
    F_mixed0, E_mixed0, q_mixed0 = sysm.get("forces"), sysm.get("energy")[0], sysm.get("charges")
    sysm.step(a.warmup, DT)
    st0 = sysm.status()

    clocks = Clocks(local)
    barrier()
    clocks.start()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    sysm.step(a.steps, DT)
    e1.record(stream)
    barrier()
    ck = clocks.stop()
    ms = max_over_ranks(e0.elapsed_time(e1), dev, world)
    st1 = sysm.status()
    n = s.n
    value = aggregate_value(n, a.steps, world, ms)
    cg_per_step = (st1["cg_iters_total"] - st0["cg_iters_total"]) / a.steps
    rebuilds = st1["rebuilds"] - st0["rebuilds"]
    # our kernel launches in the timed region: 28 per step outside the CG
    # loop (12 of them the list check/rebuild, which return at once when no
    # rebuild is due; 3 of the FP64 pass over queued atoms, which exit at
    # once when the queue is empty), 2 per CG iteration; 24 in all where one
    # kernel runs the whole solve (no update passes in the profile below)
    launches = int(28 * a.steps + 2 * (st1["cg_iters_total"] - st0["cg_iters_total"]))

    # per-kernel timing (CUDA events on the library's stream)
    ph = sysm.profile_steps(a.profile_steps, DT)
    if ph["cg_update"][1] == 0:
        launches = 24 * a.steps
    st2 = sysm.status()
    mv_ms, mv_n = ph["cg_matvec"]
    entries = st2["mean_mat"] * n   # the stored matrix entries a matrix pass streams
    bytes_mv = cg_matvec_bytes(n, entries, 4)
    peak, peak_kind = peaks()
    mv_s = mv_ms / max(mv_n, 1) / 1e3
    achieved = bytes_mv / mv_s / 1e9 if mv_n else None
    traffic = (MV_TRAFFIC_CAPTURE["bytes"] * entries / MV_TRAFFIC_CAPTURE["entries"]
               if MV_TRAFFIC_CAPTURE else None)
    total_ph = sum(t for t, _ in ph.values())
    phases = {k: {"ms_per_step": round(t / a.profile_steps, 4), "launches": c, "share": round(t / total_ph, 4)}
              for k, (t, c) in ph.items()}
    # per-phase roofline on the live lists: measured bond counts (bonds
    # inside S per atom, ordered bond pairs per atom) and the arithmetic-pipe
    # peaks measured on this GPU now
    coord = sysm.get("coordination")
    bonds, triplets = float(coord.sum()), float((coord * (coord - 1.0)).sum())
    work = phase_work(n, st2["mean_all"] * n, entries, st2["mean_cov"] * n, bonds, triplets)
    try:
        pk = ctbop.measure_peaks(local, stream.cuda_stream)
    except Exception as e:   # a report, not a requirement
        pk = {"unavailable": f"{type(e).__name__}: {e}"[:200]}
    rf_phases, rf_step = roofline_table(ph, a.profile_steps, work, pk if "fp32_tflops" in pk else None, peak)
    rf_step["bonds_per_atom"] = bonds / n
    rf_step["triplets_per_atom"] = triplets / n

    # the state the timed steps reached, with the forces of its last step
    # evaluation (the MD path's precision mode), for the FP64 comparison
    x_hot, F_hot, E_hot = sysm.get("positions"), sysm.get("forces"), sysm.get("energy")[0]
    st_hot = sysm.status()

    # end to end through the C ABI with host buffers: per step upload the
    # velocities from pinned memory, step, read back energy, positions and
    # velocities. A fresh system from the same inputs and the same warm-up,
    # so the timed steps cover the same part of the trajectory as `value`
    # (the charge solve's iteration count changes as the slab heats).
    sysm.close()
    e2e_steps = a.e2e_steps if a.e2e_steps > 0 else a.steps
    sysm = ctbop.System(P1, precision="mixed", device=local)
    sysm.set_stream(stream.cuda_stream)
    sysm.load(s, velocities=v)
    sysm.compute()
    sysm.step(a.warmup, DT)
    pin_v = torch.empty((n, 3), dtype=torch.float64).pin_memory()
    pin_x = torch.empty((n, 3), dtype=torch.float64).pin_memory()
    pin_e = torch.empty((1,), dtype=torch.float64).pin_memory()
    sysm.get("velocities", pin_v)
    barrier()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        sysm.set_velocities(pin_v)
        sysm.step(1, DT)
        sysm.get("energy", pin_e)
        sysm.get("positions", pin_x)
        sysm.get("velocities", pin_v)
    barrier()
    t_e2e = max_over_ranks(time.perf_counter() - t0, dev, world)
    e2e = {"value": aggregate_value(n, e2e_steps, world, t_e2e * 1e3), "unit": UNIT, "steps": e2e_steps,
           "h2d_bytes_per_step": 24 * n, "d2h_bytes_per_step": 48 * n + 8}
    sysm.close()
    del sysm

    fp64 = None
    if not a.no_fp64:
        s64 = ctbop.System(P1, precision="fp64", device=local)
        s64.set_stream(stream.cuda_stream)
        s64.load(s, velocities=v)
        s64.compute()
        F64, E64, q64 = s64.get("forces"), s64.get("energy")[0], s64.get("charges")
        rms = float(np.sqrt(np.mean(F64 ** 2)))
        ferr = float(np.max(np.abs(F_mixed0 - F64)) / rms)
        eerr = float(abs(E_mixed0 - E64) / n)
        qerr = float(np.max(np.abs(q_mixed0 - q64)))
        # per-component relative error with a 1e-3 eV/A floor
        cerr = float(np.max(np.abs(F_mixed0 - F64) / np.maximum(np.abs(F64), 1e-3)))
        k64 = max(2, min(a.steps, 10))
        s64.step(2, DT)
        barrier()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        s64.step(k64, DT)
        f1.record(stream)
        barrier()
        ms64 = f0.elapsed_time(f1)
        fp64 = {"value": n * k64 * world / (ms64 / 1e3), "ms_per_step": ms64 / k64, "steps": k64,
                "mixed_vs_fp64_force_err": ferr, "mixed_vs_fp64_energy_err_eV_per_atom": eerr,
                "mixed_vs_fp64_charge_err_e": qerr, "mixed_vs_fp64_force_component_rel_err_floor_1e-3": cerr}
        s64.close()
        # the same comparison at the hot state the timed MD reached: the
        # mixed forces of its last step against an FP64 evaluation there
        hot = st.Structure("hot", x_hot, s.types, s.box, s.pbc, s.frozen)
        s64 = ctbop.System(P1, precision="fp64", device=local)
        s64.set_stream(stream.cuda_stream)
        s64.load(hot)
        s64.compute()
        F64h, E64h = s64.get("forces"), s64.get("energy")[0]
        s64.close()
        rms_h = float(np.sqrt(np.mean(F64h ** 2)))
        fp64["hot_state"] = {"mixed_vs_fp64_force_err": float(np.max(np.abs(F_hot - F64h)) / rms_h),
                             "mixed_vs_fp64_force_component_rel_err_floor_1e-3":
                                 float(np.max(np.abs(F_hot - F64h) / np.maximum(np.abs(F64h), 1e-3))),
                             "rms_force_eV_per_A": rms_h,
                             "mixed_vs_fp64_energy_err_eV_per_atom": float(abs(E_hot - E64h) / n),
                             "mixed_fp64_atoms": st_hot["fp64_atoms"], "mixed_fp64_pair_bonds": st_hot["fp64_bonds"],
                             "after_steps": a.warmup + a.steps + a.profile_steps}

    if rank != 0:
        return
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": a.steps,
        "warmup": a.warmup, "ms_per_step": ms / a.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": desc, "n_atoms": n, "precision": "mixed", "dt_fs": DT, "T_K": T_K,
                   "parallelism": f"replicas{world}", "l2": "inputs larger than L2: the neighbour list and "
                   "charge-matrix entries streamed every step exceed 3 GB",
                   "cg_iters_per_step": cg_per_step, "rebuilds_in_timed_region": rebuilds,
                   "mean_entries_per_atom": st2["mean_all"], "mean_matrix_entries_per_atom": st2["mean_mat"],
                   "mean_covalent_entries": st2["mean_cov"],
                   "tuned": tuned_shapes(st2),
                   "fp64_atoms_last_step": st2["fp64_atoms"], "fp64_pair_bonds_last_step": st2["fp64_bonds"]},
        "roofline": {"kernel": "k_cg_mv (charge CG matrix pass)", "bound": "hbm", "achieved": achieved,
                     "peak": peak, "unit": "GB/s", "frac": (achieved / peak) if achieved else None,
                     "traffic": traffic, "peak_kind": peak_kind,
                     "bytes_per_launch": bytes_mv, "ms_per_launch": mv_s * 1e3},
        "phases": phases,
        "roofline_phases": rf_phases,
        "roofline_step": rf_step,
        "pipe_peaks": pk,
        "e2e": e2e,
        "gpu_launches": launches,
        "clocks": ck,
        "fp64": fp64,
    }
    if world == 1 and not a.no_sustained:
        line["sustained"] = run_sustained(dev, stream, s, v)
    if world == 1 and not a.no_nvt:
        line["nvt"] = run_nvt(dev, stream, s, v)
    if world == 1 and not a.no_ensemble:
        line["ensemble"] = run_ensemble(dev, stream)
    if world == 1 and not a.no_grad:
        line["param_grad"] = run_param_grad(dev, stream, "mixed")
        line["param_grad"]["fp64"] = run_param_grad(dev, stream, "fp64")
    if world == 1 and not a.no_screen:
        line["desorption_screen"] = run_screen(dev, stream)
    if world == 1 and not a.no_relax:
        line["relax"] = run_relax(dev, stream)
    if world == 1 and not a.no_rings:
        line["rings"] = run_rings(dev, stream)
    if world == 1 and not a.no_drift:
        line["nve_drift"] = run_nve_drift(dev, stream)
    if world == 1 and not a.no_cpu:
        line["cpu_baseline"] = cpu_baseline()
        line["cpu_baseline_all_cores"] = cpu_baseline_all_cores()
    print(json.dumps(line), flush=True)


# The oracle's bounded sample of the ~1M-atom workload: the same shape
# (stepped 4H-SiC(0001) staircase, 5% C adatoms, frozen bottom) at 4,378
# atoms, above the oracle's dense-solve limit, so it solves the charges by
# CG as it would at full size.
SAMPLE_DIMS = (16, 8, 10)


def _oracle_step_time(s, v, steps, params, warmup=0):
    """Seconds per velocity-Verlet step of the oracle, as it stands, on one
    structure: velocity_verlet with `steps` steps minus the same call with
    none (its initial evaluation, which a step does not repeat), after
    `warmup` untimed steps. Returns (seconds per step, state after warm-up)."""
    from oracle import ctbop_oracle as O
    x = s.x
    if warmup:
        x, v, _, _ = O.velocity_verlet(s.x, v, s.types, s.box, s.pbc, params, DT, warmup, s.frozen)
    t0 = time.perf_counter()
    O.velocity_verlet(x, v, s.types, s.box, s.pbc, params, DT, 0, s.frozen)
    t_init = time.perf_counter() - t0
    t0 = time.perf_counter()
    O.velocity_verlet(x, v, s.types, s.box, s.pbc, params, DT, steps, s.frozen)
    t_all = time.perf_counter() - t0
    return max(t_all - t_init, 1e-9) / steps


def _oracle_sample_rate(args):
    """Atom-steps/s of the oracle on the workload sample (a top-level
    function, so a spawn pool can run one per core)."""
    steps, warmup, seed = args
    from paper_1802_07871_gb300 import structures as st
    s = st.stepped_slab_small(*SAMPLE_DIMS)
    v = st.maxwell_boltzmann(s.types, T_K, seed=seed, frozen=s.frozen)
    return s.n / _oracle_step_time(s, v, steps, st.load_params("p1"), warmup)


def cpu_baseline(steps=10, warmup=0, configs=True):
    """The FP64 oracle, as it stands, single-threaded (BLAS/OpenMP pools
    pinned to one thread), per velocity-Verlet step: on the bounded sample
    of the ~1M-atom workload, and (configs=True) on the 512-atom 3C-SiC cell
    (100 steps at 300 K, its full run) and the 19,488-atom stepped slab (3 of
    its 2000 steps, at 2000 K)."""
    from paper_1802_07871_gb300 import structures as st
    P1 = st.load_params("p1")
    s = st.stepped_slab_small(*SAMPLE_DIMS)
    value = _oracle_sample_rate((steps, warmup, 103))
    out = {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
           "sample": f"{s.n}-atom stepped 4H-SiC slab with C adatoms (the workload's shape), {steps} "
                     f"velocity-Verlet steps at 2500 K after {warmup} untimed, time per step excluding the "
                     "initial evaluation, numpy FP64, CG charge solve (the oracle's path above 4,000 atoms)"}
    if configs:
        b = st.bulk_3c_512()
        vb = st.maxwell_boltzmann(b.types, 300.0, seed=101)
        t_b = _oracle_step_time(b, vb, 100, P1)
        m = st.stepped_slab_20k()
        vm = st.maxwell_boltzmann(m.types, 2000.0, seed=102, frozen=m.frozen)
        t_m = _oracle_step_time(m, vm, 3, P1)
        out["configs"] = {
            "3C-SiC 512 atoms, 100 NVE steps at 300 K (dense charge solve)": {"value": b.n / t_b, "unit": UNIT,
                                                                             "steps": 100},
            "stepped slab 19,488 atoms, 3 NVE steps at 2000 K (CG charge solve)": {"value": m.n / t_m,
                                                                                  "unit": UNIT, "steps": 3}}
    return out


def cpu_baseline_all_cores(steps=3):
    """The oracle on every host core at once: one process per core (spawn
    pool, one BLAS thread each), each stepping its own copy of the workload
    sample with its own velocities, as independent replicas; value = the sum
    of the per-process atom-steps/s (the processes overlap for the whole
    timed part)."""
    import multiprocessing as mp
    n = os.cpu_count() or 1
    try:
        with mp.get_context("spawn").Pool(n) as pool:
            rates = pool.map(_oracle_sample_rate, [(steps, 0, 1000 + k) for k in range(n)], chunksize=1)
    except Exception as e:   # a report, not a requirement: never fail the run for it
        return {"unavailable": f"{type(e).__name__}: {e}"[:200]}
    return {"value": float(sum(rates)), "unit": UNIT, "cores": n, "kind": "oracle",
            "sample": f"{n} processes, each {steps} steps of its own copy of the workload sample "
                      f"({SAMPLE_DIMS} stepped slab with adatoms, different velocities)",
            "per_process_min_max": [float(min(rates)), float(max(rates))]}


def run_reference(a):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cb = cpu_baseline(steps=max(1, a.steps), warmup=a.warmup, configs=False)
    line = {"metric": METRIC, "value": cb["value"], "unit": UNIT, "n_gpus": world, "steps": a.steps,
            "warmup": a.warmup, "ms_per_step": None, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOADS[a.workload], "precision": "fp64", "dt_fs": DT, "T_K": T_K,
                       "sample": "each step a bounded sample of this workload (see cpu_baseline.sample)"},
            "cpu_baseline": cb,
            "e2e": {"value": cb["value"], "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    a = args_()
    if a.impl == "reference":
        run_reference(a)
    else:
        run_ours(a)


if __name__ == "__main__":
    main()
