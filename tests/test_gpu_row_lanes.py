"""The charge-matrix assembly and the charge-force gather with several lanes
per atom (small systems) against those with a thread per atom: the same
replicas evaluated alone (8 or 32 lanes) and in a batch with a large one (a
thread per atom), at sizes that leave partial warps and blocks and replicas
that share them; and the FP64 reciprocal roots the charge kernel takes against
the library's, over the range it meets."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")
HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1802_07871_gb300", "csrc")


def _eval(structs, prec, q):
    sysm = ctbop.System(P1, precision=prec)
    sysm.load_replicas(structs)
    sysm.set_charges(q)
    sysm.compute(fixed_charges=True)
    n = [s.n for s in structs]
    out = {k: np.split(sysm.get(k), np.cumsum(n)[:-1]) for k in ("forces", "e_atom")}
    out["virial"], out["energy"], out["kinetic"] = sysm.get("virial"), sysm.get("energy"), sysm.get("kinetic")
    sysm.compute()          # and with the solve on the assembled matrix
    out["charges"] = np.split(sysm.get("charges"), np.cumsum(n)[:-1])
    sysm.close()
    return out


@pytest.mark.parametrize("prec,lanes", [("mixed", 32), ("mixed", 8), ("fp64", 32), ("fp64", 8)])
def test_lane_groups_match_a_thread_per_atom(prec, lanes):
    small = [st.sic_3c(1, 4.36, 0.1, seed=1), st.amorphous_carbon_cluster(33, 2.0, 2),
             st.sic_3c(2, 4.36, 0.05, seed=3), st.stepped_slab_small(6, 3, 4)]
    if lanes == 8:
        small = small + [st.sic_3c(9, 4.36, 0.05, seed=4)]        # 5,832 atoms more
    big = st.sic_3c(28 if prec == "mixed" else 34, 4.36, 0.05, seed=5)   # 175,616 or 314,432 atoms
    rng = np.random.default_rng(6)
    qs = [rng.normal(0.0, 0.2, s.n) for s in small]
    a = _eval(small, prec, np.concatenate(qs))
    b = _eval(small + [big], prec, np.concatenate(qs + [rng.normal(0.0, 0.2, big.n)]))
    # the sums of about 230 terms are grouped otherwise: FP64 to 1e-12 of their
    # size; FP32 forces to some tens of rounding units of the largest terms
    # (14 eV/A pair terms of 0.04 e^2), energies compensated
    ftol, etol, qtol = (1e-11, 1e-11, 1e-9) if prec == "fp64" else (2e-5, 2e-6, 1e-5)
    for r, s in enumerate(small):
        rms = max(1.0, float(np.sqrt(np.mean(b["forces"][r] ** 2))))
        assert np.max(np.abs(a["forces"][r] - b["forces"][r])) < ftol * rms
        assert np.max(np.abs(a["e_atom"][r] - b["e_atom"][r])) < etol * 10
        assert np.max(np.abs(a["charges"][r] - b["charges"][r])) < qtol
        assert abs(a["energy"][r] - b["energy"][r]) < etol * s.n
        wr = max(1.0, float(np.max(np.abs(b["virial"][r]))))
        assert np.max(np.abs(a["virial"][r] - b["virial"][r])) < (1e-11 if prec == "fp64" else 1e-5) * wr


def test_fp64_reciprocal_roots(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "roots.cu"
    src.write_text('''
#include <cstdio>
#include <cmath>
#include "internal.cuh"
__global__ void k(int n, double* o) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double x = exp10(-2.0 + 6.0 * i / (n - 1));   // 1e-2 .. 1e4
  double a = ct::rsqrt_step(x), b = ct::rcbrt_step(x);
  o[i] = fabs(fma(-a * a, x, 1.0)) * 0.5 + fabs(a * sqrt(x) - 1.0) * 0.5;
  o[n + i] = fabs(b * cbrt(x) - 1.0);
}
int main() {
  const int n = 1 << 20;
  double* o;
  cudaMallocManaged(&o, 2 * n * sizeof(double));
  k<<<n / 256, 256>>>(n, o);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  double s = 0, c = 0;
  for (int i = 0; i < n; ++i) { s = std::fmax(s, o[i]); c = std::fmax(c, o[n + i]); }
  printf("%.3e %.3e\\n", s, c);
}
''')
    exe = str(tmp_path / "roots")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC,
                    "-I", os.path.join(os.path.dirname(HERE), "include"), str(src), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    # a few units of 2^-53: the rounding of y^n, of the correction and of the check itself
    assert float(out[0]) < 8e-16 and float(out[1]) < 8e-16, out
