"""The FP32 assembly and charge-force gather on either side of the lines between
8 lanes and a thread per atom (80,896 and 197,600 atoms): small replicas
alone and in batches between the lines and above both."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


def _eval(structs, q):
    sysm = ctbop.System(P1, precision="mixed")
    sysm.load_replicas(structs)
    sysm.set_charges(q)
    sysm.compute(fixed_charges=True)
    cut = np.cumsum([s.n for s in structs])[:-1]
    out = {k: np.split(sysm.get(k), cut) for k in ("forces", "e_atom")}
    out["virial"], out["energy"] = sysm.get("virial"), sysm.get("energy")
    sysm.compute()
    out["charges"] = np.split(sysm.get("charges"), cut)
    assert sysm.status()["rc"] == "OK"
    sysm.close()
    return out


@pytest.mark.parametrize("cells", [(24, 24, 18), (30, 30, 30)])   # 82,944 and 216,000 atoms beside the small ones
def test_thread_per_atom_matches_lane_groups(cells):
    small = [st.sic_3c(1, 4.36, 0.1, seed=1), st.amorphous_carbon_cluster(33, 2.0, 2), st.sic_3c(2, 4.36, 0.05, seed=3),
             st.stepped_slab_small(6, 3, 4), st.sic_3c(9, 4.36, 0.05, seed=4)]
    big = st.sic_3c(cells, 4.36, 0.05, seed=5)
    rng = np.random.default_rng(6)
    qs = [rng.normal(0.0, 0.2, s.n) for s in small]
    a = _eval(small, np.concatenate(qs))
    b = _eval(small + [big], np.concatenate(qs + [rng.normal(0.0, 0.2, big.n)]))
    # sums of about 230 FP32 terms, grouped otherwise: forces to some tens of
    # rounding units of the largest terms (14 eV/A pair terms of 0.04 e^2),
    # energies compensated, charges to the solve's tolerance
    for r, s in enumerate(small):
        rms = max(1.0, float(np.sqrt(np.mean(b["forces"][r] ** 2))))
        assert np.max(np.abs(a["forces"][r] - b["forces"][r])) < 2e-5 * rms
        assert np.max(np.abs(a["e_atom"][r] - b["e_atom"][r])) < 2e-5
        assert abs(a["energy"][r] - b["energy"][r]) < 2e-6 * s.n
        wr = max(1.0, float(np.max(np.abs(b["virial"][r]))))
        assert np.max(np.abs(a["virial"][r] - b["virial"][r])) < 1e-5 * wr
        assert np.max(np.abs(a["charges"][r] - b["charges"][r])) < 1e-5
