"""The FP64 charge-force gather on the kernel values that the assembly keeps
against the one that computes them (an evaluation at fixed charges, which
assembles nothing): forces, energies and virial of the same charges, for 32 and
for 8 lanes per atom, rows that end inside a batch, replicas that share warps,
self images in a tiny box; and the virial read after steps."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")
KEYS = ("forces", "e_atom", "energy", "virial")


def _structs(kind):
    if kind == "ragged":
        return [st.amorphous_carbon_cluster(n, 2.0, 3 + n) for n in (2, 3, 31, 33)] + [st.sic_3c(1, 4.36, 0.1, seed=1)]
    if kind == "slab":
        return [st.stepped_slab_small(6, 3, 4)]
    return [st.sic_3c(11, 4.36, 0.05, seed=2)]      # 10,648 atoms: 8 lanes


@pytest.mark.parametrize("kind", ["ragged", "slab", "eight lanes"])
def test_stored_kernel_values_give_the_same_forces(kind):
    structs = _structs(kind)
    sysm = ctbop.System(P1, precision="fp64")
    sysm.load_replicas(structs)

    def compare(a, b):
        # the same expressions; sums of about 230 terms in the same order
        for k in KEYS:
            assert np.max(np.abs(a[k] - b[k])) <= 1e-11 * max(1.0, float(np.max(np.abs(b[k])))), k

    def read():
        return {k: sysm.get(k) for k in KEYS}

    for _ in range(2):        # direct, then from a graph
        sysm.compute()
        a = read()
        sysm.set_charges(sysm.get("charges"))
        sysm.compute(fixed_charges=True)
        compare(a, read())
    sysm.step(3, 0.5)
    a = read()                # (the virial of the stepped state: a gather of its own)
    sysm.set_charges(sysm.get("charges"))
    sysm.compute(fixed_charges=True)
    compare(a, read())
    sysm.close()
