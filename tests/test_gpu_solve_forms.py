"""The forms of the charge solve (a thread-block cluster per replica, all
blocks on one replica, two launches per iteration; picked by size) reach the
same minimiser: the same replicas are solved in batches and alone, so that
their solves take different forms, at sizes around the forms' edges: an empty
replica, one atom, replicas that share 32-atom blocks, 4096 and 4608 atoms (on
either side of the lone cluster's limit) and a batch with a replica too large
for a cluster."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


def _empty():
    return st.Structure("empty", np.zeros((0, 3)), np.zeros(0, np.int32), np.full(3, 20.0), np.zeros(3, bool))


def _one():
    return st.Structure("one", np.full((1, 3), 10.0), np.ones(1, np.int32), np.full(3, 20.0), np.zeros(3, bool))


def _solve(structs, prec, pc, steps=2):
    """Charges and energies of a batch, split by replica, after an evaluation
    and after two steps (warm starts from the solve's own history)."""
    sysm = ctbop.System(P1, precision=prec, precond=pc)
    sysm.load_replicas(structs)
    sysm.compute()
    out = []
    for k in range(2):
        if k:
            sysm.step(steps, 0.5)
        q, E = sysm.get("charges"), sysm.get("energy")
        cut = np.cumsum([s.n for s in structs])[:-1]
        out.append((np.split(q, cut), E))
    assert sysm.status()["rc"] == "OK"
    sysm.close()
    return out


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("pc", ["block", "jacobi"])
@pytest.mark.parametrize("group", ["small", "edge"])
def test_every_form_reaches_the_same_minimiser(prec, pc, group):
    big = st.sic_3c((10, 10, 11), 4.36, 0.05, seed=3)   # 8,800 atoms: too many for a cluster
    if group == "small":
        a = [_one(), st.sic_3c(2, 4.36, 0.05, seed=7), _empty(), st.amorphous_carbon_cluster(45, 2.0, 12),
             st.sic_3c((2, 2, 3), 4.36, 0.05, seed=8), st.stepped_slab_small(6, 3, 4)]
        batches = [a, a + [big], [a[1]], [a[5]]]
        where = [(0, range(len(a))), (1, range(len(a))), (2, [1]), (3, [5])]
    else:
        a = [st.sic_3c(8, 4.36, 0.05, seed=9), st.sic_3c((8, 8, 9), 4.36, 0.05, seed=10)]
        batches = [a, a + [big], [a[0]], [a[1]]]
        where = [(0, range(2)), (1, range(2)), (2, [0]), (3, [1])]
    got = [_solve(b, prec, pc) for b in batches]
    # every solve ends within the residual tolerance of the minimiser (1e-11 or
    # 1e-5 eV/e over eigenvalues of the order of 10 eV/e^2)
    qtol = 1e-9 if prec == "fp64" else 1e-5
    etol = 1e-9 if prec == "fp64" else 2e-6
    for b, names in where[1:]:
        for k, r in enumerate(names):
            for stage in range(2):
                q0, q1 = got[0][stage][0][r], got[b][stage][0][k]
                assert len(q0) == len(q1)
                if len(q0):
                    assert np.max(np.abs(q0 - q1)) < qtol
                    assert abs(q1.sum()) < 1e-9
                    assert abs(got[0][stage][1][r] - got[b][stage][1][k]) < etol * len(q0)
