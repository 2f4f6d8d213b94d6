"""Which form of the charge solve a batch takes (one kernel per solve, or two
launches per iteration; told by the update launches of the phase times), at the
batches that the tests of the forms mean to compare and on both sides of the
rule for batches of uneven replicas, whose clusters all have the size that the
largest replica wants."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


def _cell(n):
    return st.sic_3c(n, 4.36, 0.05, seed=3)   # 8 n^3 atoms


def _one_kernel(structs, prec):
    sysm = ctbop.System(P1, precision=prec)
    sysm.load_replicas(structs)
    sysm.compute()
    launches = sysm.profile_steps(1, 0.5)["cg_update"][1]
    assert sysm.status()["rc"] == "OK"
    sysm.close()
    return launches == 0


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes,one", [
    ([2], True), ([8], True), ([10], True),                        # lone: cluster, cluster, grid
    ([2, 1, 3], True), ([2, 1, 3, 11], False),                     # 10,648 atoms: too many for a cluster
    ([8] + [2] * 20, True), ([8] + [2] * 1000, False),             # few and many small ones beside a large one
    ([8, 8] + [3] * 300, False), ([6] + [2] * 100, True), ([5] * 64, True), ([2] * 500, True)])
def test_form_of_the_solve(prec, sizes, one):
    assert _one_kernel([_cell(n) for n in sizes], prec) == one


@pytest.mark.parametrize("count,one", [(4, True), (16, False)])
def test_form_of_large_replicas(count, one):
    """8,000 atoms each, mixed: seven clusters at a time."""
    assert _one_kernel([_cell(10)] * count, "mixed") == one


def test_ensembles_keep_their_clusters():
    assert _one_kernel(st.annealing_ensemble(96, n_max=3000)[0], "mixed")
    assert _one_kernel(st.differentiation_batch(192), "mixed")
    assert _one_kernel(st.differentiation_batch(24), "fp64")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_an_uneven_batch_matches_its_replicas_alone(prec):
    small = [_cell(2), st.amorphous_carbon_cluster(45, 2.0, 12)]
    batch = [_cell(8)] + small * 300
    got = []
    for structs in (batch, [_cell(8)], [small[0]], [small[1]]):
        sysm = ctbop.System(P1, precision=prec)
        sysm.load_replicas(structs)
        sysm.compute()
        got.append((sysm.get("charges"), sysm.get("energy")))
        sysm.close()
    n = [s.n for s in batch]
    q = np.split(got[0][0], np.cumsum(n)[:-1])
    # every solve ends within the residual tolerance of the minimiser (1e-11 or
    # 1e-5 eV/e over eigenvalues of the order of 10 eV/e^2)
    qtol, etol = (1e-9, 1e-9) if prec == "fp64" else (1e-5, 2e-6)
    for r, (k, e) in enumerate([(0, 1), (1, 2), (2, 3), (599, 2), (600, 3)]):
        assert np.max(np.abs(q[k] - got[e][0])) < qtol
        assert abs(got[0][1][k] - got[e][1][0]) < etol * n[k]
