"""Ring search of atoms whose surroundings overflow the table in shared memory
(160 places): in a dense C cluster the atoms within four bonds of one are up to
194, those within three at most 96, so a search for rings of up to eight atoms
takes the larger tables and one for up to six does not; both must find the same
rings of up to six atoms."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_overflowing_tables_find_the_same_rings(prec):
    structs = [st.amorphous_carbon_cluster(600, 4.5, 5), st.graphene_sheet(200, 3)]
    sysm = ctbop.System(P1, precision=prec)
    sysm.load_replicas(structs)
    sysm.compute()

    def records(max_size):
        r = sysm.rings(max_size=max_size)
        r = r[r["size"] <= 6]
        key = np.lexsort((r["centre"][:, 2], r["centre"][:, 1], r["centre"][:, 0], r["size"], r["replica"]))
        return r[key]

    a, b = records(8), records(6)
    F = sysm.get("forces")
    sysm.compute()
    assert np.allclose(sysm.get("forces"), F, rtol=0, atol=1e-4)   # (the search leaves the system usable)
    sysm.close()
    assert len(a) == len(b) and len(a) > 500
    assert np.array_equal(a["size"], b["size"]) and np.array_equal(a["replica"], b["replica"])
    assert np.array_equal(a["centre"], b["centre"])
    assert np.array_equal(a["orientation"], b["orientation"], equal_nan=True)


def _host_rings(s, cut, max_size):
    """Rings of an open cluster straight from the definition: n atoms in a
    circle of bonds, the graph distance of any two the shorter way round it.
    Tuples (size, centre)."""
    d = np.linalg.norm(s.x[:, None] - s.x[None], axis=-1)
    bond = (d < cut) & (d > 0) & (s.types[:, None] == 1) & (s.types[None] == 1)
    near = [np.nonzero(b)[0].tolist() for b in bond]
    dist = np.full((s.n, s.n), 99)
    reach = np.eye(s.n, dtype=bool)
    for k in range(max_size // 2 + 1):
        dist[reach & (dist == 99)] = k
        reach = (reach.astype(np.float32) @ bond.astype(np.float32)) > 0
    dist = dist.tolist()
    out = []

    def extend(path, n):
        t = len(path)
        if t == n:
            if path[1] < path[-1] and dist[path[0]][path[-1]] == 1:
                out.append((n, s.x[path].mean(0)))
            return
        for w in near[path[-1]]:
            if w > path[0] and w not in path and all(
                    dist[v][w] == min(t - k, n - t + k) for k, v in enumerate(path)):
                extend(path + [w], n)

    for n in range(3, max_size + 1):
        for a in range(s.n):
            extend([a], n)
    return out


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_every_ring_is_found_once_whatever_the_table(prec):
    """Against the definition, ring by ring, in a cluster whose densest atoms
    take the larger tables (56 of 600): none missing and none twice."""
    s = st.amorphous_carbon_cluster(600, 4.5, 5)
    want = _host_rings(s, P1["pair"]["CC"]["S"], 8)
    sysm = ctbop.System(P1, precision=prec)
    sysm.load(s)
    sysm.compute()
    got = sysm.rings()
    sysm.close()
    assert len(got) == len(want)
    for n in range(3, 9):
        a = np.array([c for k, c in want if k == n]).reshape(-1, 3)
        b = got["centre"][got["size"] == n]
        assert len(a) == len(b)
        # one to one, to the rounding of the bond vectors
        d = np.linalg.norm(a[:, None] - b[None], axis=-1)
        assert np.array_equal(np.sort(d.argmin(1)), np.arange(len(b))) and np.all(d.min(1) < (1e-9 if prec == "fp64" else 1e-4))
