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
