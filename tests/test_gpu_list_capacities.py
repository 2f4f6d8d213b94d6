"""Covalent capacities above the need (ctbop_options.cap_cov): the places of the
other entries come after the covalent ones that were asked for, so the lists
are sized for both and the results are those of the default capacities."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("cap_cov,cap_all", [(100, 0), (100, 64), (30, 256), (128, 256)])
def test_a_larger_covalent_capacity_leaves_room_for_the_rest(prec, cap_cov, cap_all):
    s = st.sic_3c(2, 4.36, 0.05, seed=3)
    out = []
    for kw in ({}, {"cap_cov": cap_cov, "cap_all": cap_all}):
        sysm = ctbop.System(P1, precision=prec, **kw)
        sysm.load(s)
        sysm.compute()
        d = sysm.status()
        assert d["rc"] == "OK"
        out.append((sysm.get("forces"), d["max_cov"], d["max_all"]))
        sysm.close()
    assert out[0][1:] == out[1][1:]
    # (the order of a row's entries may differ: rounding)
    assert np.max(np.abs(out[0][0] - out[1][0])) < (1e-9 if prec == "fp64" else 1e-3)
