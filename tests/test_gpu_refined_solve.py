"""FP64 charge solves that refine in cycles (one kernel per solve, by a cluster
up to 4,096 atoms of a lone system and by the whole grid above): they converge
under the iteration cap that one CG in FP64 needs from no charges; and they meet
tolerances far below the rounding of the FP64 residual, where the cycles no
longer gain and the CG has to go on in FP64 by its own recursion."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")
STRUCTS = {
    "cell8": lambda: st.sic_3c(1, 4.36, 0.1, seed=1),
    "sic64": lambda: st.sic_3c(2, 4.36, 0.08, seed=11),
    "sic512": lambda: st.sic_3c(4, 4.36, 0.05, seed=3),
    "slab582": lambda: st.stepped_slab_small(8, 4, 6),
    "sic4096": lambda: st.sic_3c(8, 4.36, 0.05, seed=9),
    "sic13824": lambda: st.sic_3c(12, 4.36, 0.05, seed=9),
}
# iterations of a CG in FP64 throughout, from zero charges to the default
# tolerance (measured with two launches per iteration and FP64 matrix passes)
CAPS = [("cell8", "block", 1), ("cell8", "jacobi", 7), ("sic64", "block", 24), ("sic64", "jacobi", 20),
        ("sic512", "block", 49), ("sic512", "jacobi", 37), ("slab582", "block", 45), ("slab582", "jacobi", 51),
        ("sic4096", "block", 53), ("sic4096", "jacobi", 52), ("sic13824", "block", 57), ("sic13824", "jacobi", 55)]


@pytest.mark.parametrize("name,pc,cap", CAPS)
def test_converges_under_the_cap_of_one_cg(name, pc, cap):
    s = STRUCTS[name]()
    sysm = ctbop.System(P1, precision="fp64", precond=pc, cg_max_iter=cap)
    sysm.load(s)
    sysm.compute()
    assert sysm.status()["rc"] == "OK", sysm.status()["cg_iters_last"]
    if (name, pc) == ("cell8", "block"):
        # (steps move the atoms under a preconditioner that was the exact inverse
        # at the last list build: one iteration is not enough for one CG either)
        sysm.close()
        return
    sysm.step(2, 0.5)
    assert sysm.profile_steps(1, 0.5)["cg_update"][1] == 0   # (the solve is one kernel)
    assert sysm.status()["rc"] == "OK"
    sysm.close()


@pytest.mark.parametrize("tol", [1e-15, 1e-17, 1e-25])
@pytest.mark.parametrize("name", ["cell8", "sic512", "slab582", "sic13824"])
def test_tolerances_below_the_residuals_rounding(name, tol):
    s = STRUCTS[name]()
    out = []
    for t in (0.0, tol):
        sysm = ctbop.System(P1, precision="fp64", cg_tol=t)
        sysm.load(s)
        sysm.compute()
        d = sysm.status()
        assert d["rc"] == "OK", d["cg_iters_last"]
        assert sysm.profile_steps(1, 0.5)["cg_update"][1] == 0
        sysm.set_positions(s.x)
        sysm.compute()
        assert sysm.status()["rc"] == "OK"
        out.append(sysm.get("charges"))
        sysm.close()
    # the default stops at 1e-11 eV/e over eigenvalues of the order of 10 eV/e^2
    assert np.max(np.abs(out[0] - out[1])) < 1e-9
    assert abs(out[1].sum()) < 1e-10
