"""Removal energies report a batch solve that did not converge: the system
itself converges under a small iteration cap (restarted from its own charges
until it has), the systems without a candidate, which start from those charges,
do not."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("count", [1, 5])
def test_an_unconverged_batch_solve_is_an_error(prec, count):
    s = st.stepped_slab_small(6, 3, 4)
    cand = np.nonzero((s.types == 0) & ~s.frozen)[0][:count]
    sysm = ctbop.System(P1, precision=prec, cg_max_iter=4)
    sysm.load(s)
    for _ in range(100):
        sysm.set_positions(s.x)
        sysm.compute()
        if sysm.status()["rc"] == "OK":
            break
    assert sysm.status()["rc"] == "OK"
    with pytest.raises(ctbop.CtbopError, match="CG_NOT_CONVERGED"):
        sysm.removal_energies(cand)
    assert sysm.status()["rc"] == "OK"   # the system's own state is as it was
    sysm.close()
    ref = ctbop.System(P1, precision=prec)
    ref.load(s)
    assert np.all(np.isfinite(ref.removal_energies(cand)))
    ref.close()
