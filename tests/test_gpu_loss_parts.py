"""The force part of the force-matching loss, summed on the device: against the
sum over the forces that the system reports, at atom counts at the edges of a
block, with several replicas, in the caller's and in a stored order."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("order", [None, "morton"])
@pytest.mark.parametrize("sizes", [(2,), (255,), (256,), (257,), (31, 1, 224, 33)])
def test_force_loss_is_the_sum_over_the_forces(sizes, order, prec):
    structs = [st.amorphous_carbon_cluster(n, 2.0, 7 + k) for k, n in enumerate(sizes)]
    sysm = ctbop.System(P1, precision=prec)
    sysm.load_replicas(structs, order=order)
    n = np.array([s.n for s in structs])
    rng = np.random.default_rng(8)
    w = rng.uniform(0.5, 2.0, len(n))
    F_ref = rng.normal(0.0, 1.0, (int(n.sum()), 3))
    loss, G = sysm.param_grad(w_F=w, F_ref=F_ref)

    def check(loss, w):   # against the forces of this very evaluation
        want = float(np.sum(np.repeat(w, n)[:, None] * (sysm.get("forces") - F_ref) ** 2))
        # 3 N positive FP64 terms summed in another order
        assert abs(loss - want) <= 1e-12 * want

    check(loss, w)
    # no weight: no loss and, as g is zero, no adjoint solve
    loss0, G0 = sysm.param_grad(w_F=0.0 * w, F_ref=F_ref)
    assert loss0 == 0.0 and not np.any(ctbop.params_vector(G0))
    # the weights enter linearly (the right-hand side doubles exactly; the
    # adjoint solve stops at its tolerance)
    loss2, G2 = sysm.param_grad(w_F=2.0 * w, F_ref=F_ref)
    g, g2 = ctbop.params_vector(G), ctbop.params_vector(G2)
    check(loss2, 2.0 * w)
    assert np.max(np.abs(g2 - 2.0 * g)) <= (1e-7 if prec == "fp64" else 1e-4) * np.max(np.abs(g2))
    sysm.close()
