"""Derivatives with respect to the cutoff radii where a third atom stands just
past the inner radius: there an FP32 cutoff rounds to 1 and its slope is all but
zero, while the slope of that slope, which the force part of the loss takes,
has already jumped. FP32 policy against FP64 on the same atoms."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


@pytest.mark.parametrize("typ,t", [(0, 4e-5), (1, 4e-5), (1, 1e-4), (1, 3e-4), (1, 0.3)])
def test_cutoff_radius_gradient_past_the_inner_radius(typ, t):
    v = ctbop.params_vector(ctbop.params_struct(P1))
    R, S = v[16 + 3 * typ], v[20 + 3 * typ]
    a, b = np.array([0.6, 0.64, 0.48]), np.array([-0.48, 0.6, -0.64])
    x = np.array([np.zeros(3), (0.85 * R) * a, (R + t * (S - R)) * b]) + 9.3
    s = st.Structure(name="three atoms", x=x, types=np.full(3, typ, dtype=np.int32), box=np.full(3, 20.0),
                     pbc=np.zeros(3, dtype=bool), frozen=np.zeros(3, dtype=bool))
    F_ref = np.random.default_rng(1).normal(0.0, 2.0, (3, 3))
    G = []
    for prec in ("fp64", "mixed"):
        sysm = ctbop.System(P1, precision=prec)
        sysm.load_replicas([s])
        _, g = sysm.param_grad(w_F=[1.0], F_ref=F_ref)
        G.append(ctbop.params_vector(g))
        sysm.close()
    # FP32 lengths near 2 A: 2e-7 A of a taper of 0.25 A, terms to some 1e-6
    # each, cancelling to a tenth of their size at worst
    k = slice(16, 24)
    assert np.max(np.abs(G[0][k])) > 0.0
    assert np.max(np.abs(G[1][k] - G[0][k])) <= 1e-4 * np.max(np.abs(G[0][k]))
