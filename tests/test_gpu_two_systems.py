"""Two systems in one process whose kernels need different amounts of shared
memory (a few and many covalent entries per atom) do not limit one another: the
allowance belongs to the kernel, not to the system that was set up last. Taken
in turn, and by two threads at once."""
import threading

import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


def _system(s, cap, prec):
    sysm = ctbop.System(P1, precision=prec, cap_cov=cap, cap_all=512)
    sysm.load(s)
    return sysm


def _use(sysm, s, k=0):
    sysm.set_positions(s.x)
    sysm.compute()
    F = sysm.get("forces")
    L, G = sysm.param_grad(w_E=[1.0], E_ref=[0.0], w_F=[0.1], F_ref=np.zeros((s.n, 3)))
    return F, L


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_in_turn(prec):
    s = st.sic_3c(2, 4.36, 0.05, seed=3)
    wide = _system(s, 100, prec)
    F0, L0 = _use(wide, s)
    narrow = _system(s, 16, prec)
    F1, L1 = _use(narrow, s)
    F2, L2 = _use(wide, s)
    wide.step(2, 0.5)
    assert wide.status()["rc"] == narrow.status()["rc"] == "OK"
    wide.close()
    narrow.close()
    tol = 1e-9 if prec == "fp64" else 1e-3
    assert np.max(np.abs(F1 - F0)) < tol and np.max(np.abs(F2 - F0)) < tol
    assert abs(L1 - L0) < tol * abs(L0) and abs(L2 - L0) < tol * abs(L0)


def test_by_two_threads():
    s = st.sic_3c(2, 4.36, 0.05, seed=3)
    systems = [_system(s, cap, "mixed") for cap in (100, 16)]
    want = [_use(y, s)[1] for y in systems]
    failed = []

    def work(k):
        try:
            for _ in range(60):
                L = _use(systems[k], s)[1]
                assert abs(L - want[k]) < 1e-3 * abs(want[k])
        except Exception as e:   # (a thread's exception would be lost)
            failed.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for y in systems:
        y.close()
    assert not failed, failed
