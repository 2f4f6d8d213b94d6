"""Neighbour lists of the FP64 policy, whose pair tests run in FP32 with the FP64
distance taken near the limits: the numbers of covalent and of all entries
against a count over all images in FP64, with pairs set a few parts in 1e9 to
1e6 inside and outside the list radii, in open, periodic and tiny boxes, and
with coordinates far from the origin."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")
SKIN = 0.3


def _counts(x, types, box, pbc, rc, rcov):
    m = [int(np.ceil(rc / L)) if p else 0 for L, p in zip(box, pbc)]
    n_all = n_cov = 0
    for a in range(-m[0], m[0] + 1):
        for b in range(-m[1], m[1] + 1):
            for c in range(-m[2], m[2] + 1):
                d = x[None, :, :] + np.array([a, b, c]) * box - x[:, None, :]
                r2 = np.sum(d * d, axis=2)
                if a == b == c == 0:
                    np.fill_diagonal(r2, np.inf)
                lim = (rcov[types[:, None] * 2 + types[None, :]]) ** 2
                n_cov += np.sum(r2 < lim)
                n_all += np.sum(r2 < np.maximum(lim, rc * rc))
    return n_all / len(x), n_cov / len(x)


@pytest.mark.parametrize("kind", ["open", "periodic", "tiny", "far"])
def test_fp64_lists_hold_the_pairs_inside_the_radii(kind):
    v = ctbop.params_vector(ctbop.params_struct(P1))
    p = ctbop.params_struct(P1)
    rc, rcov = p.r_coul + SKIN, np.array(list(p.S)) + SKIN
    assert np.array_equal(np.array(list(p.S)), v[20:24])
    rng = np.random.default_rng(3)
    box = np.full(3, 7.0 if kind == "tiny" else 26.0)
    n = 12 if kind == "tiny" else 200
    x = rng.uniform(0.0, 1.0, (n, 3)) * box
    types = rng.integers(0, 2, n).astype(np.int32)
    more, mt = [], []
    for k, rel in enumerate((1e-9, -1e-9, 3e-8, -3e-8, 1e-7, -1e-7, 3e-6, -3e-6) * 3):
        d = rng.normal(size=3)
        d /= np.linalg.norm(d)
        j, t = int(rng.integers(0, n)), int(rng.integers(0, 2))
        r = rcov[types[j] * 2 + t] if k % 2 else rc
        if kind != "tiny":
            more.append(x[j] + d * r * (1.0 + rel))
            mt.append(t)
    if more:
        x, types = np.concatenate([x, more]), np.concatenate([types, np.array(mt, dtype=np.int32)])
    if kind == "far":
        x[::2] += 400.0     # (an open box's cells reach as far as its atoms)
    pbc = np.full(3, kind in ("periodic", "tiny"))
    s = st.Structure(name=kind, x=x, types=types, box=box, pbc=pbc, frozen=np.zeros(len(x), dtype=bool))
    sysm = ctbop.System(P1, precision="fp64", skin=SKIN)
    sysm.load_replicas([s])
    try:
        sysm.compute(fixed_charges=True)
        got = sysm.status()
    finally:
        sysm.close()
    n_all, n_cov = _counts(x, types, box, pbc, rc, rcov)
    assert abs(got["mean_cov"] - n_cov) < 1e-9
    assert abs(got["mean_all"] - n_all) < 1e-9
