"""The differentiable energy takes its results on the device where torch's
current stream is ordered with the system's, and through the host elsewhere:
the same energies and gradients on the default stream, on a stream that the
system shares, and on one it does not know; again after every change of the
positions (the first evaluation and the captured ones)."""
import numpy as np
import pytest

from paper_1802_07871_gb300 import ctbop
from paper_1802_07871_gb300 import structures as st

pytestmark = pytest.mark.gpu
P1 = st.load_params("p1")


# (positions handed over from a stream that the system does not know have to be
# complete by then: float64, which needs no conversion kernel)
@pytest.mark.parametrize("where,dtype", [("default", "float64"), ("default", "float32"), ("shared", "float64"),
                                         ("shared", "float32"), ("foreign", "float64"), ("cpu", "float32")])
def test_energy_and_gradient_on_any_stream(where, dtype):
    import torch
    from paper_1802_07871_gb300.autograd import Energy
    structs = [st.amorphous_carbon_cluster(33, 2.0, 2), st.sic_3c(1, 4.36, 0.1, seed=1)]
    off = np.cumsum([0] + [s.n for s in structs])
    ref = ctbop.System(P1, precision="fp64")
    ref.load_replicas(structs)
    sysm = ctbop.System(P1, precision="fp64")
    sysm.load_replicas(structs)
    stream = torch.cuda.Stream() if where in ("shared", "foreign") else torch.cuda.current_stream()
    if where == "shared":
        sysm.set_stream(stream.cuda_stream)
    x0 = np.concatenate([s.x for s in structs])
    dt = getattr(torch, dtype)
    torch.cuda.synchronize()
    for k in range(3):
        with torch.cuda.stream(stream):
            assert sysm.ordered_with_current_stream() == (where != "foreign")
            x = torch.tensor(x0 + 0.01 * k, dtype=dt, device="cpu" if where == "cpu" else "cuda", requires_grad=True)
            E = Energy.apply(x, sysm)
            (E * torch.tensor([1.0, 2.0], dtype=dt, device=x.device)).sum().backward()
            e, g = E.detach().cpu().numpy(), x.grad.cpu().numpy()
        ref.set_positions(x.detach().cpu().to(torch.float64).numpy())
        ref.compute()
        F = ref.get("forces")
        F[off[1]:] *= 2.0
        # the same system on the same positions: sums of atomics, solve tolerance
        tol = 1e-8 if dtype == "float64" else 1e-6
        assert e.dtype == np.dtype(dtype) and g.dtype == np.dtype(dtype)
        assert np.max(np.abs(e - ref.get("energy"))) <= tol * np.max(np.abs(e))
        assert np.max(np.abs(g + F)) <= tol * max(1.0, np.max(np.abs(F)))
    sysm.close()
    ref.close()


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_positions_still_being_written_on_a_foreign_stream(dtype):
    """The system does not know the stream that writes and converts the
    positions: it has to wait for them all the same."""
    import torch
    from paper_1802_07871_gb300.autograd import Energy
    s = st.sic_3c(2, 4.36, 0.05, seed=3)
    ref = ctbop.System(P1, precision="fp64")
    ref.load(s)
    sysm = ctbop.System(P1, precision="fp64")
    sysm.load(s)
    dt = getattr(torch, dtype)
    base = torch.tensor(s.x, dtype=dt, device="cuda")
    x = base.clone().requires_grad_(True)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for k in range(2):
        with torch.cuda.stream(stream):
            torch.cuda._sleep(50_000_000)   # (some 25 ms before the positions are there)
            with torch.no_grad():
                x.copy_(base + 0.01 * (k + 1) * torch.sin(7.0 * base))
            E = Energy.apply(x, sysm)
            (g,) = torch.autograd.grad(E.sum(), x)
        stream.synchronize()
        ref.set_positions(x.detach().cpu().to(torch.float64).numpy())
        ref.compute()
        tol = 1e-8 if dtype == "float64" else 1e-6
        assert np.max(np.abs(E.detach().cpu().numpy() - ref.get("energy"))) <= tol * abs(ref.get("energy")[0])
        assert np.max(np.abs(g.cpu().numpy() + ref.get("forces"))) <= tol * max(1.0, np.max(np.abs(ref.get("forces"))))
    sysm.close()
    ref.close()
