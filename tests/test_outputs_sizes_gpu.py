"""Per-site energies and spectra at sides around the kernels' tile edges (32 x 8
columns, chunks of 4 to 32 planes, 2048 modes of a shell), odd ones whose second
field does not start on a 16-byte boundary among them, against the oracle on the
very fields that the simulation holds; and neither changes the simulation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from oracle import pycool_observables as B  # noqa: E402
from oracle import pycool_oracle as O  # noqa: E402
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("name,stencil,n,precision", [
    ("preheat32", "7pt", 1, "fp64"), ("preheat32", "iso27", 2, "fp64"),
    ("oscillon256", "4th", 5, "fp64"), ("preheat32", "7pt", 33, "fp64"),
    ("qball256", "4th", 41, "fp64"), ("qball256", "iso27", 31, "split_fp32"),
    ("preheat32", "7pt", 65, "split_fp32"), ("oscillon256", "7pt", 64, "split_dd")])
def test_on_the_fields_held(name, stencil, n, precision):
    w = I.workload(name, dt=0.005)
    phi, pi = I.white_ics(w, n=n)
    sim = P.Simulation(G.gpu_cfg(P, w, n=n, order=2, stencil=stencil, precision=precision))
    sim.set_initial(phi, pi)
    sim.evolve(2)
    before = sim.checkpoint()
    rho, prs = sim.energy_fields()
    power = [[sim.spectrum(k, f) for f in range(phi.shape[0])] for k in (0, 1)]
    assert sim.checkpoint() == before
    phi, pi = sim.get_fields()
    e = sim.energies()
    sim.close()
    st = O.State(phi=phi, pi=pi, a=e["a"], pa=e["pa"])
    orho, oprs = B.energy_fields(G.oracle_cfg(w, n=n, order=2, stencil=stencil), st)
    # some twenty roundings at the size of the terms; in the split forms the
    # differences are of fluctuations that the read-out rounds at phi0's size, so
    # G is off by 2 |d| 2^-53 |phi| per neighbour, d the differences
    size = np.abs(orho).max() + np.abs(oprs).max()
    d = max(float(np.ptp(x)) for x in phi)
    dx = w["L"] / n
    tol = 40 * G.EPS64 * (size + 8 * 2 * d * np.abs(phi).max() / (e["a"] * dx) ** 2)
    assert np.abs(rho - orho).max() <= tol and np.abs(prs - oprs).max() <= tol
    for k, arr in enumerate((phi, pi)):
        for f in range(arr.shape[0]):
            p, c = power[k][f]
            po, co = B.spectrum(arr[f])
            assert np.array_equal(c, co)
            # transforms: 3 log2 n levels of roundings at the field's norm; a shell's
            # power is quadratic, so its error is the amplitude's times twice its root
            total = float(np.mean(arr[f] ** 2))
            lev = G.EPS64 * 40 * max(1.0, 3 * np.log2(n))
            bound = lev * (2 * np.sqrt(po * total) + lev * total) + lev * po
            assert np.all(np.abs(p - po) <= bound)
