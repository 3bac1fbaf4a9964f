"""pycool_linear_evolve groups modes by the sorted magnitudes of their wave
numbers: odd and even sides, the smallest one, every stencil, and step counts
whose stages end before, at and after the end of a table chunk (64 entries),
against the oracle evolving every mode."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")
from oracle import pycool_linear as L  # noqa: E402
from oracle import pycool_oracle as O  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("n,stencil,order,steps", [
    (2, "7pt", 2, 3), (4, "4th", 4, 21), (5, "iso27", 2, 63), (6, "7pt", 2, 64),
    (9, "4th", 2, 65), (10, "iso27", 4, 43), (13, "7pt", 8, 9), (7, "7pt", 2, 0)])
def test_modes_of_every_class(n, stencil, order, steps):
    cfg = O.LatticeConfig(n=n, L=0.8 * n, model="chaotic2", params=(1.0, 50.0), dt=0.02,
                          order=order, mpl=10.0, stencil=stencil)
    rng = np.random.default_rng(n)
    phi = np.stack([b + 1e-3 * rng.standard_normal((n, n, n)) for b in (1.0, 0.2)])
    pi = np.stack([b + 1e-3 * rng.standard_normal((n, n, n)) for b in (-0.3, 0.1)])
    pa0 = O.initial_pa(cfg, 1.0, phi, pi)
    ls = L.from_lattice(cfg, phi, pi, 1.0, pa0)
    L.evolve(cfg, ls, steps)
    ophi, opi = L.to_lattice(ls)
    t = [torch.from_numpy(x).cuda() for x in (phi, pi)]
    out = [torch.empty_like(x) for x in t]
    gcfg = P.make_config(n, 0.8 * n, "chaotic2", (1.0, 50.0), 0.02, order=order, mpl=10.0,
                         stencil=stencil)
    a, pa, f0, p0 = P.pycool_linear_evolve(gcfg, 1.0, pa0, *t, steps, *out)
    assert G.rel(a, ls.a) < 1e-11 and G.rel(pa, ls.pa) < 1e-11
    stages = max(1, steps * P.pycool_stages_per_step(order))
    for g, o in zip(out, (ophi, opi)):
        for e, tol in zip(G.fluct_errors(g.cpu().numpy(), o), G.fluct_tolerances(o, stages, 1e-11)):
            assert e < tol
