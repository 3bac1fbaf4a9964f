"""The plain staging at the smallest sides, where a site's neighbours coincide and a tile's
halo ring is larger than the tile, and at sides above its other tests (two fields, tiles of
unequal width and height), against the oracle."""
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("name,stencil,n", [
    ("preheat32", "7pt", 1), ("oscillon256", "iso27", 1), ("qball256", "7pt", 2),
    ("preheat32", "iso27", 2), ("oscillon256", "7pt", 3), ("qball256", "4th", 4),
    ("preheat32", "4th", 5), ("oscillon256", "4th", 7), ("preheat32", "7pt", 100),
    ("qball256", "iso27", 101), ("oscillon256", "4th", 111)])
def test_against_the_oracle(name, stencil, n):
    w = I.workload(name, dt=0.005, order=4)
    phi, pi = I.white_ics(w, n=n)
    L = w["L"] / w["n"] * n          # the workload's spacing: stable at every side
    gphi, gpi, ge = G.run_gpu(P, G.gpu_cfg(P, dict(w, L=L), n=n, stencil=stencil), phi, pi, 2)
    st, oe = G.run_oracle(G.oracle_cfg(dict(w, L=L), n=n, stencil=stencil), phi, pi, 2)
    stages = int(ge["sweeps_done"]) + 1
    for g, o in ((gphi, st.phi), (gpi, st.pi)):
        assert all(e < t for e, t in zip(G.fluct_errors(g, o), G.fluct_tolerances(o, stages, 1e-11)))
    assert G.rel(ge["a"], st.a) < 1e-11 and G.rel(ge["rho"], oe["rho"]) < 1e-9
