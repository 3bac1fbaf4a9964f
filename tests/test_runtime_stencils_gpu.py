"""Run-time potentials at sides around the kick kernel's tiles (32 x 8 sites,
chunks of planes) with every stencil, the chaotic potential as expressions
against the oracle: the first stage of a new state sums in float64, the others
in fixed point."""
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402

CHAOTIC = ("0.5*p[0]*f0*f0 + 0.5*p[1]*f0*f0*f1*f1",
           ("p[0]*f0 + p[1]*f0*f1*f1", "p[1]*f0*f0*f1"))


@pytest.fixture(scope="module")
def model():
    return P.pycool_model_define(*CHAOTIC)


@pytest.mark.parametrize("stencil,n", [("7pt", 1), ("iso27", 2), ("4th", 4), ("7pt", 7),
                                       ("iso27", 33), ("4th", 35), ("7pt", 64), ("iso27", 40)])
def test_against_the_oracle(model, stencil, n):
    w = I.workload("preheat32", order=4)
    phi, pi = I.white_ics(w, n=n)
    cfg = P.make_config(n, w["L"] * n / 32, model, w["params"], w["dt"], order=4,
                        stencil=stencil, mpl=w["mpl"])
    gphi, gpi, ge = G.run_gpu(P, cfg, phi, pi, 4, chunks=2)
    st, oe = G.run_oracle(G.oracle_cfg(dict(w, L=w["L"] * n / 32), n=n, stencil=stencil), phi,
                          pi, 4)
    stages = int(ge["sweeps_done"]) + 1
    for g, o in ((gphi, st.phi), (gpi, st.pi)):
        assert max(G.field_errors(g, o)) < 1e-11
        assert all(e < t for e, t in zip(G.fluct_errors(g, o), G.fluct_tolerances(o, stages, 1e-11)))
    assert G.rel(ge["a"], st.a) < 1e-11 and G.rel(ge["rho"], oe["rho"]) < 1e-9
