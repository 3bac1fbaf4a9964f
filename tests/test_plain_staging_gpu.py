"""The persistent kernel's plain staging on the GPU against the oracle: lattice
sides that TMA boxes do not take (single tiles, tiles of unequal width and
height, more tiles than blocks' worth of planes) with every stencil, and the
split-FP32 form's 13-point stencil at sides that are multiples of 32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("name,stencil,n,precision", [
    ("preheat32", "7pt", 45, "fp64"), ("preheat32", "iso27", 23, "fp64"),
    ("oscillon256", "4th", 35, "fp64"), ("oscillon256", "iso27", 70, "fp64"),
    ("qball256", "7pt", 22, "fp64"), ("qball256", "4th", 50, "fp64"),
    ("preheat32", "7pt", 45, "split_fp32"), ("oscillon256", "iso27", 23, "split_fp32"),
    ("qball256", "7pt", 70, "split_fp32"), ("preheat32", "4th", 32, "split_fp32"),
    ("oscillon256", "4th", 64, "split_fp32"), ("qball256", "4th", 35, "split_fp32")])
def test_against_the_oracle(name, stencil, n, precision):
    w = I.workload(name, dt=0.005, order=4)
    phi, pi = I.white_ics(w, n=n)
    gphi, gpi, ge = G.run_gpu(P, G.gpu_cfg(P, w, n=n, stencil=stencil, precision=precision), phi,
                              pi, 3, chunks=2)
    st, oe = G.run_oracle(G.oracle_cfg(w, n=n, stencil=stencil), phi, pi, 3)
    stages = int(ge["sweeps_done"]) + 1
    for g, o in ((gphi, st.phi), (gpi, st.pi)):
        # split-FP32: its stated bound at the fluctuations' scale
        tol = (G.fluct_tolerances(o, stages, 1e-11) if precision == "fp64"
               else [1e-4] * o.shape[0])
        assert all(e < t for e, t in zip(G.fluct_errors(g, o), tol))
    assert G.rel(ge["a"], st.a) < 1e-11 and G.rel(ge["rho"], oe["rho"]) < 1e-9

