"""The FP64 persistent kernel's fixed-point stencil on the GPU.

A stage whose input's largest |phi| and |pi| are known sums D in 64-bit fixed
point, any other in float64.  A checkpoint carries the maxima (bytes 160..175
of its background record), so that one with them cleared continues in float64:
both continuations are held to the oracle's tolerance of one stage, over fields
whose values span many binades, a field that is zero, and magnitudes at the
ends of the range that the scale can take."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402

AMAX = slice(160, 176)


def _fields(kind, n, nf, seed=3):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((2, nf, n, n, n))
    if kind == "binades":      # magnitudes from 2^-60 to 1, signs mixed
        x = np.sign(x) * 2.0 ** rng.uniform(-60, 0, x.shape)
    elif kind == "background":
        x = 1.0 + 1e-6 * x
    elif kind == "zero":       # the last field and its momentum vanish everywhere
        x[:, -1] = 0.0
    elif kind == "tiny":       # below the smallest scale: stays in float64
        x = x * 2.0 ** -970
    elif kind == "small":
        x = x * 2.0 ** -400
    return x[0], x[1]


@pytest.mark.parametrize("stencil", ["7pt", "iso27", "4th"])
@pytest.mark.parametrize("model,kind,n", [
    ("free", "binades", 32), ("free", "tiny", 32), ("free", "small", 64),
    ("chaotic2", "zero", 32), ("qball", "background", 64), ("oscillon", "binades", 96)])
def test_fixed_point_against_float64(model, kind, n, stencil):
    params = {"free": (1.0,), "chaotic2": (1.0, 4.0), "qball": (1.0, -0.1, 1.0),
              "oscillon": (1.0, 1.0, 0.5)}[model]
    phi, pi = _fields(kind, n, P.MODEL_NF[P.MODELS[model]])
    w = dict(n=n, L=0.5 * n, model=model, params=params, order=2, dt=0.05, mpl=np.inf)
    sim = P.Simulation(G.gpu_cfg(P, w, stencil=stencil))
    sim.set_initial(phi, pi)
    blob = sim.checkpoint()
    known = np.frombuffer(blob[AMAX], dtype=np.uint32)[: 2 * phi.shape[0]]
    hi = np.array([[np.abs(a[f]).max() for a in (phi, pi)] for f in range(phi.shape[0])])
    assert np.array_equal(known & 0x7fffffff, (hi.ravel().view(np.uint64) >> 32).astype(np.uint32))
    out = []
    for b in (blob, blob[:160] + bytes(16) + blob[176:]):
        sim.restore(b)
        sim.evolve(1)
        assert sim.sync() == P.OK
        out.append(sim.get_fields())
    sim.close()
    st, _ = G.run_oracle(G.oracle_cfg(w, stencil=stencil), phi, pi, 1)
    # one stage: each side within 40 roundings at the field's magnitude of the
    # oracle (fluct_tolerances); a weight of 4.3 dt / dx^2 scales the stencil's
    for got in out:
        for g, o in zip(got, (st.phi, st.pi)):
            for e, t in zip(G.fluct_errors(g, o), G.fluct_tolerances(o, 1, 0.0)):
                assert e <= t, (e, t)
    if kind == "zero":
        assert all(not a[-1].any() for got in out for a in got)
