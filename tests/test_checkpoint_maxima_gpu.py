"""A restored FP64 state takes its fixed-point scale from its fields, not from the
record's maxima: a checkpoint whose fields were scaled by 2^10 evolves as set_initial
of the scaled fields does, bit for bit, and one whose maxima were set too small as the
intact one.  (m_pl infinite: the scale factor, and with it the record's sums, do not
enter.)  Staged by TMA, staged plainly, and a potential given as expressions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
import gpu_helpers as G  # noqa: E402

AMAX = slice(160, 176)   # of the background record


@pytest.mark.parametrize("model,n,stencil", [
    ("oscillon", 32, "7pt"), ("oscillon", 64, "iso27"), ("chaotic2", 32, "4th"),
    ("chaotic2", 21, "7pt"), ("oscillon", 45, "iso27"), ("expr", 32, "7pt")])
def test_edited_checkpoint(model, n, stencil):
    nf = 2 if model == "chaotic2" else 1
    params = {"chaotic2": (1.0, 4.0), "oscillon": (1.0, 1e-9, 1e-18), "expr": (1.0,)}[model]
    if model == "expr":
        model = P.pycool_model_define("0.5*p[0]*f0*f0", ("p[0]*f0",))
    rng = np.random.default_rng(11)
    phi, pi = rng.standard_normal((2, nf, n, n, n))
    w = dict(n=n, L=0.5 * n, model=model, params=params, order=2, dt=0.02, mpl=np.inf)
    sim = P.Simulation(G.gpu_cfg(P, w, stencil=stencil))

    def evolved():
        sim.evolve(2)
        assert sim.sync() == P.OK
        return sim.get_fields()

    sim.set_initial(phi, pi)
    blob = sim.checkpoint()
    want = evolved()
    small = np.frombuffer(blob[AMAX], dtype=np.uint32) - np.uint32(12 << 20)   # 2^-12 of them
    sim.restore(blob[:AMAX.start] + small.tobytes() + blob[AMAX.stop:])
    for a, b in zip(want, evolved()):
        assert np.array_equal(a, b)
    fields = 2 * nf * n ** 3 * 8
    head, body = blob[:-fields], np.frombuffer(blob[-fields:], dtype=np.float64)
    sim.restore(head + (body * 1024.0).tobytes())
    got = evolved()
    sim.set_initial(phi * 1024.0, pi * 1024.0)
    for a, b in zip(evolved(), got):
        assert np.array_equal(a, b)
    sim.close()
