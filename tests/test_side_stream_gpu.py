"""Host data that a call uploads, on a stream that does not wait for the default
one: a restored checkpoint evolved at once, and a first spectrum (whose tables are
uploaded by that call), against the same on the default stream, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("n,precision", [(96, "fp64"), (45, "fp64"), (64, "split_fp32")])
def test_restore_then_evolve(n, precision):
    w = I.workload("preheat32")
    phi, pi = I.white_ics(w, n=n)
    cfg = G.gpu_cfg(P, w, n=n, precision=precision)
    out = []
    for stream in (None, torch.cuda.Stream().cuda_stream):
        sim = P.Simulation(cfg, stream=stream)
        sim.set_initial(phi, pi)
        sim.evolve(2)
        blob = sim.checkpoint()
        sim.set_initial(pi, phi)   # another state in every buffer
        sim.evolve(1)
        sim.restore(blob)
        sim.evolve(2)
        got = sim.get_fields()
        out.append([*got, *(sim.spectrum(0, 0))])
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
