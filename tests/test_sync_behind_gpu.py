"""pycool_sync waits for the evolve, not for what the caller has queued behind it on
the same stream: with a kernel of about a second there, a sync whose deadline is half a
second returns the finished state at once (a non-blocking stream and the default one)."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("side", [True, False])
@pytest.mark.parametrize("n,precision", [(32, "fp64"), (20, "fp64"), (20, "split_fp32")])
def test_work_behind_the_evolve(n, precision, side):
    stream = torch.cuda.Stream() if side else torch.cuda.default_stream()
    w = I.workload("preheat32")
    phi, pi = I.white_ics(w, n=n)
    sim = P.Simulation(G.gpu_cfg(P, w, n=n, precision=precision), stream=stream.cuda_stream)
    sim.set_initial(phi, pi)
    sim.evolve(2)
    with torch.cuda.stream(stream):
        torch.cuda._sleep(2_000_000_000)   # SM clocks, about a second
    t0 = time.perf_counter()
    status = sim.sync(0.5)
    steps = sim.energies()["steps_done"]
    waited = time.perf_counter() - t0
    assert status == P.OK and steps == 2
    assert waited < 0.5
    gphi, _ = sim.get_fields()
    assert np.isfinite(gphi).all()
    sim.close()
