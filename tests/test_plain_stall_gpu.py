"""The plain staging's bounded waits: a grid barrier that waits for an arrival that
never comes, with a short limit, makes every block of the launch give up and return,
as the TMA staging's (test_failure_gpu.py) -- one and two fields, one and two halo
planes, few blocks and one per SM."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("name,n,stencil", [
    ("preheat32", 45, "7pt"), ("oscillon256", 19, "iso27"), ("qball256", 70, "4th")])
def test_device_wait_runs_out_and_returns_a_status(name, n, stencil):
    w = I.workload(name)
    phi, pi = I.white_ics(w, n=n)
    cfg = G.gpu_cfg(P, w, n=n, stencil=stencil)

    def run():
        s = P.Simulation(cfg)
        s.set_initial(phi, pi)
        s.evolve(2)
        out = s.get_fields()
        s.close()
        return out

    before = run()
    sim = P.Simulation(cfg)
    sim.set_initial(phi, pi)
    assert P.pycool_debug_barrier_stall(sim.handle, 1 << 20) == P.OK   # ~0.5 ms limit
    sim.evolve(2)
    t0 = time.perf_counter()
    assert sim.sync(30.0) == P.E_TIMEOUT
    assert time.perf_counter() - t0 < 10.0
    with pytest.raises(P.PycoolError) as ei:
        sim.evolve(1)
    assert ei.value.status == P.E_STATE
    sim.close()
    after = run()                      # the context is still usable: same result as before
    for a, b in zip(before, after):
        assert np.array_equal(a, b)


def test_no_persistent_kernel_no_stall():
    w = I.workload("oscillon256")
    sim = P.Simulation(G.gpu_cfg(P, w, n=45, precision="split_fp32"))
    assert P.pycool_debug_barrier_stall(sim.handle, 1 << 20) == P.E_STATE
    sim.close()
