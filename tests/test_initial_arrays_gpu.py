"""pycool_set_initial from device arrays that a copy takes and a kernel's float64 loads
do not: an address that is no multiple of 8.  And from arrays on an 8-byte boundary only,
which the kernel reads a value at a time.  Both against the aligned arrays, bit for bit."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


@pytest.mark.parametrize("shift", [4, 8, 12])
@pytest.mark.parametrize("name,n", [("preheat32", 32), ("oscillon256", 21), ("preheat32", 15)])
def test_unaligned_device_arrays(name, n, shift):
    w = I.workload(name)
    fields = I.white_ics(w, n=n)
    keep = []
    for x in fields:
        raw = torch.zeros(x.nbytes + 16, dtype=torch.uint8, device="cuda")
        raw[shift:shift + x.nbytes] = torch.from_numpy(x.reshape(-1).view(np.uint8).copy()).cuda()
        keep.append(raw)
    torch.cuda.synchronize()
    sim = P.Simulation(G.gpu_cfg(P, w, n=n))
    out = []
    for ptr in ([torch.from_numpy(x).cuda() for x in fields], keep):
        at = [t.data_ptr() + (shift if t.dtype == torch.uint8 else 0) for t in ptr]
        assert P.lib.pycool_set_initial(sim.handle, at[0], at[1], 1, 1.0, math.nan) == P.OK
        sim.evolve(2)
        out.append(sim.get_fields())
    sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
