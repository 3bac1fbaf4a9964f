"""The first transform of a process on a stream that does not wait for the default
one: nothing that the library's own transforms read may still be on its way.  Each
case is a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import numpy as np, torch
import paper_1201_5029_gb300 as P
from oracle import pycool_observables as B
n, EPS = 64, 2.0 ** -53
side = torch.cuda.Stream()
rng = np.random.default_rng(8)
f = rng.standard_normal((2, n, n, n))
# 40 roundings a level, of the field's norm
"""
SPECTRUM = HEAD + """
cfg = P.make_config(n, 0.5 * n, "chaotic2", (1.0, 4.0), 0.01, mpl=1.0)
sim = P.Simulation(cfg, stream=side.cuda_stream)
sim.set_initial(f, f[::-1].copy())
p, c = sim.spectrum(0, 1)
po, co = B.spectrum(f[1])
lev = 40 * EPS * 3 * np.log2(n)
total = float(np.mean(f[1] ** 2))
assert np.array_equal(c, co)
assert np.all(np.abs(p - po) <= lev * (2 * np.sqrt(po * total) + lev * total) + lev * po)
"""
LINEAR = HEAD + """
x, y = (torch.from_numpy(f + k).cuda() for k in (0.0, 1.0))
ox, oy = torch.empty_like(x), torch.empty_like(y)
torch.cuda.synchronize()
cfg = P.make_config(n, 0.5 * n, "chaotic2", (1.0, 4.0), 0.01, mpl=1.0)
P.pycool_linear_evolve(cfg, 1.0, -1.0, x, y, 0, ox, oy, side.cuda_stream)
tol = 40 * EPS * 6 * np.log2(n)
for a, b in ((x, ox), (y, oy)):
    assert float((a - b).norm()) <= tol * float(a.norm())
"""


@pytest.mark.parametrize("code", [SPECTRUM, LINEAR], ids=["spectrum", "linear_evolve"])
def test_first_transform_on_a_side_stream(code):
    r = subprocess.run([sys.executable, "-c", code.format(root=ROOT, tests=os.path.join(ROOT, "tests"))],
                       capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
