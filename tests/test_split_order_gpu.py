"""The order of the split-FP32 form's float32 sums.

A stage's lattice sums set the re-centring of the next one, and a float32 mean
shift below half an ulp of the fluctuations is counted again stage after stage,
so another order of summation shows in the field at some 1e-9 of itself where a
one-field background passes near zero.  tests/golden/split_fp32_order.txt holds
what the per-stage kernels (sides that are not multiples of 32, and the 13-point
stencil) and the persistent kernel with units of at least four planes give there:
phi and pi at every (n^3 // 40)-th site.  The fields are held to 1e-9 of their
norm, the bound of float64 outputs."""
import os

import numpy as np
import pytest

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "split_fp32_order.txt")
CASES = [(19, "7pt", 2, 97), (45, "iso27", 2, 97), (45, "4th", 2, 97), (32, "4th", 2, 97),
         (64, "iso27", 2, 97), (32, "7pt", 2, 97), (45, "7pt", 8, 6), (64, "7pt", 8, 6)]


def samples(n, stencil, order, steps):
    """phi and pi of the oscillon model (dx of the 256^3 workload) at the golden sites."""
    w = I.workload("oscillon256")
    phi, pi = I.white_ics(w, n=n)
    sim = P.Simulation(P.make_config(n, w["L"] / w["n"] * n, w["model"], w["params"], 0.02,
                                     order=order, precision="split_fp32", stencil=stencil,
                                     mpl=w["mpl"]))
    sim.set_initial(phi, pi)
    sim.evolve(steps)
    got = sim.get_fields()
    sim.close()
    return [a.reshape(-1)[:: n ** 3 // 40] for a in got]


def golden():
    out = {}
    with open(GOLDEN) as f:
        for line in f:
            if not line.startswith("#"):
                n, stencil, order, steps, which, *v = line.split()
                key = int(n), stencil, int(order), int(steps)
                out.setdefault(key, {})[which] = np.array([float.fromhex(x) for x in v])
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_outputs(case):
    want = golden()[case]
    for which, got in zip(("phi", "pi"), samples(*case)):
        ref = want[which]
        assert got.shape == ref.shape
        assert np.linalg.norm(got - ref) <= 1e-9 * np.linalg.norm(ref), which


@pytest.mark.parametrize("nf", [1, 2])
@pytest.mark.parametrize("n", [32, 64, 96, 128, 160])
def test_units_of_at_least_four_planes(n, nf):
    """The persistent kernel's units of the split-FP32 form (planes with one halo plane a side)."""
    for stencil in (P.STENCIL_7PT, P.STENCIL_ISO27):
        _, units, _ = P.pycool_persist_plan(n, nf, P.SPLIT_FP32, 152, 126 << 20, stencil)
        assert (units[:, 3] - 2 >= 4).all()
