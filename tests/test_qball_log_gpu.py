"""The logarithm of the FP64 form's Q-ball kick near its reference.

With K = -1 and M^2 the field's own |Phi|^2/2 the kick is m^2 Phi ln(|Phi|^2/(2 M^2)),
a logarithm near zero and nothing else (m_pl infinite, pi = 0, a spacing so large that
the Laplacian is below 1e-20): pi / (dt phi) shows its absolute error.  Site by site that
scatters by the two roundings of |Phi|^2 = phi1^2 + phi2^2, uniform over half an ulp:
with |Phi|^2 about 1.5, 2^-53/sqrt(3) and half as much for a square about 0.75, over
1.5: 0.43 2^-53.  A correction term of fewer bits would add to it; the bound is
0.5 2^-53, in every tier of the argument up to the two-digit ones."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")

LD = np.longdouble


@pytest.mark.parametrize("top", [-17, -16, -14, -12, -9])
@pytest.mark.parametrize("n", [32, 21])
def test_scatter_of_the_logarithm(n, top):
    rng = np.random.default_rng(100 - top)
    u2 = 1.5 * (1 + rng.choice((-1.0, 1.0), (n, n, n)) * 2.0 ** rng.uniform(top - 1, top, (n, n, n)))
    u2[0, 0, 0] = 1.5                       # the reference
    phi = np.sqrt(u2) * np.array([math.cos(0.7), math.sin(0.7)])[:, None, None, None]
    dt = 0.125
    sim = P.Simulation(P.make_config(n, 1e12 * n, "qball", (1.0, -1.0, math.sqrt(0.75)), dt, order=2,
                                     mpl=np.inf))
    sim.set_initial(phi, np.zeros_like(phi))
    sim.evolve(1)
    _, pi = sim.get_fields()
    sim.close()
    exact = np.log1p((phi[0].astype(LD) ** 2 + phi[1].astype(LD) ** 2) / LD(1.5) - 1)
    for f in range(2):
        err = np.float64(pi[f].astype(LD) / (phi[f].astype(LD) * dt) - exact) * 2.0 ** 53
        print("\n", n, top, f, err.std(), err.mean())
        assert err.std() <= 0.5
        assert abs(err.mean()) <= 8.0       # the reference's own logarithm and reciprocal
