"""The error of the FP64 form's integer Laplacian, site by site.

One leapfrog stage of the massless free field with pi = 0 and m_pl infinite leaves
pi = kD D[phi] with kD = dt / dx^2, so pi / kD shows D itself.  Against extended
precision D may be off by
  sum |w| / (2 den) U + 4 2^-53 |D|,
U = 2^-(63 - headroom) of the binade's end above the largest |phi|: half a unit a value
(sum |w| / den: 12, 256/30, 192/12; headroom 4, 8, 8), then D's and kD's rounding
(1/den and the products).  A lump that falls through 60 binades, signs mixed, in
which most sites are below a unit; and the pattern with the largest sum that a
lattice can have (all weights of one sign), with magnitudes up to the last float64
below the binade's end, at which an integer sum would wrap if it could."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")

LD = np.longdouble
W = {"7pt": (4, 12, 1, lambda o: {0: -6, 1: 1}.get(sum(map(abs, o)), 0)),
     "iso27": (8, 256, 30, lambda o: (-128, 14, 3, 1)[sum(map(abs, o))]),
     "4th": (8, 192, 12, None)}


def _exact(phi, stencil):
    """den D in extended precision."""
    f = phi.astype(LD)
    if stencil == "4th":
        out = -90 * f
        for ax in range(3):
            for k, w in ((1, 16), (2, -1)):
                out += w * (np.roll(f, k, ax) + np.roll(f, -k, ax))
        return out
    out = np.zeros_like(f)
    r = (-1, 0, 1)
    for o in [(z, y, x) for z in r for y in r for x in r]:
        w = W[stencil][3](o)
        if w:
            out += w * np.roll(f, o, (0, 1, 2))
    return out


def _field(kind, n):
    x = (np.arange(n) - n // 2)
    r2 = x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2
    if kind == "lump":
        s = np.sign(np.random.default_rng(2).standard_normal((n, n, n)))
        return 0.7 * s * 2.0 ** (-60.0 * r2 / (n // 2) ** 2)
    even = np.arange(n) % 2 == 0
    all_even = even[:, None, None] & even[None, :, None] & even[None, None, :]
    big = {"extreme": 1.75, "top": 2.0 - 2.0 ** -20, "last": np.nextafter(2.0, 0.0)}[kind]
    return np.where(all_even, -big, big)


@pytest.mark.parametrize("stencil", ["7pt", "iso27", "4th"])
@pytest.mark.parametrize("kind", ["lump", "extreme", "top", "last"])
@pytest.mark.parametrize("n", [32, 64, 22])
def test_error_of_d(n, kind, stencil):
    head, total, den, _ = W[stencil]
    phi = _field(kind, n)
    dt, dx = 0.125, 0.5       # kD = 1/2, exact
    sim = P.Simulation(P.make_config(n, dx * n, "free", (0.0,), dt, order=2, stencil=stencil,
                                     mpl=np.inf))
    sim.set_initial(phi[None], np.zeros((1, n, n, n)))
    sim.evolve(1)
    _, pi = sim.get_fields()
    sim.close()
    d = _exact(phi, stencil) / den
    unit = 2.0 ** (np.floor(np.log2(np.abs(phi).max())) + 1 - (63 - head))
    tol = total / (2 * den) * unit + 4 * 2.0 ** -53 * np.abs(d)
    err = np.abs(pi[0].astype(LD) / (dt / dx ** 2) - d)
    print("\n", n, kind, stencil, float((err / tol).max()))
    assert (err <= tol).all()
