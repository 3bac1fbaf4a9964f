"""The library's own transforms (sides 64, 128 and 256) on the GPU, through the
spectrum and the linearised evolution: against numpy on white noise, a homogeneous
field, one plane wave, a single site and values of very different magnitudes; and
a value that is not finite spoils every mode, as float64 transforms have it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")
from oracle import pycool_observables as B  # noqa: E402
from paper_1201_5029_gb300 import inputs as I  # noqa: E402
import gpu_helpers as G  # noqa: E402


def _field(kind, n):
    rng = np.random.default_rng(5)
    f = rng.standard_normal((n, n, n))
    if kind == "background":
        f = 0.8 + 1e-4 * f
    elif kind == "constant":
        f = np.full((n, n, n), 0.7)
    elif kind == "wave":
        f = I.plane_wave(n, (3, n // 2, 5), 1e-3, 0.4)
    elif kind == "site":
        f = np.zeros((n, n, n))
        f[1, n - 1, 3] = -2.5
    elif kind == "binades":
        f = np.sign(f) * 2.0 ** rng.uniform(-60, 0, f.shape)
    return f


@pytest.mark.parametrize("n", [64, 128, 256])
@pytest.mark.parametrize("kind", ["noise", "background", "constant", "wave", "site", "binades"])
def test_spectrum(n, kind):
    f = _field(kind, n)[None]
    cfg = P.make_config(n, 0.5 * n, "free", (1.0,), 0.01, mpl=np.inf)
    sim = P.Simulation(cfg)
    sim.set_initial(f, f[:, ::-1].copy())
    for which, arr in ((0, f[0]), (1, f[0, ::-1])):
        p, c = sim.spectrum(which, 0)
        po, co = B.spectrum(np.ascontiguousarray(arr))
        assert np.array_equal(c, co)
        # 40 roundings a level over 3 log2 n levels, of the field's norm; a shell's
        # power is quadratic in its amplitude
        lev = 40 * G.EPS64 * 3 * np.log2(n)
        total = float(np.mean(arr ** 2))
        assert np.all(np.abs(p - po) <= lev * (2 * np.sqrt(po * total) + lev * total) + lev * po)
    sim.close()


@pytest.mark.parametrize("n", [64, 128])
@pytest.mark.parametrize("kind", ["noise", "wave", "site", "binades"])
def test_there_and_back(n, kind):
    """No steps: forward, the identity on every mode, inverse."""
    f = _field(kind, n)
    x = torch.from_numpy(np.stack([f, 1.0 + f[::-1]])).cuda()
    y = torch.from_numpy(np.stack([f[:, ::-1].copy(), -f])).cuda()
    ox, oy = torch.empty_like(x), torch.empty_like(y)
    cfg = P.make_config(n, 0.5 * n, "chaotic2", (1.0, 4.0), 0.01, mpl=1.0)
    P.pycool_linear_evolve(cfg, 1.0, -1.0, x, y, 0, ox, oy)
    # norm-wise, both transforms: 6 log2 n levels of roundings
    tol = 40 * G.EPS64 * 6 * np.log2(n)
    for a, b in ((x, ox), (y, oy)):
        for u, v in zip(a, b):
            dev = u - u.mean()
            assert float((u - v).norm()) <= tol * float(dev.norm()) + 8 * G.EPS64 * float(u.norm())


def test_a_value_that_is_not_finite():
    n = 64
    x = torch.randn((2, n, n, n), dtype=torch.float64, device="cuda")
    y = torch.randn_like(x)
    x[0, 3, 4, 5] = float("inf")
    ox, oy = torch.empty_like(x), torch.empty_like(y)
    cfg = P.make_config(n, 0.5 * n, "chaotic2", (1.0, 4.0), 0.01, mpl=1.0)
    P.pycool_linear_evolve(cfg, 1.0, -1.0, x, y, 0, ox, oy)
    assert bool(torch.isnan(ox[0]).all())
