"""How exact the library's own transforms are (sides 64, 128, 256), there and back
through the linearised evolution of no steps (forward, the identity on every mode,
inverse; two fields, so that a batch has more than one array), and forward through the
spectrum at the largest amplitudes that a line's scale has to hold.

Bounds, norm-wise: a pass rounds each value once (2^-53 of it) and its block-scaled
arithmetic is some units of 2^-58 .. 2^-54 of the line's largest value, together at most
2 2^-53 a pass: 12 2^-53 for the six passes, beside the roundings of the means taken out
and added again.  Losing four bits of a line's scale would show."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")
import gpu_helpers as G  # noqa: E402

LAST = float(np.nextafter(2.0, 0.0))


def _field(kind, n, seed):
    if kind == "noise":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        return torch.randn((n, n, n), dtype=torch.float64, device="cuda", generator=g)
    i = torch.arange(n, device="cuda")
    s = {"nyquist": 1 - 2 * (i % 2), "square": 1 - 2 * (i // (n // 2)),
         "step4": 1 - 2 * ((i // 4) % 2)}[kind].double()
    return LAST * (s[:, None, None] * s[None, :, None] * s[None, None, :])


@pytest.mark.parametrize("n", [64, 128, 256])
@pytest.mark.parametrize("kind", ["noise", "nyquist", "square", "step4"])
def test_there_and_back(n, kind):
    x = torch.stack([_field(kind, n, 1), _field(kind, n, 2)])
    y = torch.stack([_field(kind, n, 3), -_field(kind, n, 4)])
    ox, oy = torch.empty_like(x), torch.empty_like(y)
    cfg = P.make_config(n, 0.5 * n, "chaotic2", (1.0, 4.0), 0.01, mpl=1.0)
    P.pycool_linear_evolve(cfg, 1.0, -1.0, x, y, 0, ox, oy)
    for a, b in ((x, ox), (y, oy)):
        for u, v in zip(a, b):
            assert float((u - v).norm()) <= (12 + 4) * G.EPS64 * float(u.norm())


@pytest.mark.parametrize("n", [64, 128, 256])
@pytest.mark.parametrize("value", [LAST, 2.0 - 2.0 ** -20])
def test_constant(n, value):
    sim = P.Simulation(P.make_config(n, 0.5 * n, "free", (1.0,), 0.01, mpl=np.inf))
    f = np.full((1, n, n, n), value)
    sim.set_initial(f, -f)
    for which in (0, 1):
        p, _ = sim.spectrum(which, 0)
        assert abs(p[0] / value ** 2 - 1) <= 2 * 6 * G.EPS64 + 4 * G.EPS64   # three passes, squared
        assert (p[1:] <= (6 * G.EPS64 * value) ** 2 * n ** 3).all()
    sim.close()
