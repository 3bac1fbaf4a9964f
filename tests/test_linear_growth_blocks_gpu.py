"""The growth functions' two block shapes: counts of k_eff^2 values at the ends of
the range that takes the wide blocks, over several table chunks.  A value's
arithmetic does not depend on its block, so each equals, bit for bit, the same
value computed among a few."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("model", ["chaotic2", "oscillon"])
@pytest.mark.parametrize("edge,off", [(64, 0), (64, 1), (320, -161), (320, -160), (320, -159)])
def test_any_count_gives_the_same_values(model, edge, off):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = sms * edge + off
    one = model == "oscillon"
    cfg = P.make_config(32, 25.6, model, (0.5, -1.0, 1.0 / 3.0) if one else (1.0, 50.0), 0.02,
                        order=4, mpl=100.0)
    f0, p0 = ([0.8], [0.1]) if one else ([1.0, 0.2], [-0.3, 0.1])
    k2 = np.linspace(0.0, 12.0, count)
    T, bg = P.pycool_linear_growth(cfg, 1.0, -1.0, f0, p0, k2, 45)
    pick = np.unique(np.r_[0:3, np.linspace(0, count - 1, 60).astype(int), count - 3:count])
    Ts, bgs = P.pycool_linear_growth(cfg, 1.0, -1.0, f0, p0, k2[pick], 45)
    assert np.isfinite(T).all() and np.array_equal(T[pick], Ts)
    assert bg[0] == bgs[0] and bg[1] == bgs[1]
