"""The serving loop's white-noise initial fields at sides around the kernel's
blocks of four normals and its 16-byte stores (odd sides: the second field starts
unaligned), against the numpy generator.  A request of no steps reports the
fields' means and variances.  Bounds: a normal is within 7e-15 of numpy's (its
own argument rounding, 5e-15, included), in the split form one float32 rounding
of at most 6.7 noise apart."""
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1201_5029_gb300")
from paper_1201_5029_gb300 import inputs as I  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "split_fp32"])
@pytest.mark.parametrize("n", [2, 3, 5, 16, 33, 64])
def test_means_and_variances(n, precision):
    w = I.workload("preheat32")
    noise, seed = 0.125, 4000 + n
    cfg = P.make_config(n, w["L"], w["model"], w["params"], w["dt"], order=2,
                        precision=precision, mpl=w["mpl"])
    srv = P.pycool_server_create(1 << 30, 2)
    try:
        t = P.pycool_server_submit(srv, cfg, P.make_ic(w["background"], w["momentum"], noise), seed, 0)
        status, e = P.pycool_server_wait(srv, t, 60.0)
    finally:
        P.pycool_server_destroy(srv)
    assert status == P.OK
    phi, _ = I.philox_white_ics(n, w["background"], w["momentum"], noise, seed)
    tol = 7e-15 * noise if precision == "fp64" else 6.7 * noise * 2.0 ** -24
    for f in range(len(w["background"])):
        scale = abs(w["background"][f]) + noise
        assert abs(e.mean[f] - phi[f].mean()) < tol + 4e-15 * scale
        # d(variance) <= 2 rms |dz| + the float64 sums
        assert abs(e.variance[f] - phi[f].var()) < 4 * noise * (tol + 4e-15 * scale)
