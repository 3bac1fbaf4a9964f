"""The plain staging's work plan (host logic, no GPU), which the kernel trusts: for
sides up to 1024, one and two fields, one and two halo planes,
  - the tiles (w x h sites, at most 512, at most 256 halo cells) partition the plane;
  - every (tile, z) pair is in exactly one unit and every unit inside the lattice;
  - at most 64 units a block and min(sms, 208) blocks, every block with a unit;
  - the kernel's index arithmetic stays in bounds: a tile's threads and halo cells reach
    each site and each cell of the halo ring exactly once."""
import numpy as np
import pytest

P = pytest.importorskip("paper_1201_5029_gb300")

L2 = 126 << 20
SIDES = list(range(1, 72)) + [79, 96, 97, 100, 127, 128, 129, 150, 160, 191, 203, 250, 256, 257,
                              333, 511, 512, 513, 777, 1023, 1024]


@pytest.mark.parametrize("stencil", [P.STENCIL_7PT, P.STENCIL_4TH])
@pytest.mark.parametrize("nf", [1, 2])
def test_plan_covers_lattice_once(nf, stencil):
    H = 2 if stencil == P.STENCIL_4TH else 1
    for n in SIDES:
        if n < 4 and H == 2:
            with pytest.raises(P.PycoolError):
                P.pycool_debug_plain_plan(n, nf, 152, L2, stencil)
            continue
        for sms in (152, 148) if n <= 160 else (152,):
            g, units, uoff = P.pycool_debug_plain_plan(n, nf, sms, L2, stencil)
            assert g["n"] == n and g["vx"] == 0 and g["halo"] == H
            assert 1 <= g["G"] <= min(sms, 208)
            assert uoff[0] == 0 and uoff[-1] == len(units) == g["nunits"]
            counts = np.diff(uoff)
            assert (counts >= 1).all() and (counts <= 64).all()
            x0, w = units[:, 0] & 0xffff, units[:, 0] >> 16
            y0, h = units[:, 1] & 0xffff, units[:, 1] >> 16
            z0, planes = units[:, 2], units[:, 3] - 2 * H
            assert (w >= 1).all() and (h >= 1).all() and (w * h <= 512).all()
            assert (2 * H * (w + 2 * H + h) <= 256).all()
            assert (x0 + w <= n).all() and (y0 + h <= n).all()
            assert (planes >= 1).all() and (z0 >= 0).all() and (z0 + planes <= n).all()
            tiles, tile = np.unique(np.stack([x0, y0, w, h]), axis=1, return_inverse=True)
            plane = np.zeros((n, n), dtype=np.int32)
            for tx, ty, tw, th in tiles.T:
                plane[ty:ty + th, tx:tx + tw] += 1
            assert (plane == 1).all()
            seen = np.zeros((tiles.shape[1], n + 1), dtype=np.int32)
            np.add.at(seen, (tile.ravel(), z0), 1)
            np.add.at(seen, (tile.ravel(), z0 + planes), -1)
            assert (np.cumsum(seen, axis=1)[:, :n] == 1).all()


@pytest.mark.parametrize("H", [1, 2])
def test_cells_of_a_tile(H):
    """The cells that plain_cells (persist_plain.cuh) gives the threads of a tile."""
    stencil = P.STENCIL_4TH if H == 2 else P.STENCIL_7PT
    shapes = set()
    for n in SIDES:
        if n >= 4 or H == 1:
            _, units, _ = P.pycool_debug_plain_plan(n, 1, 152, L2, stencil)
            shapes |= {(int(a) >> 16, int(b) >> 16) for a, b in units[:, :2]}
    for w, h in shapes:
        rs = w + 2 * H
        cells = np.zeros(((h + 2 * H) * rs,), dtype=np.int32)
        for t in range(512):
            if t < w * h:
                cells[(t // w + H) * rs + t % w + H] += 1
            if t < 2 * H * (rs + h):
                if t < 2 * H * rs:
                    r, col = divmod(t, rs)
                    row = r if r < H else h + r
                else:
                    t2 = t - 2 * H * rs
                    k = t2 % (2 * H)
                    row, col = t2 // (2 * H) + H, k if k < H else w + k
                cells[row * rs + col] += 1
        assert (cells == 1).all()
        assert cells.size <= 768 and 2 * H * (rs + h) <= 256
