"""The one-CTA pass between the key pass and the scatter (at most 16384 sub-bins)
against the general launches, on either side of the line: offsets, work lists (by the
planes they give) and the stats.  Corners are whole numbers and must agree exactly; the
planes of the compensated kernel, which goes by the tile lists, are within 2e-6 of the
plain kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_vis", [0, 1, 6000])
@pytest.mark.parametrize("tile,n_w", [(16, 16), (16, 17), (64, 1), (128, 50), (128, 51), (8, 4),
                                      (8, 5)])
def test_either_side(tile, n_w, n_vis):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    dev = torch.device("cuda", 0)
    n, fov, W = 256, 0.1, 7
    rng = np.random.default_rng(tile + n_w)
    uvw = (rng.uniform(-1.05, 1.05, (n_vis, 3)) * [n / 2 / fov, n / 2 / fov, 1.0])
    vis = (rng.normal(size=n_vis) + 1j * rng.normal(size=n_vis)).astype(np.complex64)
    t_uvw, t_vis = torch.from_numpy(uvw).to(dev), torch.from_numpy(vis).to(dev)
    planes = {}
    for precision in ("fp32", "compensated"):
        if precision == "compensated" and tile > 64:
            continue
        im = P.Imager(n, n_w, fov, support=W, tile=tile, max_vis=max(n_vis, 1), device=dev,
                      precision=precision, w_range=(-1.0, 1.0))
        im.bin(t_uvw, t_vis)
        im.grid()
        planes[precision] = im.planes.cpu().numpy()
        st, b = im.stats(), im.binned()
        off = b["offsets"].astype(np.int64)
        nt = n // tile
        assert len(off) == 4 * n_w * nt * nt + 1
        assert off[0] == 0 and off[-1] == st["n_binned"] and (np.diff(off) >= 0).all()
        assert st["n_binned"] + st["n_dropped_uv"] + st["n_dropped_w"] == n_vis
        assert st["sum_weight"] == st["n_binned"]
        ax, ay = (b["rec_cell"] & 0xFFFF).astype(int), (b["rec_cell"] >> 16).astype(int)
        w = uvw[b["perm"], 2]
        k = np.zeros(len(w), int)
        for j in range(1, n_w):
            k += w >= j * (2.0 / n_w) - 1.0
        ex, ey = ax % tile > tile - W, ay % tile > tile - W
        cls = np.where(ex, np.where(ey, 2, 1), np.where(ey, 3, 0))
        key = ((k * nt + ay // tile) * nt + ax // tile) * 4 + cls
        assert (key == np.searchsorted(off, np.arange(len(key)), side="right") - 1).all()
        assert len(np.unique(b["perm"])) == st["n_binned"]
    if len(planes) == 2 and n_vis:
        a, c = planes["fp32"], planes["compensated"]
        assert np.abs(a - c).max() <= 2e-6 * np.abs(c).max()
