"""The plain gridding kernel (one warp per 16 x 16-corner subtile) against the
compensated kernel (one CTA per uv-tile), cell by cell.

The planes do not depend on the tile side, so one compensated plan (tile 32) is
the reference of every tile.  Corners lie anywhere on the grid, on the edges of
tiles and subtiles, beyond the grid, and a thousand in one cell (a subtile of
several work items); single records and an empty set are taken too.

Bound, before the first run: both kernels form a record's contribution with the
same products (four roundings), and a cell that m records reach is a sum of at
most m terms in FP32, in any grouping: |a - b| <= 2 (m + 4) 2^-24 S, with S the
sum of the terms' magnitudes (the planes of |v|; the weights are positive).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, NW, FOV = 256, 2, 0.1


def points(rng, n_vis, W):
    x = rng.uniform(-2.0, N + 2.0, (n_vis, 2))
    k = n_vis // 4
    x[:k] = 16 * rng.integers(0, N // 16 + 1, (k, 2)) + rng.integers(-W, W + 1, (k, 2))
    x[k:2 * k] = rng.uniform(70.0, 71.0, (k, 2))
    uvw = np.empty((n_vis, 3))
    uvw[:, :2] = (x - N / 2) / FOV
    uvw[:, 2] = rng.uniform(-1.0, 1.0, n_vis)
    v = rng.normal(size=(n_vis, 2)).astype(np.float32)
    return uvw, v[:, 0] + 1j * v[:, 1]


def planes_of(P, kw, uvw, vis):
    dev = torch.device("cuda", 0)
    im = P.Imager(N, NW, FOV, w_range=(-1.0, 1.0), max_vis=max(len(vis), 1), device=dev, **kw)
    im.bin(torch.from_numpy(uvw).to(dev), torch.from_numpy(vis.astype(np.complex64)).to(dev))
    im.planes.fill_(float("nan"))  # every cell has to be written
    im.grid()
    b = im.binned() if len(vis) else None
    return im.planes.cpu().numpy(), b


@pytest.mark.parametrize("n_vis", [0, 1, 33, 5000])
@pytest.mark.parametrize("W,tile,kernel", [
    (1, 8, "kb"), (4, 8, "kb"), (8, 8, "kb"), (7, 16, "kb"), (16, 16, "kb"), (5, 32, "gauss"),
    (10, 32, "kb"), (7, 64, "kb"), (9, 64, "kb"), (16, 64, "kb"), (12, 128, "kb"), (16, 128, "kb")])
def test_planes(W, tile, kernel, n_vis):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    uvw, vis = points(np.random.default_rng(100 * W + tile + n_vis), n_vis, W)
    kw = dict(kernel=kernel, support=W)
    ref_kw = dict(kw, tile=32, precision="compensated")
    got, b = planes_of(P, dict(kw, tile=tile), uvw, vis)
    ref, _ = planes_of(P, ref_kw, uvw, vis)
    mag, _ = planes_of(P, ref_kw, uvw, np.abs(vis))
    m = np.zeros((NW, N, N))
    if n_vis:
        ax, ay = (b["rec_cell"] & 0xFFFF).astype(int), (b["rec_cell"] >> 16).astype(int)
        per_plane = 4 * (N // tile) ** 2
        k = np.searchsorted(b["offsets"][::per_plane], np.arange(len(ax)), side="right") - 1
        for jy in range(W):
            for jx in range(W):
                np.add.at(m, (k, ay + jy, ax + jx), 1)
    assert np.isfinite(got).all()
    bound = 2.0 * (m + 4) * 2.0 ** -24 * np.abs(mag)
    assert (np.abs(got - ref) <= np.sqrt(2.0) * bound).all()
