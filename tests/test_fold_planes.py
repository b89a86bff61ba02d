"""Opposite w-planes folded into one transform (symmetric w range) against every plane
by itself, through the unfused path (cuFFT and the plane sum) on the same gridding: odd
and even plane counts, one word, two words and byte flags of tiles, rows of tiles hit on
one side only, a crop, the Hermitian mirror, and a range that is not symmetric.

Bound, before the first run: both paths transform the same planes in FP32 and were held
to 2e-6 of the peak of each other before folding (tests/test_fft_fused.py measures 2 to
6e-7); the fold adds one rounding per cell, so the same 2e-6 on the tapered image."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile,n_w,image_n,mirror,w_range", [
    (256, 32, 1, None, False, (-50.0, 50.0)),
    (256, 8, 2, 160, False, (-50.0, 50.0)),
    (512, 64, 5, None, False, (-50.0, 50.0)),
    (512, 16, 16, 384, False, (-50.0, 50.0)),
    (1024, 8, 7, 770, False, (-50.0, 50.0)),     # 128 tiles a side: two words
    (2048, 8, 4, 1026, False, (-50.0, 50.0)),    # 256: byte flags
    (2048, 64, 9, None, True, None),             # the mirror's range is symmetric
    (4096, 64, 3, 2050, False, (-50.0, 50.0)),
    (8192, 64, 4, 4094, False, (-50.0, 50.0)),
    (512, 32, 6, None, False, (-50.0, 60.0)),    # not symmetric
])
def test_against_unfused(n, tile, n_w, image_n, mirror, w_range):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(n + n_w)
    fov, n_vis = 0.06, 20000
    # a track on one side, a core, cells at the first and last rows, w of both signs
    x = rng.normal(size=(n_vis, 2)) * 12.0 + n / 2
    x[:8000] = n / 2 + (n / 2 - 12.0) * rng.uniform(0.2, 1.0, (8000, 1)) * \
        np.array([[0.8, 0.59]]) + rng.uniform(-2, 2, (8000, 2))
    x[8000:8600, 1] = rng.choice([3.0, n - 5.0, tile, n / 2, n / 2 + tile], 600)
    uvw = np.empty((n_vis, 3))
    uvw[:, :2] = (x - n / 2) / fov
    uvw[:, 2] = rng.uniform(-50.0, 50.0, n_vis) * rng.choice([0.05, 1.0], n_vis)
    vis = (rng.normal(size=n_vis) + 1j * rng.normal(size=n_vis)).astype(np.complex64)
    im = P.Imager(n, n_w, fov, support=7, tile=tile, max_vis=n_vis, device=dev, image_n=image_n,
                  w_range=w_range, hermitian_mirror=mirror)
    im.bin(torch.from_numpy(uvw).to(dev), torch.from_numpy(vis).to(dev))
    im.grid()
    fused = im.fft_wcorrect(sparse=True).cpu().numpy().astype(np.float64)
    dense = im.fft_wcorrect(sparse=False).cpu().numpy().astype(np.float64)
    im.fft(+1)
    ref = im.wcorrect().cpu().numpy().astype(np.float64)
    m = image_n or n
    c = oracle.taper_row(oracle.Params(n=n, n_w=n_w, fov=fov, kernel=oracle.KB, support=7, tile=tile))
    c = (c / c[n // 2])[(n - m) // 2:(n + m) // 2]
    tt = np.outer(c, c)
    peak = np.abs(ref * tt).max()
    assert np.abs((fused - ref) * tt).max() <= 2e-6 * peak
    assert np.abs((dense - ref) * tt).max() <= 2e-6 * peak
