"""chi2 with the residuals formed and binned by the library, against the same sum as
torch operations on the model visibilities.

Bounds, before the first run: a term w |r|^2 carries at most four roundings and
torch's pairwise FP32 sum of N terms ceil(log2 N), so the losses differ by at most
(log2 N + 5) 2^-24; the gradients are the images of the same record values, whose
order of summation is free: the parity bar, 1e-5 of the largest pixel.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_vis,mirror,deterministic", [
    (1, False, False), (1023, False, False), (1025, False, False), (40001, False, False),
    (3000, True, False), (5000, False, True)])
def test_against_torch(n_vis, mirror, deterministic):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    from paper_2411_07321_gb300 import autograd as A
    rng = np.random.default_rng(n_vis)
    dev = torch.device("cuda", 0)
    n, fov = 256, 0.05
    im = P.Imager(n, 4, fov, support=7, tile=32, max_vis=n_vis, device=dev, image_n=160,
                  w_range=(-100.0, 100.0), hermitian_mirror=mirror, deterministic=deterministic)
    uvw = torch.from_numpy(rng.uniform(-1.0, 1.0, (n_vis, 3)) * [2000.0, 2000.0, 100.0]).to(dev)
    vis = torch.view_as_complex(torch.from_numpy(rng.normal(size=(n_vis, 2)).astype(np.float32))).to(dev)
    w = torch.from_numpy(rng.uniform(0.5, 1.5, n_vis).astype(np.float32)).to(dev)
    x = torch.from_numpy(rng.normal(size=(160, 160)).astype(np.float32)).to(dev).requires_grad_()
    im.bin(uvw, vis, w)
    before = vis.clone(), w.clone()
    loss = A.chi2(x, im, vis, w)
    (g,) = torch.autograd.grad(3.0 * loss, x)
    stats = im.stats()
    r = vis - A.predict(x, im)
    ref = (w * (r.real ** 2 + r.imag ** 2)).sum()
    (gref,) = torch.autograd.grad(3.0 * ref, x)
    assert type(loss.grad_fn).__name__ == "Chi2FnBackward"
    assert loss.dtype == torch.float32 and loss.shape == ()
    bound = (math.ceil(math.log2(n_vis + 1)) + 5) * 2.0 ** -24
    assert abs(float(loss) - float(ref)) <= bound * float(ref)
    assert float((g - gref).abs().max()) <= 1e-5 * float(gref.abs().max())
    assert im.stats() == stats
    assert torch.equal(vis, before[0]) and torch.equal(w, before[1])


def test_other_gradients():
    """vis_obs or weight asking for a gradient, other dtypes and conjugate views take
    the torch operations."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    from paper_2411_07321_gb300 import autograd as A
    dev = torch.device("cuda", 0)
    im = P.Imager(256, 2, 0.05, support=7, tile=32, max_vis=100, device=dev)
    uvw = torch.rand((100, 3), dtype=torch.float64, device=dev) * 100.0
    vis = torch.randn(100, dtype=torch.complex64, device=dev)
    w = torch.rand(100, device=dev)
    im.bin(uvw, vis, w)
    x = torch.zeros((256, 256), device=dev)
    v = vis.clone().requires_grad_()
    (gv,) = torch.autograd.grad(A.chi2(x, im, v, w), v)
    assert torch.allclose(gv, 2.0 * w * vis, rtol=1e-5, atol=1e-6)
    ww = w.clone().requires_grad_()
    (gw,) = torch.autograd.grad(A.chi2(x, im, vis, ww), ww)
    assert torch.allclose(gw, vis.abs() ** 2, rtol=1e-5, atol=1e-6)
    want = float((w * vis.abs() ** 2).sum())
    for a, b in ((vis.conj(), w), (vis, w.double()), (vis.to(torch.complex128), w)):
        assert abs(float(A.chi2(x, im, a, b)) - want) <= 1e-5 * want
