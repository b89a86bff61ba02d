"""chi2 and its residual kernel at their limits: sums that overflow, NaN, images that are
parameters of a module, and more visibilities than the blocks take in one go."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def setup(n_vis):
    import paper_2411_07321_gb300 as P
    from paper_2411_07321_gb300 import autograd as A
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(n_vis)
    im = P.Imager(256, 2, 0.05, support=7, tile=32, max_vis=n_vis, device=dev,
                  w_range=(-1.0, 1.0))
    uvw = (torch.rand((n_vis, 3), generator=g, device=dev, dtype=torch.float64) * 2.0 - 1.0) * \
        torch.tensor([2000.0, 2000.0, 1.0], device=dev, dtype=torch.float64)
    vis = torch.randn(n_vis, generator=g, device=dev, dtype=torch.complex64)
    w = torch.rand(n_vis, generator=g, device=dev) + 0.5
    im.bin(uvw, vis, w)
    return im, A, vis, w


@pytest.mark.parametrize("n_vis,at,value", [
    (5000, 4321, 3e19),              # a term over the largest float
    (5000, slice(None), 1e19),       # terms of 1e38, four of them a thread
    (5000, 7, float("inf")), (5000, 7, float("nan"))])
def test_not_finite(n_vis, at, value):
    """inf and NaN as the torch sum has them."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    im, A, vis, w = setup(n_vis)
    vis = torch.view_as_complex(torch.view_as_real(vis).index_put(
        (torch.arange(n_vis, device=vis.device)[at].reshape(-1), torch.tensor(0, device=vis.device)),
        torch.tensor(value, device=vis.device)))
    x = torch.zeros((256, 256), device=vis.device, requires_grad=True)
    loss = A.chi2(x, im, vis, w)
    assert type(loss.grad_fn).__name__ == "Chi2FnBackward"
    r = vis - A.predict(x, im)
    want = (w * (r.real ** 2 + r.imag ** 2)).sum().detach()
    assert not math.isfinite(float(want))
    assert torch.equal(torch.isnan(loss.detach()), torch.isnan(want))
    assert math.isnan(float(want)) or float(loss.detach()) == float(want)


def test_parameter():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    im, A, vis, w = setup(3000)
    g = torch.Generator(device=vis.device)
    g.manual_seed(1)
    x = torch.randn((256, 256), generator=g, device=vis.device)
    grads = []
    for image in (torch.nn.Parameter(x.clone()), x.clone().requires_grad_()):
        loss = A.chi2(image, im, vis, w)
        assert type(loss.grad_fn).__name__ == "Chi2FnBackward"
        loss.backward()
        grads.append(image.grad)
    assert float((grads[0] - grads[1]).abs().max()) <= 1e-5 * float(grads[1].abs().max())


@pytest.mark.parametrize("n_vis", [(1 << 20) + 1, (1 << 21) + 12345])
def test_more_than_a_round(n_vis):
    """Against an FP64 sum of the terms of the same FP32 residuals: three roundings of a
    term and one of the result, 4 x 2^-24, and the pairs' own error, below 2^-40."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    im, A, vis, w = setup(4096)
    g = torch.Generator(device=vis.device)
    g.manual_seed(2)
    vis = torch.randn(n_vis, generator=g, device=vis.device, dtype=torch.complex64)
    model = torch.randn(n_vis, generator=g, device=vis.device, dtype=torch.complex64)
    w = torch.rand(n_vis, generator=g, device=vis.device)
    r = vis - model
    want = float((w.double() * torch.view_as_real(r).double().square().sum(-1)).sum())
    got = im.chi2_residuals(vis, w, model)
    assert torch.equal(model, r)
    assert abs(float(got) - want) <= (4 * 2.0 ** -24 + 2.0 ** -40) * want
