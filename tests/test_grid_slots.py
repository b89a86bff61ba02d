"""Dense subtiles of the plain gridding kernel: their groups add up in slots, and the
slots go to the planes in FP64.

Identical records are the worst case of an FP32 sum: every partial sum is the same, so
the adds round the same way.  2^18 of them on one corner are 512 groups of 512, in chunks
of 64.  A cell's sum then passes at most 32 register adds (the narrowest warp, two
streams of a chunk), 8 adds of a warp's streams, 8 of a group's warps, 32 of a slot's
groups, and two more to the planes: 82 roundings of at most 2^-24 of the sum.  (The sums
of 512 groups one after the other at the planes drift by about 150.)  The compensated
kernel forms the same products and its sum is off by at most 2: bound 84 x 2^-24.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FOV = 0.1
BOUND = 84 * 2.0 ** -24


def corner(n, at, n_vis, dev):
    uvw = torch.empty((n_vis, 3), dtype=torch.float64, device=dev)
    uvw[:, 0], uvw[:, 1], uvw[:, 2] = (at[0] - n / 2) / FOV, (at[1] - n / 2) / FOV, 0.25
    vis = torch.full((n_vis,), 0.7310586 + 0.2689414j, dtype=torch.complex64, device=dev)
    return uvw, vis


def imager(P, n, n_w, W, max_vis, precision, dev):
    return P.Imager(n, n_w, FOV, support=W, tile=32, max_vis=max_vis, device=dev,
                    w_range=(-1.0, 1.0), precision=precision)


@pytest.mark.parametrize("W,at", [(4, (101.3, 90.6)), (7, (100.2, 131.7)), (9, (111.9, 127.4)),
                                  (12, (60.1, 60.8))])
def test_identical_records(W, at):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    dev = torch.device("cuda", 0)
    n, n_vis = 256, 1 << 18
    uvw, vis = corner(n, at, n_vis, dev)
    planes = {}
    for precision in ("compensated", "fp32"):
        im = imager(P, n, 2, W, n_vis, precision, dev)
        im.bin(uvw, vis)
        im.grid()
        planes[precision] = im.planes.clone()
    ref = planes["compensated"]
    peak = torch.view_as_real(ref).abs()
    assert (torch.view_as_real(planes["fp32"] - ref).abs() <= BOUND * peak).all()
    # the slots start anew with every call, and what they hold is added once
    im.grid()
    assert (torch.view_as_real(im.planes - ref).abs() <= BOUND * peak).all()
    P.rick.rick_grid_accumulate(im.plan, im.ws.data_ptr(), im.planes.data_ptr(), im._stream())
    assert (torch.view_as_real(im.planes - 2 * ref).abs() <= 2 * (BOUND + 2.0 ** -24) * peak).all()


def test_more_than_the_slots():
    """2100 subtiles of 8200 records want more slots than there are; the others add to the
    planes.  A cell of up to m records is a sum of at most m terms in FP32, in any
    grouping, and both kernels form the same products: |a - b| <= 2 (m + 4) 2^-24 S."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_07321_gb300 as P
    dev = torch.device("cuda", 0)
    n, W, each = 1024, 4, 8200
    g = torch.Generator(device=dev)
    g.manual_seed(5)
    s = torch.arange(2100, device=dev).repeat_interleave(each)
    x = torch.rand((len(s), 2), generator=g, device=dev, dtype=torch.float64) * 14.0 + 1.5
    uvw = torch.empty((len(s), 3), dtype=torch.float64, device=dev)
    uvw[:, 0] = ((s % 60) * 16 + 16 + x[:, 0] - n / 2) / FOV
    uvw[:, 1] = ((s // 60) * 16 + 16 + x[:, 1] - n / 2) / FOV
    uvw[:, 2] = 0.0
    vis = torch.randn(len(s), generator=g, device=dev, dtype=torch.complex64)
    planes = {}
    for name, precision, v in (("ref", "compensated", vis), ("sum", "compensated", vis.abs() + 0j),
                               ("got", "fp32", vis)):
        im = imager(P, n, 1, W, len(s), precision, dev)
        im.bin(uvw, v)
        im.grid()
        planes[name] = im.planes.clone()
        del im
    # records a cell can have: every one of the four subtiles around
    bound = 2.0 * (4 * each + 4) * 2.0 ** -24 * planes["sum"].abs()
    assert ((planes["got"] - planes["ref"]).abs() <= bound).all()
    rms = (planes["got"] - planes["ref"]).abs().pow(2).mean().sqrt()
    assert float(rms) <= 1e-5 * float(planes["ref"].abs().pow(2).mean().sqrt())
