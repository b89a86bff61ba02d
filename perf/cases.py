"""Performance cases of the imaging library: what its users have it compute.

Each case is one call (or one gradient step) through the public Python API on
synthetic observations of the shape the library is built for: baselines of a
station array with a dense core, tracked over eight hours, in rows of frequency
channels -- so consecutive visibilities fall on neighbouring grid cells and the
uv coverage piles up at the centre.  The observations are made on the GPU from
the seed alone.

``op`` says which call a case stands for:

  image     Imager.image -- bin, grid, transform of a resident visibility set
  request   Imager.image_from_host -- what one serving request does
  weighted  Imager.image_weighted -- Briggs-robust weighting and image
  rows      Imager.bin_channels + image_from_binned -- measurement-set layout
  streamed  Imager.image_streamed -- a set in pinned host memory, in chunks
  chi2      autograd.chi2 and its gradient in the image (degrid, then grid)
  vis_grad  autograd.grid_image and its gradient in the visibilities
  predict   Imager.predict -- model visibilities of a sky image

Images of an unpadded mesh carry the transform's FP32 rounding times the taper
correction in their corners, some thousandfold, and that rounding changes from
run to run with the order of the sums.  Most cases keep a crop of the mesh, as
one does who wants the corners; ``image_n`` 0 is the whole mesh.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_07321_gb300 as P
from paper_2411_07321_gb300 import autograd as A

DEG = math.pi / 180.0
NU0, DNU = 144.6e6, 12.207e3          # Hz: first channel, channel width
N_SRC = 12

BASE = {"op": "image", "n_vis": 65536, "n_chan": 1, "n_corr": 1, "n_ant": 60, "n": 256, "n_w": 8,
        "fov_deg": 2.0, "uv_fill": 0.5, "w_max": 300.0, "kernel": "kb", "support": 7, "tile": 64,
        "image_n": 0, "weights": True, "precision": "fp32", "deterministic": False,
        "mirror": False, "given_w": False, "chunk": 0, "robust": 0.0}


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # A small array on a small padded mesh with the Gaussian kernel: a call of a
        # few tens of microseconds of work, where the launches count.
        _case("image_small_256", n_vis=65536, n_ant=32, n=256, n_w=8, fov_deg=2.0, uv_fill=0.55,
              w_max=300.0, kernel="gauss", support=7, tile=32, weights=False, image_n=160),
        # The smallest request of a serving mix: host buffers in, host image out.
        _case("request_10k_512", op="request", n_vis=10007, n=512, n_w=4, fov_deg=2.0,
              uv_fill=0.7, w_max=500.0, image_n=384),
        # A middling serving job, nothing a power of two but the mesh.
        _case("image_1m_1024", n_vis=1000003, n_chan=4, n=1024, n_w=11, fov_deg=4.0, uv_fill=0.6,
              w_max=1500.0, image_n=770),
        # An 8 h LOFAR-like observation.
        _case("image_lofar_4096", n_vis=50000000, n_chan=16, n=4096, n_w=16, fov_deg=8.0,
              uv_fill=0.82, w_max=5000.0),
        # The largest single-GPU observation: 64 channels, a fine mesh, W = 9.
        _case("image_large_8192", n_vis=200000000, n_chan=64, n=8192, n_w=32, fov_deg=8.0,
              uv_fill=0.41, w_max=5000.0, support=9, image_n=7168),
        # One step of a chi^2 fit of the sky: model visibilities, then the gradient.
        _case("chi2_step_2048", op="chi2", n_vis=10000000, n_chan=4, n=2048, n_w=16, fov_deg=4.0,
              uv_fill=0.41, w_max=2500.0, image_n=1536),
        # An image differentiated in its visibilities (calibration), even W.
        _case("vis_grad_1024", op="vis_grad", n_vis=3000017, n_chan=8, n=1024, n_w=13,
              fov_deg=3.0, uv_fill=0.85, w_max=2000.0, support=8, image_n=768),
        # A robust-weighted image of single-channel data.
        _case("briggs_2048", op="weighted", n_vis=4000037, n=2048, n_w=16, fov_deg=4.0,
              uv_fill=0.7, w_max=2500.0, robust=-0.5),
        # Measurement-set rows: 16 channels of two correlations.
        _case("rows_2corr_4096", op="rows", n_vis=10000000, n_chan=16, n_corr=2, n=4096, n_w=16,
              fov_deg=8.0, uv_fill=0.82, w_max=5000.0),
        # A mesh padded about twofold with a ragged crop, which keeps the corners exact.
        _case("padded_4096", n_vis=6000011, n_chan=64, n=4096, n_w=24, fov_deg=8.0, uv_fill=0.4,
              w_max=4000.0, support=9, image_n=2050),
        # Out-of-core imaging: rows of channels in pinned host memory, in chunks.
        _case("streamed_4096", op="streamed", n_vis=32000000, n_chan=16, n=4096, n_w=16,
              fov_deg=8.0, uv_fill=0.82, w_max=5000.0, chunk=1 << 23, given_w=True),
        # The bitwise repeatable mode.
        _case("repeatable_2048", n_vis=2000003, n_chan=4, n=2048, n_w=9, fov_deg=4.0,
              uv_fill=0.6, w_max=2000.0, support=6, image_n=1792, deterministic=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["image", "image", "image", "request", "weighted", "rows", "streamed", "chi2",
                     "vis_grad", "predict"])
    n = rng.choice([256, 512, 1024, 2048, 2048, 4096, 4096, 8192])
    n_w = log_int(1, 32)
    n_vis = log_int(10000, 3000000 if op in ("request",) else 30000000)
    if n == 256:
        n_vis = min(n_vis, 4000000)
    n_chan = rng.choice([1, 1, 3, 4, 16, 24, 64])
    n_corr = 1
    if op in ("rows", "streamed"):
        n_corr = rng.choice([1, 2, 2, 4])
        n_chan = max(n_chan, 3)
        n_vis = max(n_vis // (n_chan * n_corr), 10) * n_chan
    kernel = rng.choice(["kb", "kb", "kb", "gauss"])
    support = rng.randint(4, 6) if kernel == "gauss" else rng.choice([4, 5, 6, 7, 7, 8, 9])
    image_n = 0
    if support > 5 or rng.random() < 0.5:  # a padded mesh; the wider kernels need it
        image_n = 2 * rng.randint(n // 4, (11 * n) // 32)
        if kernel == "kb" and image_n <= 0.6 * n:
            support = rng.choice([support, 9, 10, 12])
    deterministic = op in ("image", "rows") and rng.random() < 0.15
    precision = "compensated" if (not deterministic and rng.random() < 0.12) else "fp32"
    mirror = op == "image" and not deterministic and rng.random() < 0.15
    tile = rng.choice([32, 64, 64])
    fov = rng.uniform(1.0, 8.0)
    return _case(op=op, n_vis=n_vis, n_chan=n_chan, n_corr=n_corr, n_ant=rng.choice([32, 48, 60]),
                 n=n, n_w=n_w, fov_deg=round(fov, 3), uv_fill=round(rng.uniform(0.3, 0.9), 3),
                 w_max=round(rng.uniform(0.1, 0.5) * 0.35 * n / (fov * DEG), 1), kernel=kernel,
                 support=support, tile=tile, image_n=image_n, weights=rng.random() < 0.75,
                 precision=precision, deterministic=deterministic, mirror=mirror,
                 given_w=op == "streamed" and rng.random() < 0.5,
                 chunk=max(n_chan * n_corr, n_vis // rng.randint(2, 7)) if op == "streamed" else 0,
                 robust=round(rng.uniform(-1.0, 1.0), 2))


# ---------------------------------------------------------------- observations
def _rows(c):
    return -(-c["n_vis"] // c["n_chan"])


def _observation(c, seed, dev):
    """uvw of every row (float64 [rows, 3], wavelengths at the first channel), the
    channels' factors, values complex64 [rows, chan, corr] of a point-source sky
    with noise, and weights float32 of the same shape (or None)."""
    rs = np.random.RandomState(seed % (1 << 31))
    n_ant, rows, nc, nk = c["n_ant"], _rows(c), c["n_chan"], c["n_corr"]
    # half the stations in a 2 km core, the rest log-radial out to 80 km
    core = n_ant // 2
    r = np.where(np.arange(n_ant) < core, 2000.0 * np.sqrt(rs.rand(n_ant)),
                 2000.0 * np.exp(rs.rand(n_ant) * math.log(40.0)))
    t = 2.0 * math.pi * rs.rand(n_ant)
    east, north = r * np.cos(t), r * np.sin(t)
    lat, dec = 52.9 * DEG, 64.0 * DEG
    xyz = np.stack([-math.sin(lat) * north, east, math.cos(lat) * north], 1)
    ia, ib = np.triu_indices(n_ant, 1)
    bl = torch.from_numpy(xyz[ib] - xyz[ia]).to(dev)
    n_bl = bl.shape[0]
    steps = -(-rows // n_bl)
    i = torch.arange(rows, device=dev)
    H = ((i // n_bl + 0.5) / steps - 0.5) * (8.0 * 2.0 * math.pi / 24.0)
    b = bl[i % n_bl]
    sh, ch, sd, cd = torch.sin(H), torch.cos(H), math.sin(dec), math.cos(dec)
    uvw = torch.stack([sh * b[:, 0] + ch * b[:, 1],
                       -sd * ch * b[:, 0] + sd * sh * b[:, 1] + cd * b[:, 2],
                       cd * ch * b[:, 0] - cd * sh * b[:, 1] + sd * b[:, 2]], 1)
    scale = (NU0 + DNU * torch.arange(nc, device=dev, dtype=torch.float64)) / NU0
    top = float(scale[-1])
    uv_max = c["uv_fill"] * 0.5 * c["n"] / (c["fov_deg"] * DEG)
    uvw[:, :2] *= uv_max / (float(uvw[:, :2].abs().max()) * top)
    uvw[:, 2] *= c["w_max"] / (float(uvw[:, 2].abs().max()) * top)
    # the sky: log-uniform fluxes inside the kept field
    kept = (c["image_n"] / c["n"]) if c["image_n"] else 1.0
    half = 0.45 * c["fov_deg"] * DEG * kept
    l = torch.from_numpy(half * (2.0 * rs.rand(N_SRC) - 1.0)).to(dev)
    m = torch.from_numpy(half * (2.0 * rs.rand(N_SRC) - 1.0)).to(dev)
    nn = torch.sqrt(1.0 - l * l - m * m)
    amp = (torch.from_numpy(0.1 * np.exp(rs.rand(N_SRC) * math.log(100.0))).to(dev) / nn).float()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    vis = torch.empty((rows, nc, nk), dtype=torch.complex64, device=dev)
    step = max(1, (1 << 26) // (nc * N_SRC))
    cidx = torch.arange(nc, device=dev, dtype=torch.float32)
    for r0 in range(0, rows, step):
        q = uvw[r0:r0 + step]
        cyc = -(q[:, :1] * l + q[:, 1:2] * m + q[:, 2:] * (nn - 1.0))       # cycles, channel 0
        p0 = ((cyc - torch.round(cyc)) * (2.0 * math.pi)).float()[:, None, :]
        dp = (cyc * (2.0 * math.pi * DNU / NU0)).float()[:, None, :]
        ph = p0 + cidx[None, :, None] * dp
        v = torch.complex((torch.cos(ph) * amp).sum(-1), (torch.sin(ph) * amp).sum(-1))
        vis[r0:r0 + step] = v[:, :, None]
    del ph, v
    vr = torch.view_as_real(vis)
    for r0 in range(0, rows, 1 << 20):
        vr[r0:r0 + (1 << 20)] += 0.007 * torch.randn(vr[r0:r0 + (1 << 20)].shape, generator=g,
                                                     device=dev)
    wt = None
    if c["weights"]:
        wt = 0.5 + torch.rand((rows, nc, nk), generator=g, device=dev)
    return uvw, scale, vis, wt


def _flat(c, uvw, scale, vis, wt):
    """The observation with uvw per visibility, cut to exactly n_vis."""
    nv = c["n_vis"]
    full = (uvw[:, None, :] * scale[None, :, None]).reshape(-1, 3)[:nv].contiguous()
    return full, vis.reshape(-1)[:nv].contiguous(), \
        None if wt is None else wt.reshape(-1)[:nv].contiguous()


def _sky(c, seed, dev):
    """A smooth-free model image: a few hundred point sources on a faint random
    background, zero towards the mesh edges (where the taper correction is large)."""
    m = c["image_n"] or c["n"]
    g = torch.Generator(device=dev)
    g.manual_seed(seed + 77)
    x = 1e-3 * torch.randn((m, m), generator=g, device=dev)
    k = 300
    at = torch.randint(0, m, (2, k), generator=g, device=dev)
    x[at[0], at[1]] += torch.rand(k, generator=g, device=dev) * 2.0
    d = (torch.arange(m, device=dev) - m / 2).abs() * (2.0 / c["n"])
    e = torch.where(d < 0.8, 1.0, 0.0).float()
    return (x * e[:, None] * e[None, :]).contiguous()


def _pin(t):
    return None if t is None else torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _imager(c, max_vis, dev):
    w_range = (-c["w_max"], c["w_max"]) if c["given_w"] else None
    return P.Imager(c["n"], c["n_w"], c["fov_deg"] * DEG, kernel=c["kernel"],
                    support=c["support"], tile=c["tile"], w_range=w_range,
                    precision=c["precision"], max_vis=max_vis, device=dev,
                    image_n=c["image_n"] or None, hermitian_mirror=c["mirror"],
                    deterministic=c["deterministic"])


def prepare(case, seed):
    c = dict(BASE, **case)
    dev = torch.device("cuda", torch.cuda.current_device())
    op = c["op"]
    uvw, scale, vis, wt = _observation(c, seed, dev)
    s = {"op": op, "case": c}
    m = c["image_n"] or c["n"]
    if op == "rows":
        s.update(uvw=uvw, scale=scale, vis=vis, wt=wt)
        s["im"] = _imager(c, vis.shape[0] * vis.shape[1], dev)
    elif op == "streamed":
        s.update(uvw=_pin(uvw), scale=scale.cpu(), vis=_pin(vis), wt=_pin(wt))
        s["out"] = torch.empty((m, m), dtype=torch.float32, pin_memory=True)
        s["im"] = _imager(c, c["chunk"], dev)
    else:
        uvw, vis, wt = _flat(c, uvw, scale, vis, wt)
        s["im"] = _imager(c, c["n_vis"], dev)
        if op == "request":
            s.update(uvw=_pin(uvw), vis=_pin(vis), wt=_pin(wt))
            s["out"] = torch.empty((m, m), dtype=torch.float32, pin_memory=True)
        else:
            s.update(uvw=uvw, vis=vis, wt=wt)
        if op in ("chi2", "vis_grad", "predict"):
            # a solver bins its geometry once and then takes many steps
            s["im"].bin(uvw, vis, wt)
            s["x"] = _sky(c, seed, dev)
            if op == "chi2" and wt is None:
                s["wt"] = torch.ones(c["n_vis"], device=dev)
            if op == "chi2":
                s["x"].requires_grad_()
            if op == "vis_grad":
                s["vis"] = vis.clone().requires_grad_()
    torch.cuda.synchronize()
    return s


def run(s):
    im, op = s["im"], s["op"]
    if op == "image":
        return im.image(s["uvw"], s["vis"], s["wt"])
    if op == "request":
        return im.image_from_host(s["uvw"], s["vis"], s["wt"], s["out"])
    if op == "weighted":
        return im.image_weighted(s["uvw"], s["vis"], s["wt"], robust=s["case"]["robust"])
    if op == "rows":
        im.bin_channels(s["uvw"], s["scale"], s["vis"], s["wt"], n_corr=s["case"]["n_corr"])
        return im.image_from_binned()
    if op == "streamed":
        im.image_streamed(s["uvw"], s["vis"], s["wt"], s["out"], chan_scale=s["scale"],
                          n_corr=s["case"]["n_corr"])
        im.join_out()
        return s["out"]
    if op == "chi2":
        loss = A.chi2(s["x"], im, s["vis"], s["wt"])
        (g,) = torch.autograd.grad(loss, s["x"])
        return {"loss": loss.detach(), "grad": g}
    if op == "vis_grad":
        img = A.grid_image(s["vis"], im, s["wt"])
        (g,) = torch.autograd.grad(img, s["vis"], s["x"])
        return {"image": img.detach(), "grad": g}
    if op == "predict":
        return im.predict(s["x"])
    raise ValueError(op)


def work(case):
    """Inputs read once, outputs written once; the multiply-adds of Eq. 3 (two real
    ones per visibility and footprint cell) and one complex transform per image
    column and plane (5 n log2 n) with the plane's turn of every pixel.  The row
    transforms depend on the coverage and are not counted."""
    c = dict(BASE, **case)
    m = c["image_n"] or c["n"]
    nv, nval = c["n_vis"], c["n_vis"] * c["n_corr"]
    per_vis_uvw = c["op"] not in ("rows", "streamed")
    data = (24 * nv if per_vis_uvw else 24 * _rows(c)) + 8 * nval + (4 * nval if c["weights"] else 0)
    img = 4 * m * m
    grid = 4.0 * c["support"] ** 2 * nv * (2 if c["mirror"] else 1)
    cols = c["n_w"] * m * (5.0 * c["n"] * math.log2(c["n"]) + 8.0 * m)
    if c["op"] == "chi2":  # geometry (20 B), observed values and weights, image in, gradient out
        return {"bytes": nv * (20 + 8 + 4) + 2 * img, "flops": 2 * (grid + cols)}
    if c["op"] == "vis_grad":
        return {"bytes": nv * (20 + 8 + 8 + (4 if c["weights"] else 0)) + 2 * img,
                "flops": 2 * (grid + cols)}
    if c["op"] == "predict":
        return {"bytes": nv * (20 + 8) + img, "flops": grid + cols}
    return {"bytes": data + img, "flops": grid + cols}


# ---------------------------------------------------------------- 64-bit values
def _shape(c):
    """KB shape (Beatty et al. 2005, oversampling 2) or Gaussian sigma."""
    W = c["support"]
    if c["kernel"] == "kb":
        return math.pi * math.sqrt((W / 2.0) ** 2 * 1.5 ** 2 - 0.8)
    return W / 6.0


def _kernel(c, d):
    W, p = c["support"], _shape(c)
    if c["kernel"] == "kb":
        return torch.special.i0(p * torch.sqrt(torch.clamp(1.0 - (2.0 * d / W) ** 2, min=0.0))) \
            / float(torch.special.i0(torch.tensor(p, dtype=torch.float64)))
    return torch.exp(-d * d / (2.0 * p * p))


def _taper(c, nu):
    """Continuous transform of the kernel, by a 96-point Gauss-Legendre rule."""
    x, w = np.polynomial.legendre.leggauss(96)
    W = c["support"]
    d = torch.from_numpy(0.25 * W * (x + 1.0)).to(nu.device)
    g = _kernel(c, d) * torch.from_numpy(w).to(nu.device) * (0.5 * W)
    return (torch.cos(2.0 * math.pi * nu[:, None] * d[None, :]) * g).sum(1)


class _Exact:
    """W-stacked imaging and its transpose in float64, plane by plane."""

    def __init__(self, c, uvw, dev):
        self.c, self.dev = c, dev
        n, n_w, W, fov = c["n"], c["n_w"], c["support"], c["fov_deg"] * DEG
        h = (W - 1) // 2 if W % 2 else W // 2 - 1
        w = uvw[:, 2]
        if c["given_w"]:
            w0, w1 = -c["w_max"], c["w_max"]
        else:
            w0, w1 = float(w.min()), float(w.max())
        dw = (w1 - w0) / n_w
        self.wk = [w0 + (k + 0.5) * dw if dw else w0 for k in range(n_w)]
        plane = torch.zeros(w.shape, dtype=torch.int16, device=dev)
        if dw:
            for j in range(1, n_w):
                plane += (w >= j * dw + w0).to(torch.int16)
        ok = (w >= w0) & (w <= w1)
        self.a, self.f = [], []
        for ax in (0, 1):
            x = uvw[:, ax] * fov + n / 2
            cen = torch.floor(x + 0.5) if W % 2 else torch.floor(x)
            a = cen.to(torch.int32) - h
            ok &= (a >= 0) & (a + W <= n)
            self.a.append(a)
            self.f.append(x - cen)
        self.h, self.ok = h, ok
        idx = torch.nonzero(ok).reshape(-1)
        order = torch.argsort(plane[idx], stable=True)
        self.order = idx[order]
        self.count = torch.bincount(plane[idx].long(), minlength=n_w).tolist()
        m = c["image_n"] or n
        self.m, self.off = m, (n - m) // 2
        pix = torch.arange(self.off, self.off + m, device=dev, dtype=torch.float64) - n // 2
        self.l = pix * (fov / n)
        self.ctap = _taper(c, pix / n)
        self.sign = 1.0 - 2.0 * (torch.arange(n, device=dev) % 2).double()

    def planes(self):
        o = 0
        for k, cnt in enumerate(self.count):
            yield k, self.order[o:o + cnt]
            o += cnt

    def _parts(self, idx):
        """Chunks of idx with their footprint rows, columns and kernel weights."""
        W = self.c["support"]
        j = torch.arange(W, device=self.dev, dtype=torch.float64) - self.h
        for i0 in range(0, idx.numel(), 1 << 23):
            q = idx[i0:i0 + (1 << 23)]
            gx = _kernel(self.c, j[:, None] - self.f[0][q][None, :])
            gy = _kernel(self.c, j[:, None] - self.f[1][q][None, :])
            yield q, self.a[0][q].long(), self.a[1][q].long(), gx, gy

    def _turn(self, k):
        r2 = self.l[:, None] ** 2 + self.l[None, :] ** 2
        nm1 = -r2 / (1.0 + torch.sqrt(1.0 - r2))
        ph = self.wk[k] * nm1
        ph -= torch.round(ph)
        return torch.polar(torch.ones_like(ph), 2.0 * math.pi * ph)

    def scale(self, correct):
        r2 = self.l[:, None] ** 2 + self.l[None, :] ** 2
        nn = torch.sqrt(1.0 - r2)
        s = self.sign[self.off:self.off + self.m]
        return (nn if correct else 1.0 / nn) * (s / self.ctap)[:, None] * (s / self.ctap)[None, :]

    def image(self, val, correct=True):
        """Re of the plane sum of complex128 values (weights applied), scaled."""
        n, W, off, m = self.c["n"], self.c["support"], self.off, self.m
        acc = torch.zeros((m, m), dtype=torch.float64, device=self.dev)
        for k, idx in self.planes():
            if not idx.numel():
                continue
            g = torch.zeros(n * n, 2, dtype=torch.float64, device=self.dev)
            for q, ax, ay, gx, gy in self._parts(idx):
                v = torch.view_as_real(val[q])
                for jy in range(W):
                    vy = v * gy[jy][:, None]
                    for jx in range(W):
                        cell = (ay + jy) * n + ax + jx
                        g.index_add_(0, cell, vy * gx[jx][:, None])
            z = torch.view_as_complex(g).reshape(n, n) * self.sign[:, None] * self.sign[None, :]
            del g
            z = torch.fft.ifft2(z, norm="forward")[off:off + m, off:off + m]
            t = self._turn(k)
            acc += z.real * t.real - z.imag * t.imag
        return acc * self.scale(correct)

    def adjoint(self, img, n_vis, correct=True):
        """Transpose of image(): the values at every visibility (0 where dropped)."""
        n, W, off, m = self.c["n"], self.c["support"], self.off, self.m
        out = torch.zeros(n_vis, dtype=torch.complex128, device=self.dev)
        x = img.double() * self.scale(correct)
        for k, idx in self.planes():
            if not idx.numel():
                continue
            z = torch.zeros((n, n), dtype=torch.complex128, device=self.dev)
            z[off:off + m, off:off + m] = x * self._turn(k).conj()
            z = torch.fft.fft2(z) * self.sign[:, None] * self.sign[None, :]
            z = z.reshape(-1)
            for q, ax, ay, gx, gy in self._parts(idx):
                o = torch.zeros(q.numel(), dtype=torch.complex128, device=self.dev)
                for jy in range(W):
                    for jx in range(W):
                        o += z[(ay + jy) * n + ax + jx] * (gx[jx] * gy[jy])
                out[q] = o
        return out


def exact(case, seed):
    c = dict(BASE, **case)
    if c["n_vis"] * c["support"] ** 2 > 2.0e10:  # minutes of 64-bit scatter
        return None
    dev = torch.device("cuda", torch.cuda.current_device())
    op = c["op"]
    uvw, scale, vis, wt = _observation(c, seed, dev)
    if op in ("rows", "streamed"):
        nv = vis.shape[0] * vis.shape[1]
        full = (uvw[:, None, :] * scale[None, :, None]).reshape(-1, 3)
        v = vis.to(torch.complex128)
        w = torch.ones(vis.shape, dtype=torch.float64, device=dev) if wt is None else wt.double()
        val, w = (v * w).sum(-1).reshape(-1), w.sum(-1).reshape(-1)
    else:
        nv = c["n_vis"]
        full, vis, wt = _flat(c, uvw, scale, vis, wt)
        w = torch.ones(nv, dtype=torch.float64, device=dev) if wt is None else wt.double()
        val = vis.to(torch.complex128) * w
        if c["mirror"]:
            full = torch.cat([full, -full])
            val, w = torch.cat([val, val.conj()]), torch.cat([w, w])
    del uvw
    E = _Exact(c, full, dev)
    del full
    sumw = float(w[E.ok].sum())
    if op == "weighted":
        n, h = c["n"], E.h
        cell = (E.a[1].long() + h) * n + E.a[0].long() + h
        kept = torch.nonzero(E.ok).reshape(-1)
        dens = torch.zeros(n * n, dtype=torch.float64, device=dev).index_add_(0, cell[kept],
                                                                              w[kept])
        f2 = (5.0 * 10.0 ** -c["robust"]) ** 2 * sumw / float((dens * dens).sum())
        d = torch.zeros_like(w)
        d[kept] = dens[cell[kept]]
        w2 = w / (1.0 + f2 * d)
        return E.image(vis.to(torch.complex128) * w2) / float(w2[E.ok].sum())
    if op == "chi2":
        x = _sky(c, seed, dev)
        r = vis.to(torch.complex128) - E.adjoint(x, nv, correct=False)
        loss = (w * (r.real ** 2 + r.imag ** 2)).sum()
        return {"loss": loss, "grad": E.image(-2.0 * w * r, correct=False)}
    if op == "vis_grad":
        y = _sky(c, seed, dev)
        return {"image": E.image(val) / sumw, "grad": E.adjoint(y, nv) * w / sumw}
    if op == "predict":
        return E.adjoint(_sky(c, seed, dev), nv, correct=False)
    return E.image(val) / sumw
