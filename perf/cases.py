"""Workloads of the imager: what its users run, from the smallest image to the
largest, each through the package's public entry points.

A case is a dict of plain values; ``kind`` says which call it is:

* ``image``    reset, grid, image: one dirty image of device-resident data;
* ``planes``   reset, grid, grid_planes: the gridded w-planes alone;
* ``channels`` BatchImager.images: several frequency channels in one call;
* ``gradient`` dirty_image and its backward: the image and the gradient of a
  loss on it with respect to the visibilities;
* ``predict``  Imager.predict: model visibilities of a model image.

Inputs are synthetic.  ``coverage`` "track" is an Earth-rotation synthesis (a
random planar array of ``array_km``, the textbook baseline-to-uvw rotation, the
longest |u| or |v| placed at 0.45 n cells, or, with ``field_deg``, the rows that
lie in the grid of that field), "disk" u, v uniform in a disk of 0.45 n cells and
w uniform; ``order`` is the order of the rows: "random" (flagged, shuffled or
averaged data) or "time" (as a telescope writes them: integration by
integration).  Visibilities are a few point sources plus noise.
"""
import math

import numpy as np
import torch

import paper_2504_00959_gb300 as rick

C_LIGHT = 299_792_458.0
GAUSS, KB = 0, 1


def _case(name, kind, n, nw, m, **more):
    c = dict(kind=kind, n=n, nw=nw, m=m, support=7, kernel=KB, coverage="track", order="random", weights="unit",
             uniform=False, fold=False, apply_n=False, w_support=1, nchan=1, graph=False,
             array_km=20.0, field_deg=0.0)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a quick-look image (256^2, 8 planes, 1e5 visibilities, Gaussian kernel): launches and latency
        _case("image_256", "image", 256, 8, 100_000, kernel=GAUSS, coverage="disk"),
        # a grid side that is not a power of two, weighted data, the n factor of Eq. 1
        _case("image_1000", "image", 1000, 12, 600_000, support=6, weights="random", apply_n=True, order="time"),
        # an ordinary facet or survey field
        _case("image_1024", "image", 1024, 16, 1_000_000),
        # the benchmark's 4096^2 x 32-plane x 1e7-visibility image
        _case("image_4096", "image", 4096, 32, 10_000_000),
        # the benchmark's 16384^2 field of 5 degrees at an eighth of its planes and visibilities: support 8, uniform
        # weighting, an array whose longest baselines lie outside the grid
        _case("image_16384", "image", 16384, 16, 25_000_000, support=8, uniform=True, array_km=60.0, field_deg=5.0),
        # one deep channel: few cells, many visibilities
        _case("image_2048_deep", "image", 2048, 16, 20_000_000, order="time"),
        # accurate w-terms of a real sky: four planes per visibility, folded onto w >= 0
        _case("image_2048_wsupport", "image", 2048, 16, 2_000_000, w_support=4, fold=True, weights="random"),
        # gridding alone, for a caller with its own transform
        _case("planes_512", "planes", 512, 16, 500_000, support=8),
        # frequency channels of uneven depth imaged in one call
        _case("channels_2048", "channels", 2048, 16, 16_000_000, nchan=8),
        # many small channels (a spectral-line cube of a small field), replayed from a graph
        _case("channels_256", "channels", 256, 8, 800_000, nchan=16, graph=True, support=6),
        # differentiable imaging: the image and the visibility gradient of a loss on it
        _case("gradient_4096", "gradient", 4096, 32, 10_000_000),
        # self-calibration's forward model: visibilities of a model image
        _case("predict_2048", "predict", 2048, 16, 3_000_000, order="time"),
    ]


def _smooth(x):
    """The smallest even number >= x with no prime factor above 7 (a good FFT size)."""
    x = max(2, int(x) + (int(x) & 1))
    while True:
        r = x
        for p in (2, 3, 5, 7):
            while r % p == 0:
                r //= p
        if r == 1:
            return x
        x += 2


def draw(rng):
    def logu(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    kind = rng.choice(["image", "image", "image", "planes", "channels", "gradient", "predict"])
    x = logu(200, 8200)
    n = 1 << max(7, min(13, round(math.log2(x)))) if rng.random() < 0.6 else _smooth(x)
    nchan = rng.randint(2, 12) if kind == "channels" else 1
    most = max(1, min(48, int(1.5e9 / (n * n) / nchan)))  # planes
    nw = max(1, min(most, int(logu(2, 49))))
    m = int(logu(2e4, 2e7))
    w_support = rng.choice([3, 4]) if kind in ("image", "gradient", "predict") and nw >= 12 and rng.random() < 0.2 else 1
    if w_support > 1:
        m = min(m, 4_000_000)
    return _case(None, kind, n, nw, m, support=rng.randint(4, 9), kernel=rng.choice([GAUSS, KB, KB]),
                 coverage=rng.choice(["track", "track", "track", "disk"]), order=rng.choice(["random", "time"]),
                 weights=rng.choice(["unit", "random"]), uniform=kind in ("image", "gradient") and rng.random() < 0.25,
                 fold=kind in ("image", "channels") and rng.random() < 0.2, apply_n=rng.random() < 0.2,
                 w_support=w_support, nchan=nchan, graph=kind == "channels" and rng.random() < 0.5)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _track(m, order, g, freq, km):
    """u, v, w in wavelengths (float64) of m (baseline, integration) rows of 256
    antennas in a disk of km, 6 h of 10 s integrations at declination -30."""
    na, nt, lat = 256, 2160, math.radians(-30.0)
    r, th = 500.0 * km * torch.sqrt(_rand(g, na)), 2.0 * math.pi * _rand(g, na)
    east, north = r * torch.cos(th), r * torch.sin(th)
    xyz = torch.stack([-math.sin(lat) * north, east, math.cos(lat) * north])
    i, j = torch.triu_indices(na, na, offset=1, device="cuda")
    rows = torch.randint(0, i.numel() * nt, (m,), generator=g, device="cuda")
    if order == "time":
        rows = torch.sort(rows).values
    t, b = rows // i.numel(), rows % i.numel()
    L = xyz[:, j[b]] - xyz[:, i[b]]
    H = (-3.0 + (t.double() + 0.5) * 10.0 / 3600.0) * (math.pi / 12.0)
    s, c, sd, cd = torch.sin(H), torch.cos(H), math.sin(lat), math.cos(lat)
    lam = C_LIGHT / freq
    return ((s * L[0] + c * L[1]) / lam, (-sd * c * L[0] + sd * s * L[1] + cd * L[2]) / lam,
            (cd * c * L[0] - cd * s * L[1] + sd * L[2]) / lam)


def _sky(u, v, w, field, g):
    """Visibilities of 6 point sources in the central 80 % of the field, plus noise."""
    m = u.numel()
    vis = torch.view_as_complex(0.3 * torch.randn((m, 2), generator=g, device="cuda"))
    flux, lm = torch.exp(torch.randn(6, generator=g, device="cuda")), 0.4 * field * (2.0 * _rand(g, 6, 2) - 1.0)
    for f, (l, mm) in zip(flux.tolist(), lm.tolist()):
        r2 = l * l + mm * mm
        turns = -(u * l + v * mm - w * r2 / (1.0 + math.sqrt(1.0 - r2)))
        ang = (2.0 * math.pi * (turns - torch.round(turns))).float()
        vis += torch.polar(torch.full_like(ang, f), ang)
    return vis


def _flags(case):
    return (rick.GRID_CORRECT | rick.REAL_IMAGE | (rick.APPLY_N if case["apply_n"] else 0)
            | (rick.UNIFORM_WEIGHT if case["uniform"] else 0) | (rick.HERMITIAN_FOLD if case["fold"] else 0))


def _channel_sizes(case, seed):
    rs = np.random.RandomState(int(seed) % (1 << 31))
    share = np.exp(rs.uniform(0.0, math.log(8.0), case["nchan"]))
    cut = np.floor(np.concatenate([[0.0], np.cumsum(share)]) / share.sum() * case["m"]).astype(np.int64)
    cut[-1] = case["m"]
    return cut.tolist()


def _data(case, seed):
    """The problem's parameters, w-ranges and tensors."""
    g = _gen(seed)
    n, m, nchan = case["n"], case["m"], case["nchan"]
    off = _channel_sizes(case, seed) if case["kind"] == "channels" else [0, m]
    u = torch.empty(m, device="cuda", dtype=torch.float64)
    v, w = torch.empty_like(u), torch.empty_like(u)
    if case["coverage"] == "disk":
        pixel = math.radians(2.0) / n
        r, th = 0.45 * n * torch.sqrt(_rand(g, m)) / (n * pixel), 2.0 * math.pi * _rand(g, m)
        u, v, w = r * torch.cos(th), r * torch.sin(th), 50.0 * (2.0 * _rand(g, m) - 1.0)
    else:
        for c in range(nchan):
            a, b = off[c], off[c + 1]
            while a < b:
                x = _track(b - a, case["order"], g, 1.4e9 * (1.0 - 0.3 * c / nchan), case["array_km"])
                if case["field_deg"]:  # keep the rows whose footprints lie in the grid
                    lim = (n / 2 - case["support"]) / math.radians(case["field_deg"])
                    keep = torch.nonzero((x[0].abs() < lim) & (x[1].abs() < lim)).flatten()
                    x = [t[keep] for t in x]
                e = a + x[0].numel()
                u[a:e], v[a:e], w[a:e] = x
                a = e
        pixel = math.radians(case["field_deg"]) / n if case["field_deg"] else \
            0.45 / float(torch.maximum(u.abs().max(), v.abs().max()))
    if case["coverage"] == "disk" and case["order"] == "time":
        k = torch.argsort(th)
        u, v, w = u[k], v[k], w[k]
    vis = _sky(u, v, w, n * pixel, g)
    wt = torch.ones(m, device="cuda") if case["weights"] == "unit" else 0.5 + torch.rand(m, generator=g, device="cuda")
    u, v, w = u.float(), v.float(), w.float()
    ranges = []
    for c in range(nchan):
        x = w[off[c]:off[c + 1]]
        x = x.abs() if case["fold"] else x
        lo, hi = (0.0 if case["fold"] else float(x.min()), float(x.max())) if x.numel() else (-1.0, 1.0)
        hi = hi if hi > lo else lo + 1.0
        sw = case["w_support"]
        if sw > 1:  # the w-footprints need half a support of planes beyond the data
            d = (hi - lo) / (case["nw"] - sw) * sw / 2
            lo, hi = lo - d, hi + d
        ranges.append((lo, hi))
    if case["w_support"] > 1:  # keep the planes fine enough for the kernel in w: narrow the field where needed
        dw = (ranges[0][1] - ranges[0][0]) / case["nw"]
        pixel = min(pixel, math.sqrt(1.0 / dw) / n)
    params = dict(n=n, nw=case["nw"], pixel_rad=pixel, w_min=ranges[0][0], w_max=ranges[0][1], kernel=case["kernel"],
                  support=case["support"], kernel_param=0.0, flags=_flags(case), w_support=case["w_support"])
    d = dict(params=params, ranges=ranges, off=off, u=u, v=v, w=w, wt=wt, vis=vis)
    if case["kind"] == "gradient":  # a residual under the primary beam
        x = (torch.arange(n, device="cuda") - n // 2) / n
        beam = torch.exp(-(x * x) / 0.04)
        d["upstream"] = torch.randn((n, n), generator=g, device="cuda") * beam[:, None] * beam[None, :]
    if case["kind"] == "predict":  # a clean-component model
        k = max(16, n)
        at = torch.randint(n // 10, n - n // 10, (2, k), generator=g, device="cuda")
        d["model"] = torch.zeros((n, n), device="cuda")
        d["model"][at[0], at[1]] = torch.exp(torch.randn(k, generator=g, device="cuda"))
    return d


def prepare(case, seed):
    d = _data(case, seed)
    d["kind"], d["graph"] = case["kind"], case["graph"]
    if case["kind"] == "channels":
        d["imager"] = rick.BatchImager(d["params"], d["ranges"])
        d["stream"] = torch.cuda.Stream()
        d["out"] = torch.empty((case["nchan"], case["n"], case["n"]), device="cuda")
        torch.cuda.synchronize()
    else:
        d["imager"] = rick.Imager(d["params"])
    return d


def run(state):
    im, kind = state["imager"], state["kind"]
    vis, u, v, w, wt = state["vis"], state["u"], state["v"], state["w"], state["wt"]
    if kind == "channels":
        if not state["graph"]:
            return im.images(vis, u, v, w, wt, state["off"], out=state["out"])
        here, s = torch.cuda.current_stream(), state["stream"]  # a graph needs a stream of its own
        s.wait_stream(here)
        with torch.cuda.stream(s):
            im.images(vis, u, v, w, wt, state["off"], out=state["out"], use_graph=True)
        here.wait_stream(s)
        return state["out"]
    if kind == "predict":
        return im.predict(state["model"], u, v, w)
    if kind == "gradient":
        x = vis.detach().requires_grad_(True)
        img = rick.dirty_image(x, u, v, w, wt, im)
        (g,) = torch.autograd.grad(img, x, state["upstream"])
        return {"image": img.detach(), "grad": g}
    im.reset()
    im.grid(vis, u, v, w, wt)
    return im.grid_planes() if kind == "planes" else im.image()


def work(case):
    n, nw, m, S = case["n"], case["nw"] * case["nchan"], case["m"], case["support"]
    vis_bytes, pix = 24 * m, 4 * n * n * case["nchan"]
    grid_flops = 4.0 * m * S * S * case["w_support"]
    fft_flops = nw * 10.0 * n * n * math.log2(n)
    stack_flops = nw * 14.0 * n * n
    kind = case["kind"]
    if kind == "planes":
        return {"bytes": vis_bytes + 8 * nw * n * n, "flops": grid_flops}
    if kind == "predict":
        return {"bytes": 12 * m + 8 * m + pix, "flops": grid_flops + fft_flops + stack_flops}
    if kind == "gradient":
        return {"bytes": 2 * (vis_bytes + pix), "flops": 2.0 * (grid_flops + fft_flops + stack_flops)}
    return {"bytes": vis_bytes + pix, "flops": grid_flops + fft_flops + stack_flops}


# ------------------------------------------------- the same in 64 bits (torch)

def _kernel(case, x, S):
    if case["kernel"] == GAUSS:
        return torch.exp(-x * x / (2.0 * (S / 6.0) ** 2))
    return torch.special.i0(2.34 * S * torch.sqrt(torch.clamp(1.0 - (2.0 * x / S) ** 2, min=0.0)))


def _transform_of_kernel(case, S, xi):
    """Fourier transform of the kernel over [-S/2, S/2] at xi, relative to xi = 0."""
    t, q = np.polynomial.legendre.leggauss(96)
    t = torch.tensor(t * S / 2, device="cuda")
    g = _kernel(case, t, S) * torch.tensor(q, device="cuda")
    out = torch.zeros_like(xi)
    for tk, gk in zip(t.tolist(), g.tolist()):
        out += gk * torch.cos(2.0 * math.pi * tk * xi)
    return out / g.sum()


class _Exact:
    """One channel in FP64: cells and planes are decided in binary32, as the package states, everything else is float64."""

    def __init__(self, case, d, a, b, rng):
        p = d["params"]
        self.case, self.n, self.nw, self.S, self.sw = case, p["n"], p["nw"], p["support"], case["w_support"]
        n, S = self.n, self.S
        self.u, self.v, self.w = (d[k][a:b].double() for k in "uvw")
        self.flip = (self.w < 0) if case["fold"] else torch.zeros(b - a, dtype=torch.bool, device="cuda")
        sign = torch.where(self.flip, -1.0, 1.0).double()
        self.u, self.v, self.w = self.u * sign, self.v * sign, self.w * sign
        scale = n * p["pixel_rad"]
        s32 = float(np.float32(scale))
        p32 = [(x * s32 + n // 2).float() for x in (self.u, self.v)]
        first = [torch.floor(x - np.float32(S / 2)) for x in p32]
        self.ok = torch.ones(b - a, dtype=torch.bool, device="cuda")
        for f in first:
            self.ok &= (f >= -1) & (f <= n - S - 1)
        self.f = [f.long() + 1 for f in first]
        self.near = [torch.clamp(torch.floor(x + 0.5).long(), max=n - 1) for x in p32]
        self.p = [x * scale + n / 2 for x in (self.u, self.v)]
        self.w_lo, self.dw = rng[0], (rng[1] - rng[0]) / self.nw
        t32 = (self.w.float() - np.float32(rng[0])) * np.float32(1.0 / self.dw)
        if self.nw == 1:
            self.k = torch.zeros_like(self.f[0])
        elif self.sw == 1:
            self.k = torch.clamp(torch.floor(t32), 0, self.nw - 1).long()
        else:
            self.k = torch.floor(t32 - 0.5 - np.float32(self.sw / 2)).long() + 1
        self.pw = (self.w - rng[0]) / self.dw - 0.5
        self.wt = torch.where(self.ok, d["wt"][a:b].double(), 0.0)
        if case["uniform"]:
            cell = self.near[1] * n + self.near[0]
            count = torch.bincount(cell[self.ok], minlength=n * n)
            self.wt = torch.where(self.ok, self.wt / count[torch.where(self.ok, cell, 0)].clamp(min=1), 0.0)
        self.pixel = p["pixel_rad"]
        x = (torch.arange(n, device="cuda", dtype=torch.float64) - n // 2)
        r2 = (x * self.pixel)[None, :] ** 2 + (x * self.pixel)[:, None] ** 2
        self.nm1 = -r2 / (1.0 + torch.sqrt(torch.clamp(1.0 - r2, min=0.0)))
        taper = _transform_of_kernel(case, S, x / n)
        self.final = (r2 < 1.0).double() / (taper[None, :] * taper[:, None])
        if case["apply_n"]:
            self.final *= 1.0 + self.nm1
        if self.sw > 1:
            self.final /= _transform_of_kernel(case, self.sw, self.dw * self.nm1)

    def taps(self, i):
        g = []
        for f, p in zip(self.f, self.p):
            t = torch.stack([_kernel(self.case, f[i] + q - p[i], self.S) for q in range(self.S)])
            g.append(t / t.sum(0))
        return g

    def on_plane(self, k):
        """Indices of the visibilities with a tap on plane k, and those taps."""
        if self.sw == 1:
            i = torch.nonzero(self.ok & (self.k == k)).flatten()
            return i, torch.ones(i.numel(), device="cuda", dtype=torch.float64)
        i = torch.nonzero(self.ok & (self.k <= k) & (k < self.k + self.sw)).flatten()
        h = torch.stack([_kernel(self.case, self.k[i] + q - self.pw[i], self.sw) for q in range(self.sw)])
        return i, _kernel(self.case, k - self.pw[i], self.sw) / h.sum(0)

    def chunks(self, k):
        i, h = self.on_plane(k)
        for s in range(0, i.numel(), 1 << 22):
            yield i[s:s + (1 << 22)], h[s:s + (1 << 22)]

    def plane(self, k, vis):
        n, S = self.n, self.S
        P = torch.zeros((n * n, 2), device="cuda", dtype=torch.float64)
        for i, h in self.chunks(k):
            gu, gv = self.taps(i)
            a = torch.view_as_real(torch.where(self.flip[i], vis[i].conj(), vis[i]).to(torch.complex128)) * (self.wt[i] * h)[:, None]
            for r in range(S):
                for q in range(S):
                    P.index_add_(0, (self.f[1][i] + r) * n + self.f[0][i] + q, a * (gv[r] * gu[q])[:, None])
        return torch.view_as_complex(P).view(n, n)

    def screen(self, k):
        t = (self.w_lo + (k + 0.5) * self.dw) * self.nm1
        return torch.polar(torch.ones_like(t), 2.0 * math.pi * (t - torch.round(t)))

    def image(self, vis):
        acc = torch.zeros((self.n, self.n), device="cuda", dtype=torch.float64)
        for k in range(self.nw):
            P = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(self.plane(k, vis)), norm="forward"))
            acc += (P * self.screen(k)).real
            del P
        return acc * self.final / self.wt.sum()

    def degrid(self, image, wt, total):
        """Adjoint of image() (real images): wt / total times the footprint of the conjugately screened planes."""
        r = image.double() * self.final / total
        out = torch.zeros(self.u.numel(), device="cuda", dtype=torch.complex128)
        for k in range(self.nw):
            Q = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(r * self.screen(k).conj())))
            Q = Q.reshape(-1)
            for i, h in self.chunks(k):
                gu, gv = self.taps(i)
                s = torch.zeros(i.numel(), device="cuda", dtype=torch.complex128)
                for a in range(self.S):
                    for q in range(self.S):
                        s += Q[(self.f[1][i] + a) * self.n + self.f[0][i] + q] * (gv[a] * gu[q])
                s = s * (wt[i] * h)
                out[i] += torch.where(self.flip[i], s.conj(), s)
            del Q
        return out


def exact(case, seed):
    if case["m"] * case["support"] ** 2 * case["w_support"] > 2.5e9:
        return None
    d = _data(case, seed)
    x = [_Exact(case, d, a, b, r) for a, b, r in zip(d["off"], d["off"][1:], d["ranges"])] if case["kind"] == "channels" \
        else [_Exact(case, d, 0, case["m"], d["ranges"][0])]
    kind, e = case["kind"], x[0]
    if kind == "channels":
        return torch.stack([c.image(d["vis"][a:b]) for c, a, b in zip(x, d["off"], d["off"][1:])])
    if kind == "planes":
        return torch.stack([e.plane(k, d["vis"]) for k in range(case["nw"])])
    if kind == "predict":
        return e.degrid(d["model"], e.ok.double(), 1.0)
    if kind == "gradient":
        return {"image": e.image(d["vis"]), "grad": e.degrid(d["upstream"], e.wt, e.wt.sum())}
    return e.image(d["vis"])
