"""The two-pass transform of n = 1024, 2048, 4096 (row transforms of the
non-empty tiles, then the whole column transform with the w-screen and the
plane sum) and the split transform's sparse rows of n = 8192, 16384 against cuFFT's 2D plan and the separate stack (RICK_FFT_2D), where
its work depends on the data: empty tiles, tile rows and planes, every tile
side, several plane groups and more planes than one run of the screen's
rotation, several chunks of measurements (their tiles united; more than one
gridding pass: all tiles), w-support, and its adjoint.

Tolerance: the two factorisations of the FP32 transform differ by a few
roundings of ~1e-7 of a plane's RMS per pass; the other tests of two paths of
the same image hold 1e-5 of the peak (uncorrected images), and so do these.
The adjoint's planes are dense, its bound is theirs (1e-4)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

REAL = synth.FLAG_REAL


@pytest.fixture(scope="module")
def rick():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as r
    r.load()
    return r


def _problem(n, nw, m, seed, part=1.0, empty_planes=False, S=7):
    """Measurements in a disk of `part` of the grid, off its centre, on planes
    0, 3, 6, .. only with empty_planes."""
    g = torch.Generator().manual_seed(seed)
    pixel = 2e-4 / (n / 1024)
    du = 1.0 / (n * pixel)
    r = 0.45 * part * n * torch.sqrt(torch.rand(m, generator=g, dtype=torch.float64))
    th = 2 * np.pi * torch.rand(m, generator=g, dtype=torch.float64)
    off = 0.45 * (1 - part) * n
    u, v = (r * torch.cos(th) + off) * du, (r * torch.sin(th) - off) * du
    k = torch.randint(0, nw, (m,), generator=g)
    if empty_planes:
        k = k // 3 * 3
    w = (k + torch.rand(m, generator=g, dtype=torch.float64)) / nw * 400.0 - 200.0
    vis = torch.complex(torch.randn(m, generator=g), torch.randn(m, generator=g)) + 1
    wt = 0.5 + torch.rand(m, generator=g)
    p = dict(n=n, nw=nw, pixel_rad=pixel, w_min=-200.0, w_max=200.0, kernel=synth.KERNEL_KB, support=S, flags=REAL)
    return p, [t.cuda().contiguous() for t in (vis, u.float(), v.float(), w.float(), wt)]


def _run(rick, p, data, flags, chunks=1, r=None, out=None):
    vis, u, v, w, wt = data
    im = rick.Imager(dict(p, flags=flags))
    cut = [len(u) * i // chunks for i in range(chunks + 1)]
    for a, b in zip(cut, cut[1:]):
        im.grid(vis[a:b], u[a:b], v[a:b], w[a:b], wt[a:b])
    img = im.image(out=out).clone()
    grad = im.degrid(r, u, v, w, wt).clone() if r is not None else None
    im.stats()  # raises if a bounded wait ran out
    im.close()
    return img, grad


def _same(a, b, tol):
    assert (a - b).abs().max().item() <= tol * b.abs().max().item()


@pytest.mark.parametrize("n,nw,m,tile,extra", [
    (1024, 5, 3000, 16, {}),
    (1024, 5, 3000, 64, {"part": 0.3}),
    (2048, 3, 20000, 32, {"part": 0.2}),
    (2048, 70, 30000, 32, {"empty_planes": True}),     # > 2 runs of the rotation, empty planes
    (4096, 4, 300, 32, {"part": 0.9, "S": 8}),         # mostly empty tiles
    (4096, 2, 50000, 16, {"part": 0.1}),
    (4096, 33, 40000, 64, {"empty_planes": True}),     # one plane past a run
    (8192, 4, 20000, 16, {"empty_planes": True}),      # the split transform's sparse rows
    (8192, 2, 2000, 64, {"part": 0.3}),
    (16384, 2, 20000, 32, {"part": 0.5, "empty_planes": True}),
])
def test_equals_2d_plan(rick, n, nw, m, tile, extra):
    p, data = _problem(n, nw, m, 11 + n + nw + tile, **extra)
    p["tile"] = tile
    r = torch.randn((n, n), generator=torch.Generator().manual_seed(5)).cuda()
    a, ga = _run(rick, p, data, REAL, r=r)
    b, gb = _run(rick, p, data, REAL | rick.FFT_2D, r=r)
    _same(a, b, 1e-5)
    _same(ga, gb, 1e-4)


@pytest.mark.parametrize("flags,more", [
    (synth.FLAG_REAL | synth.FLAG_APPLY_N, {"plane_group": 5}),
    (0, {"plane_group": 1}),
    (synth.FLAG_REAL, {"w_support": 4, "plane_group": 7}),
    (synth.FLAG_REAL | synth.FLAG_UNIFORM, {}),
])
def test_options_equal_2d_plan(rick, flags, more):
    p, data = _problem(1024, 12, 20000, 21, part=0.6)
    p.update(more)
    r = torch.randn((1024, 1024), generator=torch.Generator().manual_seed(6)).cuda()
    r = r if flags & REAL else torch.complex(r, r.flip(0))
    a, ga = _run(rick, p, data, flags, r=r)
    b, gb = _run(rick, p, data, flags | rick.FFT_2D, r=r)
    _same(a, b, 1e-5)
    _same(ga, gb, 1e-4)


@pytest.mark.parametrize("chunks", [3, 16, 17])
def test_chunks_equal_one(rick, chunks):
    """Tiles of several lists are united; 17 chunks take two gridding passes."""
    p, data = _problem(1024, 6, 4000, 31, part=0.5)
    a, _ = _run(rick, p, data, REAL, chunks=chunks)
    b, _ = _run(rick, p, data, REAL)
    _same(a, b, 1e-5)


def test_image_of_nothing_and_unaligned_output(rick):
    p, data = _problem(1024, 3, 1000, 41)
    buf = torch.full((1024 * 1024 + 1,), 7.0, device="cuda")
    out = buf[1:].view(1024, 1024)  # 4-byte aligned only
    a, _ = _run(rick, p, data, REAL, out=out)
    b, _ = _run(rick, p, data, REAL)
    _same(a, b, 1e-5)
    im = rick.Imager(p)
    assert im.image().abs().max().item() == 0.0  # nothing gridded
    im.close()


def test_predict_only_reads_needed_tiles(rick):
    """Prediction at a handful of measurements (a few needed tiles) equals the
    2D plan's."""
    p, data = _problem(2048, 9, 40, 51)
    model = torch.randn((2048, 2048), generator=torch.Generator().manual_seed(7)).cuda()
    got = []
    for f in (REAL, REAL | rick.FFT_2D):
        im = rick.Imager(dict(p, flags=f))
        got.append(im.predict(model, *data[1:4]).clone())
        im.close()
    _same(got[0], got[1], 1e-4)
