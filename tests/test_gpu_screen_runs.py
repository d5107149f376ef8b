"""The w-screen of the two-pass transform (n = 1024, 2048, 4096) over many planes:
within a run of 32 planes it is a power of a rotation in binary32, whose error
must not add up from run to run.  Images and gradients against cuFFT's 2D plan
with the separate stack (RICK_FFT_2D), whose screen is evaluated directly every 8
planes.

Bounds, relative in the 2-norm: a binary32 rotation is off by at most 6e-8 in
modulus and phase, so 31 of them by at most 1.9e-6 on the last plane of a run;
the transforms round by a few 1e-7.  The image sums over the runs' planes (2e-6);
the gradient of the measurements on the last planes takes one plane each (3e-6).
plane_group 40 and 100: groups that begin and end within a run."""
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


def _rel(a, b):
    return ((a - b).abs().double().pow(2).sum() / b.abs().double().pow(2).sum()).sqrt().item()


@pytest.mark.parametrize("n,nw,flags,extra", [(1024, 1024, REAL, {}), (1024, 257, 0, {"plane_group": 40}),
                                              (2048, 256, REAL, {"plane_group": 100}), (4096, 65, REAL, {})])
def test_many_planes(rick, n, nw, flags, extra):
    prob = synth.disk_problem(n, nw, 200_000, synth.KERNEL_KB, 7, 6.0, 400.0, 500 + nw, fill=0.4, weights="random")
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    lo, hi = prob["params"]["w_min"], prob["params"]["w_max"]
    last = torch.nonzero(g["w"] > hi - (hi - lo) * 33 / nw).flatten()  # the last 33 planes
    r = torch.randn((n, n), generator=torch.Generator().manual_seed(n)).cuda()
    r = r if flags & REAL else torch.complex(r, r.flip(0))
    got = []
    for flag in (0, rick.FFT_2D):
        im = rick.Imager(dict(prob["params"], flags=flags | flag, **extra))
        im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
        img = im.image().clone()
        grad = im.degrid(r, *(g[k][last].contiguous() for k in ("u", "v", "w", "wt"))).clone()
        im.stats()  # raises if a bounded wait ran out
        im.close()
        got.append((img, grad))
    assert _rel(got[0][0], got[1][0]) <= 2e-6
    assert _rel(got[0][1], got[1][1]) <= 3e-6


def test_plane_range_within_a_run(rick):
    """Two halves of the planes, cut within a run, add up to the image, in
    either order on one handle, and again after the other half was imaged."""
    n, nw = 1024, 80
    prob = synth.disk_problem(n, nw, 50_000, synth.KERNEL_KB, 7, 6.0, 400.0, 90, fill=0.4)
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    im = rick.Imager(dict(prob["params"], flags=REAL))

    def image(k0, k1):
        im.reset()
        im.set_plane_range(k0, k1)
        im.set_weight_sum(1.0)
        im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
        return im.image().clone()
    whole, upper, lower, again = image(0, nw), image(45, nw), image(0, 45), image(45, nw)
    im.close()
    assert _rel(upper + lower, whole) <= 2e-6
    assert _rel(again, upper) <= 1e-6


def test_batch_many_planes(rick):
    n, nw, nchan = 1024, 70, 3
    prob = synth.channels_problem(nchan=nchan, n=n, nw=nw, m_lo=20_000, m_hi=60_000, device="cuda", seed=79)
    args = (prob["vis"], prob["u"], prob["v"], prob["w"], prob["wt"], prob["offsets"])
    bi = rick.BatchImager(dict(prob["params"], flags=REAL, plane_group=2 * nw), prob["ranges"])
    got = bi.images(*args).clone()
    bi.close()
    for c, (lo, hi) in enumerate(prob["ranges"]):
        a, b = prob["offsets"][c], prob["offsets"][c + 1]
        im = rick.Imager(dict(prob["params"], flags=REAL | rick.FFT_2D, w_min=lo, w_max=hi))
        im.grid(*(x[a:b] for x in args[:5]))
        want = im.image()
        assert _rel(got[c], want) <= 2e-6
        im.close()
