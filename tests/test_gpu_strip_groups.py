"""Which transform a single image of n = 1024, 2048 and 4096 takes by the planes in
its groups, read off the launches (two-pass: the tiles' marking once, then per
group the gridder's two, rows and columns; split: gridder, first column factor,
stack; 2D plan: gridder, stack), and the two-pass transform at the edge of the
rule against cuFFT's 2D plan: every tile side, options, groups that do not divide
the planes, several chunks of measurements, an unaligned output, nothing
gridded.  Bounds as in the other tests of two transforms of the same
uncorrected data: 1e-5 of the image's peak, 1e-4 for the adjoint."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

REAL, APPLY_N, UNIFORM = synth.FLAG_REAL, synth.FLAG_APPLY_N, synth.FLAG_UNIFORM


@pytest.fixture(scope="module")
def rick():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as r
    r.load()
    return r


def _run(rick, prob, flags, more, r=None, chunks=1, out=None):
    g = [prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")]
    m = g[1].numel()
    im = rick.Imager(dict(prob["params"], flags=flags, **more))
    cut = [m * i // chunks for i in range(chunks + 1)]
    for a, b in zip(cut, cut[1:]):
        im.grid(*(x[a:b].contiguous() for x in g))
    im.set_timing(True)
    img = im.image(out=out).clone()
    t = im.timing()
    im.set_timing(False)
    grad = im.degrid(r, *g[1:]).clone() if r is not None else None
    im.stats()  # raises if a bounded wait ran out
    im.close()
    return img, grad, (t["kernel_launches"], t["colfft_calls"])


def _same(a, b, tol):
    assert (a - b).abs().max().item() <= tol * b.abs().max().item()


def _problem(n, nw, m=20000, fill=0.3):
    return synth.disk_problem(n, nw, m, synth.KERNEL_KB, 7, 6.0, 200.0, n + nw, fill=fill, weights="random")


@pytest.mark.parametrize("n,nw,flags,more", [
    (1024, 12, REAL, {"tile": 16}),
    (1024, 13, REAL, {"tile": 64}),
    (1024, 30, REAL | APPLY_N, {"plane_group": 13}),
    (1024, 25, 0, {"plane_group": 12}),
    (1024, 28, REAL, {"w_support": 4, "plane_group": 14}),
    (1024, 12, REAL | UNIFORM, {}),
    (2048, 1, REAL, {"tile": 32}),
    (2048, 3, 0, {}),
    (2048, 11, REAL, {"plane_group": 4, "w_support": 3}),
    (4096, 2, REAL, {"tile": 64}),
    (4096, 9, REAL, {"plane_group": 4}),
])
def test_two_pass(rick, n, nw, flags, more):
    prob = _problem(n, nw)
    r = torch.randn((n, n), generator=torch.Generator().manual_seed(n + nw)).cuda()
    r = r if flags & REAL else torch.complex(r, r.flip(0))
    a, ga, launches = _run(rick, prob, flags, more, r)
    b, gb, _ = _run(rick, prob, flags | rick.FFT_2D, more, r)
    groups = -(-nw // more.get("plane_group", nw))
    assert launches == (1 + 4 * groups, 0)
    _same(a, b, 1e-5)
    _same(ga, gb, 1e-4)


@pytest.mark.parametrize("n,nw,group", [(1024, 11, 0), (1024, 24, 11), (2048, 6, 3), (4096, 5, 1)])
def test_few_planes_take_the_former_transform(rick, n, nw, group):
    prob = _problem(n, nw)
    a, _, launches = _run(rick, prob, REAL, {"plane_group": group})
    b, _, _ = _run(rick, prob, REAL | rick.FFT_2D, {"plane_group": group})
    groups = -(-nw // (group or nw))
    assert launches == ((3 * groups, 0) if n == 1024 else (4 * groups, groups))
    _same(a, b, 1e-5)


@pytest.mark.parametrize("chunks", [3, 16, 17])
def test_chunks(rick, chunks):
    """Tiles of several lists are united; 17 chunks take two gridding passes."""
    prob = _problem(1024, 12, 4000)
    a, _, _ = _run(rick, prob, REAL, {}, chunks=chunks)
    b, _, _ = _run(rick, prob, REAL | rick.FFT_2D, {})
    _same(a, b, 1e-5)


def test_unaligned_output_and_nothing_gridded(rick):
    prob = _problem(1024, 12, 1000)
    out = torch.full((1024 * 1024 + 1,), 7.0, device="cuda")[1:].view(1024, 1024)  # 4-byte aligned only
    a, _, _ = _run(rick, prob, REAL, {}, out=out)
    b, _, _ = _run(rick, prob, REAL | rick.FFT_2D, {})
    _same(a, b, 1e-5)
    im = rick.Imager(dict(prob["params"], flags=REAL))
    assert im.image().abs().max().item() == 0.0
    im.close()
