"""RICK_FFT_SPLIT takes the split transform with cuFFT's rows (k_colfft and
k_colstack / k_spreadcol) at the sizes that have kernels over what is not empty
too: n = 1024, 2048 and 4096 (k_rows and k_colimage) and 8192 (k_longrows),
single and batched; and every such transform gives the image of cuFFT's 2D plan
and separate stack (RICK_FFT_2D).

Which kernels ran is read off the phase counts (colfft: the split's first column
factor) and the launch count (k_longrows and k_occupancy are the library's,
cuFFT's rows are not).  Bounds as in the other tests of two transforms of the
same uncorrected data: 1e-5 of the image's peak, 1e-4 for the adjoint."""
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


def _same(a, b, tol):
    assert (a - b).abs().max().item() <= tol * b.abs().max().item()


@pytest.mark.parametrize("n,nw,extra", [(1024, 16, {}), (2048, 9, {"plane_group": 4}), (4096, 33, {}), (8192, 3, {})])
def test_single(rick, n, nw, extra):
    prob = synth.config2(m=100000, n=n, nw=nw)
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    r = torch.randn((n, n), generator=torch.Generator().manual_seed(n)).cuda()
    got = {}
    for name, flag in (("own", 0), ("split", rick.FFT_SPLIT), ("2d", rick.FFT_2D)):
        im = rick.Imager(dict(prob["params"], flags=REAL | flag, **extra))
        im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
        im.set_timing(True)
        img = im.image().clone()
        t = im.timing()
        im.set_timing(False)
        got[name] = (img, im.degrid(r, g["u"], g["v"], g["w"], g["wt"]).clone(), t)
        im.close()
    for name in ("own", "split"):
        _same(got[name][0], got["2d"][0], 1e-5)
        _same(got[name][1], got["2d"][1], 1e-4)
    groups = -(-nw // extra.get("plane_group", nw))
    assert got["split"][2]["colfft_calls"] == groups
    if n <= 4096:
        assert got["own"][2]["colfft_calls"] == 0
    else:
        assert got["own"][2]["kernel_launches"] == got["split"][2]["kernel_launches"] + 2


@pytest.mark.parametrize("n,nw,nchan", [(1024, 6, 5), (8192, 2, 3)])
def test_batch(rick, n, nw, nchan):
    """Pipelined groups (two channels each, both plane buffers) against single
    images by the 2D plan; with timing on the groups run one by one."""
    prob = synth.channels_problem(nchan=nchan, n=n, nw=nw, m_lo=20_000, m_hi=60_000, device="cuda", seed=78)
    args = (prob["vis"], prob["u"], prob["v"], prob["w"], prob["wt"], prob["offsets"])
    want = []
    for c, (lo, hi) in enumerate(prob["ranges"]):
        a, b = prob["offsets"][c], prob["offsets"][c + 1]
        im = rick.Imager(dict(prob["params"], flags=REAL | rick.FFT_2D, w_min=lo, w_max=hi))
        im.grid(*(x[a:b] for x in args[:5]))
        want.append(im.image().clone())
        im.close()
    for flag in (0, rick.FFT_SPLIT):
        bi = rick.BatchImager(dict(prob["params"], flags=REAL | flag, plane_group=2 * nw), prob["ranges"])
        for timed in (False, True):
            bi.set_timing(timed)
            got = bi.images(*args)
            for c in range(nchan):
                _same(got[c], want[c], 1e-5)
        assert bi.timing()["colfft_calls"] == (0 if n <= 4096 and not flag else -(-nchan // 2))
        bi.stats()  # raises if a bounded wait ran out
        bi.close()
