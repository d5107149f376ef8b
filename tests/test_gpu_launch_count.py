"""rick_timing.kernel_launches counts the library's own launches.  The sort is
count, scan and scatter, and the scan one launch up to 65536 counters, three
beyond; then per plane group the gridder's two and the stack (2D plan).  A
replayed graph counts what its capture counted."""
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


# 64^2 with tiles of side 16: 16 counters per plane
@pytest.mark.parametrize("nw,scan", [(1, 1), (4096, 1), (4097, 3)])
def test_single(rick, nw, scan):
    prob = synth.disk_problem(64, nw, 500, synth.KERNEL_KB, 5, 4.0, 50.0, 3, fill=0.4)
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    im = rick.Imager(dict(prob["params"], tile=16, flags=REAL))
    im.set_timing(True)
    im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    im.image()
    assert im.timing()["kernel_launches"] == (2 + scan) + 2 + 1
    im.set_timing(True)  # from zero
    im.degrid(torch.zeros((64, 64), device="cuda"), g["u"], g["v"], g["w"], g["wt"])
    assert im.timing()["kernel_launches"] == (2 + scan) + 2  # spread, gather
    im.close()


@pytest.mark.parametrize("n,transform", [(256, 1), (1024, 2)])
def test_batch_replay(rick, n, transform):
    nw, nchan = 4, 3
    prob = synth.channels_problem(nchan=nchan, n=n, nw=nw, m_lo=2000, m_hi=4000, device="cuda", seed=80)
    args = (prob["vis"], prob["u"], prob["v"], prob["w"], prob["wt"], prob["offsets"])
    bi = rick.BatchImager(dict(prob["params"], flags=REAL), prob["ranges"])
    out = torch.empty((nchan, n, n), device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    got = []
    with torch.cuda.stream(s):
        for graph in (False, True, True):  # direct, captured, replayed
            bi.set_timing(True)
            bi.images(*args, out=out, use_graph=graph)
            got.append(bi.timing()["kernel_launches"])
    torch.cuda.synchronize()
    bi.close()
    # the sort, the tiles' marking (two-pass transform), the gridder, the transform and stack
    assert got == [3 + (n == 1024) + 2 + transform] * 3
