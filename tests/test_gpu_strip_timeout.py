"""The error path of k_colimage's bounded waits: the host-set hook leaves the copy
of one plane's slot out, so that every thread block's wait on it runs out after
2 ms; the next stats query reports RICK_ERR_TIMEOUT (no hang), and after a reset
the same handle images correctly again.  The first slot, and one in a later run
of planes, when the stages have been through several phases."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

REAL = synth.FLAG_REAL


@pytest.mark.parametrize("n,nw,slot", [(1024, 12, 0), (1024, 40, 21), (2048, 5, 4), (4096, 3, 1)])
def test_times_out_and_recovers(n, nw, slot):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    prob = synth.config2(m=50000, n=n, nw=nw)
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    ref = rick.Imager(dict(prob["params"], flags=REAL | rick.FFT_2D))
    ref.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    want = ref.image().clone()
    ref.close()
    im = rick.Imager(dict(prob["params"], flags=REAL))
    im.debug_colstack(slot, 2_000_000)
    im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    im.image()
    torch.cuda.synchronize()
    with pytest.raises(rick.RickError) as exc:
        im.stats()
    assert exc.value.status == 5  # RICK_ERR_TIMEOUT
    im.debug_colstack(-1, 0)
    for _ in range(2):
        im.reset()
        im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
        got = im.image()
        im.stats()
        assert (got - want).abs().max().item() <= 1e-5 * want.abs().max().item()
    im.close()
