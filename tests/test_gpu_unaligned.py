"""Images that the caller provides, written (image) or read (degrid, predict), may
be aligned to their elements only: views that begin one element into a buffer
give what aligned ones give, by every transform, real and complex.  The sums are
the same ones in the same order; the bound (1e-6 of the peak) allows for the
tiles' dynamic claiming."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _shifted(t):
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    view = buf[1:].view(t.shape)
    view.copy_(t)
    assert view.data_ptr() % (2 * t.element_size()) != 0
    return view


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("n,nw,flag,group", [(256, 3, None, 0), (250, 5, None, 2), (1024, 3, "FFT_2D", 0),
                                             (2048, 4, None, 0), (2048, 4, "FFT_SPLIT", 3), (8192, 2, None, 0)])
def test_views_of_one_element_offset(n, nw, flag, group, real):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    prob = synth.disk_problem(n, nw, 3000, synth.KERNEL_KB, 7, 4.0, 60.0, n + nw, fill=0.4, weights="random")
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    flags = (synth.FLAG_REAL if real else 0) | (getattr(rick, flag) if flag else 0)
    im = rick.Imager(dict(prob["params"], flags=flags, plane_group=group))
    im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    want = im.image().clone()
    out = _shifted(torch.zeros_like(want))
    im.image(out=out)
    assert (out - want).abs().max().item() <= 1e-6 * want.abs().max().item()
    r = torch.randn((n, n), generator=torch.Generator().manual_seed(n), dtype=want.dtype).cuda()
    for call in (lambda x: im.degrid(x, g["u"], g["v"], g["w"], g["wt"]), lambda x: im.predict(x, g["u"], g["v"], g["w"])):
        a, b = call(r).clone(), call(_shifted(r)).clone()
        assert (a - b).abs().max().item() <= 1e-6 * a.abs().max().item()
    im.close()
