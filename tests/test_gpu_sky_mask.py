"""Pixels outside the sky (l^2 + m^2 >= 1) are 0 by every transform, also where
the planes' sums overflow binary32 (there the pixels inside are not finite)."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nw", [(1024, 13), (1024, 40), (2048, 2), (4096, 2), (8192, 2)])
def test_overflowing_planes(n, nw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    fov = 3.0  # radians: l^2 + m^2 = 1 lies at a third of the side from the centre
    prob = synth.disk_problem(n, nw, 20000, synth.KERNEL_KB, 7, fov * 180.0 / 3.141592653589793, 50.0, 31, fill=0.4)
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    x = (torch.arange(n, device="cuda", dtype=torch.float64) - n // 2) * prob["params"]["pixel_rad"]
    r2 = x[None, :] ** 2 + x[:, None] ** 2
    outside, inside = r2 > 1.0 + 1e-5, r2 < 1.0 - 1e-5
    assert outside.any()
    for flag in (0, rick.FFT_SPLIT, rick.FFT_2D):
        for scale in (1.0, 3e37):
            im = rick.Imager(dict(prob["params"], flags=synth.FLAG_REAL | flag))
            im.grid(g["vis"] * scale, g["u"], g["v"], g["w"], g["wt"])
            img = im.image()
            im.close()
            assert (img[outside] == 0).all()
            assert torch.isfinite(img[inside]).all() == (scale == 1.0)
