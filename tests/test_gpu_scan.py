"""The counting sort's scan at the counts where its paths meet: a part of one
tile of counters, whole tiles of the cluster's CTAs and one past them, and one
past the largest count the single launch takes.  With normalised taps the cells
of a plane sum to the weighted visibilities on it, which a wrong offset (an
entry gridded on another tile's plane, or lost) breaks; binary32 taps sum to 1
to ~1e-6, the bound is 1e-5 of the plane's sum of moduli."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw", [1, 255, 256, 257, 2048, 2049, 4096, 4097, 8192, 8193])
def test_plane_sums(nw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    n, m = 64, 4000  # 16 tiles of side 16 per plane
    prob = synth.disk_problem(n, nw, m, synth.KERNEL_KB, 5, 4.0, 50.0, 800 + nw, fill=0.4, weights="random")
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    im = rick.Imager(dict(prob["params"], tile=16, flags=synth.FLAG_REAL, plane_group=1))
    im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    assert im.stats()["n_gridded"] == m
    got = torch.cat([im.grid_planes(k, min(512, nw - k)).to(torch.complex128).sum((1, 2)) for k in range(0, nw, 512)])
    im.close()
    lo = torch.tensor(prob["params"]["w_min"], dtype=torch.float32)
    inv = torch.tensor(nw / (prob["params"]["w_max"] - prob["params"]["w_min"]), dtype=torch.float32)
    k = ((prob["w"] - lo) * inv).floor().clamp(0, nw - 1).long().cuda() if nw > 1 else torch.zeros(m, dtype=torch.long).cuda()
    x = g["vis"].to(torch.complex128) * g["wt"].double()
    want = torch.zeros(nw, dtype=torch.complex128, device="cuda").index_add_(0, k, x)
    size = torch.zeros(nw, dtype=torch.float64, device="cuda").index_add_(0, k, x.abs())
    assert ((got - want).abs() <= 1e-5 * size + 1e-30).all()
