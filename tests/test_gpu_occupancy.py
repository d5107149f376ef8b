"""The marking of the non-empty tiles where several blocks take a plane (more than
256 words of tile bits: n = 4096 with tiles of 32, all of 8192 and 16384, and
side-16 tiles from 2048 on): measurements in the first, the last, one middle tile row
or none of a plane, so that the planes' ranges come from one block, from two that
are far apart, or from none; twice on one handle (the blocks' counters start at
zero again).  Against cuFFT's 2D plan, at the bounds of the other tests of two
transforms (1e-5 of the image's peak, 1e-4 for the adjoint)."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile", [(2048, 16), (4096, 32), (4096, 16), (8192, 32), (16384, 64)])
def test_rows_at_the_ends(n, tile):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    nw, m, S = 5, 400, 7
    gen = torch.Generator().manual_seed(n + tile)
    pixel = 0.02 / n
    # v rows per plane: both ends, the first, none, the last, the middle
    centre = [(S, n - S), (S, S), None, (n - S, n - S), (n // 2, n // 2)]
    k = torch.randint(0, nw, (m,), generator=gen)
    k[k == 2] = 0
    rows = torch.tensor([c or (0, 0) for c in centre], dtype=torch.float64)[k, torch.randint(0, 2, (m,), generator=gen)]
    cells = torch.rand((2, m), generator=gen, dtype=torch.float64)
    u, v = (cells[0] - 0.5) * 0.9 * n, rows + (cells[1] - 0.5) - n / 2
    w = (k + 0.5) / nw * 100.0 - 50.0
    data = [torch.complex(torch.randn(m, generator=gen), torch.randn(m, generator=gen)), (u / (n * pixel)).float(),
            (v / (n * pixel)).float(), w.float(), torch.ones(m)]
    data = [t.cuda() for t in data]
    p = dict(n=n, nw=nw, pixel_rad=pixel, w_min=-50.0, w_max=50.0, kernel=synth.KERNEL_KB, support=S, tile=tile)
    r = torch.randn((n, n), generator=torch.Generator().manual_seed(5)).cuda()
    got = []
    for flag in (0, rick.FFT_2D):
        im = rick.Imager(dict(p, flags=synth.FLAG_REAL | flag))
        for _ in range(2):
            im.reset()
            im.grid(*data)
            img = im.image().clone()
            grad = im.degrid(r, *data[1:]).clone()
        assert im.stats()["n_gridded"] == m
        im.close()
        got.append((img, grad))
    assert (got[0][0] - got[1][0]).abs().max().item() <= 1e-5 * got[1][0].abs().max().item()
    assert (got[0][1] - got[1][1]).abs().max().item() <= 1e-4 * got[1][1].abs().max().item()
