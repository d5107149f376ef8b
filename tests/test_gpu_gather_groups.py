"""The gather's rule goes by a plane group's share of the measurements: shares of
2^18 and more by columns, shorter ones row by row, w-footprints across groups
included.  Every prediction of a long list against the same handle's of its first
thousand measurements (row by row): two orders of summation of the same binary32
terms, a few ulp of the largest value."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [4, 7, 8])
@pytest.mark.parametrize("m,group,w_support,tile", [(3 * (1 << 18) + 33, 2, 3, 64), (3 * (1 << 18) + 33, 2, 0, 16),
                                                    (3 * (1 << 18) - 300, 2, 3, 32), (1 << 18, 1, 0, 32)])
def test_shares(S, m, group, w_support, tile):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    n, nw = 130, 6
    prob = synth.disk_problem(n, nw, m, synth.KERNEL_KB, S, 4.0, 60.0, 760 + S, fill=0.5)
    u, v, w = (prob[k].cuda() for k in "uvw")
    im = rick.Imager(dict(prob["params"], flags=synth.FLAG_REAL, plane_group=group, w_support=w_support, tile=tile))
    model = torch.randn((n, n), generator=torch.Generator().manual_seed(S)).cuda()
    want = im.predict(model, u[:1000].contiguous(), v[:1000].contiguous(), w[:1000].contiguous()).clone()
    got = im.predict(model, u, v, w)
    im.close()
    assert (got[:1000] - want).abs().max().item() <= 1e-5 * want.abs().max().item()
    assert torch.isfinite(torch.view_as_real(got)).all()
