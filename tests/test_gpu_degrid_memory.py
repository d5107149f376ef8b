"""Prediction with most of the device's memory held: the sorted measurements
(20 bytes each) where they fit, else their indices (4 bytes), and the same again
at the second call, whose scratch the handle's pool still holds (which
cudaMemGetInfo counts as used).

The limits are the library's own: the scratch and 64 MB have to fit.  m =
2e7: 400 MB of entries, 80 MB of indices, tile offsets far below 1 MB.  With F
bytes free, entries are taken at the first call from 464 MB on; what they leave
free at the second is F - 400 MB, less than indices and reserve (144 MB) at the
500 MB of the first case."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

M = 20_000_000


@pytest.mark.parametrize("free_mb", [500, 300])
def test_repeated_predict(free_mb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as rick
    n, nw = 256, 4
    prob = synth.disk_problem(n, nw, 1000, synth.KERNEL_KB, 7, 4.0, 60.0, 77, fill=0.4)
    im = rick.Imager(dict(prob["params"], flags=synth.FLAG_REAL))
    u, v, w = (prob[k].cuda().repeat(M // 1000) for k in "uvw")
    model = torch.randn((n, n), generator=torch.Generator().manual_seed(9)).cuda()
    want = im.predict(model, *(x[:1000].contiguous() for x in (u, v, w))).clone()  # short list: row by row
    outs = [torch.zeros(M, dtype=torch.complex64, device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = []
    try:
        free, _ = torch.cuda.mem_get_info()
        hold.append(torch.empty(free - free_mb * 1_000_000, dtype=torch.uint8, device="cuda"))
        free, _ = torch.cuda.mem_get_info()
        assert abs(free - free_mb * 1_000_000) < 30_000_000
        for out in outs:
            im.predict(model, u, v, w, out=out)
            torch.cuda.synchronize()
    finally:
        hold.clear()
        torch.cuda.empty_cache()
        im.close()
    for out in outs:
        # two orders of summation of the same 49 binary32 terms: a few ulp of the largest value
        assert (out.view(-1, 1000) - want).abs().max().item() <= 1e-5 * want.abs().max().item()
