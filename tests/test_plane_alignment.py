"""The gridder stores pairs of cells: planes that the caller provides must be
16-byte aligned, and a call with others is refused before any launch."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2504_00959_gb300 import build
    build.build()
    from paper_2504_00959_gb300 import _lib
    return _lib.load()


def test_static_entry_refuses(lib):
    """No GPU is touched: the refusal comes with the other argument checks."""
    from paper_2504_00959_gb300 import _lib
    p = _lib.RickParams()
    assert lib.rick_params_default(ctypes.byref(p)) == 0
    err = ctypes.create_string_buffer(256)
    for offset in (4, 8, 12):
        s = lib.rick_grid_planes_static(ctypes.byref(p), None, None, None, None, None, 0, ctypes.c_void_p(4096 + offset),
                                        None, err, 256)
        assert s == 1 and b"aligned" in err.value


@pytest.mark.gpu
def test_grid_planes_refuses(lib):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_00959_gb300 as rick
    import synth
    prob = synth.disk_problem(64, 2, 100, synth.KERNEL_KB, 5, 4.0, 50.0, 3)
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    im = rick.Imager(dict(prob["params"], flags=synth.FLAG_REAL))
    im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    buf = torch.zeros(2 * 64 * 64 + 2, dtype=torch.complex64, device="cuda")
    assert lib.rick_grid_planes(im._h, 0, 2, ctypes.c_void_p(buf.data_ptr() + 8)) == 1
    assert lib.rick_grid_planes(im._h, 0, 2, ctypes.c_void_p(buf.data_ptr() + 16)) == 0
    want = im.grid_planes()
    assert (buf[2:].view(2, 64, 64) - want).abs().max().item() <= 1e-6 * want.abs().max().item()
    im.close()
