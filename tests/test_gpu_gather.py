"""The adjoint's gather, row by row for short lists and most supports and a lane
per footprint column for long lists of supports 4, 7 and 8 (at the first list
length that takes it, and at one that leaves the last warp a single
measurement), at footprints across tile edges and at the grid's edges, against the FP64
oracle's adjoint at the bar of the other adjoint tests (1e-4 of the largest
component); and the row-by-row gather that kernels with an amplifying grid
correction keep, with the gradient of an image in the well-conditioned centre."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

REAL, CORRECT = synth.FLAG_REAL, synth.FLAG_CORRECT


@pytest.fixture(scope="module")
def rick():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    import paper_2504_00959_gb300 as r
    r.load()
    return r


def _check(rick, oracle_mod, prob, flags, r, **extra):
    g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
    q = dict(prob["params"], flags=flags, **extra)
    im = rick.Imager(q)
    im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
    got = im.degrid(torch.from_numpy(r).cuda(), g["u"], g["v"], g["w"], g["wt"]).cpu().numpy()
    im.close()
    p = synth.to_numpy(prob)
    ref = oracle_mod.degrid(q, p["u"], p["v"], p["w"], p["wt"], p["vis"], r.astype(np.complex128),
                            flags=flags & ~REAL)
    assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref))


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 8, 9, 12, 16])
@pytest.mark.parametrize("m", [1, 33, 5000])
def test_supports(rick, oracle_mod, S, m):
    prob = synth.disk_problem(128, 3, m, synth.KERNEL_KB, S, 4.0, 60.0, 700 + S + m, fill=0.55, weights="random")
    r = np.random.default_rng(S).standard_normal((128, 128)).astype(np.float32)
    _check(rick, oracle_mod, prob, REAL, r)


@pytest.mark.parametrize("S", [4, 7, 8])
@pytest.mark.parametrize("m,flags,extra", [(1 << 18, REAL, {}), ((1 << 18) + 33, REAL | synth.FLAG_UNIFORM, {"tile": 16}),
                                           ((1 << 18) + 1, REAL, {"w_support": 3, "plane_group": 2, "tile": 64})])
def test_columns(rick, oracle_mod, S, m, flags, extra):
    prob = synth.disk_problem(130, 6, m, synth.KERNEL_KB, S, 4.0, 60.0, 760 + S, fill=0.55, weights="random")
    r = np.random.default_rng(S).standard_normal((130, 130)).astype(np.float32)
    _check(rick, oracle_mod, prob, flags, r, **extra)


@pytest.mark.parametrize("flags,extra", [(REAL | synth.FLAG_UNIFORM, {"tile": 16}),
                                         (REAL, {"w_support": 3, "plane_group": 2, "tile": 64})])
def test_weights_and_w_support(rick, oracle_mod, flags, extra):
    prob = synth.disk_problem(130, 6, 4000, synth.KERNEL_KB, 6, 4.0, 60.0, 731, fill=0.45, weights="random")
    r = np.random.default_rng(3).standard_normal((130, 130)).astype(np.float32)
    _check(rick, oracle_mod, prob, flags, r, **extra)


def test_row_order_kernel(rick, oracle_mod):
    """Gaussian support 8 with grid correction: the handle gathers row by row."""
    prob = synth.disk_problem(128, 3, 3000, synth.KERNEL_GAUSS, 8, 4.0, 60.0, 741, weights="random")
    x = (np.arange(128) - 64) / 128
    beam = np.exp(-(x / 0.1) ** 2)
    r = (np.random.default_rng(4).standard_normal((128, 128)) * np.outer(beam, beam)).astype(np.float32)
    _check(rick, oracle_mod, prob, REAL | CORRECT, r)
