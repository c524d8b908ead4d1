"""Matrix-free solver over few baseline-types: channels with an SM each (512
antennas and more) take a wider kernel than many channels do.  Both stop at
relative steps of 1e-6 on equations whose FP32 residuals carry about 1e-6:
the same channels, calibrated alone and among 200, agree to 3e-5.  Sides around
the first that takes it, an odd number of antennas, a grid whose vectors fit in
shared memory and one whose do not."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


@pytest.mark.parametrize("L", [7, 22, 23, 32, 47, 64])
def test_few_channels_as_among_many(gc, L):
    sel = gc.Selection("subset", L, 4096)
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(60 + L, L, 2, sel.pair_i, sel.pair_j, pt, sel.n_ubl,
                                         (sel.win_t1 - sel.win_t0)[pt], device="cuda")
    out = []
    for rep in (1, 100):
        ctx = gc.Context(0)
        g, V, st = ctx.calibrate(sums.repeat(rep, 1), sel, solver="lincal_cg")
        ctx.device_status()
        s = gc.decode_stats(st)
        assert np.all(s["status"] == gc.GC_OK)
        out.append((g[:2].cpu().numpy(), V[:2].cpu().numpy(), s["chi2"][:2]))
    (g, V, x), (h, W, y) = out
    assert np.max(np.abs(g - h) / np.abs(h)) < 3e-5
    assert np.max(np.abs(V - W)) < 3e-5 * np.max(np.abs(W))
    assert np.allclose(x, y, rtol=1e-5)
