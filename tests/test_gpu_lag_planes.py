"""The matrix-free solver's lag-plane operator (low-cadence selections) against
its pair-list operator ("cal.operator" = 1): grid sides around the eight-wide
tiles, model visibilities inside and outside the coarse space, the largest grid
whose planes fit and the first that falls back, partly occupied lattices and
warm starts.  Both stop at relative steps of 1e-6 on equations whose FP32
residuals carry about 1e-6: gains agree to 3e-5."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


def _both(gc, sel, sums, autos=None, **more):
    out = []
    for op in (0, 1):
        ctx = gc.Context(0)
        ctx.set_tuning("cal.operator", op)
        g, V, st = ctx.calibrate(sums, sel, autos, solver="lincal_cg",
                                 **{k: v.clone() if torch.is_tensor(v) else v for k, v in more.items()})
        ctx.device_status()
        s = gc.decode_stats(st)
        assert np.all(s["status"] == gc.GC_OK)
        out.append((g.cpu().numpy(), V.cpu().numpy(), s))
    return out


def _close(a, b, occ=None):
    (g, V, s), (h, W, t) = a, b
    if occ is not None:
        assert not np.any(g[:, ~occ])
        g, h = g[:, occ], h[:, occ]
    assert np.max(np.abs(g - h) / np.abs(h)) < 3e-5
    assert np.max(np.abs(V - W)) < 3e-5 * np.max(np.abs(W))
    assert np.allclose(s["chi2"], t["chi2"], rtol=1e-5)


@pytest.mark.parametrize("L,C", [(4, 3), (6, 2), (7, 2), (8, 4), (9, 1), (16, 2), (17, 2), (24, 2), (31, 1), (36, 1), (37, 1)])
def test_full_grids(gc, L, C):
    sel = gc.Selection("lowcad", L, 4096)
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(40 + L, L, C, sel.pair_i, sel.pair_j, pt, sel.n_ubl, (sel.win_t1 - sel.win_t0)[pt],
                                         device="cuda")
    a, b = _both(gc, sel, sums)
    _close(a, b)
    g, V = (torch.from_numpy(x).cuda() for x in a[:2])
    a, b = _both(gc, sel, sums, gains=g, vmodel=V, warm_start=True)
    assert np.all(a[2]["iters"] <= 3)
    _close(a, b)


@pytest.mark.parametrize("side", [3, 5, 8])
def test_hexagons(gc, side):
    L, mask = synth.hex_mask(side)
    sel = gc.Selection("lowcad", L, 4096, mask=mask, lattice="triangular")
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(90 + side, L, 2, sel.pair_i, sel.pair_j, pt, sel.n_ubl,
                                         (sel.win_t1 - sel.win_t0)[pt], device="cuda")
    a, b = _both(gc, sel, sums)
    _close(a, b, mask.astype(bool))
