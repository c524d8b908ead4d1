"""Warm starts of the matrix-free solver with elements of exactly zero: one
visibility, all of them, a gain, several gains, gains and visibilities at once,
through the lag planes, the gather over the grid and the pair list.  All reach the
solution that a start without zeros reaches: gains and visibilities agree to 3e-5
(both runs stop at relative steps of 1e-6 on equations whose FP32 residuals
carry about 1e-6)."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu

STARTS = {
    "one visibility": ([], [3]),
    "all visibilities": ([], slice(None)),
    "one gain": ([17], []),
    "gains": ([0, 17, 18, 40], []),
    "gains and visibilities": ([5, 41], [0, 1, 4]),
}


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


def problem(gc, kind):
    if kind == "hexagon":
        L, mask = synth.hex_mask(5)
        sel = gc.Selection("lowcad", L, 4096, mask=mask, lattice="triangular")
    else:
        L, mask = (12 if kind == "subset" else 9), None
        sel = gc.Selection(kind, L, 4096)
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(60 + L, L, 3, sel.pair_i, sel.pair_j, pt, sel.n_ubl,
                                         (sel.win_t1 - sel.win_t0)[pt], device="cuda")
    occ = np.arange(L * L) if mask is None else np.flatnonzero(np.asarray(mask).reshape(-1))
    return sel, sums, occ


@pytest.mark.parametrize("start", list(STARTS))
@pytest.mark.parametrize("kind,operator", [("lowcad", 0), ("lowcad", 1), ("hexagon", 0), ("hexagon", 1),
                                           ("subset", 0), ("subset", 1)])
def test_zeros_are_left(gc, kind, operator, start):
    sel, sums, occ = problem(gc, kind)
    ctx = gc.Context(0)
    ctx.set_tuning("cal.operator", operator)
    g, V, _ = ctx.calibrate(sums, sel, solver="lincal_cg")
    ref, Vref = g.cpu().numpy(), V.cpu().numpy()
    ants, vis = STARTS[start]
    g0, V0 = g.clone(), V.clone()
    g0[1:, torch.as_tensor(occ[ants], device="cuda")] = 0   # channel 0 keeps its gains
    V0[1:, vis] = 0
    h, W, st = ctx.calibrate(sums, sel, solver="lincal_cg", warm_start=True, gains=g0, vmodel=V0)
    ctx.device_status()
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    h, W = h.cpu().numpy(), W.cpu().numpy()
    assert np.max(np.abs(h - ref)[:, occ] / np.abs(ref)[:, occ]) < 3e-5
    assert np.max(np.abs(W - Vref)) < 3e-5 * np.max(np.abs(Vref))
