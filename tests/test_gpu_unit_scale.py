"""The matrix-free solver on data and starts far from unity, through the lag planes
and the gather over the grid: visibilities scaled by s have the same gains and
scaled models, and a warm start may split them otherwise between gains and
visibilities.  Tolerances of two converged runs (3e-5); chi^2 scales with s^2 and
keeps its FP32 residuals' accuracy."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


@pytest.fixture(scope="module", params=["subset 12", "subset 40", "lowcad 6", "lowcad 9", "lowcad 24", "hexagon 3", "hexagon 5"])
def problem(gc, request):
    kind, n = request.param.split()
    n = int(n)
    if kind == "hexagon":
        L, mask = synth.hex_mask(n)
        sel = gc.Selection("lowcad", L, 4096, mask=mask, lattice="triangular")
    else:
        L, mask = n, None
        sel = gc.Selection(kind, L, 4096)
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(60 + L, L, 2, sel.pair_i, sel.pair_j, pt, sel.n_ubl,
                                         (sel.win_t1 - sel.win_t0)[pt], device="cuda")
    occ = np.arange(L * L) if mask is None else np.flatnonzero(np.asarray(mask).reshape(-1))
    ctx = gc.Context(0)
    g, V, st = ctx.calibrate(sums, sel, solver="lincal_cg")
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    return ctx, sel, sums, occ, g, V, st


def same(gc, problem, out, s=1.0):
    ctx, sel, sums, occ, g, V, st = problem
    h, W, su = out
    ctx.device_status()
    su = gc.decode_stats(su)
    assert np.all(su["status"] == gc.GC_OK)
    ref, h = g.cpu().numpy()[:, occ], h.cpu().numpy()[:, occ]
    assert np.max(np.abs(h - ref) / np.abs(ref)) < 3e-5
    Vref = V.cpu().numpy().astype(np.complex128)
    assert np.max(np.abs(W.cpu().numpy() / s - Vref)) < 3e-5 * np.max(np.abs(Vref))
    assert np.allclose(su["chi2"] / s / s, gc.decode_stats(st)["chi2"], rtol=1e-4)


@pytest.mark.parametrize("s", [1e-20, 1e-13, 1e-7, 1e-3, 1e2, 1e3, 3e4, 1e6, 1e12])
def test_scaled_data(gc, problem, s):
    ctx, sel, sums = problem[:3]
    same(gc, problem, ctx.calibrate(sums * s, sel, solver="lincal_cg"), s)


@pytest.mark.parametrize("a", [1e-9, 1e-3, 0.1, 30.0, 1e3, 1e9])
def test_rescaled_warm_start(gc, problem, a):
    ctx, sel, sums, _, g, V, _ = problem
    same(gc, problem, ctx.calibrate(sums, sel, solver="lincal_cg", warm_start=True, gains=g * a, vmodel=V / a / a))


def test_scaled_data_and_no_visibilities(gc, problem):
    ctx, sel, sums, _, g, V, _ = problem
    same(gc, problem, ctx.calibrate(sums * 1e-20, sel, solver="lincal_cg", warm_start=True, gains=g.clone(),
                                    vmodel=torch.zeros_like(V)), 1e-20)
