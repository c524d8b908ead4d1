"""The direct lincal solver at the edges of its blocks: fewer antennas than a
block of 16, whole and ragged block counts, the largest band that stays in shared
memory and the first that does not, zero and rescaled warm starts.  Small arrays against
the FP64 oracle, large ones against the matrix-free solver.  Tolerances: the
gains are binary32 (rounding 6e-8, 1e-6 with margin for the oracle's own
convergence); the FP32 form stops at steps of 1e-6 and the matrix-free solver
at the same, on systems that amplify a gradient error by a few tens."""
import numpy as np
import pytest
import torch

from oracle import calib as oc
from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


@pytest.fixture(scope="module")
def ctx(gc):
    return gc.Context(0)


def _problem(gc, L, C, T=2048):
    sel = gc.Selection("subset", L, T)
    pt = sel.pair_type()
    tp = (sel.win_t1 - sel.win_t0)[pt]
    sums, gains, V = synth.make_visibilities(70 + L, L, C, sel.pair_i, sel.pair_j, pt, sel.n_ubl, tp)
    return sel, pt, tp, sums


def _rel(a, b):
    return float(np.max(np.abs(a - b) / np.abs(b)))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-6), ("fp32", 1e-4)])
@pytest.mark.parametrize("L,C", [(3, 3), (4, 5), (5, 1), (8, 2), (11, 2), (16, 2), (17, 1)])
def test_matches_oracle(gc, ctx, L, C, precision, tol):
    sel, pt, tp, sums = _problem(gc, L, C)
    g, V, st = ctx.calibrate(sums.cuda(), sel, solver="lincal", precision=precision)
    ctx.device_status()
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    for c in range(C):
        ref, Vr, _, ok = oc.calibrate(sums[c].numpy().astype(np.complex128) / tp, sel.pair_i, sel.pair_j, pt,
                                      [tuple(t) for t in sel.types.tolist()], L,
                                      "lincal")
        assert ok
        assert _rel(g[c].cpu().numpy().astype(np.complex128), ref) < tol
        assert _rel(V[c].cpu().numpy().astype(np.complex128), Vr) < tol


@pytest.mark.parametrize("L", [32, 39, 40, 41, 49])
def test_large_bands_match_matrix_free(gc, ctx, L):
    sel, pt, tp, sums = _problem(gc, L, 3)
    v = sums.cuda()
    g, V, st = ctx.calibrate(v, sel, solver="lincal")
    h, W, su = ctx.calibrate(v, sel, solver="lincal_cg")
    ctx.device_status()
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK) and np.all(gc.decode_stats(su)["status"] == gc.GC_OK)
    assert _rel(h.cpu().numpy(), g.cpu().numpy()) < 3e-5
    assert _rel(W.cpu().numpy(), V.cpu().numpy()) < 3e-5


def test_warm_starts_with_zero_and_rescaled_values(gc, ctx):
    """A zero gain and a zero visibility are left by the first step; gains of
    another overall scale and data far from unity change nothing."""
    L = 12
    sel, pt, tp, sums = _problem(gc, L, 2)
    v = sums.cuda()
    g, V, _ = ctx.calibrate(v, sel, solver="lincal")
    ref = g.cpu().numpy()
    g0, V0 = g.clone(), V.clone()
    g0[:, 17] = 0
    V0[:, 3] = 0
    h, _, st = ctx.calibrate(v, sel, solver="lincal", warm_start=True, gains=g0, vmodel=V0)
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    assert _rel(h.cpu().numpy(), ref) < 1e-6
    h, _, st = ctx.calibrate(v, sel, solver="lincal", warm_start=True, gains=g * 1e-6, vmodel=V * 1e12)
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    assert _rel(h.cpu().numpy(), ref) < 1e-6
    h, _, st = ctx.calibrate(v * 1e-20, sel, solver="lincal")
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    assert _rel(h.cpu().numpy(), ref) < 1e-6
