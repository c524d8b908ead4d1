"""Kernels that walk several work items: what a CTA leaves of one must not reach
the next.  Channels repeat a few different ones, many more than fit the chip at
once, so that a CTA's consecutive items differ; each repetition has the bits of
the first (the pair-list X-engine, the direct solver) or the solution of its
channel alone (the lag planes, whose sums are not ordered: 3e-5 between two
runs that stop at relative steps of 1e-6)."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu

D = 7   # different channels


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


def tile(x, C):
    return x[torch.arange(C, device=x.device) % x.shape[0]].contiguous()


def repeats(x, n=D):
    """Every channel equal, bit for bit, to the first with its data."""
    b = torch.view_as_real(x) if x.is_complex() else x
    return torch.equal(b, tile(b[:n], b.shape[0]))


@pytest.mark.parametrize("autos", [True, False])
@pytest.mark.parametrize("fmt", ["c64", "c32h", "i4c"])
@pytest.mark.parametrize("L,C,T,hexside", [(5, 3000, 60, 0), (8, 1500, 130, 0), (17, 300, 400, 0), (0, 1500, 90, 4)])
def test_xengine_lists(gc, fmt, L, C, T, hexside, autos):
    if hexside:
        L, mask = synth.hex_mask(hexside)
        sel = gc.Selection("lowcad", L, T, mask=mask, lattice="triangular")
    else:
        sel = gc.Selection("lowcad", L, T)
    g = torch.Generator(device="cuda").manual_seed(L + T)
    if fmt == "i4c":
        v = torch.randint(0, 256, (D, T, L * L), generator=g, device="cuda", dtype=torch.uint8)
    else:
        x = torch.randn(D, T, L * L, 2, generator=g, device="cuda")
        v = torch.view_as_complex(x) if fmt == "c64" else x.half()
    ctx = gc.Context(0)
    out = ctx.reduce(tile(v, C), sel, autos=autos)
    few = ctx.reduce(v, sel, autos=autos)
    ctx.device_status()
    out, few = (out, few) if autos else ((out,), (few,))
    for a, b in zip(out, few):
        assert repeats(a)
        if fmt == "i4c":
            assert torch.equal(a[:D], b)
        else:   # fewer channels may be split in time: other order, FP32 sums of up to T products
            assert (a[:D] - b).abs().max() <= 1e-5 * b.abs().max()


def sums_of(gc, scheme, L):
    sel = gc.Selection(scheme, L, 1024)
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(20 + L, L, D, sel.pair_i, sel.pair_j, pt, sel.n_ubl,
                                         (sel.win_t1 - sel.win_t0)[pt], device="cuda")
    return sel, sums


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("L,C", [(3, 3000), (8, 2000), (12, 900), (21, 400), (41, 200)])
def test_direct_solver(gc, L, C, precision):
    sel, sums = sums_of(gc, "subset", L)
    ctx = gc.Context(0)
    g, V, st = ctx.calibrate(tile(sums, C), sel, solver="lincal", precision=precision)
    h, W, _ = ctx.calibrate(sums, sel, solver="lincal", precision=precision)
    ctx.device_status()
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    assert repeats(g) and repeats(V)
    assert torch.equal(torch.view_as_real(g[:D]), torch.view_as_real(h))
    assert torch.equal(torch.view_as_real(V[:D]), torch.view_as_real(W))


# (from 153 channels on the smaller of these arrays run two CTAs of half the threads an SM)
@pytest.mark.parametrize("L,C", [(4, 800), (8, 800), (9, 153), (16, 400), (24, 200)])
def test_lag_planes(gc, L, C):
    sel, sums = sums_of(gc, "lowcad", L)
    ctx = gc.Context(0)
    g, V, st = ctx.calibrate(tile(sums, C), sel, solver="lincal_cg")
    h, W, _ = ctx.calibrate(sums, sel, solver="lincal_cg")
    ctx.device_status()
    assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    h, W = tile(h, C), tile(W, C)
    assert float(((g - h).abs() / h.abs()).max()) < 3e-5
    assert float((V - W).abs().max() / W.abs().max()) < 3e-5
