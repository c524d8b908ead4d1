"""Every calibration solver at its device-side time limit.  A tolerance below
rounding keeps each channel iterating until the limit, which every thread of a
CTA has to leave on at the same pass: all channels report GC_ETIMEOUT and the
context stays usable.  More channels than fit at once for the small arrays."""
import numpy as np
import pytest

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu

STOP = dict(tol=1e-300, max_iter=10 ** 9, time_limit_ms=3)


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


def sums_of(gc, scheme, L, C):
    sel = gc.Selection(scheme, L, 1024)
    pt = sel.pair_type()
    sums, _, _ = synth.make_visibilities(30 + L, L, C, sel.pair_i, sel.pair_j, pt, sel.n_ubl,
                                         (sel.win_t1 - sel.win_t0)[pt], device="cuda")
    return sel, sums


def check(gc, ctx, stats, redo):
    with pytest.raises(gc.GridcorrError) as e:
        ctx.device_status()
    assert e.value.status == gc.GC_ETIMEOUT
    for st in stats:
        assert np.all(gc.decode_stats(st)["status"] == gc.GC_ETIMEOUT)
    for st in redo():   # cleared, and the context still works
        assert np.all(gc.decode_stats(st)["status"] == gc.GC_OK)
    ctx.device_status()


@pytest.mark.parametrize("solver,scheme,L,C,operator,precision", [
    ("lincal", "subset", 8, 700, 0, "fp64"),
    ("lincal", "subset", 8, 700, 0, "fp32"),
    ("lincal", "subset", 33, 20, 0, "fp64"),
    ("lincal", "subset", 41, 3, 0, "fp64"),
    ("lincal_cg", "subset", 8, 700, 0, "fp32"),
    ("lincal_cg", "lowcad", 8, 700, 0, "fp32"),
    ("lincal_cg", "lowcad", 8, 700, 1, "fp32"),
    ("omnical", "subset", 8, 700, 0, "fp32"),
])
def test_one_array(gc, solver, scheme, L, C, operator, precision):
    sel, sums = sums_of(gc, scheme, L, C)
    ctx = gc.Context(0)
    ctx.set_tuning("cal.operator", operator)
    _, _, st = ctx.calibrate(sums, sel, solver=solver, precision=precision, **STOP)
    check(gc, ctx, [st], lambda: [ctx.calibrate(sums, sel, solver=solver, precision=precision)[2]])


def test_batched(gc):
    ctx = gc.Context(0)
    arrays = [dict(zip(("sel", "vred"), sums_of(gc, scheme, L, C)))
              for scheme, L, C in (("subset", 8, 400), ("subset", 16, 40), ("lowcad", 6, 200))]
    out = ctx.calibrate_batched(arrays, **STOP)
    check(gc, ctx, [o[2] for o in out], lambda: [o[2] for o in ctx.calibrate_batched(arrays)])
