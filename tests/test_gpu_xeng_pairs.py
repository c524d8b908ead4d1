"""The pair-list X-engine (selections with several windows) at the edges of its
tiles: entries per thread and blocks per window (small and large grids),
grid samples that bulk copies cannot take, windows split into time slices,
ragged stages, with and without autos, full and partly occupied lattices.
4+4-bit sums are compared bit for bit; floating-point sums with the bound of
the X-engine tests, |dS_p| <= 1e-5 sqrt(A_i A_j)."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


@pytest.fixture(scope="module")
def ctx(gc):
    return gc.Context(0)


def _selection(gc, L, T, hexside):
    if hexside:
        L, mask = synth.hex_mask(hexside)
        return gc.Selection("lowcad", L, T, mask=mask, lattice="triangular")
    return gc.Selection("lowcad", L, T)


# (L, C, T, side of a hexagon or 0): one warp of entries; a grid sample of 25
# elements (plain staging); several slices per window (few channels, long
# windows); 11264 entries per window; 12 windows of unequal entry counts
CASES = [(4, 3, 130, 0), (5, 2, 333, 0), (8, 1, 6000, 0), (32, 1, 520, 0), (17, 2, 700, 0), (0, 2, 411, 4)]


@pytest.mark.parametrize("fmt", ["c64", "c32h", "i4c"])
@pytest.mark.parametrize("L,C,T,hexside", CASES)
def test_lists_match_oracle(gc, ctx, orc, fmt, L, C, T, hexside):
    sel = _selection(gc, L, T, hexside)
    assert sel.n_cycle > 1
    N = sel.L * sel.L
    rng = np.random.default_rng(31 * N + T)
    pt = sel.pair_type()
    t0, t1 = sel.win_t0[pt], sel.win_t1[pt]
    used = sel.n_cycle * sel.t_int
    if fmt == "i4c":
        re, im = rng.integers(-8, 8, (C, T, N)), rng.integers(-8, 8, (C, T, N))
        v = torch.from_numpy((((re & 15) << 4) | (im & 15)).astype(np.uint8)).cuda()
        held = re + 1j * im
    else:
        x = (rng.standard_normal((C, T, N)) + 1j * rng.standard_normal((C, T, N))).astype(np.complex64)
        v = torch.from_numpy(x).cuda()
        held = x.astype(np.complex128)
        if fmt == "c32h":
            v = torch.view_as_real(v).half().contiguous()
            held = torch.view_as_complex(v.double()).cpu().numpy()
    vr, au = ctx.reduce(v, sel)
    alone = ctx.reduce(v, sel, autos=False)
    ctx.device_status()
    assert torch.equal(alone, vr)
    vr, au = vr.cpu().numpy(), au.cpu().numpy()
    for c in range(C):
        a = np.sum(np.abs(held[c][:used]) ** 2, axis=0)
        if fmt == "i4c":
            ref = orc.xengine_i4c(v[c].cpu().numpy(), sel.pair_i, sel.pair_j, t0, t1)
            assert np.array_equal(vr[c].astype(np.int64), ref)
            assert np.array_equal(au[c].astype(np.int64), np.rint(a).astype(np.int64))
        else:
            ref = orc.xengine_c64(held[c], sel.pair_i, sel.pair_j, t0, t1)
            aw = {w: np.sum(np.abs(held[c][w * sel.t_int:(w + 1) * sel.t_int]) ** 2, axis=0) for w in range(sel.n_cycle)}
            w = t0 // sel.t_int
            bound = np.sqrt(np.array([aw[k][i] * aw[k][j] for k, i, j in zip(w, sel.pair_i, sel.pair_j)]))
            assert np.max(np.abs(vr[c] - ref) / bound) < TOL
            assert np.max(np.abs(au[c] - a) / a) < TOL
