"""The pair-list X-engine with few channels, where windows are cut into many short
time slices and into several blocks: every format against sums in FP64 (4+4 bits
exactly; floating point within 1e-5 sqrt(A_i A_j) of the window), with and
without autocorrelations, which must not change the sums."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["c64", "c32h", "i4c"])
@pytest.mark.parametrize("L,C,T,hexside", [(3, 8, 4096, 0), (5, 1, 8192, 0), (6, 4, 3001, 0), (8, 1, 8192, 0), (11, 1, 256, 0),
                                           (16, 1, 1000, 0), (24, 1, 4096, 0), (32, 1, 256, 0), (32, 1, 4100, 0), (0, 1, 3000, 4)])
def test_few_channels(fmt, L, C, T, hexside):
    from paper_2005_03060_gb300 import gridcorr
    if hexside:
        L, mask = synth.hex_mask(hexside)
        sel = gridcorr.Selection("lowcad", L, T, mask=mask, lattice="triangular")
    else:
        sel = gridcorr.Selection("lowcad", L, T)
    g = torch.Generator(device="cuda").manual_seed(7 * L + T)
    if fmt == "i4c":
        re, im = (torch.randint(-8, 8, (C, T, L * L), generator=g, device="cuda") for _ in range(2))
        v = (((re & 15) << 4) | (im & 15)).to(torch.uint8)
        held = torch.complex(re.double(), im.double())
    else:
        x = torch.randn(C, T, L * L, 2, generator=g, device="cuda")
        v = torch.view_as_complex(x) if fmt == "c64" else x.half()
        held = torch.view_as_complex(x.double() if fmt == "c64" else v.double())
    ctx = gridcorr.Context(0)
    out, autos = ctx.reduce(v, sel)
    alone = ctx.reduce(v, sel, autos=False)
    ctx.device_status()
    assert torch.equal(alone, out)
    pt = torch.as_tensor(sel.pair_type(), device="cuda").long()
    pi, pj = (torch.as_tensor(a, device="cuda").long() for a in (sel.pair_i, sel.pair_j))
    win = torch.as_tensor(sel.win_t0 // sel.t_int, device="cuda")[pt]
    total = torch.zeros(C, L * L, dtype=torch.float64, device="cuda")
    for w in range(sel.n_cycle):
        s = held[:, w * sel.t_int:(w + 1) * sel.t_int]
        m = torch.einsum("cti,ctj->cij", s, s.conj())
        a = torch.diagonal(m, dim1=1, dim2=2).real
        total += a
        q = torch.nonzero(win == w).flatten()
        ref, got = m[:, pi[q], pj[q]], out[:, q]
        if fmt == "i4c":
            assert torch.equal(got.double(), torch.view_as_real(ref).round())
        else:
            assert float(((got - ref).abs() / (a[:, pi[q]] * a[:, pj[q]]).sqrt()).max()) < 1e-5
    if fmt == "i4c":
        assert torch.equal(autos.double(), total.round())
    else:
        assert float(((autos - total).abs() / total).max()) < 1e-5
