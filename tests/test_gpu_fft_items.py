"""More work items than resident CTAs in the FFT-correlator, so that each CTA
takes several in a row: what an item leaves on the chip must not reach the
next.  Every channel holds the same voltages and gains, so all spectra have the
same bits; the first is checked against the FP64 oracle within the lag-sum bound of
the FP32 path.  Grids short of their FFT configuration's largest side and, for
each configuration, that side."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def lag_err(got, ref, nd, n):
    return float(np.max(np.abs(got - ref) * nd) / (n * abs(ref[ref.shape[0] // 2, ref.shape[1] // 2])))


def pair_counts(mask, L):
    m = mask.reshape(L, L).astype(float)
    f = np.abs(np.fft.fft2(m, (2 * L, 2 * L))) ** 2
    return np.round(np.fft.fftshift(np.fft.ifft2(f).real)[1:, 1:])


@pytest.fixture(scope="module")
def gridcorr():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr


def draw(orc, fmt, L, T):
    """One channel's voltages in `fmt`, what the format holds of them, its gains."""
    volt, gains, _ = synth.make_voltages(800 + L, L, 1, T, n_src=20)
    if fmt == "i4c":
        v = torch.from_numpy(orc.quantize(volt[0].numpy())[0])[None]
        held = orc.unpack_i4c(v[0].numpy())
    elif fmt == "c32h":
        v = torch.view_as_real(volt).to(torch.float16).contiguous()
        held = torch.view_as_complex(v[0].to(torch.float64)).numpy()
    else:
        v, held = volt, volt[0].numpy()
    return v, held, gains


def repeat(x, C):
    return x.cuda().expand(C, *x.shape[1:]).contiguous()


def check(out, ref, nd, n):
    bits = torch.view_as_real(out)
    assert torch.equal(bits, bits[:1].expand_as(bits))
    assert lag_err(out[0].cpu().numpy(), ref, nd, n) < TOL


SIZES = [(1, 4000), (3, 4000), (7, 4000), (8, 4000), (9, 4000), (13, 4000), (16, 4000), (21, 2000), (32, 1000), (33, 400),
         (37, 400), (63, 300), (64, 300)]


@pytest.mark.parametrize("L,C", SIZES)
@pytest.mark.parametrize("fmt", ["c64", "c32h", "i4c"])
def test_channels_agree(gridcorr, orc, fmt, L, C):
    T = 18 if L > 1 else 20
    v, held, gains = draw(orc, fmt, L, T)
    ctx = gridcorr.Context(0)
    g, v = repeat(gains, C), repeat(v, C)
    ref = orc.fx(held, gains[0].numpy(), L)
    r = L - np.abs(np.arange(-(L - 1), L))
    nd = r[:, None] * r[None, :]
    for path, shape in ((0, 0), (1, 0), (1, 1)):   # path 1: the CUDA cores for 4+4 bits too
        ctx.set_tuning("fft.path", path)
        ctx.set_tuning("fft.shape", shape)
        out = ctx.correlate(v, g)
        ctx.device_status()
        check(out, ref, nd, L * L)
    f = gridcorr.lib().gc_correlate_noalloc
    f.argtypes = [ctypes.c_void_p] + [ctypes.c_int] * 4 + [ctypes.c_void_p] * 4
    f.restype = ctypes.c_int
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.empty_like(out)
    st = f(v.data_ptr(), {"c64": 0, "i4c": 1, "c32h": 2}[fmt], L, C, T, g.data_ptr(), out.data_ptr(), status.data_ptr(),
           torch.cuda.current_stream().cuda_stream)
    assert st == gridcorr.GC_OK and int(status.item()) == 0
    check(out, ref, nd, L * L)


@pytest.mark.parametrize("side,C", [(2, 4000), (4, 4000), (7, 4000), (11, 2000), (19, 300)])
@pytest.mark.parametrize("fmt", ["c64", "c32h", "i4c"])
def test_masked_channels_agree(gridcorr, orc, fmt, side, C):
    L, mask = synth.hex_mask(side)
    v, held, gains = draw(orc, fmt, L, 18)
    ctx = gridcorr.Context(0)
    out = ctx.correlate(repeat(v, C), repeat(gains, C), mask=mask)
    ctx.device_status()
    occ = np.asarray(mask).reshape(-1).astype(bool)
    nd = pair_counts(occ, L)
    sums = orc.fx(np.where(occ, held, 0), gains[0].numpy(), L)
    r = L - np.abs(np.arange(-(L - 1), L))
    ref = sums * (r[:, None] * r[None, :]) / np.maximum(nd, 1)   # means over the pairs that are there
    check(out, ref, nd, int(occ.sum()))
