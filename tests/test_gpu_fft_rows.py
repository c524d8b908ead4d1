"""Ragged voltage rows of the FFT-correlator: aligned tensors are staged with
bulk copies and split into rows on the chip, tensors whose base is not a
multiple of 16 bytes with plain loads; both give the same bits, within the lag-sum
bound of the FP32 path of the FP64 oracle.  Row lengths around the kernels'
sizes, sample counts that leave a part of a stage, and channel counts that the
finalising kernel's tiles do not divide."""
import numpy as np
import pytest
import torch

from paper_2005_03060_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def lag_err(got, ref, L):
    N = L * L
    r = np.arange(-(L - 1), L)
    nd = (L - np.abs(r))[:, None] * (L - np.abs(r))[None, :]
    return float(np.max(np.abs(got - ref) * nd) / (N * abs(ref[L - 1, L - 1])))


@pytest.fixture(scope="module")
def gc():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr.Context(0)


@pytest.mark.parametrize("fmt,L,C,T", [
    ("c64", 17, 3, 1), ("c64", 19, 2, 33), ("c64", 31, 3, 257), ("c64", 33, 1, 7), ("c64", 63, 1, 5),
    ("c32h", 17, 2, 3), ("c32h", 21, 3, 130), ("c32h", 31, 1, 257), ("c32h", 33, 2, 9), ("c32h", 62, 1, 4),
    ("i4c", 17, 3, 5), ("i4c", 21, 2, 131), ("i4c", 32, 5, 64), ("i4c", 33, 1, 9), ("i4c", 63, 1, 6),
    ("i4c", 65, 1, 3), ("i4c", 101, 1, 5), ("i4c", 127, 1, 2), ("i4c", 128, 1, 3)])
def test_bulk_rows(gc, orc, fmt, L, C, T):
    volt, gains, _ = synth.make_voltages(700 + L, L, C, T, n_src=20)
    if fmt == "i4c":
        v = torch.from_numpy(np.stack([orc.quantize(x.numpy())[0] for x in volt])).cuda()
        held = [orc.unpack_i4c(x) for x in v.cpu().numpy()]
    elif fmt == "c32h":
        v = torch.view_as_real(volt).to(torch.float16).contiguous().cuda()
        held = list(torch.view_as_complex(v.cpu().to(torch.float64)).numpy())
    else:
        v = volt.cuda()
        held = list(volt.numpy())
    g = gains.cuda()
    off = 2 if fmt == "c32h" else 1   # one voltage past a 16-byte boundary
    flat = torch.empty(v.numel() + off, dtype=v.dtype, device=v.device)
    moved = flat[off:].view(v.shape)
    moved.copy_(v)
    got, same = gc.correlate(v, g), gc.correlate(moved, g)
    gc.device_status()
    assert torch.equal(torch.view_as_real(got), torch.view_as_real(same))
    for c in range(C):
        assert lag_err(got[c].cpu().numpy(), orc.fx(held[c], gains[c].numpy(), L), L) < TOL, c
