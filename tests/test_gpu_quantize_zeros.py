"""The quantiser on data that is zero in places: components, samples, threads'
whole shares and channels.  Scales and bytes equal to the oracle's to the last
bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["real", "imaginary", "first half", "one sample", "every fourth", "vanishing beside zeros"])
@pytest.mark.parametrize("T,N", [(6, 4), (130, 64), (400, 1024)])
def test_zeros(orc, T, N, kind):
    from paper_2005_03060_gb300 import gridcorr
    rng = np.random.default_rng(T + N)
    x = (rng.standard_normal((2, T * N)) + 1j * rng.standard_normal((2, T * N))).astype(np.complex64)
    if kind == "real":
        x.imag = 0
    elif kind == "imaginary":
        x.real = -0.0
    elif kind == "first half":
        x[:, :T * N // 2] = 0
    elif kind == "one sample":
        x[:, :-1] = 0
    elif kind == "every fourth":
        x[:, np.arange(T * N) % 4 > 0] = 0
    else:
        x[:, ::2] = 0
        x *= np.float32(1e-22)
    x = x.reshape(2, T, N)
    q, s = gridcorr.Context(0).quantize(torch.from_numpy(x).cuda())
    for c in range(2):
        ref, sc = orc.quantize(x[c])
        assert np.float32(sc) == s[c].item()
        assert np.array_equal(q[c].cpu().numpy(), ref)
