"""The quantiser's sum of squares over FP32's whole range of magnitudes, where
the float pairs it is summed in hand over to FP64, and at ragged sizes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2005_03060_gb300 import gridcorr
    return gridcorr.Context(0)


@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e25, 0.0])
@pytest.mark.parametrize("C,T,N", [(2, 3, 2), (1, 1030, 64), (3, 257, 1024)])
def test_quantiser_sum_of_squares(ctx, orc, C, T, N, scale):
    """Scales equal to the last bit, over FP32's whole range of magnitudes (one
    channel mixes large and vanishing values)."""
    rng = np.random.default_rng(C * T + N)
    x = ((rng.standard_normal((C, T, N)) + 1j * rng.standard_normal((C, T, N))) * scale).astype(np.complex64)
    x[0, :, ::2] *= np.float32(1e-9)
    q, s = ctx.quantize(torch.from_numpy(x).cuda())
    q, s = q.cpu().numpy(), s.cpu().numpy()
    for c in range(C):
        if scale == 0.0:
            assert s[c] == 0 and not q[c].any()
            continue
        ref, sc = orc.quantize(x[c])
        assert np.float32(sc) == s[c]
        assert np.array_equal(q[c], ref)
