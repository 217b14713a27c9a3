"""Gaussian low-pass multiply: the 16-byte chunk kernel and the per-element
one against the formula in 64 bits, at the edges of both (partial row blocks,
one-chunk rows, odd widths, unaligned buffers), in both storage types."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]

# FP32: each factor is expf of an argument with two roundings (|arg| <= 16 here
# with sigma = side/4: absolute argument error below 16 * 2^-23, so relative
# factor error below 2e-6 for the tails and 2 ulp at the centre); in the
# 2-norm, where the centre dominates, 1e-6 holds with room.  Half: one
# rounding to 11 bits, 2^-11.
TOL = {"c64": 1e-6, "h16": 2.0 ** -11}


def _factor(n, sigma):
    k = np.arange(n, dtype=np.float64)
    d = np.minimum(k, n - k)
    return np.exp(-d * d / (2.0 * sigma * sigma))


@pytest.mark.parametrize("kind", ["c64", "h16"])
@pytest.mark.parametrize("rows,cols,skip", [
    (1, 1, 0), (3, 2, 0), (7, 4, 0), (1025, 4, 0), (9, 8, 0), (17, 1024, 0), (8, 2048, 0),
    (5, 6, 0), (40, 1000, 0), (33, 512, 1), (1024, 64, 0), (2, 16384, 0)])
def test_lowpass_every_shape(kind, rows, cols, skip):
    import paper_1505_08019_gb300 as fft
    g = torch.Generator(device="cuda").manual_seed(7)
    n = rows * cols
    dtype = torch.float32 if kind == "c64" else torch.float16
    buf = torch.randn(n + skip, 2, generator=g, device="cuda").to(dtype)
    x = buf[skip:]                       # skip = 1: not 16-byte aligned
    before = x.double().cpu().numpy().reshape(rows, cols, 2)
    sr, sc = max(rows / 4, 1.0), max(cols / 4, 1.0)
    fft.fft2d_lowpass(rows, cols, fft.FFT2D_C64 if kind == "c64" else fft.FFT2D_C32H,
                      x.data_ptr(), sr, sc)
    got = x.double().cpu().numpy().reshape(rows, cols, 2)
    want = before * (_factor(rows, sr)[:, None] * _factor(cols, sc)[None, :])[..., None]
    assert np.linalg.norm(got - want) <= TOL[kind] * np.linalg.norm(want)
