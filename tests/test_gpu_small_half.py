"""Small half2 images in one launch, bit for bit the two passes: the complex64
row and column passes (other kernels, the same FP32 arithmetic) on the
dequantised values, with the stored rounding and exponents of each pass
redone in torch."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


def _pow2(e):
    return torch.ldexp(torch.ones_like(e, dtype=torch.float32), e)


def _factor(e, axis):
    f = _pow2(e)
    return f[:, None, None] if axis == 0 else f[None, :, None]


def _store(y, axis):
    """y (rows, cols, 2) as half2 with one exponent per line of `axis`: the
    line's largest component is f 2^k, f in [0.5, 1), and e = k - 14."""
    m = y.abs().amax(dim=(1 - axis, 2))
    e = torch.where(m > 0, torch.frexp(m)[1] - 14, 0).to(torch.int32)
    return (y * _factor(-e, axis)).half(), e


@pytest.mark.parametrize("direction", ["FFT2D_FORWARD", "FFT2D_INVERSE"])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("rows,cols", [(2, 2), (4, 64), (64, 4), (16, 16), (64, 64), (32, 128), (128, 512),
                                       (256, 256), (2048, 32), (16, 4096), (4096, 16), (2, 4096), (4096, 2)])
def test_small_half_bits(rows, cols, axis, direction):
    import paper_1505_08019_gb300 as fft
    d = getattr(fft, direction)
    g = torch.Generator(device="cuda").manual_seed(rows * 7 + cols)
    q = torch.randn(rows, cols, 2, generator=g, device="cuda").half()
    e = torch.randint(-6, 7, (rows if axis == 0 else cols,), generator=g, dtype=torch.int32, device="cuda")
    q[rows // 2] = 0                                   # a zero row
    out, oe = torch.empty_like(q), torch.empty(cols, dtype=torch.int32, device="cuda")
    with fft.Plan(rows, cols, d, fft.FFT2D_C32H) as p:
        fft.fft2d_exec_h16(p.handle, q, e, axis, out, oe)
    with fft.Plan(rows, cols, d) as p:
        x = q.float() * _factor(e, axis)
        y = torch.empty_like(x)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_ROWS, x, y)
        h, he = _store(y, 0)
        x = h.float() * _factor(he, 0)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, y)
        want, we = _store(y, 1)
    assert torch.equal(oe, we)
    assert torch.equal(out, want)
