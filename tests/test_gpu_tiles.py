"""Column passes on both sides of the lines between tile sizes: the widths at
which a column length changes kernel, one complex column up, widths of less
than a tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]

# (rows, widths around the lines): 128 CTAs of 2^12 and of 2^13 values
EDGES = [(64, (2, 64, 128)), (128, (2, 16, 32, 4096, 8192)), (256, (4, 2048, 4096)),
         (512, (2, 1024, 2048, 4096)), (1024, (2, 512, 1024, 2048, 4096)),
         (2048, (2, 256, 512, 1024, 2048)), (4096, (2, 128, 256, 512, 1024))]
CASES = [(r, c) for r, cs in EDGES for c in cs]


def _rel(got, want):
    return float(np.linalg.norm(got - want) / np.linalg.norm(want))


@pytest.mark.parametrize("rows,cols", CASES)
def test_column_tiles_c64(rows, cols):
    """The default of every width gives the plain kernel's bits."""
    import paper_1505_08019_gb300 as fft
    x = torch.view_as_complex(torch.randn(rows, cols, 2, device="cuda"))
    with fft.Plan(rows, cols, fft.FFT2D_INVERSE) as p:
        got, want = torch.empty_like(x), torch.empty_like(x)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, got)
        fft.fft2d_plan_set_variant(p.handle, fft.FFT2D_PASS_COLS, 0)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, want)
        assert torch.equal(got, want)


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("rows,cols", CASES)
def test_column_tiles_dct(rows, cols, inverse):
    """Against scipy's DCT-II (twice the unnormalised one) and its inverse in
    64 bits; 1e-5 is the FP32 bound of the other GPU tests."""
    fftpack = pytest.importorskip("scipy.fft")
    import paper_1505_08019_gb300 as fft
    x = torch.randn(rows, cols, device="cuda")
    x64 = x.double().cpu().numpy()
    want = fftpack.idct(2 * x64, axis=0) / cols if inverse else fftpack.dct(x64, axis=0) / 2
    with fft.Plan(rows, cols, fft.FFT2D_INVERSE if inverse else fft.FFT2D_FORWARD,
                  fft.FFT2D_R32_DCT2) as p:
        out = torch.empty_like(x)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, out)
        assert _rel(out.double().cpu().numpy(), want) <= 1e-5
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, x)        # in place
        assert torch.equal(x, out)


# the half2 TMA line: 2^22 values, and above 8192 columns
HALF_WIDE = [(512, 4096), (512, 8192), (512, 16384), (1024, 8192), (1024, 16384), (2048, 4096)]


@pytest.mark.parametrize("rows,cols", [(r, c) for r, c in CASES if r > 64] + HALF_WIDE)
def test_column_tiles_half(rows, cols):
    """Whole half2 transform against 64 bits within the half2 tests' 5e-3, and
    the stored range of every column."""
    import paper_1505_08019_gb300 as fft
    q = torch.randn(rows, cols, 2, device="cuda").half()
    e = torch.zeros(rows, dtype=torch.int32, device="cuda")
    out, oe = torch.empty_like(q), torch.empty(cols, dtype=torch.int32, device="cuda")
    with fft.Plan(rows, cols, fft.FFT2D_FORWARD, fft.FFT2D_C32H) as p:
        fft.fft2d_exec_h16(p.handle, q, e, 0, out, oe)
        got = out.double() * torch.pow(2.0, oe.double())[None, :, None]
        want = torch.view_as_real(torch.fft.fft2(torch.view_as_complex(q.double())))
        assert float((got - want).norm() / want.norm()) <= 5e-3
        top = out.abs().amax(dim=(0, 2)).float()
        assert bool(((top >= 2.0 ** 13) & (top <= 2.0 ** 14)).all())
