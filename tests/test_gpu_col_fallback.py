"""Column passes that TMA cannot feed (buffers of less than 16-byte alignment,
fewer columns than a tile), or that fill no tile, run the kernel that serves
their length best then, with the plain kernel's bits."""
import pytest

from _graph import launches

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


@pytest.mark.parametrize("rows,cols,odd", [(512, 1, 0), (512, 2, 0), (512, 4, 1), (1024, 1, 0), (1024, 2, 0),
                                           (1024, 4, 1), (1024, 8, 1), (1024, 64, 1), (1024, 1024, 1),
                                           (1024, 16384, 1)])
def test_narrow_tiles(rows, cols, odd):
    """512 rows: fewer columns than a tile of the default kernel; 1024 rows:
    images that TMA cannot feed."""
    import paper_1505_08019_gb300 as fft
    P, L = fft.FFT2D_PASS_COLS, rows.bit_length() - 1
    names = [fft.fft2d_variant_name(P, L, v) for v in range(fft.fft2d_variant_count(P, L))]
    buf = torch.view_as_complex(torch.randn(rows * cols + 1, 2, device="cuda"))
    x = buf[odd:odd + rows * cols].view(rows, cols)

    def geometry(p, out):
        fft.fft2d_exec_pass(p.handle, P, x, out)
        return launches(lambda s: fft.fft2d_exec_pass(p.handle, P, x, out, s))

    with fft.Plan(rows, cols) as p:
        got, narrow, plain = (torch.empty_like(x) for _ in range(3))
        default = geometry(p, got)
        fft.fft2d_plan_set_variant(p.handle, P, names.index("narrow"))
        assert default == geometry(p, narrow)
        fft.fft2d_plan_set_variant(p.handle, P, names.index("plain"))
        assert default != geometry(p, plain)
        assert torch.equal(got, narrow) and torch.equal(got, plain)


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("rows,cols,threads", [(2048, 4, 256), (2048, 1024, 512), (2048, 2048, 1024),
                                               (4096, 4, 256), (4096, 512, 512), (4096, 1024, 1024),
                                               (4096, 4096, 1024)])
def test_dct_tiles_of_long_columns(rows, cols, threads, inverse):
    """An image of 8-byte alignment: tiles of 2^14 values (16 a thread) where
    the aligned one is TMA-fed, the smaller tiles of narrow images below that.
    The result is the aligned one's within the FP32 bound of the other GPU
    tests."""
    import paper_1505_08019_gb300 as fft
    if inverse and (rows, cols) == (4096, 4):
        threads = 512                  # the inverse has no tiles of 2^12 values here
    buf = torch.randn(rows * cols + 2, device="cuda")
    x = buf[2:].view(rows, cols)
    with fft.Plan(rows, cols, fft.FFT2D_INVERSE if inverse else fft.FFT2D_FORWARD,
                  fft.FFT2D_R32_DCT2) as p:
        P = fft.FFT2D_PASS_COLS
        want, got = torch.empty_like(x), torch.empty_like(buf)[2:].view(rows, cols)
        fft.fft2d_exec_pass(p.handle, P, x.clone(), want)
        fft.fft2d_exec_pass(p.handle, P, x, got)
        (_, block, _), = launches(lambda s: fft.fft2d_exec_pass(p.handle, P, x, got, s))
        assert block[0] == threads
        assert float((got - want).norm() / want.norm()) <= 1e-5
