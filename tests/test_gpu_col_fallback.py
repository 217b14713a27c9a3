"""Column passes that TMA cannot feed (buffers of less than 16-byte alignment,
fewer columns than a tile) run the kernel that serves their length best
without it, with the plain kernel's bits."""
import pytest

from _graph import launches

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


@pytest.mark.parametrize("cols,odd", [(1, 0), (2, 0), (4, 1), (8, 1), (64, 1), (1024, 1), (16384, 1)])
def test_1024_rows_run_narrow_tiles(cols, odd):
    import paper_1505_08019_gb300 as fft
    P = fft.FFT2D_PASS_COLS
    names = [fft.fft2d_variant_name(P, 10, v) for v in range(fft.fft2d_variant_count(P, 10))]
    buf = torch.view_as_complex(torch.randn(1024 * cols + 1, 2, device="cuda"))
    x = buf[odd:odd + 1024 * cols].view(1024, cols)

    def geometry(p, out):
        fft.fft2d_exec_pass(p.handle, P, x, out)
        return launches(lambda s: fft.fft2d_exec_pass(p.handle, P, x, out, s))

    with fft.Plan(1024, cols) as p:
        got, narrow, plain = (torch.empty_like(x) for _ in range(3))
        default = geometry(p, got)
        fft.fft2d_plan_set_variant(p.handle, P, names.index("narrow"))
        assert default == geometry(p, narrow)
        fft.fft2d_plan_set_variant(p.handle, P, names.index("plain"))
        assert default != geometry(p, plain)
        assert torch.equal(got, narrow) and torch.equal(got, plain)
