"""A launch that the runtime refuses is that call's error and no later one's."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


def test_refused_launch_does_not_fail_the_next_call():
    import paper_1505_08019_gb300 as fft
    rows, cols = 70000, 16            # one grid row per image row: 65535 is the most
    big = torch.zeros(rows, cols, dtype=torch.complex64, device="cuda")
    x = torch.view_as_complex(torch.randn(64, 128, 2, device="cuda"))
    with fft.Plan(64, 128) as p:
        want = p(x)
    with pytest.raises(fft.FFT2DError) as ei:
        fft.fft2d_lowpass(rows, cols, fft.FFT2D_C64, big, 100.0, 10.0)
    assert ei.value.status == fft.FFT2D_ERR_CUDA
    out = torch.empty_like(x)
    fft.fft2d_exec_noalloc(64, 128, fft.FFT2D_FORWARD, x, out)
    scale = float(want.abs().max())
    assert float((out - want).abs().max()) <= 1e-5 * scale
