"""Failure path of the TMA-fed kernels of 1024-row columns: CTA 0 never issues
one load of its first tile, its bounded wait gives up, the host reads
FFT2D_ERR_TIMEOUT, and the same plan then transforms correctly."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


@pytest.mark.parametrize("cols,variant", [(64, None), (256, "tma32g5"), (256, "tma64w8")])
def test_withheld_load_of_1024_rows(cols, variant):
    import paper_1505_08019_gb300 as fft
    P = fft.FFT2D_PASS_COLS
    names = [fft.fft2d_variant_name(P, 10, v) for v in range(fft.fft2d_variant_count(P, 10))]
    x = torch.view_as_complex(torch.randn(1024, cols, 2, device="cuda"))
    out, want = torch.empty_like(x), torch.empty_like(x)
    with fft.Plan(1024, cols) as p:
        fft.fft2d_plan_set_variant(p.handle, P, names.index("plain"))
        fft.fft2d_exec_pass(p.handle, P, x, want)
        fft.fft2d_plan_set_variant(p.handle, P, -1 if variant is None else names.index(variant))
        fft.fft2d_sync_status(p.handle)
        fft.fft2d_selftest_withheld_load(p.handle, x, out)
        with pytest.raises(fft.FFT2DError) as ei:
            fft.fft2d_sync_status(p.handle)
        assert ei.value.status == fft.FFT2D_ERR_TIMEOUT
        fft.fft2d_sync_status(p.handle)                      # cleared
        fft.fft2d_exec_pass(p.handle, P, x, out)
        fft.fft2d_sync_status(p.handle)
        assert torch.equal(out, want)


def test_unaligned_1024_rows_are_refused():
    """From an odd pixel on the pass runs a kernel without TMA."""
    import paper_1505_08019_gb300 as fft
    x = torch.zeros(1024 * 64 + 1, dtype=torch.complex64, device="cuda")[1:].view(1024, 64)
    with fft.Plan(1024, 64) as p:
        with pytest.raises(fft.FFT2DError) as ei:
            fft.fft2d_selftest_withheld_load(p.handle, x, x)
        assert ei.value.status == fft.FFT2D_ERR_ARG
