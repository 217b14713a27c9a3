"""Columns of 8192 and 16384 rows through the L2-resident strip: every column
is independent of the image's width, so a wide image (several chunks of
strips) must give the bits of the narrow ones cut from it, down to one complex
column (partly filled strips); complex64 also the bits of the cluster
kernels, and one DCT column of each kind the oracle's definition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]

TOL = 1e-5      # relative L2, the FP32 bound of the other GPU tests


def _columns(fft, kind, rows, x, out=None):
    """Column pass of x (rows x complex columns) through a plan of its width."""
    cols = x.shape[1]
    if kind == "c64":
        p = fft.Plan(rows, cols, fft.FFT2D_INVERSE)
    else:
        d = fft.FFT2D_FORWARD if kind == "dct" else fft.FFT2D_INVERSE
        p = fft.Plan(rows, 2 * cols, d, fft.FFT2D_R32_DCT2)
    out = torch.empty_like(x) if out is None else out
    fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, out)
    torch.cuda.synchronize()
    p.close()
    return out


@pytest.mark.parametrize("kind", ["c64", "dct", "idct"])
@pytest.mark.parametrize("rows", [8192, 16384])
def test_strip_columns_do_not_depend_on_the_width(rows, kind):
    import paper_1505_08019_gb300 as fft
    g = torch.Generator(device="cuda").manual_seed(rows)
    x = torch.view_as_complex(torch.randn(rows, 1024, 2, generator=g, device="cuda"))
    wide = _columns(fft, kind, rows, x)
    inplace = x.clone()
    _columns(fft, kind, rows, inplace, inplace)
    assert torch.equal(inplace, wide)
    for n in (1, 2, 8, 16, 32, 64, 512):
        part = _columns(fft, kind, rows, x[:, 1024 - n:].contiguous())
        # the inverse scale is a power of two, so other widths are exact multiples
        f = 1.0 if kind == "dct" else n / 1024
        assert torch.equal(part * f, wide[:, 1024 - n:]), n


@pytest.mark.parametrize("rows,other", [(8192, "pairl2"), (16384, "quadl2")])
def test_strip_equals_the_cluster_kernel(rows, other):
    import paper_1505_08019_gb300 as fft
    L = rows.bit_length() - 1
    x = torch.view_as_complex(torch.randn(rows, 64, 2, device="cuda"))
    got = []
    names = [fft.fft2d_variant_name(fft.FFT2D_PASS_COLS, L, v)
             for v in range(fft.fft2d_variant_count(fft.FFT2D_PASS_COLS, L))]
    with fft.Plan(rows, 64) as p:
        for name in ("stripl2", other):
            fft.fft2d_plan_set_variant(p.handle, fft.FFT2D_PASS_COLS, names.index(name))
            out = torch.empty_like(x)
            fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, x, out)
            got.append(out)
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("rows,kind", [(8192, "dct"), (8192, "idct"), (16384, "dct"), (16384, "idct")])
def test_strip_dct_column_against_the_oracle(rows, kind, orc):
    import paper_1505_08019_gb300 as fft
    x = torch.zeros(rows, 1, dtype=torch.complex64, device="cuda")
    x.real = torch.randn(rows, 1, generator=torch.Generator(device="cuda").manual_seed(3),
                         device="cuda")
    got = torch.view_as_real(_columns(fft, kind, rows, x)).cpu().numpy().reshape(rows, 2)
    want = orc.dct1d(x.real.cpu().numpy().reshape(rows).astype(np.float64), inverse=kind == "idct")
    if kind == "idct":
        want = np.asarray(want) / 2      # the pass carries the whole 1 / (rows cols), cols = 2
    assert np.linalg.norm(got[:, 0] - want) <= TOL * np.linalg.norm(want)
    assert np.linalg.norm(got[:, 1]) <= TOL * np.linalg.norm(want)
