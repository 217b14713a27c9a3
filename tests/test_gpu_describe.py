"""A plan's description names the one-launch kernel exactly where the transform
takes it, as counted from the captured call."""
import pytest

from _graph import launches

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


@pytest.mark.parametrize("rows,cols", [(2, 2), (64, 32), (256, 256), (4096, 16), (512, 256), (1, 64), (8192, 4)])
def test_description_follows_the_launches(rows, cols):
    import paper_1505_08019_gb300 as fft
    x = torch.view_as_complex(torch.randn(rows, cols, 2, device="cuda"))
    out = torch.empty_like(x)

    def check(p):
        p(x, out)
        found = launches(lambda s: p(x, out, s))
        text = fft.fft2d_plan_describe(p.handle)
        one = rows > 1 and cols > 1 and len(found) == 1
        assert ("exec:small" in text) == one, text
        if one:
            assert f"exec:small(ctas={found[0][0][0]},ept=16,default)" in text
        return one

    with fft.Plan(rows, cols) as p:
        small = check(p)
        assert small == (1 < rows <= 4096 and cols > 1 and rows * cols <= 1 << 16)
        if small:                       # a forced variant is one of two launches
            fft.fft2d_plan_set_variant(p.handle, fft.FFT2D_PASS_ROWS, 0)
            assert not check(p)


@pytest.mark.parametrize("rows,cols", [(64, 64), (256, 256), (512, 256)])
def test_half_plans_too(rows, cols):
    import paper_1505_08019_gb300 as fft
    q = torch.randn(rows, cols, 2, device="cuda").half()
    e = torch.zeros(rows, dtype=torch.int32, device="cuda")
    out, oe = torch.empty_like(q), torch.empty(cols, dtype=torch.int32, device="cuda")
    with fft.Plan(rows, cols, fft.FFT2D_FORWARD, fft.FFT2D_C32H) as p:
        def call(s):
            fft.fft2d_exec_h16(p.handle, q, e, 0, out, oe, s)
        call(torch.cuda.current_stream())
        n = len(launches(call))
        assert ("exec:small" in fft.fft2d_plan_describe(p.handle)) == (n == 1) == (rows * cols <= 1 << 16)
