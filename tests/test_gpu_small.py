"""Small images in one launch: bit for bit the two single passes, at every
axis length the one-launch kernel holds, at the ends of its pixel range and
on both sides of its line, in both storage types and directions, in place and
out of place, on several streams at once and from a captured graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]

# every column length, every row length, one pixel to the largest cluster,
# partly filled CTAs (below 4096 pixels), and the first shapes beyond the line
SHAPES = [(2, 2), (2, 64), (64, 2), (4, 8), (16, 16), (32, 32), (64, 64), (128, 64), (128, 128),
          (256, 128), (256, 256), (512, 128), (64, 1024), (2048, 32), (16, 4096), (4096, 16),
          (4096, 2), (2, 4096), (8, 2048), (1024, 8), (512, 256), (8192, 8), (8, 8192)]


def _input(rows, cols, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(rows, cols, 2, generator=g, device="cuda")


@pytest.mark.parametrize("direction", ["FFT2D_FORWARD", "FFT2D_INVERSE"])
@pytest.mark.parametrize("rows,cols", SHAPES)
def test_small_equals_the_two_passes(rows, cols, direction):
    import paper_1505_08019_gb300 as fft
    x = torch.view_as_complex(_input(rows, cols, rows * 5 + cols))
    with fft.Plan(rows, cols, getattr(fft, direction)) as p:
        want = torch.empty_like(x)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_ROWS, x, want)
        fft.fft2d_exec_pass(p.handle, fft.FFT2D_PASS_COLS, want, want)
        assert torch.equal(p(x), want)
        y = x.clone()
        p(y, y)
        assert torch.equal(y, want)


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("rows,cols", SHAPES)
def test_small_half_equals_grouped(rows, cols, axis):
    """The grouped half2 kernels of the serving loop run the same CTA work."""
    import paper_1505_08019_gb300 as fft
    q = _input(rows, cols, rows * 3 + cols).half()
    lines = rows if axis == 0 else cols
    e = torch.randint(-6, 7, (lines,), dtype=torch.int32, device="cuda",
                      generator=torch.Generator(device="cuda").manual_seed(lines))
    p = fft.fft2d_plan(rows, cols, fft.FFT2D_C32H, fft.FFT2D_FORWARD)
    try:
        out, oe = torch.empty_like(q), torch.empty(cols, dtype=torch.int32, device="cuda")
        fft.fft2d_exec_h16(p, q, e, axis, out, oe)
        f = torch.pow(2.0, e.double())
        x = q.double() * (f[:, None, None] if axis == 0 else f[None, :, None])
        want = torch.view_as_real(torch.fft.fft2(torch.view_as_complex(x)))
        got = out.double() * torch.pow(2.0, oe.double())[None, :, None]
        # two stored roundings of 2^-11 relative to a line's largest value,
        # within the bound the half2 tests use
        assert float((got - want).norm() / want.norm()) <= 5e-3
        # in place, the same bits
        inq, ine = q.clone(), torch.empty_like(oe)
        fft.fft2d_exec_h16(p, inq, e, axis, inq, ine)
        assert torch.equal(inq, out) and torch.equal(ine, oe)
    finally:
        fft.fft2d_destroy(p)


def test_small_on_streams_and_from_a_graph():
    import paper_1505_08019_gb300 as fft
    x = torch.view_as_complex(_input(256, 256, 9))
    with fft.Plan(256, 256) as p:
        want = p(x)
        outs = [torch.empty_like(x) for _ in range(8)]
        streams = [torch.cuda.Stream() for _ in outs]
        torch.cuda.synchronize()
        for _ in range(20):
            for s, o in zip(streams, outs):
                p(x, o, s)
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in outs)
        y = torch.empty_like(x)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p(x, y)
            p(y, y)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, p(want))
        assert np.isfinite(torch.view_as_real(y).sum().item())


def test_autotune_keeps_the_bits():
    import paper_1505_08019_gb300 as fft
    x = torch.view_as_complex(_input(64, 256, 3))
    with fft.Plan(64, 256) as p:
        want = p(x)
        fft.fft2d_autotune(p.handle)
        assert torch.equal(p(x), want)


def test_forced_variants_keep_the_two_launches():
    import paper_1505_08019_gb300 as fft
    x = torch.view_as_complex(_input(128, 128, 4))
    with fft.Plan(128, 128) as p:
        want = p(x)
        for v in range(fft.fft2d_variant_count(fft.FFT2D_PASS_COLS, 7)):
            fft.fft2d_plan_set_variant(p.handle, fft.FFT2D_PASS_COLS, v)
            assert torch.equal(p(x), want)
