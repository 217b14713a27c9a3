"""Small batches through the launch for any axis length: every image gets the
bits of its own transform, whatever lengths, directions and storage types
share the batch, at the ends of the length range, beside images that take
other launches, over more images than one table, and with a forced variant."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]

MIXES = {
    "tiny": [(2, 2), (2, 64), (16, 4), (32, 32), (8, 8), (1, 8), (8, 1)],
    "ends": [(4096, 2), (2, 4096), (2048, 64), (64, 2048), (512, 512), (4096, 64), (128, 128)],
    "long": [(8192, 4), (4, 8192), (256, 256), (16384, 2), (64, 64)],
    "many": [(1 << (2 + i % 7), 1 << (2 + i % 5)) for i in range(150)],
    "beyond": [(2048, 2048), (2048, 1024), (1024, 2048), (128, 64), (64, 128)],     # over 2^23 values
}


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("mix", sorted(MIXES))
def test_batch_equals_single_images(mix, forced):
    import paper_1505_08019_gb300 as fft
    g = torch.Generator(device="cuda").manual_seed(len(mix))
    shapes = MIXES[mix]
    plans = {(s, d): fft.Plan(s[0], s[1], d) for s in set(shapes)
             for d in (fft.FFT2D_FORWARD, fft.FFT2D_INVERSE)}
    use = [plans[s, fft.FFT2D_INVERSE if i % 3 == 1 else fft.FFT2D_FORWARD]
           for i, s in enumerate(shapes)]
    xs = [torch.view_as_complex(torch.randn(*s, 2, generator=g, device="cuda")) for s in shapes]
    want = [p(x) for p, x in zip(use, xs)]
    before = fft.fft2d_batch_get_variant(fft.FFT2D_PASS_COLS, 6)
    if forced:
        fft.fft2d_batch_set_variant(fft.FFT2D_PASS_COLS, 6, 1)
    try:
        outs = [torch.empty_like(x) for x in xs]
        fft.fft2d_exec_batched([p.handle for p in use], xs, outs)
        inplace = [x.clone() for x in xs]
        fft.fft2d_exec_batched([p.handle for p in use], inplace, inplace)
        for s, o, y, w in zip(shapes, outs, inplace, want):
            assert torch.equal(o, w) and torch.equal(y, w), s
    finally:
        if forced:
            fft.fft2d_batch_set_variant(fft.FFT2D_PASS_COLS, 6, -1)
            assert fft.fft2d_batch_get_variant(fft.FFT2D_PASS_COLS, 6) == before


def test_served_half2_equals_the_plan():
    import paper_1505_08019_gb300 as fft
    shapes = [(16, 64), (64, 16), (2, 128), (256, 64), (512, 512), (1024, 256), (2048, 16), (2, 2)]
    srv = fft.fft2d_serve_create(1 << 30, 2)
    try:
        jobs = []
        for i, (r, c) in enumerate(shapes):
            q = torch.randn(r, c, 2, generator=torch.Generator().manual_seed(i)).half().pin_memory()
            e = torch.randint(-4, 5, (r,), dtype=torch.int32).pin_memory()
            out, oe = torch.empty_like(q).pin_memory(), torch.empty(c, dtype=torch.int32).pin_memory()
            t = fft.fft2d_serve_submit(srv, fft.FFT2D_OP_FORWARD, r, c, fft.FFT2D_C32H, q, out, e, oe)
            jobs.append((r, c, q, e, out, oe, t))
        for r, c, q, e, out, oe, t in jobs:
            fft.fft2d_serve_wait(srv, t)
            dq, de = q.cuda(), e.cuda()
            want, we = torch.empty_like(dq), torch.empty(c, dtype=torch.int32, device="cuda")
            with fft.Plan(r, c, fft.FFT2D_FORWARD, fft.FFT2D_C32H) as p:
                fft.fft2d_exec_h16(p.handle, dq, de, 0, want, we)
                assert torch.equal(want.cpu(), out) and torch.equal(we.cpu(), oe), (r, c)
    finally:
        fft.fft2d_serve_destroy(srv)
