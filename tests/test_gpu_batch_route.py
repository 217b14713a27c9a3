"""Which launches a batch makes, counted from a captured graph of the call."""
import pytest

from _graph import launches

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA GPU")]


def batch(shapes):
    import paper_1505_08019_gb300 as fft
    plans = {s: fft.Plan(*s) for s in set(shapes)}
    xs = [torch.view_as_complex(torch.randn(*s, 2, device="cuda")) for s in shapes]
    outs = [torch.empty_like(x) for x in xs]
    handles = [plans[s].handle for s in shapes]
    fft.fft2d_exec_batched(handles, xs, outs)        # first launches outside the capture
    return plans, handles, xs, outs


def test_tuning_keeps_a_small_batch_in_one_launch_per_pass():
    import paper_1505_08019_gb300 as fft
    plans, handles, xs, outs = batch([(64, 128), (128, 64), (64, 64), (128, 128)] * 4)

    def count():
        return len(launches(lambda s: fft.fft2d_exec_batched(handles, xs, outs, s)))

    want = [o.clone() for o in outs]
    scratch = [x.clone() for x in xs]
    try:
        assert count() == 2
        fft.fft2d_autotune_batched(handles, scratch, [torch.empty_like(x) for x in xs])
        assert count() == 2
        fft.fft2d_exec_batched(handles, xs, outs)
        assert all(torch.equal(o, w) for o, w in zip(outs, want))
        # a forced variant is a choice of the length's own launch
        fft.fft2d_batch_set_variant(fft.FFT2D_PASS_COLS, 6, 1)
        assert count() == 3
        fft.fft2d_exec_batched(handles, xs, outs)
        assert all(torch.equal(o, w) for o, w in zip(outs, want))
        # and the next tuning replaces it
        fft.fft2d_autotune_batched(handles, scratch, [torch.empty_like(x) for x in xs])
        assert count() == 2
    finally:
        for length in range(1, 15):
            for pass_ in (fft.FFT2D_PASS_ROWS, fft.FFT2D_PASS_COLS):
                fft.fft2d_batch_set_variant(pass_, length, -1)


@pytest.mark.parametrize("n,want", [(128, 2), (129, 2), (512, 2), (513, 4)])
def test_a_batch_of_many_images_shares_its_launches(n, want):
    """Up to 512 images in one launch per pass, each with its own transform's
    bits, whichever job table holds it."""
    import paper_1505_08019_gb300 as fft
    plans, handles, xs, outs = batch([(16, 64), (64, 32), (32, 16)] * (n // 3) + [(8, 128)] * (n % 3))
    assert len(launches(lambda s: fft.fft2d_exec_batched(handles, xs, outs, s))) == want
    one = {s: torch.empty(s, dtype=torch.complex64, device="cuda") for s in plans}
    for x, o in zip(xs, outs):
        s = tuple(x.shape)
        assert torch.equal(plans[s](x, one[s]), o)


@pytest.mark.parametrize("shapes", [[(1024, 1024)], [(2048, 256)] * 4, [(1024, 512)] * 3 + [(1024, 1024)],
                                    [(8192, 64)] * 2, [(1024, 512), (2048, 512)]])
def test_columns_in_launches_of_their_own(shapes):
    """Rows in the launch for any length and columns in one launch of their
    own (which follows on the caller's stream) or in two (which do not): the
    bits of each image's own transform, call after call on the same buffers."""
    import paper_1505_08019_gb300 as fft
    plans, handles, xs, outs = batch(shapes)
    want = [plans[tuple(x.shape)](x) for x in xs]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for _ in range(20):
            for o in outs:
                o.zero_()
            fft.fft2d_exec_batched(handles, xs, outs)
            fft.fft2d_exec_batched(handles, xs, outs)
            got = [o.clone() for o in outs]
    torch.cuda.synchronize()
    assert all(torch.equal(g, w) for g, w in zip(got, want))
    if shapes[0][0] < 8192:
        assert len(launches(lambda s: fft.fft2d_exec_batched(handles, xs, outs, s))) \
            == len({s[0] for s in shapes}) + 1
