"""Performance cases of the 2D FFT library: what its users have it do.

Each case is one call (or the few calls) a program makes through the public
binding, at sizes of the paper's Table 1, of the test-suite and of
``bench.py``.  Sides are powers of two, the only ones the library accepts, so
the ragged part of the range is its aspect ratios: long strips, 1:4 images and
batches of uneven shapes.

kinds
  fft     one complex64 image on the device, forward or inverse (``Plan``)
  filter  FFT -> Gaussian low-pass (sigma = side/8) -> inverse FFT, on the device
  half    one half2 image with per-line exponents (``fft2d_exec_h16``); forward
          reads per-row exponents, inverse the per-column ones of a spectrum
  dct     one real image, DCT-II forward or DCT-III inverse
  batch   many uneven images in one ``fft2d_exec_batched`` call
  serve   a burst of mixed requests on host buffers through the serving loop
"""
from __future__ import annotations

import math
import random

import torch

import paper_1505_08019_gb300 as fft

FWD, INV = fft.FFT2D_FORWARD, fft.FFT2D_INVERSE


def listed():
    return [
        # the smallest plain image of the benchmark's configurations: bound by
        # launches and latency
        {"name": "fft_256", "kind": "fft", "rows": 256, "cols": 256, "dir": FWD},
        # the paper's own size, back from a spectrum
        {"name": "ifft_1024", "kind": "fft", "rows": 1024, "cols": 1024, "dir": INV},
        # image filtering, the use that motivates the paper, at Table 1's largest size
        {"name": "filter_2048", "kind": "filter", "rows": 2048, "cols": 2048},
        # the headline workload of bench.py
        {"name": "fft_4096", "kind": "fft", "rows": 4096, "cols": 4096, "dir": FWD},
        # a tall strip: the longest columns, short rows
        {"name": "ifft_strip_16384x1024", "kind": "fft", "rows": 16384, "cols": 1024, "dir": INV},
        # the largest image the library takes
        {"name": "fft_16384", "kind": "fft", "rows": 16384, "cols": 16384, "dir": FWD},
        # large image in half2 storage
        {"name": "half_8192", "kind": "half", "rows": 8192, "cols": 8192, "dir": FWD},
        # a 1:4 half2 image as the serving loop takes them, spectrum -> image
        {"name": "ihalf_256x1024", "kind": "half", "rows": 256, "cols": 1024, "dir": INV},
        # the DCT workload of bench.py
        {"name": "dct_4096", "kind": "dct", "rows": 4096, "cols": 4096, "dir": FWD},
        # the largest image, from its cosine coefficients
        {"name": "idct_16384", "kind": "dct", "rows": 16384, "cols": 16384, "dir": INV},
        # the batched workload of bench.py: 64 images, sides 128 .. 2048
        {"name": "batch_64", "kind": "batch", "images": 64, "lo": 7, "hi": 11, "shapes": 0},
        # a burst on the serving loop: half squares, half 1:4, 70 % complex64, 30 % half2
        {"name": "serve_24", "kind": "serve", "requests": 24, "lo": 6, "hi": 10, "shapes": 0},
    ]


def draw(rng):
    kind = rng.choices(["fft", "filter", "half", "dct", "batch", "serve"],
                       [0.36, 0.12, 0.18, 0.18, 0.1, 0.06])[0]
    if kind == "batch":
        lo = rng.randint(6, 8)
        return {"kind": kind, "images": rng.randint(8, 64), "lo": lo,
                "hi": rng.randint(lo + 1, 11), "shapes": rng.randint(1, 1 << 20)}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(4, 24), "lo": 6,
                "hi": rng.randint(8, 10), "shapes": rng.randint(1, 1 << 20)}
    most = {"fft": 28, "filter": 26, "half": 27, "dct": 28}[kind]
    while True:
        lr, lc = rng.randint(4, 14), rng.randint(4, 14)
        if 12 <= lr + lc <= most:
            break
    case = {"kind": kind, "rows": 1 << lr, "cols": 1 << lc}
    if kind != "filter":
        case["dir"] = rng.choice([FWD, INV])
    return case


# ------------------------------------------------------------------- inputs
def _gray(rows, cols, seed):
    """A gray image on the GPU: eight Gaussian blobs and uniform [0, 1) noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(4, 8, generator=g, device="cuda")
    side = min(rows, cols)
    amp, s = 0.5 + 1.5 * u[0], side / 32 + side * (1 / 4 - 1 / 32) * u[1]

    def bells(n, mid):
        t = torch.arange(n, device="cuda", dtype=torch.float32)[:, None]
        return torch.exp(-((t - mid * n) ** 2) / (2 * s * s))

    x = torch.rand(rows, cols, generator=g, device="cuda")
    r, c = bells(rows, u[2]) * amp, bells(cols, u[3])
    for b in range(8):
        x.addcmul_(r[:, b:b + 1], c[None, :, b])
    return x


def _image(rows, cols, seed):
    return _gray(rows, cols, seed).to(torch.complex64)


def _complex_input(case, seed):
    x = _image(case["rows"], case["cols"], seed)
    return torch.fft.fft2(x) if case.get("dir", FWD) == INV else x


def _exponents(x, axis):
    """One power-of-two exponent per row (axis 0) or column (axis 1): every
    stored component of the line stays below 2^14."""
    m = torch.view_as_real(x).abs().amax(dim=(1 - axis, 2))
    return torch.where(m > 0, torch.frexp(m)[1] - 14, 0).to(torch.int32)


def _pow2(e, axis):
    """2^e of every line as float64, exact, shaped to multiply (rows, cols, 2)."""
    f = ((e.long() + 1023) << 52).view(torch.float64)
    return f[:, None, None] if axis == 0 else f[None, :, None]


def _pack(x, axis):
    e = _exponents(x, axis)
    return (torch.view_as_real(x) * _pow2(-e, axis).float()).half(), e


def _unpack(q, e, axis):
    return torch.view_as_complex(q.double() * _pow2(e, axis))


def _half_input(case, seed):
    axis = 0 if case["dir"] == FWD else 1
    return _pack(_complex_input(case, seed), axis) + (axis,)


def _dct_input(case, seed):
    x = _gray(case["rows"], case["cols"], seed)
    return _dct2d(x, FWD).float() if case["dir"] == INV else x


def _batch_shapes(case):
    r = random.Random(case["shapes"])
    return [(1 << r.randint(case["lo"], case["hi"]), 1 << r.randint(case["lo"], case["hi"]))
            for _ in range(case["images"])]


def _requests(case):
    """(op, rows, cols, dtype) of every request of a burst."""
    r = random.Random(case["shapes"])
    got = []
    for _ in range(case["requests"]):
        long_side = 1 << r.randint(case["lo"], case["hi"])
        short = long_side if r.random() < 0.5 else long_side // 4
        rows, cols = (long_side, short) if r.random() < 0.5 else (short, long_side)
        op = fft.FFT2D_OP_FORWARD if r.random() < 0.5 else fft.FFT2D_OP_LOWPASS
        got.append((op, rows, cols, fft.FFT2D_C64 if r.random() < 0.7 else fft.FFT2D_C32H))
    return got


class _Server:
    """A serving loop that lives as long as the state that holds it."""

    def __init__(self):
        self.handle = fft.fft2d_serve_create(1 << 32, 4)

    def __del__(self):
        if getattr(self, "handle", None):
            fft.fft2d_serve_destroy(self.handle)
            self.handle = None


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fft":
        x = _complex_input(case, seed)
        return {"kind": kind, "plan": fft.Plan(case["rows"], case["cols"], case["dir"]), "x": x,
                "out": torch.empty_like(x)}
    if kind == "filter":
        rows, cols = case["rows"], case["cols"]
        x = _image(rows, cols, seed)
        return {"kind": kind, "rows": rows, "cols": cols, "fwd": fft.Plan(rows, cols, FWD),
                "inv": fft.Plan(rows, cols, INV), "x": x, "spectrum": torch.empty_like(x),
                "out": torch.empty_like(x)}
    if kind == "half":
        q, e, axis = _half_input(case, seed)
        return {"kind": kind, "axis": axis, "x": q, "x_exp": e, "out": torch.empty_like(q),
                "plan": fft.Plan(case["rows"], case["cols"], case["dir"], fft.FFT2D_C32H),
                "out_exp": torch.empty(case["cols"], dtype=torch.int32, device="cuda")}
    if kind == "dct":
        x = _dct_input(case, seed)
        return {"kind": kind, "x": x, "out": torch.empty_like(x),
                "plan": fft.Plan(case["rows"], case["cols"], case["dir"], fft.FFT2D_R32_DCT2)}
    if kind == "batch":
        shapes = _batch_shapes(case)
        plans = {s: fft.Plan(s[0], s[1], FWD) for s in set(shapes)}
        xs = [_image(r, c, seed * 1000 + i) for i, (r, c) in enumerate(shapes)]
        return {"kind": kind, "keep": plans, "plans": [plans[s].handle for s in shapes], "x": xs,
                "out": [torch.empty_like(x) for x in xs]}
    reqs = []
    for i, (op, rows, cols, dtype) in enumerate(_requests(case)):
        x = _image(rows, cols, seed * 1000 + i)
        if dtype == fft.FFT2D_C64:
            x = x.cpu().pin_memory()
            reqs.append((op, rows, cols, dtype, x, torch.empty_like(x).pin_memory(), None, None))
        else:
            q, e = (t.cpu().pin_memory() for t in _pack(x, 0))
            reqs.append((op, rows, cols, dtype, q, torch.empty_like(q).pin_memory(), e,
                         torch.empty(cols, dtype=torch.int32).pin_memory()))
    return {"kind": kind, "server": _Server(), "requests": reqs}


# --------------------------------------------------------------------- run
def run(state):
    kind = state["kind"]
    if kind in ("fft", "dct"):
        return state["plan"](state["x"], state["out"])
    if kind == "filter":
        rows, cols = state["rows"], state["cols"]
        state["fwd"](state["x"], state["spectrum"])
        fft.fft2d_lowpass(rows, cols, fft.FFT2D_C64, state["spectrum"], rows / 8, cols / 8)
        return state["inv"](state["spectrum"], state["out"])
    if kind == "half":
        fft.fft2d_exec_h16(state["plan"].handle, state["x"], state["x_exp"], state["axis"],
                           state["out"], state["out_exp"])
        return {"out": state["out"], "exp": state["out_exp"]}
    if kind == "batch":
        fft.fft2d_exec_batched(state["plans"], state["x"], state["out"])
        return state["out"]
    srv = state["server"].handle
    tickets = [fft.fft2d_serve_submit(srv, op, rows, cols, dtype, x, out, e, out_e)
               for op, rows, cols, dtype, x, out, e, out_e in state["requests"]]
    for t in tickets:
        fft.fft2d_serve_wait(srv, t)
    return [{"out": r[5]} if r[7] is None else {"out": r[5], "exp": r[7]}
            for r in state["requests"]]


def work(case):
    """Input and output once each; 5 N log2 N per complex transform (half for real data)."""
    kind = case["kind"]

    def flops(rows, cols):
        n = rows * cols
        return 5.0 * n * math.log2(n)

    if kind == "batch":
        shapes = _batch_shapes(case)
        return {"bytes": sum(16 * r * c for r, c in shapes),
                "flops": sum(flops(r, c) for r, c in shapes)}
    if kind == "serve":
        reqs = _requests(case)
        return {"bytes": sum(r * c * (16 if d == fft.FFT2D_C64 else 8) for _, r, c, d in reqs),
                "flops": sum(flops(r, c) * (1 if op == fft.FFT2D_OP_FORWARD else 2)
                             for op, r, c, _ in reqs)}
    rows, cols = case["rows"], case["cols"]
    n = rows * cols
    if kind == "fft":
        return {"bytes": 16 * n, "flops": flops(rows, cols)}
    if kind == "filter":
        return {"bytes": 16 * n, "flops": 2 * flops(rows, cols)}
    if kind == "half":
        lines = (rows if case["dir"] == FWD else cols) + cols
        return {"bytes": 8 * n + 4 * lines, "flops": flops(rows, cols)}
    return {"bytes": 8 * n, "flops": flops(rows, cols) / 2}


# ------------------------------------------------------------------- exact
def _dct_lines(x, dir):
    """DCT-II (or its inverse) of every row of a float64 matrix, through one
    complex FFT of the reordered line (Makhoul, 1980)."""
    n = x.shape[1]
    k = torch.arange(n, device=x.device, dtype=torch.float64)
    turn = torch.polar(torch.ones_like(k), math.pi * k / (2 * n))
    if dir == FWD:
        v = torch.cat([x[:, 0::2], x[:, 1::2].flip(1)], dim=1)
        return (torch.fft.fft(v) * turn.conj()).real
    mirror = torch.cat([torch.zeros_like(x[:, :1]), x[:, 1:].flip(1)], dim=1)
    v = torch.fft.ifft(torch.complex(x, -mirror) * turn).real
    out = torch.empty_like(x)
    out[:, 0::2] = v[:, :(n + 1) // 2]
    out[:, 1::2] = v[:, (n + 1) // 2:].flip(1)
    return out


def _dct2d(x, dir):
    """The same over both axes, a slab of lines at a time, in 64 bits."""
    out = x.double()
    for _ in range(2):
        step = max(1, (1 << 26) // out.shape[1])
        out = torch.cat([_dct_lines(s, dir) for s in out.split(step)]).t().contiguous()
    return out


def _lowpass(spectrum):
    rows, cols = spectrum.shape

    def gauss(n):
        k = torch.arange(n, device=spectrum.device, dtype=torch.float64)
        d = torch.minimum(k, n - k)
        return torch.exp(-d * d / (2 * (n / 8) ** 2))

    return spectrum * gauss(rows)[:, None] * gauss(cols)[None, :]


def _exact_half(x):
    e = _exponents(x, 1)
    return {"out": torch.view_as_real(x) * _pow2(-e, 1), "exp": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "fft":
        x = _complex_input(case, seed).to(torch.complex128)
        return torch.fft.fft2(x) if case["dir"] == FWD else torch.fft.ifft2(x)
    if kind == "filter":
        x = _image(case["rows"], case["cols"], seed).to(torch.complex128)
        return torch.fft.ifft2(_lowpass(torch.fft.fft2(x)))
    if kind == "half":
        x = _unpack(*_half_input(case, seed))
        return _exact_half(torch.fft.fft2(x) if case["dir"] == FWD else torch.fft.ifft2(x))
    if kind == "dct":
        return _dct2d(_dct_input(case, seed), case["dir"])
    if kind == "batch":
        return [torch.fft.fft2(_image(r, c, seed * 1000 + i).to(torch.complex128))
                for i, (r, c) in enumerate(_batch_shapes(case))]
    got = []
    for i, (op, rows, cols, dtype) in enumerate(_requests(case)):
        x = _image(rows, cols, seed * 1000 + i)
        x = x.to(torch.complex128) if dtype == fft.FFT2D_C64 else _unpack(*_pack(x, 0), 0)
        y = torch.fft.fft2(x)
        if op == fft.FFT2D_OP_LOWPASS:
            y = torch.fft.ifft2(_lowpass(y))
        got.append({"out": y} if dtype == fft.FFT2D_C64 else _exact_half(y))
    return got
