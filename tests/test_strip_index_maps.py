"""The index maps of the two-phase strip column kernel (columns of 8192 and
16384 rows), rebuilt in numpy from the formulas of its source and checked on
the CPU: which row a thread loads, the shared-memory slots between its stage
groups, the scratch rows between the phases, the partners k and N - k of the
DCT kinds, and the row every result goes to.  Each slot must be written once
and read by the thread that expects it, and the result must be the transform.
"""
import numpy as np
import pytest

LA = 7
NA = 1 << LA
COLS = 2            # data columns carried along (the kernel's w)


def brev(x, bits):
    return int(format(x, f"0{bits}b")[::-1], 2)


class Slots:
    """A buffer whose slots are written once before they are read."""

    def __init__(self, n):
        self.v = np.full((n, COLS), np.nan + 0j)
        self.writes = np.zeros(n, int)

    def put(self, i, x):
        self.v[i] = x
        self.writes[i] += 1

    def get(self, i):
        assert self.writes[i] == 1, i
        return self.v[i]

    def full(self):
        return self.writes.min() == 1 and self.writes.max() == 1


def stages(a, base, groups, factor):
    """Stages t < groups on a[base .. base + 2^groups): factor(t, m)."""
    for t in range(groups):
        for r in range(1 << groups):
            if r & (1 << t):
                continue
            d = factor(t, r & ((1 << t) - 1)) * a[base + (r | 1 << t)]
            a[base + (r | 1 << t)] = a[base + r] - d
            a[base + r] = a[base + r] + d


def rot(sign, stage, j):
    """The plan's table: W of 2^stage to the j."""
    assert 0 <= j < 1 << (stage - 1)
    return np.exp(sign * 2j * np.pi * j / (1 << stage))


def dct_row(n, N):
    return 2 * n if n < N // 2 else 2 * (N - 1 - n) + 1


def dct_pair(zk, zp, cs):
    c, s = cs.real / 2, cs.imag / 2
    sr, dr, si, di = zk.real + zp.real, zp.real - zk.real, zk.imag + zp.imag, zk.imag - zp.imag
    return (c * sr + s * di) + 1j * (c * si + s * dr), (s * sr - c * di) + 1j * (s * si - c * dr)


def idct_pre(za, zb, cs):
    ux, uy, vx, vy = za.real + zb.imag, za.imag - zb.real, zb.real + za.imag, zb.imag - za.real
    c, s = cs.real, cs.imag
    return (c * ux - s * uy) + 1j * (s * ux + c * uy), (s * vx - c * vy) + 1j * (c * vx + s * vy)


def post(k, N):
    assert 0 <= k <= N // 2
    return np.exp(1j * np.pi * k / (2 * N))


def phase1(X, LB, kind, sign):
    NB, N = 1 << LB, NA << LB
    scratch, read = Slots(N), np.zeros(N, int)
    for pi in range(NB // 2):
        c0, c1 = pi, NB // 2 if pi == 0 else NB - pi
        sm = Slots(2 * NA)
        a = {}

        def load(row):
            read[row] += 1
            return X[row].copy()

        if kind == "idct":
            i_of = {(u, j): brev(j % 8, 3) * 16 + (u if j < 8 else 15 - u)
                    for u in range(16) for j in range(16)}
            for u in range(16):
                a[u] = [load((c0 if j < 8 else c1) + NB * i_of[u, j]) for j in range(16)]
            if pi:
                for u in range(16):
                    for r in range(8):
                        k = c0 + NB * (brev(r, 3) * 16 + u)
                        assert (c1 + NB * i_of[u, 15 - r]) == N - k
                        x0, x1 = a[u][r], a[u][15 - r]
                        if r % 2 == 0:
                            a[u][r], a[u][15 - r] = idct_pre(x0, x1, post(k, N))
                        else:
                            a[u][15 - r], a[u][r] = idct_pre(x1, x0, post(N - k, N))
            else:
                pre = Slots(2 * NA)
                for u in range(16):
                    for j in range(16):
                        pre.put(j // 8 << LA | i_of[u, j], a[u][j])
                for u in range(16):
                    for j in range(16):
                        i = i_of[u, j]
                        im = (NA - i) & (NA - 1) if j < 8 else NA - 1 - i
                        k = (0 if j < 8 else NB // 2) + NB * i
                        if k == 0:
                            continue
                        assert (0 if j < 8 else NB // 2) + NB * im == N - k
                        o = pre.get(j // 8 << LA | im)
                        if k <= N // 2:
                            a[u][j] = idct_pre(a[u][j], o, post(k, N))[0]
                        else:
                            a[u][j] = idct_pre(o, a[u][j], post(N - k, N))[1]
            for u in range(16):
                for v in range(2):
                    stages(a[u], 8 * v, 3, lambda t, m: rot(sign, t + 1, m))
                    hi = brev(15 - u if v else u, 4)
                    for r in range(8):
                        sm.put(v << LA | r | hi << 3, a[u][8 * v + r])
            assert sm.full()
            for u in range(16):
                s, lo = u >> 3, u & 7
                y = [sm.get(s << LA | lo | r << 3).copy() for r in range(16)]
                stages(y, 0, 4, lambda t, m: rot(sign, t + 4, lo + 8 * m))
                for r in range(16):
                    scratch.put(brev(c1 if s else c0, LB) << LA | lo | r << 3, y[r])
        else:
            for u in range(16):
                s, hib = u >> 3, u & 7
                n = [(c1 if s else c0) + NB * (brev(r, 4) * 8 + hib) for r in range(16)]
                if kind == "dct":
                    assert all((n[r] < N // 2) == (r % 2 == 0) for r in range(16))
                y = [load(dct_row(q, N) if kind == "dct" else q) for q in n]
                stages(y, 0, 4, lambda t, m: rot(sign, t + 1, m))
                for r in range(16):
                    sm.put(s << LA | r | brev(hib, 3) << 4, y[r])
            assert sm.full()
            for u in range(16):
                for v in range(2):
                    y = [sm.get(v << LA | u | r << 4).copy() for r in range(8)]
                    stages(y, 0, 3, lambda t, m: rot(sign, t + 5, u + 16 * m))
                    for r in range(8):
                        scratch.put(brev(c1 if v else c0, LB) << LA | u | r << 4, y[r])
    assert read.min() == 1 and read.max() == 1 and scratch.full()
    return scratch


def phase2(scratch, LB, kind, sign):
    NB, N = 1 << LB, NA << LB
    out = Slots(N)
    threads = 16 if LB == 7 else 8
    GL = LB - 3
    RL = 1 << GL
    for li in range(NA // 2):
        lo = (li, NA // 2 if li == 0 else NA - li)
        sm = Slots(2 * NB)
        for u in range(threads):
            where = [(u >> 3, j | (u & 7) << 4) if LB == 7 else (j // 8, j % 8 | u << 3)
                     for j in range(16)]
            y = [scratch.get(b << LA | lo[s]).copy() for s, b in where]
            if LB == 7:
                stages(y, 0, 4, lambda t, m: rot(sign, LA + t + 1, lo[u >> 3] + NA * m))
                for r in range(16):
                    sm.put(u >> 3 << LB | r | (u & 7) << 4, y[r])
            else:
                for v in range(2):
                    stages(y, 8 * v, 3, lambda t, m: rot(sign, LA + t + 1, lo[v] + NA * m))
                    for r in range(8):
                        sm.put(v << LB | r | u << 3, y[8 * v + r])
        assert sm.full()
        last, ex = {}, Slots(2 * NB)
        for u in range(threads):
            y = []
            for v in range(2):
                rl = RL - 1 - u if v else u
                z = [sm.get(v << LB | rl | r << GL).copy() for r in range(8)]
                stages(z, 0, 3, lambda t, m: rot(sign, LA + GL + t + 1, lo[v] + NA * (rl + RL * m)))
                y += z
            last[u] = y
            for j in range(16):
                ex.put(j // 8 << LB | (RL - 1 - u if j >= 8 else u) | (j % 8) << GL, y[j])
        assert ex.full()
        for u in range(threads):
            K = [lo[j // 8] + NA * ((RL - 1 - u if j >= 8 else u) | (j % 8) << GL) for j in range(16)]
            y = list(last[u])
            if kind == "dct" and li:
                for r in range(8):
                    assert K[15 - r] == N - K[r] and (K[r] < N // 2) == (r < 4)
                    x0, x1 = last[u][r], last[u][15 - r]
                    if r < 4:
                        y[r], y[15 - r] = dct_pair(x0, x1, post(K[r], N))
                    else:
                        y[15 - r], y[r] = dct_pair(x1, x0, post(N - K[r], N))
            elif kind == "dct":
                for j in range(16):
                    v = j // 8
                    b = (RL - 1 - u if v else u) | (j % 8) << GL
                    bm = NB - 1 - b if v else (NB - b) & (NB - 1)
                    assert lo[v] + NA * bm == (N - K[j]) % N
                    o = ex.get(v << LB | bm)
                    y[j] = dct_pair(last[u][j], o, post(K[j], N))[0] if K[j] <= N // 2 \
                        else dct_pair(o, last[u][j], post(N - K[j], N))[1]
            for j in range(16):
                if kind == "idct":
                    assert (K[j] < N // 2) == (j % 8 < 4)
                out.put(dct_row(K[j], N) if kind == "idct" else K[j], y[j])
    assert out.full()
    return out.v


@pytest.mark.parametrize("kind,sign", [("c64", -1), ("c64", 1), ("dct", -1), ("idct", 1)])
@pytest.mark.parametrize("LB", [6, 7])
def test_strip_maps(LB, kind, sign):
    N = NA << LB
    rng = np.random.default_rng(LB)
    X = rng.standard_normal((N, COLS)) + 1j * rng.standard_normal((N, COLS))
    got = phase2(phase1(X, LB, kind, sign), LB, kind, sign)
    if kind == "c64":
        want = np.fft.fft(X, axis=0) if sign < 0 else np.fft.ifft(X, axis=0) * N
    elif kind == "dct":
        # both real columns of a complex one: X[k] = Re(exp(-i pi k / 2N) V[k])
        v = np.concatenate([X[0::2], X[1::2][::-1]])
        k = np.arange(N)[:, None]
        turn = np.exp(-1j * np.pi * k / (2 * N))
        want = (turn * np.fft.fft(v.real, axis=0)).real + 1j * (turn * np.fft.fft(v.imag, axis=0)).real
    else:
        # x[n] = X[0] + 2 sum X[k] cos(pi k (2n + 1) / 2N), at sampled rows
        rows = np.sort(rng.choice(N, 64, replace=False))
        k = np.arange(N)[None, :]
        C = np.cos(np.pi * k * (2 * rows[:, None] + 1) / (2 * N)) * np.where(k == 0, 1.0, 2.0)
        want, got = C @ X, got[rows]
    assert np.abs(got - want).max() <= 1e-11 * np.abs(want).max()
