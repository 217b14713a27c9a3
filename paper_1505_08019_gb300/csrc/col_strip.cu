// col_strip.cu -- column pass for columns of 2^13 and 2^14 rows in two phases
// per strip of 32 complex columns, the strip's intermediate held in L2.
//
// A column this long fits no SM next to its neighbours, so its values change
// SMs once.  The DIT stages (Section 2 eqs. 2-3) split at any stage: with
// L = LA + LB, position p + 2^LA b of the scrambled column holds row
// c + 2^LB rev(p) with c = rev(b), so
//   phase 1, stages 1 .. LA:    for each residue c, 2^LA rows that lie 2^LB
//                               apart -> scratch row 2^LA b + p,
//   phase 2, stages LA+1 .. L:  for each lo < 2^LA, the 2^LB scratch rows
//                               lo + 2^LA r -> output index lo + 2^LA r.
// Both phases touch whole 128-byte (or 256-byte) row segments, need 16 values
// per thread and 32 KB of shared memory per CTA, and four CTAs share an SM,
// so loads, exchanges and stores of different items overlap -- against one
// CTA per SM in lockstep with its cluster in the kernels of col_group.cuh.
//
// An item is a pair of residues (phase 1) or of lo values (phase 2) times 16
// or 32 columns: 4096 complex values, 256 threads x 16.  The pairs are {c,
// C - c}, and {0, C/2}: then the DCT's partners k and N - k (two real columns
// per complex line, see dct.cu) are in one item, and in one thread except in
// the item of 0 and C/2.
//
// Launches.  Launch j runs phase 1 of chunk j and phase 2 of chunk j - 1,
// whose items alternate in the grid (reads of the image from HBM beside
// writes to it); a chunk is kChunk strips, so that the two chunks of scratch
// in use stay in L2.  The kernel boundary is the only synchronisation:
// chained launches (launch_chained).  One persistent launch whose
// items waited for counters published with release increments took 0.84 -
// 0.94 ms where this takes 0.69 (16384^2 inverse DCT): every publication waits
// until the item's scattered stores are performed.
//
// What bounds it: L2 traffic.  Each value crosses the SM - L2 boundary four
// times (image in, scratch out and in, image out).  A copy that stays in L2
// runs at 8.1 TB/s on a GB300 (read + written), HBM at 6.0 - 6.8; the 16384^2
// DCT column pass moves its 4.3 GB at 6.3 TB/s.  The output goes past L2's
// normal priority (st.global.cs) so that the scratch stays: 0.75 -> 0.69 ms.
// Measured, column pass, before (cluster kernels) / here: 16384^2 inverse DCT
// 1.37 / 0.69 ms, forward 0.80 / 0.68; 8192^2 DCT 0.20 / 0.17; 16384x1024
// inverse DCT 100 / 45 us; 8192x64 DCT 19 / 6.5 us (complex64: kernels_col.cu).
// 5 CTAs per SM (48 registers) changed nothing, 6 spilled and took 1.1 ms.
#include <cstdint>

#include "dct_math.cuh"
#include "line_fft.cuh"
#include "passes.h"

namespace fft2d {

namespace {

constexpr int kStripCols = 32;            // complex columns of a strip
constexpr long long kChunkBytes = 32ll << 20;   // scratch of a chunk; two are in use

enum { kStripC64 = 0, kStripDct = 1, kStripIdct = 2 };

struct StripArgs {
    const float2 *in;
    float2 *out;
    long long ld;                         // row pitch in complex values
    int cols;                             // complex columns
    const float2 *tw, *post;
    float scale;
    // first strip, items and scratch of each phase in this launch
    int strip[2], items[2];
    float2 *scratch[2];
};

// Stages t = 0 .. G-1 of one unit a[base + r], r < 2^G, with the factors of
// stage t from fetch(t, m); the same butterflies as run_stages_g.
template <int G, bool FIRST, class F>
__device__ __forceinline__ void unit_stages(float2 (&a)[16], int base, float p, F fetch)
{
#pragma unroll
    for (int t = 0; t < G; t++) {
#pragma unroll
        for (int r = 0; r < (1 << G); r++) {
            if (r & (1 << t))
                continue;
            const int m = r & ((1 << t) - 1);
            float2 &x0 = a[base + r];
            float2 &x1 = a[base + (r | (1 << t))];
            if (FIRST && m == 0) {
                const float2 d = x1;
                x1 = make_float2(__fsub_rn(x0.x, d.x), __fsub_rn(x0.y, d.y));
                x0 = make_float2(__fadd_rn(x0.x, d.x), __fadd_rn(x0.y, d.y));
            } else if (t >= 1 && m >= (1 << (t - 1))) {
                const int m0 = m - (1 << (t - 1));
                const float2 w = FIRST && m0 == 0 ? make_float2(1.f, 0.f) : fetch(t, m0);
                butterfly_w(x0, x1, quarter_turn(w, p));
            } else {
                butterfly_w(x0, x1, fetch(t, m));
            }
        }
    }
}

template <int LA, int LB>
struct StripCfg {
    static constexpr int L = LA + LB, N = 1 << L;
    static constexpr int NA = 1 << LA, NB = 1 << LB;      // points of phases 1 and 2
    static constexpr int W1 = 2048 / NA, W2 = 2048 / NB;  // columns of an item
    static constexpr int N1 = NB / 2 * (kStripCols / W1); // items per strip and phase
    static constexpr int N2 = NA / 2 * (kStripCols / W2);
    static constexpr long long SLOT = (long long)N * kStripCols;
    static constexpr int CHUNK = (int)(kChunkBytes / (SLOT * 8));   // strips
    static_assert(N1 == N2, "the phases have equal items");
    static_assert(LA == 7 && (LB == 6 || LB == 7), "stage splits 7 + 6 and 7 + 7");
};

// Row of the image that element n of the (reordered) column comes from or
// goes to; lower: n < N/2, known at compile time where this is called.
template <int N>
__device__ __forceinline__ int dct_row(int n, bool lower)
{
    return lower ? 2 * n : 2 * (N - 1 - n) + 1;
}

template <int MODE, int LA, int LB>
__global__ void __launch_bounds__(256, 4) col_strip_kernel(const StripArgs g)
{
    using S = StripCfg<LA, LB>;
    constexpr int N = S::N, NB = S::NB;
    __shared__ float2 sm[4096];
    __shared__ float2 tw1[S::NA];            // stages 1 .. LA
    __shared__ float2 tw2[2 * NB];           // stages LA+1 .. L of the item's two lo
    const int tid = threadIdx.x;

    pdl_wait();
    // items of the two phases alternate as long as there are both
    const int both = 2 * (g.items[0] < g.items[1] ? g.items[0] : g.items[1]);
    const int blk = (int)blockIdx.x;
    const int phase = blk < both ? 1 - (blk & 1) : g.items[0] > g.items[1] ? 0 : 1;
    const int item = blk < both ? blk >> 1 : blk - both / 2;
    constexpr int PER = S::N1;               // items per strip, either phase
    const int rel = item / PER, idx = item % PER;
    const int strip = (phase ? g.strip[1] : g.strip[0]) + rel;
    const float p = -__ldg(g.tw + 2).y;      // sign of the quarter turn
    float2 a[16];
    float2 *slot = (phase ? g.scratch[1] : g.scratch[0]) + rel * S::SLOT;
    if (phase == 0) {
        if (tid < S::NA - 1)
            tw1[tid] = __ldg(g.tw + tid);   // read after the exchange barrier
        constexpr int W = S::W1;         // 16: half-warps run over columns
        const int w = tid % W, u = tid / W;
        const int pi = idx / (kStripCols / W);
        const int wb = idx % (kStripCols / W) * W + w;    // column of the strip
        const int col = strip * kStripCols + wb;
        const bool live = col < g.cols;
        const int c0 = pi, c1 = pi == 0 ? NB / 2 : NB - pi;  // the two residues
        const float2 *src = g.in + col;
        if constexpr (MODE == kStripIdct) {
            // units (c0, hib) and (c1, 15 - hib), 3 stages; position
            // index r holds row c + NB i, i = rev3(r) 16 | hib
            const float2 z = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 8; r++) {
                const int i0 = brev_c(r, 3) * 16 + u, i1 = brev_c(r, 3) * 16 + 15 - u;
                a[r] = live ? ld_stream(src + (long long)(c0 + NB * i0) * g.ld) : z;
                a[8 + r] = live ? ld_stream(src + (long long)(c1 + NB * i1) * g.ld) : z;
            }
            if (pi != 0) {
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    const int k = c0 + NB * (brev_c(r, 3) * 16 + u);
                    const float2 x0 = a[r], x1 = a[15 - r];       // k and N - k
                    if (r % 2 == 0)                                // k < N/2
                        idct_pre(x0, x1, __ldg(g.post + k), a[r], a[15 - r]);
                    else
                        idct_pre(x1, x0, __ldg(g.post + (N - k)), a[15 - r], a[r]);
                }
            } else {
                // residues 0 and NB/2 are their own mirrors, in other
                // threads: partners through shared memory
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int i = brev_c(j % 8, 3) * 16 + (j < 8 ? u : 15 - u);
                    sm[(j / 8 << LA | i) * W + w] = a[j];
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int i = brev_c(j % 8, 3) * 16 + (j < 8 ? u : 15 - u);
                    const int im = j < 8 ? (S::NA - i) & (S::NA - 1) : S::NA - 1 - i;
                    const int k = (j < 8 ? 0 : NB / 2) + NB * i;
                    if (k == 0)
                        continue;                                  // X[N] = 0
                    const float2 o = sm[(j / 8 << LA | im) * W + w];
                    float2 yk, yp;
                    if (k <= N / 2) {
                        idct_pre(a[j], o, __ldg(g.post + k), yk, yp);
                        a[j] = yk;
                    } else {
                        idct_pre(o, a[j], __ldg(g.post + (N - k)), yk, yp);
                        a[j] = yp;
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int v = 0; v < 2; v++) {
                unit_stages<3, true>(a, 8 * v, p,
                                     [&](int t, int m) { return __ldg(g.tw + (1 << t) - 1 + m); });
                const int hi = brev_rt(v ? 15 - u : u, 4);
#pragma unroll
                for (int r = 0; r < 8; r++)
                    sm[((v << LA) | r | (hi << 3)) * W + w] = a[8 * v + r];
            }
            __syncthreads();
            const int set = u >> 3, lo = u & 7;
#pragma unroll
            for (int r = 0; r < 16; r++)
                a[r] = sm[((set << LA) | lo | (r << 3)) * W + w];
            unit_stages<4, false>(a, 0, p,
                                  [&](int t, int m) { return tw1[(8 << t) - 1 + lo + 8 * m]; });
            const int b = brev_rt(set ? c1 : c0, LB);
            float2 *dst = slot + ((b << LA) | lo) * kStripCols + wb;
#pragma unroll
            for (int r = 0; r < 16; r++)
                dst[(r << 3) * kStripCols] = a[r];
        } else {
            // unit (set, hib), 4 stages; index r holds element
            // n = c + NB i, i = rev4(r) 8 | hib
            const int set = u >> 3, hib = u & 7;
            const int c = set ? c1 : c0;
#pragma unroll
            for (int r = 0; r < 16; r++) {
                const int n = c + NB * (brev_c(r, 4) * 8 + hib);
                const int row = MODE == kStripDct ? dct_row<N>(n, r % 2 == 0) : n;
                a[r] = live ? ld_stream(src + (long long)row * g.ld) : make_float2(0.f, 0.f);
            }
            unit_stages<4, true>(a, 0, p,
                                 [&](int t, int m) { return __ldg(g.tw + (1 << t) - 1 + m); });
            const int hi = brev_rt(hib, 3);
#pragma unroll
            for (int r = 0; r < 16; r++)
                sm[((set << LA) | r | (hi << 4)) * W + w] = a[r];
            __syncthreads();
#pragma unroll
            for (int v = 0; v < 2; v++) {
#pragma unroll
                for (int r = 0; r < 8; r++)
                    a[8 * v + r] = sm[((v << LA) | u | (r << 4)) * W + w];
                unit_stages<3, false>(a, 8 * v, p,
                                      [&](int t, int m) { return tw1[(16 << t) - 1 + u + 16 * m]; });
                const int b = brev_rt(v ? c1 : c0, LB);
                float2 *dst = slot + ((b << LA) | u) * kStripCols + wb;
#pragma unroll
                for (int r = 0; r < 8; r++)
                    dst[(r << 4) * kStripCols] = a[8 * v + r];
            }
        }
    } else {
        constexpr int W = S::W2;         // 16, or a whole warp of columns
        const int w = tid % W, u = tid / W;
        const int li = idx / (kStripCols / W);
        const int wb = idx % (kStripCols / W) * W + w;
        const int col = strip * kStripCols + wb;
        const bool live = col < g.cols;
        const int lo0 = li, lo1 = li == 0 ? S::NA / 2 : S::NA - li;
        // value index j of this thread: unit v = j / 8 (7 + 7: one unit
        // of 16), scratch row lo + 2^LA b
#pragma unroll
        for (int j = 0; j < 16; j++) {
            const int set = LB == 7 ? u >> 3 : j / 8;
            const int b = LB == 7 ? j | (u & 7) << 4 : j % 8 | u << 3;
            a[j] = ld_l2(slot + ((b << LA) | (set ? lo1 : lo0)) * kStripCols + wb);
        }
        if (tid < 2 * (NB - 1)) {
            const int set = tid / (NB - 1), e = tid % (NB - 1) + 1;
            const int t = 31 - __clz(e), m = e - (1 << t);
            tw2[set * NB + e - 1] =
                __ldg(g.tw + (S::NA << t) - 1 + (set ? lo1 : lo0) + S::NA * m);
        }
        __syncthreads();
        if constexpr (LB == 7) {
            const int set = u >> 3, rhi = u & 7;
            unit_stages<4, false>(a, 0, p,
                                  [&](int t, int m) { return tw2[set * NB + (1 << t) - 1 + m]; });
#pragma unroll
            for (int r = 0; r < 16; r++)
                sm[((set << LB) | r | (rhi << 4)) * W + w] = a[r];
        } else {
#pragma unroll
            for (int v = 0; v < 2; v++) {
                unit_stages<3, false>(a, 8 * v, p,
                                      [&](int t, int m) { return tw2[v * NB + (1 << t) - 1 + m]; });
#pragma unroll
                for (int r = 0; r < 8; r++)
                    sm[((v << LB) | r | (u << 3)) * W + w] = a[8 * v + r];
            }
        }
        __syncthreads();
        // last three stages: units (lo0, rl) and (lo1, mirrored rl)
        constexpr int GL = LB - 3, RL = 1 << GL;
#pragma unroll
        for (int v = 0; v < 2; v++) {
            const int rl = v ? RL - 1 - u : u;
#pragma unroll
            for (int r = 0; r < 8; r++)
                a[8 * v + r] = sm[((v << LB) | rl | (r << GL)) * W + w];
            unit_stages<3, false>(a, 8 * v, p,
                                  [&](int t, int m) { return tw2[v * NB + (RL << t) - 1 + rl + RL * m]; });
        }
        float2 *dst = g.out + col;
        if constexpr (MODE == kStripDct) {
            // output K = lo + 2^LA b, partner N - K: index 15 - j of the
            // same thread, or (lo 0 and 2^LA / 2) through shared memory
            if (li != 0) {
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    const int K = lo0 + S::NA * (u | r << GL);
                    const float2 x0 = a[r], x1 = a[15 - r];
                    if (r < 4)                                   // K < N/2
                        dct_pair(x0, x1, __ldg(g.post + K), g.scale, a[r], a[15 - r]);
                    else
                        dct_pair(x1, x0, __ldg(g.post + (N - K)), g.scale, a[15 - r], a[r]);
                }
            } else {
                __syncthreads();
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int v = j / 8, rl = v ? RL - 1 - u : u;
                    sm[((v << LB) | rl | ((j % 8) << GL)) * W + w] = a[j];
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int v = j / 8, rl = v ? RL - 1 - u : u;
                    const int b = rl | (j % 8) << GL;
                    const int K = (v ? lo1 : 0) + S::NA * b;
                    const int bm = v ? NB - 1 - b : (NB - b) & (NB - 1);
                    const float2 o = sm[((v << LB) | bm) * W + w];
                    float2 xk, xp;
                    if (K <= N / 2) {
                        dct_pair(a[j], o, __ldg(g.post + K), g.scale, xk, xp);
                        a[j] = xk;
                    } else {
                        dct_pair(o, a[j], __ldg(g.post + (N - K)), g.scale, xk, xp);
                        a[j] = xp;
                    }
                }
            }
        }
        if (live) {
#pragma unroll
            for (int j = 0; j < 16; j++) {
                const int v = j / 8, r = j % 8, rl = v ? RL - 1 - u : u;
                const int n = (v ? lo1 : lo0) + S::NA * (rl | r << GL);
                const int row = MODE == kStripIdct ? dct_row<N>(n, r < 4) : n;
                const float f = MODE == kStripDct ? 1.f : g.scale;
                st_stream(dst + (long long)row * g.ld, make_float2(a[j].x * f, a[j].y * f));
            }
        }
    }
}

template <int MODE, int LA, int LB>
cudaError_t strip_launch(const StripPass &a, cudaStream_t s)
{
    using S = StripCfg<LA, LB>;
    if (a.cols < 1 ||
        ((reinterpret_cast<uintptr_t>(a.in) | reinterpret_cast<uintptr_t>(a.out)) & 7))
        return cudaErrorNotSupported;
    StripArgs g;
    g.in = a.in;
    g.out = a.out;
    g.ld = a.ld;
    g.cols = a.cols;
    g.tw = a.tw;
    g.post = a.post;
    g.scale = a.scale;
    auto k = col_strip_kernel<MODE, LA, LB>;
    const int nstrips = (a.cols + kStripCols - 1) / kStripCols;
    // two chunks of scratch, smaller ones where the device has no room
    int per = nstrips < S::CHUNK ? nstrips : S::CHUNK;
    void *block = nullptr;
    cudaError_t e;
    for (;; per = (per + 1) / 2) {
        const size_t chunks = per < nstrips ? 2 : 1;
        e = scratch_take(&block, chunks * per * S::SLOT * sizeof(float2), s);
        if (e != cudaErrorMemoryAllocation)
            break;
        cudaGetLastError();
        if (per == 1)
            return cudaErrorNotSupported;
    }
    if (e != cudaSuccess)
        return e;
    const int nchunks = (nstrips + per - 1) / per;
    auto strips = [&](int c) {   // of chunk c
        return c < 0 || c >= nchunks ? 0 : nstrips - c * per < per ? nstrips - c * per : per;
    };
    for (int j = 0; j <= nchunks && e == cudaSuccess; j++) {
        for (int ph = 0; ph < 2; ph++) {
            const int c = j - ph;
            g.strip[ph] = c * per;
            g.items[ph] = strips(c) * S::N1;
            g.scratch[ph] = static_cast<float2 *>(block) + (c & 1) * per * S::SLOT;
        }
        e = launch_chained(k, dim3((unsigned)(g.items[0] + g.items[1])), 256, 0, s, 1, g);
    }
    const cudaError_t f = cudaFreeAsync(block, s);
    return e != cudaSuccess ? e : f;
}

}  // namespace

cudaError_t launch_col_strip(StripKind kind, int L, const StripPass &a, cudaStream_t s)
{
    if (L != 13 && L != 14)
        return cudaErrorNotSupported;
    switch (kind) {
    case StripKind::C64:
        return L == 13 ? strip_launch<kStripC64, 7, 6>(a, s) : strip_launch<kStripC64, 7, 7>(a, s);
    case StripKind::Dct:
        return L == 13 ? strip_launch<kStripDct, 7, 6>(a, s) : strip_launch<kStripDct, 7, 7>(a, s);
    case StripKind::Idct:
        return L == 13 ? strip_launch<kStripIdct, 7, 6>(a, s) : strip_launch<kStripIdct, 7, 7>(a, s);
    }
    return cudaErrorNotSupported;
}

}  // namespace fft2d
