// any_axis.cuh -- one CTA's line transforms with the axis length chosen at run
// time: 2^12 values (256 threads x 16, 64 registers, 32 KB of shared memory)
// whatever the length, so that one kernel serves every length from 2 to 4096
// points.  A CTA takes 2^(12-L) rows or 2^(12-L) adjacent columns; the body is
// the line engine of the single-length kernels, so the bits are theirs.
#pragma once

#include "line_fft.cuh"

namespace fft2d {

constexpr int kAnyL = 12;   // log2 of the values per CTA

// Exchange buffer of 2^12 values, or (axes of up to 16 points: no exchange)
// the half2 exponent reduction of up to 2^11 lines; with an exchange, at most
// 2^7 lines reduce behind it.
constexpr int kAnySmem = (1 << kAnyL) * 8 + 128 * 4;

template <int L, bool ROW, class IO>
__device__ __forceinline__ void any_axis_of(const IO &io, const float2 *__restrict__ tw, float scale,
                                           int cta, int lines, int ld)
{
    using C = LineCfg<L, ROW ? 0 : kAnyL - L, ROW ? kAnyL - L : 0>;
    constexpr int PER = 1 << (kAnyL - L);   // lines per CTA
    const long long l0 = (long long)cta * PER;
    line_fft<C, ROW, true, IO>(io, ROW ? Geo{l0, 1, 0, ld} : Geo{0, 1, l0, ld}, tw, scale, L,
                               lines - l0);
}

template <bool ROW, class IO>
__device__ __forceinline__ void any_axis(int L, const IO &io, const float2 *__restrict__ tw,
                                            float scale, int cta, int lines, int ld)
{
    switch (L) {
    case 1: return any_axis_of<1, ROW>(io, tw, scale, cta, lines, ld);
    case 2: return any_axis_of<2, ROW>(io, tw, scale, cta, lines, ld);
    case 3: return any_axis_of<3, ROW>(io, tw, scale, cta, lines, ld);
    case 4: return any_axis_of<4, ROW>(io, tw, scale, cta, lines, ld);
    case 5: return any_axis_of<5, ROW>(io, tw, scale, cta, lines, ld);
    case 6: return any_axis_of<6, ROW>(io, tw, scale, cta, lines, ld);
    case 7: return any_axis_of<7, ROW>(io, tw, scale, cta, lines, ld);
    case 8: return any_axis_of<8, ROW>(io, tw, scale, cta, lines, ld);
    case 9: return any_axis_of<9, ROW>(io, tw, scale, cta, lines, ld);
    case 10: return any_axis_of<10, ROW>(io, tw, scale, cta, lines, ld);
    case 11: return any_axis_of<11, ROW>(io, tw, scale, cta, lines, ld);
    case 12: return any_axis_of<12, ROW>(io, tw, scale, cta, lines, ld);
    }
}

}  // namespace fft2d
