// dct_math.cuh -- the arithmetic between a complex line and the two real DCT
// lines that share it (the reduction is described in dct.cu).
#pragma once

#include <cuda_runtime.h>

namespace fft2d {

// The "two for one" split of Z = DFT(v_a + i v_b) into the DCT-II outputs of
// the real lines a and b (Makhoul's reduction): from Z[k], Z[k'] (k' = N - k)
// and (c, s) = (cos, sin)(pi k / (2N)),
//   xk = (X_a[k], X_b[k]),  xp = (X_a[k'], X_b[k']),  both times scale.
__device__ __forceinline__ void dct_pair(float2 zk, float2 zp, float2 cs, float scale,
                                         float2 &xk, float2 &xp)
{
    const float c = cs.x * 0.5f * scale, s = cs.y * 0.5f * scale;
    const float sr = zk.x + zp.x, dr = zp.x - zk.x;   // Zr[k] + Zr[k'], Zr[k'] - Zr[k]
    const float si = zk.y + zp.y, di = zk.y - zp.y;   // Zi[k] + Zi[k'], Zi[k] - Zi[k']
    xk = make_float2(c * sr + s * di, c * si + s * dr);     // (X_a[k], X_b[k])
    xp = make_float2(s * sr - c * di, s * si - c * dr);     // (X_a[k'], X_b[k'])
}

// The inverse's rotation before its DFT, for the partners k and N - k (0 < k
// <= N/2) of the spectrum z = X_a + i X_b: Z[k] and Z[N-k] (formulas in
// dct.cu), (c, s) = (cos, sin)(pi k / (2N)).
__device__ __forceinline__ void idct_pre(float2 za, float2 zb, float2 cs, float2 &yk, float2 &yp)
{
    const float ux = za.x + zb.y, uy = za.y - zb.x;
    const float vx = zb.x + za.y, vy = zb.y - za.x;
    yk = make_float2(cs.x * ux - cs.y * uy, cs.y * ux + cs.x * uy);
    yp = make_float2(cs.y * vx - cs.x * vy, cs.x * vx + cs.y * vy);
}

}  // namespace fft2d
