// filter.cu -- Gaussian low-pass multiply of an unshifted 2D spectrum, the
// "filter" step of the FFT -> filter -> inverse FFT image operation (the
// paper's motivating use, image filtering, Section 1).
//
// H[k][l] = exp(-d_k^2 / (2 s_r^2)) * exp(-d_l^2 / (2 s_c^2)),
// d_k = min(k, rows - k), d_l = min(l, cols - l), with s_r, s_c the caller's
// widths in frequency bins (side/8 in the serving workload).  H is real and
// <= 1, so for half2 storage the per-column exponents stay valid.
#include <cuda_fp16.h>

#include "async_copy.cuh"
#include "passes.h"

namespace fft2d {

namespace {

__device__ __forceinline__ float gauss_factor(int k, int n, float inv2s2)
{
    const int d = k < n - k ? k : n - k;
    return expf(-(float)d * (float)d * inv2s2);
}

__device__ __forceinline__ float2 scaled(float2 v, float h)
{
    return make_float2(v.x * h, v.y * h);
}
__device__ __forceinline__ __half2 scaled(__half2 q, float h)
{
    const float2 v = __half22float2(q);
    return __floats2half2_rn(v.x * h, v.y * h);
}

// Any width, height and alignment: one element per access.
template <class T>
__global__ void lowpass_kernel(T *x, int rows, int cols, float inv2sr2, float inv2sc2)
{
    const int row = blockIdx.y;
    const float hr = gauss_factor(row, rows, inv2sr2);
    T *line = x + (long long)row * cols;
    pdl_wait();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += gridDim.x * blockDim.x)
        line[c] = scaled(line[c], hr * gauss_factor(c, cols, inv2sc2));
}

// The same multiply bound by memory traffic: a thread owns one 16-byte chunk
// of columns (2 complex64 or 4 half2 pixels) of kLowpassRows rows, computes
// its columns' factors once, and has all its loads in flight before the
// first store.  The rows' factors are computed once per block in shared
// memory, while the kernel is still waiting for the previous one.  Factors
// and products are those of lowpass_kernel, bit for bit.  8 rows: 128 bytes
// of loads in flight per thread, and 1024 blocks at 2048^2.  Measured, images
// in turn: 4096^2 complex64 55.4 -> 40.1 us (6.7 TB/s read and written, the
// copy rate), half2 49.3 -> 21.3; 2048^2 16.5 -> 11.5, half2 12.3 -> 4.1;
// 1024^2 6.2 -> 3.9, half2 6.2 -> 3.1.
// Block: bx chunks of a row times 256 / bx rows; grid: (chunks / bx, rows / rows per block).
constexpr int kLowpassRows = 8;

template <class T>
__global__ void __launch_bounds__(256) lowpass_chunk_kernel(T *x, int rows, int cols, int bx,
                                                            float inv2sr2, float inv2sc2)
{
    constexpr int VEC = 16 / (int)sizeof(T);
    union Chunk {
        float4 v;
        T t[VEC];
        __device__ Chunk() {}
    };
    __shared__ float hr[256 * kLowpassRows];
    const int by = 256 / bx;                     // rows in step
    const int row0 = blockIdx.y * by * kLowpassRows;
    for (int i = threadIdx.x; i < by * kLowpassRows; i += 256)
        hr[i] = row0 + i < rows ? gauss_factor(row0 + i, rows, inv2sr2) : 0.f;
    const int tx = threadIdx.x % bx, ty = threadIdx.x / bx;
    const int c = (blockIdx.x * bx + tx) * VEC;
    float hc[VEC];
#pragma unroll
    for (int j = 0; j < VEC; j++)
        hc[j] = gauss_factor(c + j, cols, inv2sc2);
    __syncthreads();
    pdl_wait();
    T *p = x + (long long)(row0 + ty) * cols + c;
    Chunk q[kLowpassRows];
#pragma unroll
    for (int k = 0; k < kLowpassRows; k++)
        if (row0 + ty + k * by < rows)
            q[k].v = *reinterpret_cast<const float4 *>(p + (long long)k * by * cols);
#pragma unroll
    for (int k = 0; k < kLowpassRows; k++) {
        if (row0 + ty + k * by >= rows)
            continue;
#pragma unroll
        for (int j = 0; j < VEC; j++)
            q[k].t[j] = scaled(q[k].t[j], hr[ty + k * by] * hc[j]);
        *reinterpret_cast<float4 *>(p + (long long)k * by * cols) = q[k].v;
    }
}

template <class T>
cudaError_t lowpass_launch(T *x, int rows, int cols, float ir, float ic, cudaStream_t s)
{
    constexpr int VEC = 16 / (int)sizeof(T);
    const int chunks = cols / VEC;
    // whole chunks, and chunks per row a divisor or a multiple of the block
    if (rows <= 65535 && cols % VEC == 0 && !(reinterpret_cast<uintptr_t>(x) & 15) &&
        (chunks % 256 == 0 || 256 % chunks == 0)) {
        const int bx = chunks < 256 ? chunks : 256;
        const int per = 256 / bx * kLowpassRows;
        return launch_chained(lowpass_chunk_kernel<T>, dim3(chunks / bx, (rows + per - 1) / per), 256, 0,
                              s, 1, x, rows, cols, bx, ir, ic);
    }
    int bx = (cols + 255) / 256;
    if (bx > 16)
        bx = 16;
    return launch_chained(lowpass_kernel<T>, dim3(bx, rows), 256, 0, s, 1, x, rows, cols, ir, ic);
}

}  // namespace

cudaError_t launch_lowpass(bool half2, void *x, int rows, int cols, float sigma_r, float sigma_c,
                           cudaStream_t s)
{
    const float ir = 1.0f / (2.0f * sigma_r * sigma_r);
    const float ic = 1.0f / (2.0f * sigma_c * sigma_c);
    return half2 ? lowpass_launch(static_cast<__half2 *>(x), rows, cols, ir, ic, s)
                 : lowpass_launch(static_cast<float2 *>(x), rows, cols, ir, ic, s);
}

}  // namespace fft2d
