// small.cu -- the whole 2D transform of a small image in one launch.
//
// Up to 2^16 pixels an image is a few microseconds of launch and latency, not
// of bandwidth: two launches of 8 to 16 CTAs each.  Here one cluster of at
// most 16 CTAs holds the image, 4096 values (256 threads x 16) per CTA: every
// CTA transforms its 4096 / cols rows into `out` (which stays in L2), one
// cluster barrier orders that before the reads of the column phase, and every
// CTA transforms its 4096 / rows columns in place.  Both phases are the
// per-CTA line transforms of the two-launch path, so the results are its
// results bit for bit.  The axis lengths are chosen at run time inside the
// kernel (both phases have the same CTA shape whatever the length).
//
// What bounds it: the latency of two load - exchange - store chains and the
// barrier between them.  Measured, calls in a row: a 256^2 forward transform
// takes 5.0 us against 10.1 in two launches.  Why 4096 values per CTA: the same 64-register,
// 32 KB configuration serves every axis from 2 to 4096 points, and 16 CTAs
// spread 2^16 pixels over as many SMs as one cluster may span.
#include "any_axis.cuh"
#include "passes.h"

namespace fft2d {

namespace {

constexpr int kSmallMaxCtas = 16;         // largest cluster (non-portable above 8)

// The column phase reads what other CTAs of the cluster have just written.
struct StoreC64Shared : StoreC64 {
    static constexpr bool CG = true;
};
template <int IA>
struct StoreH16Shared : StoreH16T<IA> {
    static constexpr bool CG = true;
};

// One cluster = the whole grid.  rio / cio: the storage of the two phases.
template <class RIO, class CIO>
__global__ void __launch_bounds__(256, 4) small_kernel(const RIO rio, const CIO cio,
                                                       const float2 *__restrict__ tw_rows,
                                                       const float2 *__restrict__ tw_cols, int rows,
                                                       int cols, int Lr, int Lc, float scale)
{
    const int cta = (int)blockIdx.x;
    any_axis<true>(Lc, rio, tw_rows, 1.0f, cta, rows, cols);
    // every row is in `out` before any column is read, and the exchange
    // buffer is free again
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    any_axis<false>(Lr, cio, tw_cols, scale, cta, cols, cols);
}

int small_ctas(int Lr, int Lc) { return Lr + Lc > kAnyL ? 1 << (Lr + Lc - kAnyL) : 1; }

// Whether the device takes the kernel in clusters of `ctas`: above 8 they are
// opt-in, and a device may refuse them.
template <class RIO, class CIO>
bool small_cluster_ok(int ctas)
{
    if (ctas <= 8)
        return true;
    auto k = small_kernel<RIO, CIO>;
    static DeviceCache ok;   // 1: usable, 2: not
    const int d = device_current();
    if (!ok.get(d)) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        int n = 0;
        if (e == cudaSuccess) {
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = kSmallMaxCtas;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kSmallMaxCtas);
            cfg.blockDim = dim3(256);
            cfg.dynamicSmemBytes = kAnySmem;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
        }
        if (e != cudaSuccess)
            cudaGetLastError();
        ok.set(d, e == cudaSuccess && n > 0 ? 1 : 2);
    }
    return ok.get(d) == 1;
}

template <class RIO, class CIO>
cudaError_t small_launch(const RIO &rio, const CIO &cio, const SmallArgs &a, cudaStream_t s)
{
    const int ctas = small_ctas(a.Lr, a.Lc);
    if (!small_cluster_ok<RIO, CIO>(ctas))
        return cudaErrorNotSupported;
    return launch_chained(small_kernel<RIO, CIO>, dim3(ctas), 256, kAnySmem, s,
                          LaunchHow((unsigned)ctas), rio, cio, a.tw_rows, a.tw_cols, 1 << a.Lr,
                          1 << a.Lc, a.Lr, a.Lc, a.scale);
}

}  // namespace

// 2^16 pixels is the most that one cluster holds at 4096 values per CTA.
bool small_image(int Lr, int Lc)
{
    return Lr >= 1 && Lc >= 1 && Lr <= kAnyL && Lc <= kAnyL && Lr + Lc <= kAnyL + 4;
}

int small_image_ctas(bool half2, int Lr, int Lc)
{
    if (!small_image(Lr, Lc))
        return 0;
    const int ctas = small_ctas(Lr, Lc);
    const bool ok = half2 ? small_cluster_ok<StoreH16T<0>, StoreH16Shared<0>>(ctas)
                          : small_cluster_ok<StoreC64, StoreC64Shared>(ctas);
    return ok ? ctas : 0;
}

cudaError_t launch_small(const SmallArgs &a, const float2 *in, float2 *out, cudaStream_t s)
{
    StoreC64Shared c;
    c.in = out;
    c.out = out;
    return small_launch(StoreC64{in, out}, c, a, s);
}

cudaError_t launch_small_h16(const SmallArgs &a, const __half2 *in, const int *in_exp, int in_axis,
                             __half2 *out, int *row_exp, int *out_exp, cudaStream_t s)
{
    StoreH16Shared<0> c;
    c.in = out;
    c.out = out;
    c.in_exp = row_exp;
    c.in_axis = 0;
    c.out_exp = out_exp;
    return in_axis == 0 ? small_launch(StoreH16T<0>{in, out, in_exp, 0, row_exp}, c, a, s)
                        : small_launch(StoreH16T<1>{in, out, in_exp, 1, row_exp}, c, a, s);
}

}  // namespace fft2d
