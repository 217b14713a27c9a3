// batch_any.cu -- grouped launches over images of any axis lengths: one row
// launch and one column launch for a whole batch (any_axis.cuh), where the
// per-length launches of batch.cu took one per (pass, length, direction) on
// four streams joined by events.  A batch of small images is bound by its
// launches and events on the host and by the gaps between small kernels on
// the device, not by its traffic.
#include "any_axis.cuh"
#include "batch_job.cuh"
#include "passes.h"

namespace fft2d {

namespace {

template <bool ROW, class Table>
__global__ void __launch_bounds__(256, 4) batch_any_kernel(const __grid_constant__ Table t)
{
    const BatchJob &jb = t.job[find_job(t)];
    any_axis<ROW>(jb.L, StoreC64{jb.in, jb.out}, jb.tw, jb.scale, (int)blockIdx.x - jb.first_cta,
                  jb.lines, (int)jb.ld);
}

template <bool ROW, int IA>
__global__ void __launch_bounds__(256, 4) batch_any_h16_kernel(const __grid_constant__ BatchTableH16 t)
{
    const BatchJobH16 &jb = t.job[find_job(t)];
    any_axis<ROW>(jb.L, StoreH16T<IA>{jb.in, jb.out, jb.in_exp, IA, jb.out_exp}, jb.tw, jb.scale,
                  (int)blockIdx.x - jb.first_cta, jb.lines, (int)jb.ld);
}

template <class Table>
int fill_ctas(Table &t)
{
    int ctas = 0;
    for (int i = 0; i < t.n; i++) {
        const int per = 1 << (kAnyL - t.job[i].L);   // lines per CTA
        t.job[i].first_cta = ctas;
        ctas += (t.job[i].lines + per - 1) / per;
    }
    return ctas;
}

template <class Table>
cudaError_t any_launch(bool row, Table &t, cudaStream_t s)
{
    const int ctas = fill_ctas(t);
    if (ctas == 0)
        return cudaSuccess;
    return launch_chained(row ? batch_any_kernel<true, Table> : batch_any_kernel<false, Table>,
                          dim3((unsigned)ctas), 256, kAnySmem, s, 1, t);
}

}  // namespace

cudaError_t launch_batch_any(bool row, BatchTable &t, cudaStream_t s)
{
    return any_launch(row, t, s);
}

cudaError_t launch_batch_any(bool row, BatchTableWide &t, cudaStream_t s)
{
    return any_launch(row, t, s);
}

cudaError_t launch_batch_any_h16(bool row, BatchTableH16 &t, int in_axis, cudaStream_t s)
{
    const int ctas = fill_ctas(t);
    if (ctas == 0)
        return cudaSuccess;
    auto k = !row           ? batch_any_h16_kernel<false, 0>
             : in_axis == 0 ? batch_any_h16_kernel<true, 0>
                            : batch_any_h16_kernel<true, 1>;
    return launch_chained(k, dim3((unsigned)ctas), 256, kAnySmem, s, 1, t);
}

}  // namespace fft2d
