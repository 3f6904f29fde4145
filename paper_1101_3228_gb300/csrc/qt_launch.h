// qt_launch.h -- dispatch from run-time (form, dimension class, samples per
// thread) to the compiled instantiations of the forward kernel.
#pragma once
#include <cuda_runtime.h>

#include "qt_internal.h"

namespace qt {

// Leave for `dyn` bytes of dynamic shared memory beside `fixed` bytes that the kernel declares:
// up to 48 KB in all need none (the call takes a host microsecond of every launch).
template <typename F>
cudaError_t allow_dynamic_smem(F kernel, size_t dyn, size_t fixed = 1024)
{
    if (fixed + dyn <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
}

bool forward_variant_exists(int form, int dm, int S, bool streamed);

// Launches one persistent grid (SM count x resident CTAs per SM).
cudaError_t forward_launch(int form, int dm, int S, bool streamed, const ForwardParams& p, int block, int dyn_smem,
                           int num_sms, int* blocks_per_sm, cudaStream_t st);

// per-file dispatchers (qt_forward_*.cu)
cudaError_t launch_f32_small(int dm, int S, const ForwardParams& p, int block, int dyn, int num_sms, int* bps,
                             cudaStream_t st);
cudaError_t launch_f32_large(int dm, int S, const ForwardParams& p, int block, int dyn, int num_sms, int* bps,
                             cudaStream_t st);
cudaError_t launch_f64(int dm, int S, const ForwardParams& p, int block, int dyn, int num_sms, int* bps,
                       cudaStream_t st);
cudaError_t launch_router_forward(int dm, const ForwardParams& p, int num_sms, int* bps, cudaStream_t st);
// draw, screen and certificate of the items [p.item_lo, p.item_hi)
cudaError_t launch_tc_forward(int dm, const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st);
// Algorithm II (path-wise): compiled variants, default paths per thread, launch
bool pathwise_variant_exists(int dm, int S, bool f32, bool streamed);
int pathwise_default_spt(int dm, bool f32, bool streamed, long long M, long long ctas);
cudaError_t launch_pathwise(int dm, int S, bool f32, bool streamed, const ForwardParams& p, int dyn, int num_sms,
                            int* bps, cudaStream_t st);
// located search (d <= 2): table building, then Algorithm III / given samples or Algorithm II
cudaError_t launch_build_cells(int dm, const ForwardParams& p, int num_sms, cudaStream_t st);
cudaError_t launch_forward_cells(int dm, const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st);
cudaError_t launch_path_cells(int dm, int S, const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st);
// grid builder: sample Lloyd of n <= kKmJobs sizes, and the layer grids
int kmeans_dim_class(int d);
cudaError_t launch_kmeans(const KmJobs& jobs, int n, int d, int iters, int num_sms, cudaStream_t st);
cudaError_t launch_map_grids(int d, int layers, long long maxN, const MapLayer* tab, const double* m, const double* L,
                             double* out, cudaStream_t st);
cudaError_t launch_f32_streamed(int dm, int S, const ForwardParams& p, int block, int dyn, int num_sms, int* bps,
                                cudaStream_t st);

}  // namespace qt
