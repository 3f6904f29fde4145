// qt_path_cells.cu -- Algorithm II of Pages & Wilbertz (arXiv:1101.3228, Sec. 3; the
// path-wise estimator, qt_pathwise.cu) on the located search of qt_cells.cuh, d <= 2.
//
// A CTA of 1024 threads carries a tile of paths (up to S per thread, states and
// cells in registers) through every layer.  The tables of consecutive grids (95 KB
// at most) alternate between two shared-memory buffers: while one layer is
// searched, the bulk copy of the next is in flight.  The tile is M over the CTAs
// of one wave, not a power of two, so that all SMs finish together.  What bounds
// it: the issue slots of the step (one Philox call, one or two Box-Muller pairs
// and the map) and of one search and count.  2-factor workload, 100 layers x 10^6
// paths: 1.65 ms (57% of the issue slots, 417 instructions a step; the CTA waits for its
// slowest warp at every layer), against 8.23 ms for brute force over N_{k+1} = 500 points.
#include "qt_cells.cuh"
#include "qt_launch.h"
#include "qt_path_step.cuh"

namespace qt {

template <int DM, int S, bool F32>
__global__ void __launch_bounds__(kCellThreads, 1) path_cells_kernel(const __grid_constant__ ForwardParams p)
{
    using T = typename SampleType<F32>::T;
    extern __shared__ __align__(128) unsigned char dsm_pc[];
    __shared__ __align__(8) unsigned long long s_bar[2];
    __shared__ CellGrid s_G;
    __shared__ int s_abort;
    const int tid = threadIdx.x;
    const int n = p.n;
    const uint32_t buf_bytes = (uint32_t)p.smem_grid_bytes / 2u;
    const bool euler = p.pathwise_euler != 0;
    if (tid == 0) {
        mbar_init(smem_u32(&s_bar[0]), 1);
        mbar_init(smem_u32(&s_bar[1]), 1);
        fence_proxy_async();
        s_abort = 0;
    }
    __syncthreads();
    // grids of one point need no table; the others are loaded in order, load c into
    // buffer c & 1 (staging cursor sg: thread 0)
    int sg = 0;
    long long staged = 0, used = 0;
    auto stage_next = [&]() {
        while (sg <= n && p.cells[sg].N <= 1) ++sg;
        if (sg > n) return;
        const CellGrid& G = p.cells[sg];
        const uint32_t bar = smem_u32(&s_bar[staged & 1]);
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, cell_stage_bytes<DM>(G));
        cell_stage<DM>(p, G, smem_u32(dsm_pc) + (uint32_t)(staged & 1) * buf_bytes, bar);
        ++staged;
        ++sg;
    };
    for (long long item = blockIdx.x; item < p.total_items; item += gridDim.x) {
        __syncthreads();
        if (tid == 0) {
            sg = 0;
            stage_next();
            stage_next();
        }
        const unsigned long long m0 = (unsigned long long)item * (unsigned long long)p.cell_tile;
        const unsigned long long m1 = min(p.M, m0 + (unsigned long long)p.cell_tile);
        T x[S][DM];
        int cell[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const unsigned long long m = m0 + (unsigned long long)(s * kCellThreads + tid);
            cell[s] = 0;
            if (m < m1) {
                if constexpr (F32) path_start_f32<DM>(p.params_f, DM, p.seed, m, x[s]);
                else path_start_f64<DM>(p.params_d, DM, p.seed, m, x[s]);
            }
        }
        for (int g = 0; g <= n; ++g) {
            const int k = g - 1;
            const CellGrid& G = p.cells[g];
            const int N = G.N;
            const unsigned char* sm = dsm_pc + (uint32_t)(used & 1) * buf_bytes;
            if (N > 1) {
                const int b = (int)(used & 1);
                for (int e = tid; e < (int)(sizeof(CellGrid) / 4); e += kCellThreads)
                    reinterpret_cast<int*>(&s_G)[e] = reinterpret_cast<const int*>(&G)[e];
                const uint32_t par = (uint32_t)((used >> 1) & 1);
                if (!mbar_wait_bounded(smem_u32(&s_bar[b]), par, p.spin_budget)) {
                    record_error(p.status, 4 /* QT_ETIMEOUT */, 51);
                    s_abort = 1;
                    mbar_wait_bounded(smem_u32(&s_bar[b]), par, kDrainUs);
                }
                ++used;
                __syncthreads();
                if (s_abort) break;
            }
            const float* gpf = p.params_f + (long long)max(k, 0) * p.params_stride;
            const double* gpd = p.params_d + (long long)max(k, 0) * p.params_stride;
            const long long coff = k >= 0 ? p.layers[k].coff : 0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const unsigned long long m = m0 + (unsigned long long)(s * kCellThreads + tid);
                if (m >= m1) continue;
                long long row = -1;                  // dump row of this path at layer k
                if (p.dump_count > 0 && k >= 0 && (m % (unsigned long long)p.dump_stride) == 0ull) {
                    const unsigned long long t = m / (unsigned long long)p.dump_stride;
                    if (t < (unsigned long long)p.dump_count) row = (long long)k * p.dump_count + (long long)t;
                }
                if (row >= 0)
                    for (int l = 0; l < DM; ++l) p.dumpX[row * DM + l] = (double)x[s][l];
                if (k >= 0) {
                    if constexpr (F32) path_step_f32<DM>(gpf, DM, euler, p.seed, k, m, x[s]);
                    else path_step_f64<DM>(gpd, DM, euler, p.seed, k, m, x[s]);
                }
                int j = 0;
                if (N > 1) {
                    float a[DM];
#pragma unroll
                    for (int l = 0; l < DM; ++l) {
                        if constexpr (F32) a[l] = __fsub_rn(x[s][l], s_G.mu[l]);
                        else a[l] = __double2float_rn(__dsub_rn(x[s][l], (double)s_G.mu[l]));
                    }
                    uint64_t e;
                    bool need;
                    j = cell_search<DM>(s_G, sm, p.cell_pool, a, 1.0f, e, need);
                    if (need) {
                        double z[DM];
#pragma unroll
                        for (int l = 0; l < DM; ++l) z[l] = (double)x[s][l];
                        atomicAdd(&p.status->rechecks, 1ull);
                        j = cell_exact<DM, true>(s_G, cell_records(s_G, sm), a, z, e, p.cell_pool, p.g64 + G.goff * DM);
                    }
                }
                if ((unsigned)j >= (unsigned)N) {
                    record_error(p.status, 6 /* QT_EDEVICE */, 53);
                    cell[s] = 0;
                    continue;
                }
                if (k >= 0) count_add(p.counts, p.counts_u32, coff + (long long)cell[s] * N + j, 1u);
                if (row >= 0) {
                    for (int l = 0; l < DM; ++l) p.dumpY[row * DM + l] = (double)x[s][l];
                    p.dumpI[row] = cell[s];
                    p.dumpJ[row] = j;
                }
                cell[s] = j;
            }
            if (N > 1) {
                __syncthreads();                     // every warp is done with buffer b
                if (tid == 0) stage_next();
            }
        }
        if (s_abort) break;
    }
    // after a timeout the copies still in flight land before the CTA leaves
    if (s_abort && tid == 0)
        for (long long c = used; c < staged; ++c)
            mbar_wait_bounded(smem_u32(&s_bar[c & 1]), (uint32_t)((c >> 1) & 1), kDrainUs);
    __syncthreads();
}

template <int DM, int S, bool F32>
static cudaError_t launch_pc(const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    auto kern = path_cells_kernel<DM, S, F32>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    if (e != cudaSuccess) return e;
    *bps = 1;
    long long grid = num_sms;
    if (grid > p.total_items) grid = p.total_items;
    if (grid < 1) grid = 1;
    kern<<<(unsigned)grid, kCellThreads, dyn, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_path_cells(int dm, int S, const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    const bool f32 = p.prec == 1;
#define QT_CASE(D, SS, F) \
    if (dm == D && S == SS && f32 == F) return launch_pc<D, SS, F>(p, dyn, num_sms, bps, st);
    QT_CASE(1, 1, true) QT_CASE(1, 8, true) QT_CASE(2, 1, true) QT_CASE(2, 8, true)
    QT_CASE(1, 1, false) QT_CASE(1, 4, false) QT_CASE(2, 1, false) QT_CASE(2, 4, false)
#undef QT_CASE
    return cudaErrorInvalidValue;
}

}  // namespace qt
