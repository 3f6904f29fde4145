// qt_kmeans.cu -- sample Lloyd for the grid builder: seeded N(0, I_d) training draws,
// and per iteration the nearest centre of every draw and the centroids.  All distinct
// grid sizes of a model go through each launch together (blockIdx.y = grid).
//
// What bounds it: the distances.  A nearest centre is the first minimum over j of the
// FP32 chain acc <- fma(z_l - c_jl, z_l - c_jl, acc), l ascending; 2 d FP32 operations
// a distance.  One draw per thread with loops over a run-time d gave 1.9e11 distances/s
// at d = 4 (125 us for 1e5 draws and 600 centres) and left 120 launches of it, 120 of
// the update and 240 memsets to a model of six sizes.  Now the operations come in
// packed pairs (two centres, the same roundings), a centre loaded from shared memory
// serves several draws, and only the minimum of 16 distances is tracked: which of the
// 16 it was is found once per draw, by repeating the best group.  The six sizes of
// a 4-asset basket (1e5 draws, 20 iterations): 16.7 -> 2.9 ms; a launch over their 3650
// centres takes 139 us, 2.6e12 distances/s.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "qt_internal.h"
#include "qt_launch.h"
#include "qt_sampler.cuh"

namespace qt {

namespace {

constexpr int kKmBlock = 128;
constexpr int kKmTileBytes = 48 * 1024;

__device__ __forceinline__ uint64_t km_pack(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void km_unpack(uint64_t v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}

// c_j - z (z negated in nz) for a pair of centres, squared and added: the sign of the
// difference does not reach the square.
template <int DM>
__device__ __forceinline__ uint64_t km_pair(const uint64_t (&c)[DM], const uint64_t (&nz)[DM])
{
    uint64_t acc = 0;
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        uint64_t df;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(df) : "l"(c[l]), "l"(nz[l]));
        if (l == 0)
            asm("mul.rn.f32x2 %0, %1, %1;" : "=l"(acc) : "l"(df));
        else
            asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(acc) : "l"(df), "l"(acc));
    }
    return acc;
}

template <int DM>
__device__ __forceinline__ void km_load(const float* p, uint64_t (&c)[DM])
{
    if constexpr (DM % 2 == 0) {
#pragma unroll
        for (int l = 0; l < DM; l += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p + 2 * l);
            c[l] = v.x;
            c[l + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int l = 0; l < DM; ++l) c[l] = *reinterpret_cast<const uint64_t*>(p + 2 * l);
    }
}

// Training draws of the layer index 0xFFFF (apart from the forward step's streams) as
// Z[l][t]; the first N are the starting centres, in pairs [N/2][DM][2] padded with
// infinities to whole groups of 16; the sums start at zero.
__global__ void __launch_bounds__(256) km_draw_kernel(const __grid_constant__ KmJobs jobs, int d, int dm)
{
    const KmJob& J = jobs.j[blockIdx.y];
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    float g[kDMax];
    if (t < J.S) {
        normals_f32<kDMax>(J.seed, 0xFFFF, (unsigned long long)t, d, g);
#pragma unroll
        for (int l = 0; l < kDMax; ++l)
            if (l < d) J.Z[l * J.S + t] = g[l];
    }
    if (t < J.Npad) {
        float* c = J.C + (t >> 1) * 2 * dm + (t & 1);
#pragma unroll
        for (int l = 0; l < kDMax; ++l)
            if (l < dm) c[2 * l] = t < J.N ? (l < d ? g[l] : 0.0f) : __int_as_float(0x7F800000);
        if (t < J.N)
            for (int c = 0; c < J.copies; ++c)
                for (int l = 0; l <= d; ++l) J.sums[((long long)c * J.N + t) * (d + 1) + l] = 0ull;
    }
}

// Nearest centre (training assignment; exactness is not needed here) and fixed-point
// sums (scale 2^36), so that the centroids do not depend on the order of the atomics.
// A CTA takes 128 R draws and passes the centres through shared memory, 48 KB at a time.
template <int DM, int R>
__global__ void __launch_bounds__(kKmBlock) km_assign_kernel(const __grid_constant__ KmJobs jobs, int d)
{
    extern __shared__ __align__(16) float s_c[];
    const KmJob& J = jobs.j[blockIdx.y];
    const long long t0 = (long long)blockIdx.x * (kKmBlock * R) + threadIdx.x;
    if (t0 - threadIdx.x >= J.S) return;
    constexpr int kGroup = 16 * DM;                                   // floats of a group
    constexpr int kTile = kKmTileBytes / (kGroup * (int)sizeof(float));   // groups of a tile
    uint64_t nz[R][DM];
    float best[R];
    int bg[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const long long t = min(t0 + r * kKmBlock, J.S - 1);
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            const float z = l < d ? -J.Z[l * J.S + t] : 0.0f;
            nz[r][l] = km_pack(z, z);
        }
        best[r] = __int_as_float(0x7F800000);
        bg[r] = 0;
    }
    const int groups = J.Npad / 16;
    for (int g0 = 0; g0 < groups; g0 += kTile) {
        const int ng = min(kTile, groups - g0);
        if (g0 > 0) __syncthreads();
        const float4* src = reinterpret_cast<const float4*>(J.C + (long long)g0 * kGroup);
        for (int e = threadIdx.x; e < ng * (kGroup / 4); e += kKmBlock) reinterpret_cast<float4*>(s_c)[e] = src[e];
        __syncthreads();
        for (int g = 0; g < ng; ++g) {
            float m[R];
#pragma unroll
            for (int r = 0; r < R; ++r) m[r] = __int_as_float(0x7F800000);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                uint64_t c[DM];
                km_load<DM>(s_c + g * kGroup + q * 2 * DM, c);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float a, b;
                    km_unpack(km_pair<DM>(c, nz[r]), a, b);
                    m[r] = fminf(m[r], fminf(a, b));
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (m[r] < best[r]) {
                    best[r] = m[r];
                    bg[r] = g0 + g;
                }
        }
    }
    unsigned long long* sums = J.sums;
    if (J.copies > 1) sums += (long long)(blockIdx.x % (unsigned)J.copies) * J.N * (d + 1);
    // the first centre of the best group that has its minimum: the same distances again
    const float* base = groups <= kTile ? s_c : J.C;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float* p = base + (long long)bg[r] * kGroup;
        int idx = 0;
#pragma unroll 2
        for (int q = 7; q >= 0; --q) {
            uint64_t c[DM];
            km_load<DM>(p + q * 2 * DM, c);
            float a, b;
            km_unpack(km_pair<DM>(c, nz[r]), a, b);
            if (b == best[r]) idx = 2 * q + 1;
            if (a == best[r]) idx = 2 * q;
        }
        if (t0 + r * kKmBlock < J.S) {
            unsigned long long* s = sums + (long long)(bg[r] * 16 + idx) * (d + 1);
#pragma unroll
            for (int l = 0; l < DM; ++l)
                if (l < d) {
                    float z, z2;
                    km_unpack(nz[r][l], z, z2);
                    atomicAdd(s + l, (unsigned long long)__double2ll_rn(-(double)z * 68719476736.0));
                }
            atomicAdd(s + d, 1ull);
        }
    }
}

// Centroids (an empty cell keeps its centre); leaves the sums at zero.
__global__ void __launch_bounds__(128) km_update_kernel(const __grid_constant__ KmJobs jobs, int d, int dm)
{
    const KmJob& J = jobs.j[blockIdx.y];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= J.N) return;
    unsigned long long* s = J.sums + (long long)j * (d + 1);
    const long long copy = (long long)J.N * (d + 1);
    // of all copies, left at zero
    auto total = [&](int l) {
        unsigned long long v = 0;
#pragma unroll 4
        for (int q = 0; q < J.copies; ++q) v += s[q * copy + l];
        for (int q = 0; q < J.copies; ++q) s[q * copy + l] = 0ull;
        return v;
    };
    const unsigned long long c = total(d);
    if (c == 0) return;
    float* ctr = J.C + (long long)(j >> 1) * 2 * dm + (j & 1);
    for (int l = 0; l < d; ++l) ctr[2 * l] = (float)(((double)(long long)total(l) / 68719476736.0) / (double)c);
}

template <int DM>
cudaError_t assign(const KmJobs& jobs, int n, int d, long long S, int N, int num_sms, cudaStream_t st)
{
    // four draws a thread (two above d = 6, for registers) use a loaded centre best; half
    // as many where that leaves fewer than four CTAs an SM
    constexpr int kR = DM <= 6 ? 4 : 2;
    const size_t smem = std::min<size_t>((size_t)N * DM * sizeof(float), kKmTileBytes);
    const long long per = kKmBlock * kR, wide = (S + per - 1) / per;
    if (wide * n >= 4ll * num_sms)
        km_assign_kernel<DM, kR><<<dim3((unsigned)wide, (unsigned)n), kKmBlock, smem, st>>>(jobs, d);
    else
        km_assign_kernel<DM, kR / 2><<<dim3((unsigned)((S + per / 2 - 1) / (per / 2)), (unsigned)n), kKmBlock, smem, st>>>(
            jobs, d);
    return cudaGetLastError();
}

}  // namespace

int kmeans_dim_class(int d)
{
    return d <= 6 ? d : (d <= 8 ? 8 : (d <= 10 ? 10 : (d <= 12 ? 12 : kDMax)));
}

cudaError_t launch_kmeans(const KmJobs& jobs, int n, int d, int iters, int num_sms, cudaStream_t st)
{
    const int dm = kmeans_dim_class(d);
    long long S = 0;
    int N = 0;
    for (int i = 0; i < n; ++i) {
        S = std::max(S, jobs.j[i].S);
        N = std::max(N, jobs.j[i].Npad);
    }
    km_draw_kernel<<<dim3((unsigned)((std::max<long long>(S, N) + 255) / 256), (unsigned)n), 256, 0, st>>>(jobs, d, dm);
    cudaError_t e = cudaGetLastError();
    for (int it = 0; it < iters && e == cudaSuccess; ++it) {
        switch (dm) {
            case 1: e = assign<1>(jobs, n, d, S, N, num_sms, st); break;
            case 2: e = assign<2>(jobs, n, d, S, N, num_sms, st); break;
            case 3: e = assign<3>(jobs, n, d, S, N, num_sms, st); break;
            case 4: e = assign<4>(jobs, n, d, S, N, num_sms, st); break;
            case 5: e = assign<5>(jobs, n, d, S, N, num_sms, st); break;
            case 6: e = assign<6>(jobs, n, d, S, N, num_sms, st); break;
            case 8: e = assign<8>(jobs, n, d, S, N, num_sms, st); break;
            case 10: e = assign<10>(jobs, n, d, S, N, num_sms, st); break;
            case 12: e = assign<12>(jobs, n, d, S, N, num_sms, st); break;
            default: e = assign<kDMax>(jobs, n, d, S, N, num_sms, st); break;
        }
        if (e != cudaSuccess) break;
        km_update_kernel<<<dim3((unsigned)((N + 127) / 128), (unsigned)n), 128, 0, st>>>(jobs, d, dm);
        e = cudaGetLastError();
    }
    return e;
}

namespace {

// Layer grids from base grids: x = m_k + L_k g.  The base grid is FP64 [N][d], or the
// k-means centres (FP32 pairs [N/2][dm][2]), or the origin (a layer of one point).
__global__ void __launch_bounds__(256) map_grids_kernel(int d, int dm, int layers, const MapLayer* __restrict__ tab,
                                                        const double* __restrict__ m, const double* __restrict__ L,
                                                        double* __restrict__ out)
{
    for (int k = blockIdx.y; k < layers; k += gridDim.y) {
        const MapLayer T = tab[k];
        const double* mk = m + (long long)k * d;
        const double* Lk = L + (long long)k * d * d;
        for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < T.N; j += gridDim.x * blockDim.x) {
            double g[kDMax];
            for (int q = 0; q < d; ++q)
                g[q] = T.f64 ? T.f64[(long long)j * d + q]
                             : (T.f32 ? (double)T.f32[(long long)(j >> 1) * 2 * dm + 2 * q + (j & 1)] : 0.0);
            for (int l = 0; l < d; ++l) {
                double acc = mk[l];
                for (int q = 0; q <= l; ++q) acc += Lk[l * d + q] * g[q];
                out[T.off + (long long)j * d + l] = acc;
            }
        }
    }
}

}  // namespace

cudaError_t launch_map_grids(int d, int layers, long long maxN, const MapLayer* tab, const double* m, const double* L,
                             double* out, cudaStream_t st)
{
    const unsigned bx = (unsigned)std::min<long long>((maxN + 255) / 256, 1 << 16);
    map_grids_kernel<<<dim3(bx, (unsigned)std::min(layers, 65535)), 256, 0, st>>>(d, kmeans_dim_class(d), layers, tab, m, L,
                                                                                 out);
    return cudaGetLastError();
}

}  // namespace qt
