// qt_kernels_misc.cu -- small kernels around the forward step: preparation of
// the screened grid records, the backward induction of Sec. 2, the swing recursion
// and the root price.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "qt_internal.h"
#include "qt_launch.h"
#include "qt_sampler.cuh"

namespace qt {

// ------------------------------------------------------------------ grid records
//
// FP32 record of point c of grid g (centre mu_g, an FP32 vector):
//   [ fl32(|c - mu|^2 computed in FP64), fl32(c_0 - mu_0), ..., 0 ... ]
// padded rows (j >= N_g) carry cc = +inf so that they never win the screen.
// FP64 record: [c_0 .. c_{d-1}, 0 ...] (rec64 doubles).
// R_g = max_j |fl32(c_j - mu)| rounded up, accumulated with an integer max on
// the bits of a non-negative float.
__global__ void prep_records_kernel(const double* __restrict__ g64, GridInfo* gi, int ngrids, int d,
                                    int rec_floats, int rec64, long long total_recs, float* rec32,
                                    double* rec64out)
{
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= total_recs) return;
    int lo = 0, hi = ngrids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (gi[mid].roff <= r) lo = mid; else hi = mid - 1;
    }
    const GridInfo& G = gi[lo];
    const long long j = r - G.roff;
    if (rec32) {
        float* out = rec32 + r * rec_floats;
        if (j < G.N) {
            const double* c = g64 + (G.goff + j) * d;
            double cc = 0.0, nr = 0.0;
            for (int l = 0; l < d; ++l) {
                const double t = c[l] - (double)G.mu[l];
                cc += t * t;
                const float tf = __double2float_rn(t);
                out[1 + l] = tf;
                nr += (double)tf * (double)tf;
            }
            for (int l = d + 1; l < rec_floats; ++l) out[l] = 0.0f;
            out[0] = __double2float_rn(cc);
            const float R = __double2float_ru(sqrt(nr) * (1.0 + 0x1p-50));
            atomicMax(reinterpret_cast<unsigned int*>(&gi[lo].R), __float_as_uint(R));
        } else {
            out[0] = __int_as_float(0x7F800000);
            for (int l = 1; l < rec_floats; ++l) out[l] = 0.0f;
        }
    }
    if (rec64out) {
        double* out = rec64out + r * rec64;
        if (j < G.N) {
            const double* c = g64 + (G.goff + j) * d;
            for (int l = 0; l < d; ++l) out[l] = c[l];
            for (int l = d; l < rec64; ++l) out[l] = 0.0;
        } else {
            for (int l = 0; l < rec64; ++l) out[l] = __longlong_as_double(0x7FF0000000000000LL);
        }
    }
}

// ------------------------------------------------------------------ backward induction
//
// V_k(i) = max(phi_k(i), (sum_j p_ij V_{k+1}(j)) / p_i), p_i = sum_j p_ij; empty
// rows keep phi_k(i).  One warp per row: lane l adds p_ij V_{k+1}(j) for j = l,
// l+32, ... in ascending order (one fused multiply-add each), then a butterfly
// over offsets 16, 8, 4, 2, 1 combines the lanes, so every run gives the same
// bits.
//
// What bounds it: the FP64 pipe.  An operation holds a warp's quarter of the SM for 65
// cycles, whether 1 or 32 lanes take part, so that the conversion, multiply and add of
// every entry and the division of every row cost more than the counts' bytes (8-d tree,
// 7 layers of 4000 x 4000 64-bit counts: 0.9 GB, 132 us).  Most counts are zero, and a
// zero adds nothing: every lane first puts its non-zero counts of 32 columns a lane (1024
// of the row) aside in shared memory, in order, from loads that are all in flight
// together, and then runs through them with one FP64 operation each (906 -> 262 us).  A
// count that does not fit 27 bits, or a V that is not finite (where a zero count gives
// NaN), takes the plain walk over every entry.

constexpr int kRowSlots = 32;          // columns per lane and batch
constexpr int kRowBatch = 32 * kRowSlots;
constexpr int kRowWarps = 8;           // warps of the per-layer kernels
constexpr int kBackVMax = 12288;       // doubles of V in shared memory (96 KB)

// (double)c, c > 0, on the integer pipe: the FP64 pipe is the scarce one
__device__ __forceinline__ double count_f64(uint32_t c)
{
    const int z = __clz((int)c);
    const uint32_t m = c << z;                      // leading one at bit 31: it adds 1 to the exponent
    return __hiloint2double((int)(((uint32_t)(1053 - z) << 20) + (m >> 11)), (int)(m << 21));
}

// The quotient of a row's sum by its number of paths with the bits of __ddiv_rn, which
// takes 560 cycles of a warp's FP64 pipe (an operation takes 65, of one lane or of 32):
// q = a y, then q + (a - q c) y (P. Markstein, IBM J. Res. Dev. 34, 1990), y of relative
// error below 2^-43.  The corrected q is off by less than 2^-32 ulp before its rounding,
// and a quotient by a whole number c < 2^30 is at least 1 / (2 c) ulp > 2^-31 ulp away
// from where the rounding changes.  row_recip: 0 for other row sums, which divide.
__device__ __forceinline__ double row_recip(long long c)
{
    if (c <= 0 || c >= (1ll << 30)) return 0.0;
    const double y = (double)__fdividef(1.0f, (float)(uint32_t)c);
    return __fma_rn(y, __fma_rn(-count_f64((uint32_t)c), y, 1.0), y);
}

__device__ __forceinline__ double row_quotient(double a, double y, long long c)
{
    const double q = __dmul_rn(a, y);
    const double r = __fma_rn(__fma_rn(-q, count_f64((uint32_t)c), a), y, q);
    // the correction needs ordinary magnitudes (or a zero sum)
    const int ex = (__double2hiint(q) >> 20) & 0x7FF;
    const bool plain = __double2hiint(y) == 0 || ((ex < 200 || ex > 1900) && __double_as_longlong(a) != 0);
    return plain ? __ddiv_rn(a, (double)c) : r;
}

__device__ __forceinline__ bool finite_f64(double v)
{
    return (__double2hiint(v) & 0x7FF00000) != 0x7FF00000;
}

// One batch of a row: `n` <= 1024 columns at c0.  All loads first, then the list.
template <typename C>
__device__ __forceinline__ void row_load(const C* __restrict__ c0, int n, int lane, C (&c)[kRowSlots])
{
#pragma unroll
    for (int q = 0; q < kRowSlots; ++q) {
        const int j = lane + 32 * q;
        c[q] = j < n ? __ldcs(c0 + j) : (C)0;
    }
}

// Adds the lane's share of the row sum to ci and puts its non-zero entries (count |
// slot << 27) into lst[.][lane]; returns their number, or -1 when a count needs more
// than 27 bits.
template <typename C>
__device__ __forceinline__ int row_list(const C (&c)[kRowSlots], int lane, uint32_t (*lst)[32], long long& ci)
{
    int cnt = 0;
    bool wide = false;
#pragma unroll
    for (int q = 0; q < kRowSlots; ++q) {
        ci += (long long)c[q];
        if (c[q] != (C)0) {
            wide = wide || (unsigned long long)c[q] >= (1ull << 27);
            lst[cnt][lane] = (uint32_t)c[q] | ((uint32_t)q << 27);
            ++cnt;
        }
    }
    return wide ? -1 : cnt;
}

template <typename C>
__device__ __forceinline__ int row_batch(const C* __restrict__ c0, int n, int lane, uint32_t (*lst)[32], long long& ci)
{
    C c[kRowSlots];
    row_load(c0, n, lane, c);
    return row_list(c, lane, lst, ci);
}

// acc[q] += c_ij v[q * vs + j], q < nq, over the n columns of a batch in ascending j
// per lane, from the batch's list (cnt entries of this lane), or over every entry.
template <typename C, int NQ>
__device__ __forceinline__ void row_accumulate(const C* __restrict__ c0, int n, int lane, uint32_t (*lst)[32], int cnt,
                                               bool dense, const double* v, int vs, int nq, double (&acc)[NQ])
{
    if (__any_sync(0xFFFFFFFFu, cnt < 0) || dense) {
        for (int j = lane; j < n; j += 32) {
            const double cv = (double)c0[j];
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nq) acc[q] = __fma_rn(cv, v[(long long)q * vs + j], acc[q]);
        }
        return;
    }
#pragma unroll 2
    for (int s = 0; s < cnt; ++s) {
        const uint32_t e = lst[s][lane];
        const int j = lane + 32 * (int)(e >> 27);
        const double cv = count_f64(e & 0x07FFFFFFu);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (q < nq) acc[q] = __fma_rn(cv, v[(long long)q * vs + j], acc[q]);
    }
}

__device__ __forceinline__ void row_reduce(double& acc, long long& ci)
{
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, off));
        ci += __shfl_xor_sync(0xFFFFFFFFu, ci, off);
    }
}

// One layer, one warp per row; V_{k+1} in shared memory (dynamic: Nk1 doubles) when
// `staged`, else read from L2 by the lists' entries.
template <typename C>
__global__ void __launch_bounds__(kRowWarps * 32) backward_layer_kernel(const C* __restrict__ counts, long long coff,
                                                                        int Nk, int Nk1, int staged,
                                                                        const double* __restrict__ phik,
                                                                        const double* Vnext, double* __restrict__ Vk)
{
    extern __shared__ __align__(16) double s_v[];
    __shared__ uint32_t s_lst[kRowWarps][kRowSlots][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    bool odd = false;
    for (int j = threadIdx.x; j < Nk1; j += kRowWarps * 32) {
        const double v = Vnext[j];
        odd = odd || !finite_f64(v);
        if (staged) s_v[j] = v;
    }
    const bool dense = __syncthreads_or(odd) != 0;
    const double* V = staged ? s_v : Vnext;
    for (int i = blockIdx.x * kRowWarps + warp; i < Nk; i += gridDim.x * kRowWarps) {
        const C* row = counts + coff + (long long)i * Nk1;
        double acc[1] = {0.0};
        long long ci = 0;
        for (int j0 = 0; j0 < Nk1; j0 += kRowBatch) {
            const int n = min(kRowBatch, Nk1 - j0);
            const int cnt = row_batch(row + j0, n, lane, s_lst[warp], ci);
            row_accumulate<C, 1>(row + j0, n, lane, s_lst[warp], cnt, dense, V + j0, 0, 1, acc);
            __syncwarp();
        }
        row_reduce(acc[0], ci);
        if (lane == 0) {
            const double ph = phik[i];
            const double cont = ci == 0 ? ph : row_quotient(acc[0], row_recip(ci), ci);
            Vk[i] = ph > cont ? ph : cont;
        }
    }
}

constexpr size_t kListBytes = sizeof(uint32_t) * kRowWarps * kRowSlots * 32;   // the lists of a CTA

cudaError_t launch_backward_layer(const void* counts, int u32, long long coff, int Nk, int Nk1, const double* phik,
                                  const double* Vnext, double* Vk, int num_sms, cudaStream_t st)
{
    const int staged = Nk1 <= kBackVMax;
    const size_t dyn = staged ? (size_t)Nk1 * sizeof(double) : 0;
    // the CTAs of a large layer take several rows each, so that V is read once for each
    const int per_sm = dyn <= 40 * 1024 ? 3 : (dyn <= 72 * 1024 ? 2 : 1);
    int blocks = (Nk + kRowWarps - 1) / kRowWarps;
    if (blocks > num_sms * per_sm) blocks = num_sms * per_sm;
    cudaError_t e;
    if (u32) {
        e = allow_dynamic_smem(backward_layer_kernel<uint32_t>, dyn, kListBytes);
        if (e != cudaSuccess) return e;
        backward_layer_kernel<uint32_t><<<(unsigned)blocks, kRowWarps * 32, dyn, st>>>((const uint32_t*)counts, coff, Nk,
                                                                                      Nk1, staged, phik, Vnext, Vk);
    } else {
        e = allow_dynamic_smem(backward_layer_kernel<long long>, dyn, kListBytes);
        if (e != cudaSuccess) return e;
        backward_layer_kernel<long long><<<(unsigned)blocks, kRowWarps * 32, dyn, st>>>((const long long*)counts, coff,
                                                                                       Nk, Nk1, staged, phik, Vnext, Vk);
    }
    return cudaGetLastError();
}

// All layers of a small tree in one cooperative launch.  What bounds it is the chain of
// one layer's values to the next: a launch per layer took 10 us each (365 dates of 500
// points: 3.7 ms), and so did one kernel whose CTAs met at a grid-wide count between
// layers (now 0.73 ms).  So
//  - the values are their own flags: the exchange X[layer][CTA][8] starts as all-ones
//    words (a NaN that is never put there) and a CTA polls the values themselves into
//    shared memory, without a fence or a count.  A CTA writes its rows in one piece into
//    64 bytes of its own: a line that 16 warps write one after the other while every SM
//    polls it changes hands between the two halves of L2 each time (4.7 us a layer with
//    the values polled in V, 2.6 in one piece side by side, 2.3 with 64 bytes each);
//  - a row's counts do not wait for V: three groups of producer warps read the counts of
//    every third layer, put the non-zero ones aside and prepare the reciprocal of the row
//    sum, one to three layers ahead of the consumer warps, which only run through the
//    lists.
// Every wait is bounded; one that gives up records QT_ETIMEOUT (site 60) in the status block
// ahead of the layer table and leaves NaN in the values that depend on it.
constexpr int kBackRows = 2;           // rows of a warp, at most
constexpr int kTreeWarps = 4;          // consumer warps, and warps of a producer group
constexpr int kTreeGroups = 3;
constexpr int kTreeThreads = 32 * kTreeWarps * (1 + kTreeGroups);
constexpr int kTreeMaxN = 1024;
constexpr unsigned long long kUnset = ~0ull;

struct RowHead {
    double inv, phi;                   // 1 / row sum (0: take the division), phi_k(i)
    long long ci;
};

__device__ __forceinline__ void bar_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ bool bar_or(int id, int threads, bool v)
{
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %3, 0;\n\tbar.red.or.pred q, %1, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(id), "r"(threads), "r"((int)v)
        : "memory");
    return r != 0;
}
// v <- *p where `want`; no branch, so that several loads are in flight together
__device__ __forceinline__ void ld_value(unsigned long long& v, const double* p, bool want)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p ld.relaxed.gpu.global.u64 %0, [%1];\n\t}"
                 : "+l"(v)
                 : "l"(p), "r"((int)want)
                 : "memory");
}
__device__ __forceinline__ void st_value(double* p, double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b == kUnset) b = 0x7FF8000000000000ull;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}

template <typename C>
__global__ void __launch_bounds__(kTreeThreads) backward_tree_kernel(const C* __restrict__ counts, int n, int rows,
                                                                     const TreeLayer* __restrict__ layers,
                                                                     const double* __restrict__ phi, double* V,
                                                                     double* X, DevStatus* status, long long budget_us)
{
    extern __shared__ uint32_t s_dyn[];                 // lists [group][rows][warp][slot][lane]
    __shared__ double s_val[kBackRows * kTreeWarps];
    __shared__ double s_V[2][kTreeMaxN];
    __shared__ RowHead s_head[kTreeGroups][kBackRows][kTreeWarps];
    __shared__ int8_t s_cnt[kTreeGroups][kBackRows][kTreeWarps][32];
    constexpr int kHalf = 32 * kTreeWarps;              // threads of a role
    const int lane = threadIdx.x & 31;
    const int role = (threadIdx.x >> 5) / kTreeWarps, warp = (threadIdx.x >> 5) % kTreeWarps;
    const int gw = blockIdx.x * kTreeWarps + warp, W = gridDim.x * kTreeWarps;
    auto list = [&](int grp, int r) { return (uint32_t (*)[32])(s_dyn + ((grp * rows + r) * kTreeWarps + warp) * kRowBatch); };
    // barriers: 1 + group: its buffer is full; 4 + group: it is free again; 7: the consumers
    if (role > 0) {
        const int grp = role - 1;
        for (int s = grp; s < n; s += kTreeGroups) {
            const TreeLayer L = layers[n - 1 - s];
            const int Nk1 = layers[n - s].N;
            for (int r = 0; r < rows; ++r) {
                const int i = gw + r * W;
                C c[kRowSlots];
                double ph = 0.0;
                if (i < L.N) {
                    row_load(counts + L.coff + (long long)i * Nk1, Nk1, lane, c);
                    ph = phi[L.goff + i];
                }
                if (r == 0 && s >= kTreeGroups) bar_sync(4 + grp, 2 * kHalf);
                if (i < L.N) {
                    long long ci = 0;
                    s_cnt[grp][r][warp][lane] = (int8_t)row_list(c, lane, list(grp, r), ci);
#pragma unroll
                    for (int off = 16; off >= 1; off >>= 1) ci += __shfl_xor_sync(0xFFFFFFFFu, ci, off);
                    if (lane == 0) {
                        s_head[grp][r][warp] = RowHead{row_recip(ci), ph, ci};
                    }
                }
            }
            bar_arrive(1 + grp, 2 * kHalf);
        }
        return;
    }
    const int t = threadIdx.x;
    // a negative budget gives up without waiting, as every bounded wait does
    bool gave_up = budget_us < 0;
    auto record = [&]() {
        if (atomicCAS(&status->code, 0, 4 /* QT_ETIMEOUT */) == 0) status->where = 60;
    };
    if (gave_up) record();
    TreeLayer Ln = layers[n], L = layers[n - 1];
    for (int i = blockIdx.x * kHalf + t; i < Ln.N; i += gridDim.x * kHalf) V[Ln.goff + i] = phi[Ln.goff + i];
    for (int s = 0; s < n; ++s) {
        const int k = n - 1 - s, grp = s % kTreeGroups;
        const TreeLayer Lp = layers[k > 0 ? k - 1 : 0];
        // V_{k+1} into shared memory: phi_n, or the values as they appear
        unsigned long long v[kTreeMaxN / kHalf];
#pragma unroll
        for (int q = 0; q < kTreeMaxN / kHalf; ++q) v[q] = t + q * kHalf < Ln.N ? kUnset : 0ull;
        unsigned long long t0 = 0;
        for (int polls = 0;; ++polls) {
#pragma unroll
            for (int q = 0; q < kTreeMaxN / kHalf; ++q) {
                const int j = t + q * kHalf, r = j >= W ? 1 : 0, jr = j - r * W;
                const double* from = s == 0 ? phi + Ln.goff + j
                                            : X + ((long long)(k + 1) * gridDim.x + (jr >> 2)) * 8 + 4 * r + (jr & 3);
                ld_value(v[q], from, v[q] == kUnset);
            }
            bool missing = false;
#pragma unroll
            for (int q = 0; q < kTreeMaxN / kHalf; ++q) missing |= v[q] == kUnset;
            if (!missing || s == 0 || gave_up) break;
            if ((polls & 255) == 255) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                gave_up = now - t0 > (unsigned long long)budget_us * 1000ull;
                if (gave_up) record();
            }
        }
        bool odd = false;
#pragma unroll
        for (int q = 0; q < kTreeMaxN / kHalf; ++q) {
            const double x = __longlong_as_double((long long)v[q]);
            if (t + q * kHalf < Ln.N) s_V[s & 1][t + q * kHalf] = x;
            odd = odd || !finite_f64(x);
        }
        // values that are not finite meet every entry (a zero count times infinity is NaN)
        const bool dense = bar_or(7, kHalf, odd);
        bar_sync(1 + grp, 2 * kHalf);
        const double* Vn = s_V[s & 1];
        for (int r = 0; r < rows; ++r) {
            const int i = gw + r * W;
            if (i >= L.N) break;
            const RowHead H = s_head[grp][r][warp];
            const int cnt = s_cnt[grp][r][warp][lane];
            double acc = 0.0;
            if (__any_sync(0xFFFFFFFFu, cnt < 0) || dense) {
                const C* row = counts + L.coff + (long long)i * Ln.N;
                for (int j = lane; j < Ln.N; j += 32) acc = __fma_rn((double)row[j], Vn[j], acc);
            } else {
                const uint32_t (*lst)[32] = list(grp, r);
#pragma unroll 4
                for (int e = 0; e < cnt; ++e) {
                    const uint32_t w = lst[e][lane];
                    acc = __fma_rn(count_f64(w & 0x07FFFFFFu), Vn[lane + 32 * (int)(w >> 27)], acc);
                }
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, off));
            if (lane == 0) {
                double val = H.phi;
                if (H.ci != 0) {
                    const double q = row_quotient(acc, H.inv, H.ci);
                    val = val > q ? val : q;
                }
                s_val[r * kTreeWarps + warp] = val;
            }
        }
        bar_sync(7, kHalf);
        if (t < rows * kTreeWarps) {
            const int i = blockIdx.x * kTreeWarps + (t & 3) + (t >> 2) * W;
            if (i < L.N) {
                st_value(X + ((long long)k * gridDim.x + blockIdx.x) * 8 + t, s_val[t]);
                V[L.goff + i] = s_val[t];
            }
        }
        if (s + kTreeGroups < n) bar_arrive(4 + grp, 2 * kHalf);
        Ln = L;
        L = Lp;
    }
}

bool backward_tree_fits(int n, const int64_t* N, int num_sms)
{
    // two rows a warp, 1024 columns, enough layers to pay for the launch, and an exchange
    // (64 bytes for every four rows and layer) of at most 1 GiB
    if (n < 3 || (long long)n * num_sms * 64 > (1ll << 30)) return false;
    for (int k = 0; k <= n; ++k)
        if (N[k] > kTreeMaxN || N[k] > (int64_t)num_sms * kTreeWarps * kBackRows) return false;
    return true;
}

int backward_tree_blocks(int maxN, int num_sms) { return std::min((maxN + kTreeWarps - 1) / kTreeWarps, num_sms); }

cudaError_t launch_backward_tree(const void* counts, int u32, int n, int maxN, const void* layers, const double* phi,
                                 double* V, double* X, DevStatus* status, long long budget_us, int num_sms,
                                 cudaStream_t st)
{
    const int blocks = backward_tree_blocks(maxN, num_sms), rows = maxN > blocks * kTreeWarps ? 2 : 1;
    cudaError_t e = cudaMemsetAsync(X, 0xFF, (size_t)n * blocks * 8 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    const void* f = u32 ? (const void*)backward_tree_kernel<uint32_t> : (const void*)backward_tree_kernel<long long>;
    const size_t dyn = sizeof(uint32_t) * kRowBatch * kTreeWarps * kTreeGroups * rows;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&counts, (void*)&n, (void*)&rows, (void*)&layers, (void*)&phi, (void*)&V, (void*)&X,
                    (void*)&status, (void*)&budget_us};
    return cudaLaunchCooperativeKernel(f, dim3((unsigned)blocks), dim3(kTreeThreads), args, dyn, st);
}

// ------------------------------------------------------------------ swing option
//
// Eq. (stochCtrl) with the bang-bang BDP of Sec. 2: controls x in {0, 1} at
// dates k = 0..n-1, consumption state Q, chi(Q, x) = Q + x, x admissible at
// (k, Q) when F(k+1, Q + x), F(k, Q) = (Q <= Qmax and Q + n - k >= Qmin):
//   P_k(i, Q) = max over admissible x of x v_k(i) + C_k(i, Q + x),
//   C_k(i, Q') = (sum_j p^k_ij P_{k+1}(j, Q')) / p^k_i   (0 for an empty row),
// -inf where no x is admissible.  P blocks are Q-major: [Qmax + 1][N].  One
// warp per (row i, chunk of kSwingQ consumption states): it puts the row's non-zero
// counts aside once and adds all nine continuations of the chunk from them, with
// P_{k+1} of the chunk in shared memory.  Every continuation is summed in the order
// of backward_layer_kernel (lanes j mod 32 ascending, then the fixed butterfly),
// which makes the one-right swing (Qmax = 1) the Bermudan of qt_backward bit for bit.
// The butterfly of eight values keeps half of them on each side of every exchange:
// 12 additions for the nine values where nine butterflies take 45 (an addition commutes,
// so the bits are the same), and the nine quotients are one.  2-factor tree, 100 dates,
// Q in [20, 60]: 21.0 -> 2.9 ms.
__device__ __forceinline__ bool swing_feasible(int n, int k, int Q, int Qmin, int Qmax)
{
    return Q <= Qmax && Q + (n - k) >= Qmin;
}

__global__ void swing_terminal_kernel(int Nn, int n, int Qmin, int Qmax, double* __restrict__ Pn)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)(Qmax + 1) * Nn) return;
    const int Q = (int)(e / Nn);
    Pn[e] = swing_feasible(n, n, Q, Qmin, Qmax) ? 0.0 : __longlong_as_double(0xFFF0000000000000LL);
}

template <typename C>
__global__ void __launch_bounds__(kRowWarps * 32) swing_layer_kernel(const C* __restrict__ counts, long long coff, int Nk,
                                                                     int Nk1, int staged, const double* __restrict__ vk,
                                                                     const double* __restrict__ Pnext,
                                                                     double* __restrict__ Pk, int n, int k, int Qmin,
                                                                     int Qmax)
{
    extern __shared__ __align__(16) double s_P[];      // [kSwingQ + 1][Nk1]
    __shared__ uint32_t s_lst[kRowWarps][kRowSlots][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q0 = (int)blockIdx.x * kSwingQ;
    // consumption states of the chunk whose continuation is feasible at date k + 1
    const int lo = max(0, Qmin - (n - k - 1) - q0), hi = min(kSwingQ, Qmax - q0);
    const double ninf = __longlong_as_double(0xFFF0000000000000LL);
    bool odd = false;
    for (int q = lo; q <= hi; ++q)
        for (int j = threadIdx.x; j < Nk1; j += kRowWarps * 32) {
            const double v = Pnext[(long long)(q0 + q) * Nk1 + j];
            odd = odd || !finite_f64(v);
            if (staged) s_P[q * Nk1 + j] = v;
        }
    const bool dense = __syncthreads_or(odd) != 0;
    const double* P = staged ? s_P : Pnext + (long long)q0 * Nk1;
    for (int i = blockIdx.y * kRowWarps + warp; i < Nk; i += gridDim.y * kRowWarps) {
        const C* row = counts + coff + (long long)i * Nk1;
        double acc[kSwingQ + 1];
#pragma unroll
        for (int q = 0; q <= kSwingQ; ++q) acc[q] = 0.0;
        long long ci = 0;
        for (int j0 = 0; j0 < Nk1; j0 += kRowBatch) {
            const int m = min(kRowBatch, Nk1 - j0);
            const int cnt = row_batch(row + j0, m, lane, s_lst[warp], ci);
            if (__any_sync(0xFFFFFFFFu, cnt < 0) || dense) {
                for (int j = lane; j < m; j += 32) {
                    const double cv = (double)row[j0 + j];
#pragma unroll
                    for (int q = 0; q <= kSwingQ; ++q)
                        if (q >= lo && q <= hi) acc[q] = __fma_rn(cv, P[(long long)q * Nk1 + j0 + j], acc[q]);
                }
            } else {
                for (int s = 0; s < cnt; ++s) {
                    const uint32_t e = s_lst[warp][s][lane];
                    const double* Pj = P + j0 + lane + 32 * (int)(e >> 27);
                    const double cv = count_f64(e & 0x07FFFFFFu);
#pragma unroll
                    for (int q = 0; q <= kSwingQ; ++q)
                        if (q >= lo && q <= hi) acc[q] = __fma_rn(cv, Pj[(long long)q * Nk1], acc[q]);
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) ci += __shfl_xor_sync(0xFFFFFFFFu, ci, off);
        // butterflies: value q = 0-7 ends up in lanes 4 q and 4 q + 1, value 8 in the others
        static_assert(kSwingQ == 8, "three halving exchanges");
        double last = acc[kSwingQ];
#pragma unroll
        for (int off = 16; off >= 4; off >>= 1) last = __dadd_rn(last, __shfl_xor_sync(0xFFFFFFFFu, last, off));
#pragma unroll
        for (int w = 4; w >= 1; w >>= 1) {
            const bool up = (lane & (4 * w)) != 0;
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const double keep = up ? acc[q + w] : acc[q], give = up ? acc[q] : acc[q + w];
                acc[q] = __dadd_rn(keep, __shfl_xor_sync(0xFFFFFFFFu, give, 4 * w));
            }
        }
        const bool eighth = (lane & 2) != 0;
        double sum = __dadd_rn(eighth ? last : acc[0], __shfl_xor_sync(0xFFFFFFFFu, eighth ? acc[0] : last, 2));
        sum = __dadd_rn(sum, __shfl_xor_sync(0xFFFFFFFFu, sum, 1));
        const int q = lane >> 2, Q = q0 + q;
        const double c_cur = ci == 0 ? 0.0 : row_quotient(sum, row_recip(ci), ci);
        const double c_next = __shfl_sync(0xFFFFFFFFu, c_cur, q == kSwingQ - 1 ? 2 : ((lane & 28) + 4) & 31);
        double best = ninf;
        if (swing_feasible(n, k + 1, Q, Qmin, Qmax)) best = c_cur;                  // x = 0
        if (swing_feasible(n, k + 1, Q + 1, Qmin, Qmax)) {                          // x = 1
            const double val = __dadd_rn(vk[i], c_next);
            if (val > best) best = val;
        }
        if ((lane & 3) == 0 && Q <= Qmax) Pk[(long long)Q * Nk + i] = best;
    }
}

cudaError_t launch_swing_layer(const void* counts, int u32, long long coff, int Nk, int Nk1, const double* vk,
                               const double* Pnext, double* Pk, int n, int k, int Qmin, int Qmax, int num_sms,
                               cudaStream_t st)
{
    const int chunks = Qmax / kSwingQ + 1;
    const size_t need = (size_t)(kSwingQ + 1) * Nk1 * sizeof(double);
    const int staged = need <= 160 * 1024;
    const size_t dyn = staged ? need : 0;
    // as many row blocks as fill the SMs (a CTA loads the chunk's P once for all its rows)
    const int per_sm = dyn <= 40 * 1024 ? 3 : (dyn <= 72 * 1024 ? 2 : 1);
    int by = (Nk + kRowWarps - 1) / kRowWarps;
    const int most = (num_sms * per_sm + chunks - 1) / chunks;
    if (by > most) by = most;
    const dim3 grid((unsigned)chunks, (unsigned)by);
    cudaError_t e;
    if (u32) {
        e = allow_dynamic_smem(swing_layer_kernel<uint32_t>, dyn, kListBytes);
        if (e != cudaSuccess) return e;
        swing_layer_kernel<uint32_t><<<grid, kRowWarps * 32, dyn, st>>>((const uint32_t*)counts, coff, Nk, Nk1, staged,
                                                                       vk, Pnext, Pk, n, k, Qmin, Qmax);
    } else {
        e = allow_dynamic_smem(swing_layer_kernel<long long>, dyn, kListBytes);
        if (e != cudaSuccess) return e;
        swing_layer_kernel<long long><<<grid, kRowWarps * 32, dyn, st>>>((const long long*)counts, coff, Nk, Nk1, staged,
                                                                        vk, Pnext, Pk, n, k, Qmin, Qmax);
    }
    return cudaGetLastError();
}

// Status of one launch folded into an accumulator (the fused price mode runs
// one launch per layer pair, each clearing its own status block): the first
// error code and site are kept, the counters are summed.  One thread.
__global__ void fold_status_kernel(const DevStatus* __restrict__ src, DevStatus* acc)
{
    if (acc->code == 0 && src->code != 0) {
        acc->code = src->code;
        acc->where = src->where;
    }
    acc->rechecks += src->rechecks;
    acc->candidates += src->candidates;
    acc->done_items += src->done_items;
    acc->spare[0] = src->spare[0];
    for (int q = 1; q < 4; ++q) acc->spare[q] += src->spare[q];
}

// Root value: sum_i (p^0_i / M) V_0(i): lane l adds rows l, l+32, ... in ascending
// order, then the butterfly.  The row sums (whole numbers, any order) come from the
// CTA's 32 warps, 1024 rows at a time; one lane walking the only row of a
// deterministic start took 28 us for 500 columns.
__global__ void __launch_bounds__(1024) root_price_kernel(const void* __restrict__ counts, int u32, int N0, int N1,
                                                          const double* __restrict__ V0, double* out)
{
    __shared__ long long s_sum[1024];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t* c32 = reinterpret_cast<const uint32_t*>(counts);
    const long long* c64 = reinterpret_cast<const long long*>(counts);
    double acc = 0.0;
    long long tot = 0;
    for (int i0 = 0; i0 < N0; i0 += 1024) {
        const int rows = min(1024, N0 - i0);
        if (rows == 1) {
            // one row: all warps together
            const long long at = (long long)i0 * N1;
            long long ci = 0;
            for (int j = threadIdx.x; j < N1; j += 1024) ci += u32 ? (long long)c32[at + j] : c64[at + j];
            for (int off = 16; off >= 1; off >>= 1) ci += __shfl_xor_sync(0xFFFFFFFFu, ci, off);
            if (lane == 0) s_sum[warp] = ci;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < 32; ++w) ci += s_sum[w];
                s_sum[0] = ci;
            }
        } else {
            for (int r = warp; r < rows; r += 32) {
                const long long at = (long long)(i0 + r) * N1;
                long long ci = 0;
                for (int j = lane; j < N1; j += 32) ci += u32 ? (long long)c32[at + j] : c64[at + j];
                for (int off = 16; off >= 1; off >>= 1) ci += __shfl_xor_sync(0xFFFFFFFFu, ci, off);
                if (lane == 0) s_sum[r] = ci;
            }
        }
        __syncthreads();
        if (warp == 0)
            for (int r = lane; r < rows; r += 32) {
                tot += s_sum[r];
                acc = __dadd_rn(acc, __dmul_rn((double)s_sum[r], V0[i0 + r]));
            }
        __syncthreads();
    }
    if (warp != 0) return;
    for (int off = 16; off >= 1; off >>= 1) {
        acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, off));
        tot += __shfl_xor_sync(0xFFFFFFFFu, tot, off);
    }
    if (lane == 0) *out = tot > 0 ? __ddiv_rn(acc, (double)tot) : 0.0;
}

}  // namespace qt
