// qt_forward_tc.cuh -- the forward step of Algorithm III (Pages & Wilbertz,
// arXiv:1101.3228, Sec. 4) with the nearest-cell screen on the 5th-generation
// tensor cores (tcgen05.mma, accumulators in tensor memory).
//
// The screen scores s_j = |g_j|^2 - 2 x^.g_j (g_j, x^ centred on the grid's
// FP32 centre) are one GEMM per 128 samples x 128 grid points: sample rows
// [a_hi, a_hi, a_lo, 1, 1] times grid rows [g_hi, g_lo, g_hi, cc_hi, cc_lo],
// a = -2 sigma x^, g = sigma g^, cc = sigma^2 |g^|^2, each split into an FP16
// head and an FP16 tail, sigma = 2^tc_exp so that the grid fits in [-1, 1].
// Each group of coordinates takes DM columns (the dimension class, zero
// padded), so K = 16 holds 3 DM + 2 columns for DM <= 4 and K = 32 for
// DM <= 10.  The three cross products reproduce the FP32 score to about
// 2^-21 relative (the tail x tail product is below 2^-22).
//
// Three kernels per window of work items (layer k, 128 samples each; at most 1 GiB
// of samples and states, handed over in device memory):
//   tc_draw_kernel     draws the pairs (one thread per pair, high occupancy) and
//                      writes the centred FP32 samples of both grids;
//   forward_tc_kernel  the screen: four persistent CTAs of one warpgroup per SM.  A
//                      CTA writes its 128 samples' operand rows to shared memory,
//                      streams the 128-point operand tiles of Gamma_k, then of
//                      Gamma_{k+1}, through a small ring (bulk copies), has the last
//                      warp to have read a tile issue the next tile's MMA into its
//                      128 columns of tensor memory, takes the minimum of every 16 scores with the
//                      tensor-memory loads, keeps the best two chunks and the
//                      smallest other minimum in registers, and writes them out.  Its
//                      warps meet only at mbarriers; while one CTA waits for its MMA
//                      or a barrier, the other three keep the tensor pipe busy;
//   tc_certify_kernel  re-scores, certifies, rechecks and counts (high occupancy).
//
// What bounds it, and why it is built so.  An MMA issued from one lane of a diverged
// warp costs, with its commit, 584 cycles per 256 points at K = 16 (713 at K = 32)
// however few points it has; issued by a converged warp that elects one lane, 128
// (256), the rate of the pipe.  With the pipe free, the next limits are the reads of
// tensor memory (193 scores per SM and cycle: 85 cycles per 128 x 128 tile) and the
// issue slots of the chunk tracking (about 50 half-rate instructions per thread and
// tile); what is left is the round trip of the 512 columns of tensor memory (issue,
// MMA, arrival, read, hand-over: 1350 cycles for the SM's four tiles at d = 8, 337 a tile).
// 8-d tree, 12 dates of 4000 points, 2e6 paths: 21.3 -> 19.3 ms; 4-d, 50 dates of
// 200 to 2000 points, 1e6 paths: 19.1 -> 13.7 ms (draw 1.35, screen 9.7, certify
// 2.6 ms of it); 10-d, 6 dates of 8000 points, 1e6 paths: 9.7 -> 8.7 ms; 3-d given
// samples: 0.55 -> 0.38 ms.
// The hand-over costs 2 (8 DM + 40) bytes of traffic per pair and reads of
// them, 0.3 KB at d = 8, and buys kernels that each fit their registers: one kernel
// that draws, screens and certifies kept the screen's loop in local memory, for
// which operands in shared memory leave no L1 (500 to 1000 cycles a tile in three
// variants: one CTA of 16 warps with a role each, two CTAs of two warpgroups, four
// CTAs of one).
//
// Exactness: the best chunk is re-scored on the CUDA cores in FP32 (and the
// second one where the certificate needs it), and the pick is certified against
// the exact FP64 distance with the FP32 bound inside the re-scored chunks and
// the tensor-core bound outside them; uncertified samples go to the exact
// window search (FP32 screen of the whole grid, exact FP64 distances inside
// the certified window).
#pragma once
#include <cuda_fp16.h>

#include "qt_forward.cuh"
#include "qt_launch.h"

namespace qt {

namespace {

__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    // tcgen05 shared-memory matrix descriptor, canonical K-major layout, no swizzle
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Minima of four consecutive 16-column chunks of this thread's accumulator row
// (columns taddr .. taddr + 63): tcgen05.ld.red loads 16 columns and returns
// their minimum; the loaded values themselves go to scratch registers local to
// this block, which also waits for the loads, so nothing outside it can touch
// registers the loads are still writing.
__device__ __forceinline__ void tc_chunk_min4(uint32_t taddr, float& m0, float& m1, float& m2, float& m3)
{
    asm volatile(
        "{\n\t.reg .f32 a<16>, b<16>, c<16>, e<16>;\n\t"
        "tcgen05.ld.red.sync.aligned.32x32b.x16.min.f32 {a0,a1,a2,a3,a4,a5,a6,a7,a8,a9,a10,a11,a12,a13,a14,a15}, %0, [%4];\n\t"
        "tcgen05.ld.red.sync.aligned.32x32b.x16.min.f32 {b0,b1,b2,b3,b4,b5,b6,b7,b8,b9,b10,b11,b12,b13,b14,b15}, %1, [%5];\n\t"
        "tcgen05.ld.red.sync.aligned.32x32b.x16.min.f32 {c0,c1,c2,c3,c4,c5,c6,c7,c8,c9,c10,c11,c12,c13,c14,c15}, %2, [%6];\n\t"
        "tcgen05.ld.red.sync.aligned.32x32b.x16.min.f32 {e0,e1,e2,e3,e4,e5,e6,e7,e8,e9,e10,e11,e12,e13,e14,e15}, %3, [%7];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n\t}"
        : "=f"(m0), "=f"(m1), "=f"(m2), "=f"(m3)
        : "r"(taddr), "r"(taddr + 16u), "r"(taddr + 32u), "r"(taddr + 48u)
        : "memory");
}

// Bound on |tensor-core score - exact score| in FP32-score units for a grid
// point at distance r from the centre (A = |x^|): the FP32 bound (d+2) 2^-24
// plus 32 FP32 additions of the MMA (2^-23 each, counted as truncations), the
// dropped tail product and the head/tail representation (3 * 2^-22), and the
// absolute floor of the FP16 tails (2^-25 each) divided by sigma^2.
__device__ __forceinline__ float tc_bound(float sqrt_d, float A, float r, float sigma, float inv_sigma)
{
    const float rel = 1.5f * 0x1p-18f;
    const float absf = (0x1p-23f * sqrt_d * (A + r) * sigma + 0x1p-24f) * inv_sigma * inv_sigma;
    return rel * (r * r + 2.0f * A * r) + absf;
}

__device__ __forceinline__ float cc_bound(int d, float A, float r)
{
    return (float)(d + 2) * 0x1p-24f * (1.0f + 0x1p-10f) * (r * r + 2.0f * A * r);
}

// FP32 re-score of chunk ch of 16 points for the sample of lane src by a quad of
// lanes: lane q of it scores points 4q .. 4q+3 (one 16-byte load per coordinate; the
// quad's loads cover 64 consecutive bytes of the chunk's coordinate row) and two
// exchanges combine the quad: smallest score, second smallest, first point of the
// smallest.  rows: the chunk-major records [chunk][DM + 1][16] (cc first), cert: the
// warp's centred samples [DM][128].
template <int DM>
__device__ __forceinline__ void quad_score(const float* __restrict__ rows, const float* cert, int q, int src, int ch,
                                           float& best, float& second, int& idx)
{
    const float4* c4 = reinterpret_cast<const float4*>(rows) + (long long)ch * ((DM + 1) * 4) + q;
    float4 g[DM + 1];
#pragma unroll
    for (int l = 0; l <= DM; ++l) g[l] = c4[l * 4];
    float4 sc = g[0];
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        const float x = cert[l * kTcTileM + src];
        sc.x = __fmaf_rn(x, g[1 + l].x, sc.x);
        sc.y = __fmaf_rn(x, g[1 + l].y, sc.y);
        sc.z = __fmaf_rn(x, g[1 + l].z, sc.z);
        sc.w = __fmaf_rn(x, g[1 + l].w, sc.w);
    }
    // smallest (lowest point first) and second smallest of the lane's four
    const bool xy = sc.y < sc.x, zw = sc.w < sc.z;
    const float m0 = fminf(sc.x, sc.y), m1 = fminf(sc.z, sc.w);
    const bool hi = m1 < m0;
    best = fminf(m0, m1);
    idx = hi ? (zw ? 3 : 2) : (xy ? 1 : 0);
    second = fminf(fmaxf(m0, m1), hi ? fmaxf(sc.z, sc.w) : fmaxf(sc.x, sc.y));
    idx += ch * kChunk + 4 * q;
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        const float ob = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        const float o2 = __shfl_xor_sync(0xFFFFFFFFu, second, o);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, idx, o);
        second = fminf(fminf(second, o2), fmaxf(best, ob));
        const bool take = ob < best || (ob == best && oi < idx);
        best = take ? ob : best;
        idx = take ? oi : idx;
    }
}

// Every lane's chunk, the quad's four samples in turn.  A lane that fetched its own
// chunk record by record touched 32 lines with every warp load, 1536 L1 wavefronts per
// warp and search; this takes 288.  Whole warp.
template <int DM>
__device__ __forceinline__ void quad_rescore(const float* __restrict__ rows, const float* cert, int lane, int chunk,
                                             float& best, float& second, int& idx)
{
    constexpr int kUnroll = DM <= 4 ? 2 : 1;   // two chunks' loads in flight where the registers allow it
#pragma unroll kUnroll
    for (int s = 0; s < 4; ++s) {
        const int src = (lane & ~3) | s;
        const int ch = __shfl_sync(0xFFFFFFFFu, chunk, src);
        float b, s2;
        int bi;
        quad_score<DM>(rows, cert, lane & 3, src, max(ch, 0), b, s2, bi);
        if ((lane & 3) == s) {
            best = b;
            second = s2;
            idx = bi;
        }
    }
}

// The chunks of the lanes that want it only, a quad for each, eight at a time: 9% of
// the searches at d = 8 need a second chunk, so some lane of nearly every warp does,
// and with all four samples of every quad in turn the kernel took 631 against 582 us for
// the 1e7 pairs of 50 dates at d = 4.
template <int DM>
__device__ __forceinline__ void quad_rescore_some(const float* __restrict__ rows, const float* cert, int lane, bool want,
                                                  int chunk, float& best, float& second, int& idx)
{
    unsigned todo = __ballot_sync(0xFFFFFFFFu, want);
    const int rank = __popc(todo & ((1u << lane) - 1u));
    for (int r0 = 0; todo; r0 += 8) {
        int src = __ffs(todo) - 1;                     // quads without a sample repeat the first
#pragma unroll 1
        for (int i = 0; i < 8 && todo; ++i, todo &= todo - 1)
            if (i == lane >> 2) src = __ffs(todo) - 1;
        const int ch = __shfl_sync(0xFFFFFFFFu, chunk, src);
        float b, s2;
        int bi;
        quad_score<DM>(rows, cert, lane & 3, src, ch, b, s2, bi);
        const int from = ((rank - r0) & 7) * 4;
        b = __shfl_sync(0xFFFFFFFFu, b, from);
        s2 = __shfl_sync(0xFFFFFFFFu, s2, from);
        bi = __shfl_sync(0xFFFFFFFFu, bi, from);
        if (want && rank >= r0 && rank < r0 + 8) {
            best = b;
            second = s2;
            idx = bi;
        }
    }
}

// Mixed certificate: FP32 scores inside the two best chunks (best, S1: the
// smallest other FP32 score there), tensor-core scores outside them (B2tc: a lower
// bound of the other chunks' minima, FP32-score units); R bounds every |g|.
// Bit 0 of the result: the FP32 scores inside do not single out the best; bit 1: a
// point outside may be nearer.
__device__ __forceinline__ int tc_uncertified(int d, float A, float best, float S1, float B2tc, float R,
                                              float sqrt_d, float sigma, float inv_sigma)
{
    const float Ap = A * (1.0f + 0x1p-18f);
    const float E1 = cc_bound(d, Ap, R * (1.0f + 0x1p-18f));
    const float U = best + E1;
    const float A2 = Ap * Ap;
    const float eta = 0x1p-44f * (A2 + fabsf(best) + E1);
    const float rad = fmaxf(A2 + U + 0x1p-18f * (A2 + fabsf(U)) + eta, 0.0f);
    const float rho = Ap + __fsqrt_rn(rad);
    const float lo_in = S1 - cc_bound(d, Ap, rho);
    const float lo_out = B2tc - tc_bound(sqrt_d, Ap, rho, sigma, inv_sigma);
    const float rhs = U + eta;
    // additive slack for the FP32 evaluation of both sides
    const bool ok_in = lo_in - rhs > 0x1p-20f * (fabsf(lo_in) + fabsf(rhs)) + eta || lo_in == __int_as_float(0x7F800000);
    const bool ok_out = lo_out - rhs > 0x1p-20f * (fabsf(lo_out) + fabsf(rhs)) + eta || lo_out == __int_as_float(0x7F800000);
    return (ok_in ? 0 : 1) | (ok_out ? 0 : 2);
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// Number of arrivals at a shared-memory counter before this one.
__device__ __forceinline__ uint32_t count_arrival(uint32_t ctr)
{
    uint32_t old;
    asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(ctr) : "memory");
    return old;
}

// Bounded wait with one outcome for the whole warp (tcgen05.ld and the ballots need
// converged warps).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, long long budget)
{
    return __all_sync(0xFFFFFFFFu, mbar_wait_bounded(bar, parity, budget));
}

// The warps of a CTA meet at an mbarrier (one arrival each), bounded.  By the arrival's own
// token, not a parity that the loop around it would carry (as a function of its own it costs
// the screen 10%).
__device__ __forceinline__ bool warps_meet(uint32_t bar, long long budget_us)
{
    bool ok = false;
    __syncwarp();
    if (elect_one()) {
        unsigned long long state;
        asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(state) : "r"(bar) : "memory");
        const unsigned long long t0 = global_ns();
        while (budget_us >= 0 && !ok) {
            uint32_t done;
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(done)
                : "r"(bar), "l"(state)
                : "memory");
            ok = done != 0;
            if (!ok && global_ns() - t0 > (unsigned long long)budget_us * 1000ull) break;
        }
    }
    return __any_sync(0xFFFFFFFFu, ok);
}

__device__ __forceinline__ int layer_of(const ForwardParams& p, long long item)
{
    int lo = 0, hi = p.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.layers[mid].item_begin <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Per sample, over the tiles seen so far: the two smallest chunk minima and the
// smallest of the others.  A key is a chunk minimum with its chunk's number within
// the tile (eight chunks) in the lowest three mantissa bits, so that minima and
// maxima alone carry it: 46 instructions per tile of 128 points against 80 with the
// number in a register of its own.  Only which tile a key came from is tracked by
// comparisons, once per tile.  A key is within 2^-20 of its minimum.
struct KeyTrack {
    float B1, Bs, B3;
    int t1, ts;                        // tiles of B1 and Bs
    __device__ __forceinline__ void reset()
    {
        B1 = Bs = B3 = 3.0e38f;
        t1 = ts = 0;
    }
    __device__ __forceinline__ void merge4(float a, float b, float c, float d)
    {
        const float p = fminf(a, b), q = fmaxf(a, b), r = fminf(c, d), s = fmaxf(c, d);
        const float l1 = fminf(p, r), x = fmaxf(p, r), y = fminf(q, s);
        const float l2 = fminf(x, y), l3 = fmaxf(x, y);      // the three smallest of the four
        B3 = fminf(min3f(B3, l3, fmaxf(Bs, l1)), fmaxf(B1, l2));
        Bs = min3f(Bs, l2, fmaxf(B1, l1));
        B1 = fminf(B1, l1);
    }
    __device__ __forceinline__ void add_tile(const float (&m)[8], int tile)
    {
        float k[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) k[q] = __int_as_float((__float_as_int(m[q]) & ~7) | q);
        const float o1 = B1, os = Bs;
        merge4(k[0], k[1], k[2], k[3]);
        merge4(k[4], k[5], k[6], k[7]);
        ts = Bs == os ? ts : (Bs == o1 ? t1 : tile);
        t1 = B1 == o1 ? t1 : tile;
    }
    static __device__ __forceinline__ int chunk(float key, int tile) { return tile * 8 + (__float_as_int(key) & 7); }
    // a lower bound of the chunk minimum that the key stands for
    static __device__ __forceinline__ float low(float key) { return key - 0x1p-19f * fabsf(key); }
};

}  // namespace

// Draw of one work item's sample row t (Algorithm III: the pair (X_k, X_{k+1})
// of the AR(1) step): the centred, scaled FP32 coordinates -2 (x - mu) of both grids
// with their norm, [grid][DM + 1][128] at `cert` (sign bit of the norm set when a
// coordinate leaves the FP16 range of the operands).  Parameters and grid centres
// are read from global memory (the same addresses for every thread: broadcast
// loads that stay in L1).
template <int DM>
__device__ __forceinline__ void draw_row(const ForwardParams& p, int k, const LayerDesc& L, unsigned long long m, int t,
                                         float* cert)
{
    const int d = p.d;
    const GridInfo& GA = p.grids[L.gridA];
    const GridInfo& GB = p.grids[L.gridB];
    float muA[DM], muB[DM];
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        muA[l] = GA.mu[l];
        muB[l] = GB.mu[l];
    }
    const float* spf = p.params_f ? p.params_f + (long long)k * p.params_stride : nullptr;
    const double* spd = p.params_d ? p.params_d + (long long)k * p.params_stride : nullptr;
    const Centred<DM> cs = centred_sample_inl<DM>(p, spf, spd, muA, muB, k, m);
#pragma unroll
    for (int gr = 0; gr < 2; ++gr) {
        const float* x = gr == 0 ? cs.xa : cs.yb;
        const float A = gr == 0 ? cs.Aa : cs.Ab;
        const float sg = ldexpf(1.0f, gr == 0 ? GA.tc_exp : GB.tc_exp);
        bool big = false;
#pragma unroll
        for (int l = 0; l < DM; ++l)
            if (l < d) big = big || !(fabsf(sg * x[l]) <= 16384.0f);
        float* cx = cert + gr * (DM + 1) * kTcTileM + t;
#pragma unroll
        for (int l = 0; l < DM; ++l) cx[l * kTcTileM] = l < d ? x[l] : 0.0f;
        cx[DM * kTcTileM] = __int_as_float(__float_as_int(A) | (big ? (int)0x80000000 : 0));
    }
}

// Operand row t of one grid from its centred sample (cert: [DM + 1][128]):
// [a_hi (DM), a_hi (DM), a_lo (DM), 1, 1], a = sigma x, core-matrix layout, K columns.
template <int DM, int K>
__device__ __forceinline__ void operand_row(const float* cert, int t, int exp, unsigned char* ops)
{
    const float sg = ldexpf(1.0f, exp);
    const bool big = (__float_as_int(cert[DM * kTcTileM + t]) & (int)0x80000000) != 0;
    uint32_t hi[DM], lo[DM];
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        const float v = big ? 0.0f : sg * cert[l * kTcTileM + t];
        const __half h = __float2half_rn(v);
        hi[l] = __half_as_ushort(h);
        lo[l] = __half_as_ushort(__float2half_rn(v - __half2float(h)));
    }
    const uint32_t one = __half_as_ushort(__float2half_rn(1.0f));
    uint32_t w[K / 2];
#pragma unroll
    for (int q = 0; q < K; q += 2) {
        uint32_t h2[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = q + u;
            h2[u] = c < DM ? hi[c] : (c < 2 * DM ? hi[c - DM] : (c < 3 * DM ? lo[c - 2 * DM] : (c < 3 * DM + 2 ? one : 0u)));
        }
        w[q / 2] = h2[0] | (h2[1] << 16);
    }
#pragma unroll
    for (int kb = 0; kb < K / 8; ++kb)
        *reinterpret_cast<uint4*>(ops + (((t >> 3) * (K / 8) + kb) * 64 + (t & 7) * 8) * 2) =
            make_uint4(w[4 * kb], w[4 * kb + 1], w[4 * kb + 2], w[4 * kb + 3]);
}

// Record of a work item between the kernels: the centred samples [2][DM + 1][128]
// (draw_row), then per grid and row the two best chunks and lower bounds of the
// second best and of all other chunk minima, [2][4][128].
template <int DM>
struct TcItem {
    static constexpr int kCert = 2 * (DM + 1) * kTcTileM;
    static constexpr int kFloats = kCert + 2 * 4 * kTcTileM;
};

// Layer of a work item: every layer has the same number of items, or one layer has all.
__device__ __forceinline__ int tc_layer(const ForwardParams& p, long long item)
{
    return p.tc_ipl > 0 ? (int)(item / p.tc_ipl) : layer_of(p, item);
}

// SPLIT: the work units are not items but the two grids of an item (unit 2 i + g), where items
// are so few that the SMs hold all of them at once and an item's tiles, one round trip after
// another, are the launch (one item of 2 x 4000 points at d = 4: 27 -> 15 us).  Units without a
// tile (grids of one point) make the warps meet, which costs the screen's loop 0.3% and
// is left out of the other variant: that one takes no layers of one point by one.
template <int DM, int KT, bool SPLIT>
__global__ void __launch_bounds__(kTcThreads, kTcCtas) forward_tc_kernel(const __grid_constant__ ForwardParams p)
{
    constexpr int K = 16 * KT;
    static_assert(3 * DM + 2 <= K, "operand row");
    constexpr uint32_t kTileBytes = kTcTileN * K * 2;
    constexpr uint32_t kCertBytes = TcItem<DM>::kCert * 4;
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(kTcTileN >> 3) << 17) | ((uint32_t)(kTcTileM >> 4) << 24);
    extern __shared__ __align__(128) unsigned char dsm_tc[];
    __shared__ __align__(8) unsigned long long s_tfull[kTcMaxSlots], s_cfull[2];
    __shared__ __align__(8) unsigned long long s_accfull, s_meet;
    __shared__ uint32_t s_arrived;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;

    const int t = threadIdx.x;
    const int warp = __shfl_sync(0xFFFFFFFFu, t >> 5, 0);
    const int RS = p.tc_slots;
    const long long G = gridDim.x;
    // dynamic shared memory: [tile ring][operand rows of one grid][centred samples: two items]
    unsigned char* ops = dsm_tc + (size_t)RS * kTileBytes;
    float* cert0 = reinterpret_cast<float*>(ops + kTcTileM * K * 2);
    const uint32_t ring_u = smem_u32(dsm_tc), cert_u = smem_u32(cert0);
    const uint32_t accfull = smem_u32(&s_accfull), arrived = smem_u32(&s_arrived);
    const uint32_t tfull = smem_u32(&s_tfull[0]), cfull = smem_u32(&s_cfull[0]);

    if (t == 0) {
        for (int i = 0; i < kTcMaxSlots; ++i) mbar_init(tfull + (uint32_t)(8 * i), 1);
        mbar_init(cfull, 1);
        mbar_init(cfull + 8, 1);
        mbar_init(accfull, 1);
        mbar_init(smem_u32(&s_meet), kTcThreads / 32);
        s_arrived = 0;
        s_abort = 0;
        fence_proxy_async();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"((uint32_t)kTcTileN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    const uint64_t adesc = smem_desc(smem_u32(ops), 128, K * 16);
    const uint64_t bdesc = smem_desc(ring_u, 128, K * 16);
    const long long budget = p.spin_budget;
    bool ok = true;

    // ---- tile loads: a cursor over the tiles of this CTA's items, grid A's then grid B's
    // of each (a one-point grid needs none), kept by every thread; whichever warp issues
    // a tile's MMAs starts the copy that refills the slot before it
    constexpr int kSplit = SPLIT ? 1 : 0;
    const long long unit_lo = p.item_lo << kSplit, unit_hi = p.item_hi << kSplit;
    // tiles of a unit's grid A, and of both
    auto tiles_of = [&](long long unit, const GridInfo& GA, const GridInfo& GB, int& a, int& all) {
        a = GA.N > 1 && !(SPLIT && (unit & 1) != 0) ? GA.tc_tiles : 0;
        all = a + (GB.N > 1 && !(SPLIT && (unit & 1) == 0) ? GB.tc_tiles : 0);
    };
    long long ld_item = unit_lo + blockIdx.x, ld_end = 0;
    int ld_a = 0, ld_b = 0;                            // tile numbers of the cursor's layer
    int ld_i = 0, ld_tA = 0, ld_nT = 0;
    // number of the next tile to load, -1 after the last one
    auto next_tile = [&]() -> int {
        while (ld_i == ld_nT) {                        // the next item with tiles
            if (ld_nT > 0) ld_item += G;
            ld_i = 0;
            if (ld_item >= unit_hi) {
                ld_nT = 0;
                return -1;
            }
            if (SPLIT || ld_nT == 0 || ld_item >= ld_end) {
                const LayerDesc& L = p.layers[tc_layer(p, ld_item >> kSplit)];
                const GridInfo& GA = p.grids[L.gridA];
                const GridInfo& GB = p.grids[L.gridB];
                ld_end = L.item_begin + L.items;
                tiles_of(ld_item, GA, GB, ld_tA, ld_nT);
                ld_a = (int)GA.tc_toff;
                ld_b = (int)GB.tc_toff - ld_tA;
                if (ld_nT == 0) ld_item += G;
            }
        }
        const int src = (ld_i < ld_tA ? ld_a : ld_b) + ld_i;
        ++ld_i;
        return src;
    };
    auto load_tile = [&](int src, int to) {
        const uint32_t bar = tfull + (uint32_t)(8 * to);
        mbar_arrive_expect_tx(bar, kTileBytes);
        bulk_g2s(ring_u + (uint32_t)to * kTileBytes,
                 reinterpret_cast<const unsigned char*>(p.tc_tiles) + (long long)src * kTileBytes, kTileBytes, bar);
    };
    auto load_samples = [&](long long n) {
        const long long unit = unit_lo + blockIdx.x + n * G, item = unit >> kSplit;
        if (unit >= unit_hi) return;
        const uint32_t bar = cfull + (uint32_t)(8 * (n & 1));
        mbar_arrive_expect_tx(bar, kCertBytes);
        bulk_g2s(cert_u + (uint32_t)(n & 1) * kCertBytes,
                 p.tc_items + (item - p.item_lo) * (long long)(TcItem<DM>::kFloats * 4), kCertBytes, bar);
    };
    if (t == 0) load_samples(0);
    for (int i = 0; i < RS; ++i) {
        const int src = next_tile();
        if (t == 0 && src >= 0) load_tile(src, i);
    }

    int slot = 0;                                      // ring slot and parity of the next tile
    uint32_t ph = 0, accph = 0;
    long long lend = 0;
    int tA = 0, nT = 0, expA = 0, expB = 0;
    long long n = 0;
    for (;; ++n) {
        const long long unit = unit_lo + blockIdx.x + n * G, item = unit >> kSplit;
        if (unit >= unit_hi) break;
        if (__shfl_sync(0xFFFFFFFFu, *(volatile int*)&s_abort, 0)) {
            ok = false;
            break;
        }
        if (SPLIT || n == 0 || item >= lend) {
            const LayerDesc& L = p.layers[tc_layer(p, item)];
            const GridInfo& GA = p.grids[L.gridA];
            const GridInfo& GB = p.grids[L.gridB];
            lend = L.item_begin + L.items;
            tiles_of(unit, GA, GB, tA, nT);
            expA = GA.tc_exp;
            expB = GB.tc_exp;
        }
        // this item's samples have landed; the next item's go to the other buffer, which
        // every warp has left (all have read the last tile of the item before)
        if (!warp_wait(cfull + (uint32_t)(8 * (n & 1)), (uint32_t)((n >> 1) & 1), budget)) {
            ok = false;
            break;
        }
        if (t == 0) load_samples(n + 1);
        const float* cert = cert0 + (n & 1) * TcItem<DM>::kCert;
        float* state = reinterpret_cast<float*>(p.tc_items) + (item - p.item_lo) * (long long)TcItem<DM>::kFloats + TcItem<DM>::kCert + t;
        // operand rows of one grid: the MMAs of the grid before are complete (every warp
        // has waited for its last tile); fenced for the tensor core's reads
        auto operands = [&](int gr) {
            operand_row<DM, K>(cert + gr * (DM + 1) * kTcTileM, t, gr == 0 ? expA : expB, ops);
            fence_proxy_async();
        };
        // Called by every warp when it has read the accumulator and written its operand
        // rows: the last of the four issues the next tile's MMAs (one elected lane) once
        // the tile has landed, and refills the slot `old` (its tile is read) with tile
        // src.  (A separate issuing warp behind an mbarrier took 630 cycles more for this.)
        auto arrive_and_issue = [&](int old, int src) -> bool {
            tc_fence_before();
            __syncwarp();
            uint32_t c = 0;
            if (elect_one()) c = count_arrival(arrived);
            if ((__reduce_max_sync(0xFFFFFFFFu, c) & 3u) != 3u) return true;
            if (!warp_wait(tfull + (uint32_t)(8 * slot), ph, budget)) return false;
            tc_fence_after();
            const uint64_t bd = bdesc + (uint64_t)((uint32_t)slot * (kTileBytes >> 4));
            if (elect_one()) {
#pragma unroll
                for (int s = 0; s < KT; ++s) tc_mma(tmem, adesc + (uint64_t)(s * 16), bd + (uint64_t)(s * 16), idesc, s > 0 ? 1u : 0u);
                tc_commit(accfull);
                if (src >= 0) load_tile(src, old);
            }
            __syncwarp();
            return true;
        };
        KeyTrack tr;
        tr.reset();
        auto put = [&](int gr) {
            float* o = state + gr * 4 * kTcTileM;
            o[0] = __int_as_float(KeyTrack::chunk(tr.B1, tr.t1));
            o[kTcTileM] = __int_as_float(KeyTrack::chunk(tr.Bs, tr.ts));
            o[2 * kTcTileM] = KeyTrack::low(tr.Bs);
            o[3 * kTcTileM] = KeyTrack::low(tr.B3);
            tr.reset();
        };
        if (nT > 0) {
            operands(tA > 0 ? 0 : 1);
            ok = arrive_and_issue(0, -1);
        } else if constexpr (SPLIT) {
            // no tile holds the warps together, and a warp that still waited for these samples
            // when those after the next arrive would wait for the wrong phase
            ok = warps_meet(smem_u32(&s_meet), budget);
        }
#pragma unroll 1
        for (int i = 0; i < nT; ++i) {
            ok = warp_wait(accfull, accph, budget) && ok;
            if (!ok) break;
            accph ^= 1u;
            tc_fence_after();
            // all minima first, so that the accumulator goes back before the tracking; a
            // loop, not two copies: the compiler gives every load scratch registers of its
            // own, 128 in all, and spills the rest for them
            float mc[8];
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                float m0, m1, m2, m3;
                tc_chunk_min4(trow + (uint32_t)(64 * h), m0, m1, m2, m3);
                if (h == 0) {
                    mc[0] = m0;
                    mc[1] = m1;
                    mc[2] = m2;
                    mc[3] = m3;
                } else {
                    mc[4] = m0;
                    mc[5] = m1;
                    mc[6] = m2;
                    mc[7] = m3;
                }
            }
            const int old = slot, src = next_tile();
            if (++slot == RS) {
                slot = 0;
                ph ^= 1u;
            }
            if (i + 1 == tA && tA < nT) operands(1);
            if (i + 1 < nT) ok = arrive_and_issue(old, src);
            else if (t == 0 && src >= 0) load_tile(src, old);      // the item's last tile: every MMA is complete
            tr.add_tile(mc, i < tA ? i : i - tA);
            if (i + 1 == tA) put(0);
        }
        if (!ok) break;
        if (nT > tA) put(1);
    }
    if (!ok && (t & 31) == 0) {
        record_error(p.status, 4 /* QT_ETIMEOUT */, 26);
        *(volatile int*)&s_abort = 1;
    }
    // every MMA issued completes before the memory is released: whichever warp issued,
    // its tile's barrier; after a timeout the wait for it runs on, bounded
    if (!ok) mbar_wait_bounded(accfull, accph, kDrainUs / 10);
    tc_fence_before();
    __syncthreads();
    if (t == 0 && s_abort) {
        // after a timeout the copies still in flight land too (a slot that nothing is
        // loading runs its second out)
        for (int q = 0; q < 2; ++q) mbar_wait_bounded(cfull + (uint32_t)(8 * ((n + q) & 1)), (uint32_t)(((n + q) >> 1) & 1), 1000000);
        for (int q = 0; q < RS; ++q) {
            mbar_wait_bounded(tfull + (uint32_t)(8 * slot), ph, 1000000);
            if (++slot == RS) {
                slot = 0;
                ph ^= 1u;
            }
        }
    }
    __syncthreads();
    tc_fence_after();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kTcTileN) : "memory");
    }
}

// Exact FP64 argmin over one point per lane (j >= N: none), lowest index among equal
// distances, for the sample of lane src.
template <int DM>
__device__ __noinline__ int chunk_exact(const double (&z)[DM], int src, int j, const double* __restrict__ g64, int N,
                                        int d)
{
    double zz[DM];
#pragma unroll
    for (int l = 0; l < DM; ++l) zz[l] = __shfl_sync(0xFFFFFFFFu, z[l], src);
    double best = __longlong_as_double(0x7FF0000000000000LL);
    int bi = 0x7FFFFFFF;
    if (j < N) {
        best = dist64<DM>(zz, g64 + (long long)j * d, d);
        bi = j;
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        const double ob = __shfl_xor_sync(0xFFFFFFFFu, best, off);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, off);
        if (ob < best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
        }
    }
    return bi;
}

// The last kernel of a window: persistent CTAs of 128 threads over its work items,
// thread t for row t; the records come two items ahead by bulk copies (one CTA per
// item, its loads one after the other, took 280 us for 9375 items at d = 8, all of it
// latency).  The best chunk is re-scored in FP32, the second one where the certificate
// needs it; the exact window search takes what neither certifies; then the counts.
constexpr int kCertifyCtas = 6;

template <int DM>
__global__ void __launch_bounds__(kTcTileM, kCertifyCtas) tc_certify_kernel(const __grid_constant__ ForwardParams p)
{
    constexpr uint32_t kBytes = TcItem<DM>::kFloats * 4;
    extern __shared__ __align__(128) float dsm_cf[];   // two records, then the counts of a small layer
    __shared__ __align__(8) unsigned long long s_full[2];
    __shared__ GridInfo s_G[2];
    __shared__ float s_sigma[2][2];                    // 2^tc_exp and its inverse
    const int t = threadIdx.x, lane = t & 31;
    const int d = p.d;
    // the screen gave up: its states are not valid.  One answer for the whole CTA: another
    // CTA may be recording an error while this one starts
    if (__syncthreads_or(*((volatile int32_t*)&p.status->code) != 0)) return;
    const uint32_t full = smem_u32(&s_full[0]), buf = smem_u32(dsm_cf);
    auto load = [&](long long n) {
        const long long item = p.item_lo + blockIdx.x + n * (long long)gridDim.x;
        if (item >= p.item_hi) return;
        const uint32_t bar = full + (uint32_t)(8 * (n & 1));
        mbar_arrive_expect_tx(bar, kBytes);
        bulk_g2s(buf + (uint32_t)(n & 1) * kBytes, p.tc_items + (item - p.item_lo) * (long long)kBytes, kBytes, bar);
    };
    if (t == 0) {
        mbar_init(full, 1);
        mbar_init(full + 8, 1);
        fence_proxy_async();
        load(0);
        load(1);
    }
    __syncthreads();
    int k = -1;
    LayerDesc L;
    // counts of a layer of a few hundred entries are gathered in shared memory first: the L2
    // reductions of all CTAs meet on them (1e6 given pairs on 16 x 16 points: 375 -> 330 us)
    uint32_t* hist = reinterpret_cast<uint32_t*>(dsm_cf + 2 * TcItem<DM>::kFloats);
    int live = 0;                                      // entries gathered there, 0: none
    auto flush = [&]() {
        for (int e = t; e < live; e += kTcTileM)
            if (hist[e]) count_add(p.counts, p.counts_u32, L.coff + e, hist[e]);
    };
    const float sqrt_d = sqrtf((float)d);
    for (long long n = 0;; ++n) {
        const long long item = p.item_lo + blockIdx.x + n * (long long)gridDim.x;
        if (item >= p.item_hi) break;
        const int ki = tc_layer(p, item);
        if (ki != k) {
            flush();                                   // (every warp is done with the item before)
            k = ki;
            L = p.layers[k];
            live = L.hist_smem ? L.NA * L.NB : 0;
            __syncthreads();
            for (int e = t; e < live; e += kTcTileM) hist[e] = 0;
            for (int e = t; e < (int)(sizeof(GridInfo) / 4); e += kTcTileM) {
                reinterpret_cast<int*>(&s_G[0])[e] = reinterpret_cast<const int*>(p.grids + L.gridA)[e];
                reinterpret_cast<int*>(&s_G[1])[e] = reinterpret_cast<const int*>(p.grids + L.gridB)[e];
            }
            if (t < 4) {
                const int e = p.grids[t < 2 ? L.gridA : L.gridB].tc_exp;
                s_sigma[t >> 1][t & 1] = ldexpf(1.0f, (t & 1) ? -e : e);
            }
            __syncthreads();
        }
        // the records were written by earlier kernels: the copy always lands (if it did not,
        // the copy of the next item is waited for too before the CTA leaves)
        if (!mbar_wait_bounded(full + (uint32_t)(8 * (n & 1)), (uint32_t)((n >> 1) & 1), kDrainUs)) {
            record_error(p.status, 4 /* QT_ETIMEOUT */, 27);
            mbar_wait_bounded(full + (uint32_t)(8 * ((n + 1) & 1)), (uint32_t)(((n + 1) >> 1) & 1), 1000000);
            return;
        }
        const float* rec = dsm_cf + (n & 1) * TcItem<DM>::kFloats;
        const unsigned long long ms = (unsigned long long)(item - L.item_begin) * kTcTileM + (unsigned long long)t;
        const bool valid = ms < p.M;
        __syncwarp();
        int cell[2] = {0, 0};
#pragma unroll 1
        for (int gr = 0; gr < 2; ++gr) {
            const GridInfo& Gi = s_G[gr];
            if (Gi.N <= 1) continue;
            const float* cert = rec + gr * (DM + 1) * kTcTileM + (t & 96);
            const float* st = rec + TcItem<DM>::kCert + gr * 4 * kTcTileM + t;
            const int c0 = __float_as_int(st[0]), c1 = __float_as_int(st[kTcTileM]);
            const float* rows = p.tc_rows + Gi.tc_toff * (long long)(kTcTileN * (DM + 1));
            const float Araw = cert[DM * kTcTileM + lane];
            const bool big = (__float_as_int(Araw) & (int)0x80000000) != 0;
            const float A = fabsf(Araw);
            const float sg = s_sigma[gr][0], inv_sg = s_sigma[gr][1], inv2 = inv_sg * inv_sg;
            const float second = st[2 * kTcTileM] * inv2, rest = st[3 * kTcTileM] * inv2;
            float best, in2;
            int idx;
            quad_rescore<DM>(rows, cert, lane, c0, best, in2, idx);
            // FP32 inside the best chunk, tensor-core scores outside it
            int why = tc_uncertified(d, A, best, in2, fminf(second, rest), Gi.R, sqrt_d, sg, inv_sg);
            // the second chunk competes: FP32 inside both, tensor-core scores outside
            const bool two = valid && (why & 2) != 0 && c1 != c0;
            if (__any_sync(0xFFFFFFFFu, two)) {
                float best2 = 0.0f, S12 = 0.0f;
                int idx2 = 0;
                quad_rescore_some<DM>(rows, cert, lane, two, c1, best2, S12, idx2);
                if (two) {
                    if (best2 < best || (best2 == best && idx2 < idx)) {
                        in2 = fminf(S12, best);
                        best = best2;
                        idx = idx2;
                    } else {
                        in2 = fminf(in2, best2);
                    }
                    why = tc_uncertified(d, A, best, in2, rest, Gi.R, sqrt_d, sg, inv_sg);
                }
            }
            const bool rng_ok = idx < Gi.N && !big;
            const bool need = valid && (why != 0 || !rng_ok);
            if (need) atomicAdd(&p.status->spare[!rng_ok ? 3 : ((why & 1) ? 1 : 2)], 1ull);
            // exact FP64 distances for the lanes in `need`, the whole warp for one sample: to
            // the points of the re-scored chunks where no other can be nearer (nearly always:
            // two points tie within the FP32 bound), by the window search of the whole grid
            // otherwise (its latency, 32 rounds of loads for 4000 points, ends the kernel)
            unsigned mask = __ballot_sync(0xFFFFFFFFu, need);
            if (mask) {
                const float* gpf = p.params_f ? p.params_f + (long long)k * p.params_stride : nullptr;
                const double* gpd = p.params_d ? p.params_d + (long long)k * p.params_stride : nullptr;
                const double* g64 = p.g64 + Gi.goff * d;
                const bool inside = (why & 2) == 0 && rng_ok;
                // an FP64 operation takes a warp as long for one lane as for all that need it
                double z[DM];
                if (need) exact_sample<DM>(p, gpf, gpd, k, ms, gr == 1, z);
                while (mask) {
                    const int src = __ffs(mask) - 1;
                    mask &= mask - 1;
                    int r;
                    if (__shfl_sync(0xFFFFFFFFu, (int)inside, src)) {
                        const int a = __shfl_sync(0xFFFFFFFFu, c0, src), b = __shfl_sync(0xFFFFFFFFu, two ? c1 : c0, src);
                        const int ch = lane < 16 ? a : b;
                        r = chunk_exact<DM>(z, src, ch * kChunk + (lane & 15), g64, Gi.N, d);
                    } else {
                        float x[DM];
#pragma unroll
                        for (int l = 0; l < DM; ++l) x[l] = cert[l * kTcTileM + lane];
                        r = warp_window_nn<DM>(x, A, z, src, p.rec32 + Gi.roff * Rec32<DM>::kFloats, Gi.Npad, g64, Gi.N, d);
                    }
                    if (lane == src) idx = r;
                    if (lane == 0) atomicAdd(&p.status->rechecks, 1ull);
                }
            }
            cell[gr] = idx;
        }
        // ---- counters p^k_ij
        const int ci = cell[0], cj = cell[1];
        if (valid && ((unsigned)ci >= (unsigned)L.NA || (unsigned)cj >= (unsigned)L.NB)) {
            record_error(p.status, 6 /* QT_EDEVICE */, 13);
        } else if (valid) {
            if (live) atomicAdd(&hist[ci * L.NB + cj], 1u);
            else count_add(p.counts, p.counts_u32, L.coff + (long long)ci * L.NB + cj, 1u);
            if (p.cellsA) {
                p.cellsA[ms] = ci;
                p.cellsB[ms] = cj;
            }
            if (p.dump_count > 0 && (ms % (unsigned long long)p.dump_stride) == 0ull) {
                const unsigned long long tt = ms / (unsigned long long)p.dump_stride;
                if (tt < (unsigned long long)p.dump_count) {
                    const long long row = (long long)k * p.dump_count + (long long)tt;
                    const float* gpf = p.params_f ? p.params_f + (long long)k * p.params_stride : nullptr;
                    const double* gpd = p.params_d ? p.params_d + (long long)k * p.params_stride : nullptr;
                    double z[DM];
                    exact_sample<DM>(p, gpf, gpd, k, ms, false, z);
                    for (int l = 0; l < d; ++l) p.dumpX[row * d + l] = z[l];
                    exact_sample<DM>(p, gpf, gpd, k, ms, true, z);
                    for (int l = 0; l < d; ++l) p.dumpY[row * d + l] = z[l];
                    p.dumpI[row] = ci;
                    p.dumpJ[row] = cj;
                }
            }
        }
        __syncthreads();                               // every warp is done with this record (and s_G)
        if (t == 0) load(n + 2);
    }
    flush();
}

// Screen of the items [p.item_lo, p.item_hi).
template <int DM, int KT, bool SPLIT>
cudaError_t launch_tc(const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    auto kern = forward_tc_kernel<DM, KT, SPLIT>;
    cudaError_t e = allow_dynamic_smem(kern, dyn);
    if (e != cudaSuccess) return e;
    if (p.tc_slots < 2 || p.tc_slots > kTcMaxSlots) return cudaErrorInvalidValue;
    // four CTAs share an SM: registers (launch bounds), shared memory (make_plan_full)
    // and tensor memory (128 of 512 columns each) are taken so that they fit
    *bps = kTcCtas;
    long long grid = (long long)kTcCtas * num_sms;
    const long long units = (p.item_hi - p.item_lo) * (SPLIT ? 2 : 1);
    if (grid > units) grid = units;
    if (grid < 1) return cudaSuccess;
    kern<<<(unsigned)grid, kTcThreads, dyn, st>>>(p);
    return cudaGetLastError();
}

}  // namespace qt
