// qt_cells.cuh -- located nearest-cell search for d <= 2: a table of small boxes
// ("bins") over each grid, every bin holding the few grid points whose Voronoi
// cell can meet it, so that a search evaluates one to four distances instead of
// all N_k (Sec. 3.2 of Pages & Wilbertz, arXiv:1101.3228, searches by brute
// force; its kd-tree attempt is the prior art for a located search).
//
// Table of a grid (built per call by build_cells_kernel, one 64-bit entry per
// bin): up to six 10-bit point indices in increasing order and their number in
// the top four bits; kCellPool = a longer list in the pool (offset in bits 0-31,
// length in bits 32-47); kCellScan = every point of the grid.  A point j is left
// out of a bin only if one other point is nearer by more than every rounding
// below, everywhere in the bin enlarged by a sixteenth of its width, so that the
// exact FP64 argmin and everything tied with it is always in the list.
//
// Certificate: with a = x - mu in FP32 and g = fl32(c - mu), D~ = sum (a - g)^2
// satisfies |D~ - D| <= err(D) = sqrt(d) (kappa D + e^2 / kappa) + d e^2 +
// (d + 6) 2^-24 D, e the sum of both coordinates' errors, for any kappa > 0
// (2 sqrt(D) e <= kappa D + e^2 / kappa).  The best candidate is the exact argmin
// when second - best > 2 err(second).  A sample whose e is f <= 1 times the grid's bound
// takes f kappa: 2 err(D) = f (c1 D + c2) + c3 D, kappa for distances of a bin and e for
// the whole box.  What that does not certify is tried with the square root itself and
// with the rounding of this sample and of points at this distance, u (2 |a| + sqrt(D)) in
// the place of the box's (cell_doubt): that holds on the scale of any cell, for grids whose
// points lie much closer together than their box tells, and outside the box.  Otherwise
// the exact FP64 distances of the bin's candidates decide.
//
// Outside the box the first and last bins go on.  For d = 1 they do for 2^20 bins without
// further ado: D_j - D_i = (g_i - g_j)(2 x - g_i - g_j) only grows there.  For d = 2 a point
// further out than the witness may be dropped from such a bin only if it is further away all
// along the 4096 bins beyond.  (Further out distances tie in FP64, 2^-52 r^2; a point is
// dropped for being 5 u D nearer at least, D the squared distance from the bin, or u R h.)
// Beside the box |a| <= R + sqrt(D), and the excess of 4 sqrt(d D) u (2 R + 3 sqrt(D)) over
// the box's bound is the 12 sqrt(d) u D that c3 has more.  Beyond that the whole grid is
// searched.  An axis along which all points are equal has one bin of 2^14 of the other's:
// what it adds to the distances is the same number for all points.
//
// Why bins: brute force spends 2 d flops on each of N_k + N_{k+1} candidates (1000
// on the 2-factor workload), and only the few points around a sample can be its
// cell.  About 20 bins per point (104 x 104 at most, split by the grid's extents: two
// tables fit one CTA's shared memory) leave 3.2 candidates per search on average and 5.5
// for the slowest lane of a warp (samples of N(0, I) on a quantizer of 500 points, counted on
// the CPU); 64 x 64 bins leave 6.1 and 12.6.
#pragma once
#include "qt_forward.cuh"

namespace qt {

constexpr int kCellInline = 6;         // indices held in an entry
constexpr int kCellBeyond = 4096;      // d = 2: bins beyond the table that its first and last ones serve
constexpr int kCellPool = 15;          // entry refers to the pool
constexpr int kCellScan = 14;          // entry stands for the whole grid
constexpr uint64_t kCellScanEntry = (uint64_t)kCellScan << 60;

__device__ __forceinline__ float cell_dist(const float* __restrict__ rec, int j, const float (&a)[1])
{
    const float dx = a[0] - rec[j];
    return dx * dx;
}
__device__ __forceinline__ float cell_dist(const float* __restrict__ rec, int j, const float (&a)[2])
{
    const float2 g = reinterpret_cast<const float2*>(rec)[j];
    const float dx = a[0] - g.x, dy = a[1] - g.y;
    return __fmaf_rn(dy, dy, dx * dx);
}

// A sample's 2 err(D) with the square root: linear in r = sqrt(D) beside r^2.
struct CellDoubt {
    float c, s, q;                     // 2 err(D) = c + s r + q D
    __device__ __forceinline__ float operator()(float D) const
    {
        float r;
        asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(D));
        return __fmaf_rn(q, D, __fmaf_rn(s, r, c));
    }
    // D~_best + this much and more is beyond doubt: K >= 2 err(b + K) for K = max(4 s^2,
    // 2.1 (c + s sqrt(b) + q b)), because s sqrt(b + K) <= s sqrt(b) + s sqrt(K) and
    // s sqrt(K) <= K / 2 (q K, q < 2^-17, is in the 2.1)
    __device__ __forceinline__ float window(float b) const { return fmaxf(4.04f * s * s, 2.12f * (*this)(b)); }
};

// f: the share of the grid's bound that the search takes.  e = the part beyond FP32
// rounding (f's e less the box's rounding) + u (2 |a| + r), 1.01 for this arithmetic.
template <int DM>
__device__ __forceinline__ CellDoubt cell_doubt(const CellGrid& G, const float (&a)[DM], float f)
{
    constexpr float sq = DM == 1 ? 1.0f : 1.41421357f, u = 0x1p-24f;
    float m = fabsf(a[0]);
    if constexpr (DM == 2) m += fabsf(a[1]);
    const float e0 = 1.01f * (fmaxf(__fmaf_rn(f, G.e, -G.ebox), 0.0f) + 0x1p-22f * G.e + 2.0f * u * m);
    // 4 sq (e0 + u r) r + 2 DM (e0 + u r)^2 + 2 (DM + 6) u D
    return CellDoubt{__fmaf_rn(2.05f * DM * e0, e0, 0x1p-120f), 4.1f * sq * e0, (4.1f * sq + 2.05f * (DM + 6)) * u};
}

// One step of a running minimum: smallest, second smallest, index of the smallest.
__device__ __forceinline__ void cell_take(float D, int j, float& best, float& second, int& bi)
{
    second = fminf(second, fmaxf(D, best));
    bi = D < best ? j : bi;
    best = fminf(best, D);
}

// Smallest distance to eight consecutive points (every lane reads the same ones: 16-byte
// broadcasts).
template <int DM>
__device__ __forceinline__ float cell_min8(const float* __restrict__ rec, const float (&a)[DM])
{
    float m = __int_as_float(0x7F800000);
#pragma unroll
    for (int v = 0; v < 8 * DM; v += 4) {
        const float4 r = *reinterpret_cast<const float4*>(rec + v);
        if constexpr (DM == 1) {
            const float x = a[0] - r.x, y = a[0] - r.y, z = a[0] - r.z, w = a[0] - r.w;
            m = fminf(fminf(m, fminf(x * x, y * y)), fminf(z * z, w * w));
        } else {
            const float x = a[0] - r.x, y = a[1] - r.y, z = a[0] - r.z, w = a[1] - r.w;
            m = fminf(m, fminf(__fmaf_rn(y, y, x * x), __fmaf_rn(w, w, z * z)));
        }
    }
    return m;
}

// Smallest and second smallest distance over the whole grid, eight points at a time: only
// the minimum of the eight is tracked; which point it was, and the second within its eight,
// come from that group at the end.  About 4.6 instructions a point for d = 2, as many as the
// brute-force screen takes: a grid that no table serves costs no more than without one.
template <int DM>
__device__ __forceinline__ void cell_scan(const float* __restrict__ rec, int N, const float (&a)[DM], float& best,
                                          float& second, int& bi)
{
    const float inf = __int_as_float(0x7F800000);
    float b1 = inf, b2 = inf;
    int g1 = 0;
    const int N8 = N & ~7;
    for (int j = 0; j < N8; j += 8) {
        const float m = cell_min8<DM>(rec + j * DM, a);
        b2 = fminf(b2, fmaxf(m, b1));
        g1 = m < b1 ? j : g1;
        b1 = fminf(b1, m);
    }
    // the best group's points in order, then the last N mod 8
    best = inf;
    second = inf;
    bi = 0;
    if (N8 > 0)
        for (int q = 0; q < 8; ++q) cell_take(cell_dist(rec, g1 + q, a), g1 + q, best, second, bi);
    second = fminf(second, b2);
    for (int j = N8; j < N; ++j) cell_take(cell_dist(rec, j, a), j, best, second, bi);
}

// Lists longer than an entry: the pool's, or the whole grid (records in shared
// memory), which also serves samples outside the box.  Returns the index, with the top
// bit set when the distances do not certify it, and above it the smallest distance.
template <int DM>
__device__ __noinline__ uint64_t cell_long_list(const CellGrid& G, const float* __restrict__ rec,
                                                const uint16_t* __restrict__ pool, uint64_t e, float a0, float a1, float f)
{
    float a[DM];
    a[0] = a0;
    if constexpr (DM == 2) a[1] = a1;
    float best = __int_as_float(0x7F800000), second = best;
    int bi = 0;
    if ((int)(e >> 60) == kCellScan) {
        cell_scan<DM>(rec, G.N, a, best, second, bi);
    } else {
        const uint16_t* lst = pool + (uint32_t)e;
        const int cnt = (int)((e >> 32) & 0xFFFFu);
#pragma unroll 4
        for (int q = 0; q < cnt; ++q) {
            const int j = (int)lst[q];
            cell_take(cell_dist(rec, j, a), j, best, second, bi);
        }
    }
    const bool need = !(second - best > cell_doubt<DM>(G, a, f)(second));
    return (uint32_t)bi | (need ? 0x80000000u : 0u) | ((uint64_t)__float_as_uint(best) << 32);
}

// A grid's records, after its table.
__device__ __forceinline__ const float* cell_records(const CellGrid& G, const unsigned char* sm)
{
    return reinterpret_cast<const float*>(sm + (size_t)((uint32_t)G.nb0 * (uint32_t)G.nb1 * 8u));
}

// Number of the bin of coordinate a along one axis: the FMA rounds a / h + origin to
// the nearest integer in the low bits of a float near 2^23; whatever lies outside
// the axis (or is not finite) gives a number outside [0, nb).
__device__ __forceinline__ uint32_t cell_bin(float a, float inv_h, float org)
{
    return (uint32_t)__float_as_int(__fmaf_rn(a, inv_h, org)) - 0x4B000000u;
}

// Nearest candidate of the centred sample `a` in the grid G (shared memory: G, and
// its table and records at `sm`); f: the sample's error as a share of the grid's
// bound.  `entry` is its bin's list, `need` is set when the FP32 distances do not
// certify the pick.
template <int DM>
__device__ __forceinline__ int cell_search(const CellGrid& G, const unsigned char* sm, const uint16_t* __restrict__ pool,
                                           const float (&a)[DM], float f, uint64_t& entry, bool& need)
{
    const float4 axes = *reinterpret_cast<const float4*>(G.inv_h);
    uint32_t b = cell_bin(a[0], axes.x, axes.z);
    bool in = b < (uint32_t)G.nb0;
    if constexpr (DM == 1) {
        if (!in) {
            // beside the table: the first and last bins go on for 2^20 more
            const float v = __fmaf_rn(a[0], axes.x, axes.z) - 8388608.0f;
            in = fabsf(v) <= 1048576.0f;
            b = v > 0.0f ? (uint32_t)G.nb0 - 1u : 0u;
        }
    } else {
        uint32_t b1 = cell_bin(a[1], axes.y, axes.w);
        in = in && b1 < (uint32_t)G.nb1;
        if (!in) {
            // beside the table: the first and last bins go on for kCellBeyond more
            const float v0 = __fmaf_rn(a[0], axes.x, axes.z) - 8388608.0f, v1 = __fmaf_rn(a[1], axes.y, axes.w) - 8388608.0f;
            in = fabsf(v0) <= (float)kCellBeyond && fabsf(v1) <= (float)kCellBeyond;
            b = (uint32_t)fminf(fmaxf(v0, 0.0f), (float)G.nb0 - 1.0f);
            b1 = (uint32_t)fminf(fmaxf(v1, 0.0f), (float)G.nb1 - 1.0f);
        }
        b += b1 * (uint32_t)G.nb0;
    }
    uint64_t e = kCellScanEntry;
    if (in) e = reinterpret_cast<const uint64_t*>(sm)[b];
    entry = e;
    const int cnt = (int)(e >> 60);
    int idx = (int)(e & 1023u);
    need = false;
    const float* rec = cell_records(G, sm);
    if (cnt > kCellInline) {
        const uint64_t r = cell_long_list<DM>(G, rec, pool, e, a[0], DM == 2 ? a[DM - 1] : 0.0f, f);
        idx = (int)((uint32_t)r & 0x7FFFFFFFu);
        need = ((uint32_t)r >> 31) != 0;
        if (cnt == kCellScan) entry = kCellScanEntry | (r >> 32);
    } else if (cnt > 1) {
        float best = cell_dist(rec, idx, a), second = __int_as_float(0x7F800000);
        uint64_t r = e;
        for (int q = 1; q < cnt; ++q) {
            r >>= 10;
            const int j = (int)(r & 1023u);
            const float D = cell_dist(rec, j, a);
            second = fminf(second, fmaxf(D, best));
            idx = D < best ? j : idx;
            best = fminf(best, D);
        }
        need = !(second - best > __fmaf_rn(f, __fmaf_rn(G.c1, second, G.c2), G.c3 * second));
        if (need) need = !(second - best > cell_doubt<DM>(G, a, f)(second));
    }
    return idx;
}

// Exact FP64 argmin over a bin's candidates (lowest index among equal distances), for a
// search that the FP32 distances did not certify: only those that they leave in doubt,
// D~_j <= D~_best + window, are evaluated in FP64 (two of them nearly always; an FP64
// operation holds a warp's quarter of the SM for 65 cycles whether one lane takes part or
// all, so the points in doubt are put into an entry first and evaluated side by side).  A
// sample without a finite distance has no cell: the index is out of range, and the callers
// refuse it, as in the other forms.
// a: the sample z in FP32, centred.  KNOWN: an entry that stands for the whole grid has the
// smallest distance from it in its low word.
template <int DM, bool KNOWN>
__device__ __noinline__ int cell_exact(const CellGrid& G, const float* __restrict__ rec, const float (&a)[DM],
                                       const double (&z)[DM], uint64_t e, const uint16_t* __restrict__ pool,
                                       const double* __restrict__ g64)
{
    const int kind = (int)(e >> 60);
    const int cnt = kind == kCellScan ? G.N : (kind == kCellPool ? (int)((e >> 32) & 0xFFFFu) : kind);
    auto at = [&](int q) {
        return kind == kCellScan ? q : (kind == kCellPool ? (int)pool[(uint32_t)e + q] : (int)((e >> (10 * q)) & 1023u));
    };
    float b = __int_as_float(0x7F800000);
    if (KNOWN && kind == kCellScan) {
        b = __uint_as_float((uint32_t)e);
    } else {
#pragma unroll 4
        for (int q = 0; q < cnt; ++q) b = fminf(b, cell_dist(rec, at(q), a));
    }
    const float lim = b + cell_doubt<DM>(G, a, 0.0f).window(b);   // rounding alone: a is z's own
    uint64_t in_doubt = 0;
    int n = 0;
    auto look = [&](int j) {
        if (cell_dist(rec, j, a) > lim) return;
        if (n < kCellInline) in_doubt |= (uint64_t)j << (10 * n);
        ++n;
    };
    if (kind == kCellScan) {
        const int N8 = G.N & ~7;
        for (int j = 0; j < N8; j += 8)
            if (!(cell_min8<DM>(rec + j * DM, a) > lim))
                for (int q = 0; q < 8; ++q) look(j + q);
        for (int j = N8; j < G.N; ++j) look(j);
    } else {
        for (int q = 0; q < cnt; ++q) look(at(q));
    }
    double best = __longlong_as_double(0x7FF0000000000000LL);
    int bi = 0x7FFFFFFF;
    const bool all = n > kCellInline;
    for (int q = 0; q < (all ? cnt : n); ++q) {
        const int j = all ? at(q) : (int)((in_doubt >> (10 * q)) & 1023u);
        if (all && cell_dist(rec, j, a) > lim) continue;
        const double dj = dist64<DM>(z, g64 + (long long)j * DM, DM);
        if (dj < best) {
            best = dj;
            bi = j;
        }
    }
    return bi;
}

// Bulk copies of a grid's table and records into `dst` (one thread); returns the bytes.
template <int DM>
__device__ __forceinline__ uint32_t cell_stage_bytes(const CellGrid& G)
{
    return G.N > 1 ? (uint32_t)G.nb0 * G.nb1 * 8u + (uint32_t)((G.N * DM + 3) / 4 * 4) * 4u : 0u;
}
template <int DM>
__device__ __forceinline__ void cell_stage(const ForwardParams& p, const CellGrid& G, uint32_t dst, uint32_t bar)
{
    if (G.N <= 1) return;
    const uint32_t tb = (uint32_t)G.nb0 * G.nb1 * 8u;
    bulk_g2s(dst, p.cell_tab + G.toff, tb, bar);
    bulk_g2s(dst + tb, p.cell_rec + G.roff, (uint32_t)((G.N * DM + 3) / 4 * 4) * 4u, bar);
}

// ------------------------------------------------------------------ FP32 stand-in of the FP64 pair draw
//
// FP64 samples cost the FP64 pipe about 250 operations a pair, at 1/64 of the
// FP32 rate: 3.0 ms for the 10^7 pairs of the 1-d workload.  The cells of nearly
// all of them need far fewer digits: the pair is drawn from the same Philox words
// with FP32 logarithm, square root, sine and cosine, mapped by matrices already
// combined and centred in FP64 on the host, and the certificate carries the error
// (qt_near.h); the uncertified few are drawn again in FP64.
//
// Each normal lies within 2^-20 of its radius, radius <= 8.6.  The logarithm: s has the
// roundings of f - 1, f + 1 and the division (2 ulp), 1.5 2^-22 in all, so ln f is within
// 1.75 2^-22 of itself, |ln f| < 0.35; where u <= 0.7071 (-ln u > 0.346) u's rounding and
// e ln 2 add 2.1 2^-24: 3.2 2^-22 of -ln u at its smallest, half of that after the square
// root, 0.47 2^-20 with its rounding.  The angle, truncated and rounded to FP32, is within
// 1.6 2^-24 and the polynomials within 1.5 2^-24: 0.19 2^-20.  0.72 2^-20 with the last
// product; 2^24 pairs and the extreme words stay below 2^-20 (tests/cuda/near_normals.cu).

__device__ __forceinline__ float box_muller_near(const Philox4& w, float& g0, float& g1)
{
    const unsigned long long n0 = 2ull * (((unsigned long long)(w.v[0] >> 6) << 26) | (w.v[1] >> 6)) + 1ull;
    const float u = __ull2float_rn(n0) * 0x1p-53f;
    // ln u = e ln 2 + 2 atanh((f - 1)/(f + 1)); near 1 the difference 1 - u is
    // taken from the integer, so that nothing cancels
    float fm1, el2;
    if (u > 0.70710678f) {
        fm1 = -(__ull2float_rn((1ull << 53) - n0) * 0x1p-53f);
        el2 = 0.0f;
    } else {
        const uint32_t bits = __float_as_uint(u);
        int e = (int)(bits >> 23) - 127;
        float f = __uint_as_float((bits & 0x007FFFFFu) | 0x3F800000u);
        if (f > 1.41421354f) {
            f *= 0.5f;
            e += 1;
        }
        fm1 = f - 1.0f;
        el2 = (float)e * 0.693147182f;
    }
    const float s = __fdividef(fm1, fm1 + 2.0f);
    const float z = s * s;
    float q = __fmaf_rn(z, 1.0f / 11.0f, 1.0f / 9.0f);
    q = __fmaf_rn(q, z, 1.0f / 7.0f);
    q = __fmaf_rn(q, z, 1.0f / 5.0f);
    q = __fmaf_rn(q, z, 1.0f / 3.0f);
    const float lnf = 2.0f * __fmaf_rn(s * z, q, s);
    const float rad = __fsqrt_rn(-2.0f * (el2 + lnf));
    // angle 2 pi u1: the quarter is the top two bits, x the next 32 of u1's 52 bits
    const uint32_t quarter = w.v[2] >> 30;
    const uint32_t x = ((w.v[2] << 2) & 0xFFFFFF00u) | (w.v[3] >> 24);
    const float f = (float)x * 0x1p-32f;
    const bool fold = f > 0.5f;
    const float th = (fold ? 1.0f - f : f) * 1.57079633f;
    const float t2 = th * th;
    float ps = __fmaf_rn(t2, 1.0f / 362880.0f, -1.0f / 5040.0f);
    ps = __fmaf_rn(ps, t2, 1.0f / 120.0f);
    ps = __fmaf_rn(ps, t2, -1.0f / 6.0f);
    const float st = __fmaf_rn(th * t2, ps, th);
    float pc = __fmaf_rn(t2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
    pc = __fmaf_rn(pc, t2, -1.0f / 720.0f);
    pc = __fmaf_rn(pc, t2, 1.0f / 24.0f);
    pc = __fmaf_rn(pc, t2, -0.5f);
    const float ct = __fmaf_rn(t2, pc, 1.0f);
    const float s0 = fold ? ct : st, c0 = fold ? st : ct;
    const float sa = (quarter & 1u) ? c0 : s0, ca = (quarter & 1u) ? s0 : c0;
    const float sn = (quarter & 2u) ? -sa : sa;
    const float cs = (quarter == 1u || quarter == 2u) ? -ca : ca;
    g0 = rad * cs;
    g1 = rad * sn;
    return rad;
}

// Centred pair (X - mu_A, Y - mu_B) of an FP64 layer within its dA, dB: block P =
// [cA (DM), L (DM^2), cB (DM), A L (DM^2), T (DM^2)].  Returns the largest radius as
// a share of the 8.6 that dA and dB allow for.
template <int DM>
__device__ __forceinline__ float pair_near(const float* __restrict__ P, uint64_t seed, int k, uint64_t m,
                                          float (&a)[DM], float (&b)[DM])
{
    float g[2 * DM], rad = 0.0f;
#pragma unroll
    for (int r = 0; r < DM; ++r) {
        const Philox4 w = philox4x32_10((uint32_t)m, (uint32_t)(m >> 32), (uint32_t)k, (uint32_t)r, (uint32_t)seed,
                                        (uint32_t)(seed >> 32));
        rad = fmaxf(rad, box_muller_near(w, g[2 * r], g[2 * r + 1]));
    }
    const float* pL = P + DM;
    const float* pc = pL + DM * DM;
    const float* pAL = pc + DM;
    const float* pT = pAL + DM * DM;
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        a[l] = P[l];
        b[l] = pc[l];
#pragma unroll
        for (int q = 0; q < DM; ++q) {
            a[l] = __fmaf_rn(pL[l * DM + q], g[q], a[l]);
            b[l] = __fmaf_rn(pAL[l * DM + q], g[q], b[l]);
            b[l] = __fmaf_rn(pT[l * DM + q], g[DM + q], b[l]);
        }
    }
    return rad * (1.0001f / 8.6f);
}

}  // namespace qt
