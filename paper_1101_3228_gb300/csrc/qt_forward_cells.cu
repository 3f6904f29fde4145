// qt_forward_cells.cu -- located search (qt_cells.cuh) for d <= 2: the tables of
// every grid, and Algorithm III (Pages & Wilbertz, arXiv:1101.3228, Sec. 4) or
// the counting of given samples on them.
#include "qt_cells.cuh"
#include "qt_launch.h"

namespace qt {

namespace {

constexpr int kBuildThreads = 256;
constexpr int kBuildWarps = kBuildThreads / 32;
constexpr int kBuildList = 24;            // kept points of a bin held by its lane
constexpr int kPatchX = 8, kPatchY = 4;   // bins of a patch, one per lane (d = 1: 32 x 1)

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

}  // namespace

// Table of grid p.cell_g0 + blockIdx.x (patches blockIdx.y, blockIdx.y + gridDim.y, ...).
// A warp takes a patch of 32 bins: it finds the points that can be nearest
// somewhere in the patch (about 25 of 500), then every lane tests those against
// its own bin.  Point j is dropped from a box with centre c and half-widths h when,
// against the point i nearest to c (for a bin also against the second nearest),
//   D_j(x) - D_i(x) = |g_j - c|^2 - |g_i - c|^2 - 2 (x - c).(g_j - g_i)
// is positive on the whole box by more than the FP32 rounding of the points and of this
// test, u = 2^-24: a point's coordinates are off by u R (R bounds |g|) and its differences
// t from c by u |t|, so D is off by (DM + 4) u D + 2 u R sum |t| and, with sum |t| <=
// sqrt(DM) (D / s + s) / 2 for any s > 0 (s = the widest half-width here),
//   error <= u (DM + 4 + R sqrt(DM) / s) (D_j + D_i) + u R (2 sqrt(DM) s + 4 sum h)
//            + 8 u slack.
// Twice that is allowed for.  (A bound of 2^-18 S^2 for every bin, S the size of the box,
// kept 16 points in every bin of a 1-d grid of 1000.)
//
// What bounds it: latency with few grids (a warp has one patch: 30 us for two grids of 1000
// points, 9 for five of 64), issue slots with many (366 grids of 500 points: 275 us, 66%).
template <int DM>
__global__ void __launch_bounds__(kBuildThreads) build_cells_kernel(const __grid_constant__ ForwardParams p)
{
    __shared__ float s_g[kCellMaxN * DM];
    __shared__ uint16_t s_surv[kBuildWarps][kCellMaxN];
    __shared__ float s_red[kBuildWarps][2 * DM + 1];
    __shared__ int s_some[kBuildWarps];
    CellGrid& G = p.cells[p.cell_g0 + blockIdx.x];
    const int N = G.N;
    if (N <= 1) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const double* g64 = p.g64 + G.goff * DM;
    // centred points, their extent and norm.  A grid far from the host's centre (given samples
    // come with none, and the path-wise form's model states the first layer's only) is
    // centred on its own middle instead: rounding is relative to the distance from it
    float mn[DM], mx[DM], mu[DM], r2;
    bool flat[DM];
    const long long* g0bits = reinterpret_cast<const long long*>(g64);
#pragma unroll
    for (int l = 0; l < DM; ++l) mu[l] = G.mu0[l];
    for (int pass = 0;; ++pass) {
        r2 = 0.0f;
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            mn[l] = __int_as_float(0x7F800000);
            mx[l] = -__int_as_float(0x7F800000);
            flat[l] = DM == 2;
        }
#pragma unroll 4
        for (int j = tid; j < N; j += kBuildThreads) {
            float n2 = 0.0f;
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                const long long bits = g0bits[(long long)j * DM + l];
                const float v = __double2float_rn(__dsub_rn(__longlong_as_double(bits), (double)mu[l]));
                flat[l] = flat[l] && bits == g0bits[l];
                s_g[j * DM + l] = v;
                mn[l] = fminf(mn[l], v);
                mx[l] = fmaxf(mx[l], v);
                n2 = __fmaf_rn(v, v, n2);
                if (blockIdx.y == 0) p.cell_rec[G.roff + (long long)j * DM + l] = v;
            }
            r2 = fmaxf(r2, n2);
        }
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            mn[l] = warp_min(mn[l]);
            mx[l] = warp_max(mx[l]);
            if (lane == 0) {
                s_red[warp][2 * l] = mn[l];
                s_red[warp][2 * l + 1] = mx[l];
            }
        }
        r2 = warp_max(r2);
        if (lane == 0) s_red[warp][2 * DM] = r2;
        int some = 0;                                  // bit l: axis l is not flat
#pragma unroll
        for (int l = 0; l < DM; ++l) some |= flat[l] ? 0 : 1 << l;
        some = (int)__reduce_or_sync(0xFFFFFFFFu, (unsigned)some);
        if (lane == 0) s_some[warp] = some;
        __syncthreads();
        for (int w = 0; w < kBuildWarps; ++w) {
            some |= s_some[w];
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                mn[l] = fminf(mn[l], s_red[w][2 * l]);
                mx[l] = fmaxf(mx[l], s_red[w][2 * l + 1]);
            }
            r2 = fmaxf(r2, s_red[w][2 * DM]);
        }
#pragma unroll
        for (int l = 0; l < DM; ++l) flat[l] = (some & (1 << l)) == 0;
        if (pass > 0 || !p.cell_recentre) break;
        bool off = false;
        float mid[DM];
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            mid[l] = (float)((double)mu[l] + 0.5 * ((double)mn[l] + (double)mx[l]));
            off = off || fabsf(mn[l] + mx[l]) > 4.0f * (mx[l] - mn[l]);
        }
        // (sizes that are not finite stay with the host's centre; the same in every CTA)
        if (!off || !(fabsf(mid[0]) < 1e30f) || !(fabsf(mid[DM - 1]) < 1e30f)) break;
#pragma unroll
        for (int l = 0; l < DM; ++l) mu[l] = mid[l];
        __syncthreads();
    }
    // the box: the grid's own, a quarter of its width wider on every side (quantizers
    // reach about 3 standard deviations, so the box reaches 4.5); bin b of an axis is
    // centred on (b - K) h, K an integer.  The enlarged bins must cover the error of the
    // centred sample and of its bin number, so an axis along which the grid is narrow (a
    // product grid with one point, two factors of very different size) or a grid far from
    // its centre takes wider bins than its share of the box
    const float R = __fsqrt_rn(r2) * 1.0001f;
    int nb[2] = {G.nb, DM == 2 ? G.nb : 1};
    float K[DM], h[DM], ext[DM], S = 0.0f;
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        ext[l] = fmaxf(mx[l] - mn[l], 1e-30f);
        const float far_ = fmaxf(fabsf(mn[l]), fabsf(mx[l])) + ext[l];
        S = __fmaf_rn(far_, far_, S);
    }
    if constexpr (DM == 2) {
        // about as wide as high, where the extents differ by more than two: Voronoi cells are
        // (ten times as long as high, 1000 points: 6 candidates a bin against 3)
        const float room = (float)(nb[0] * nb[0]), r = ext[0] / ext[DM - 1];
        float n0 = r > 2.0f || r < 0.5f ? (float)nb[0] * __fsqrt_rn(r) : (float)nb[0];
        if (flat[0] != flat[DM - 1]) n0 = flat[0] ? 8.0f : 0.25f * room;
        nb[0] = (int)(fminf(fmaxf(n0, 8.0f), 0.125f * room) * 0.125f) * 8;
        nb[1] = (int)(room / (float)nb[0] * 0.25f) * 4;
    }
    // (the wider bins make S larger by less than a quarter: 32 2^-21 8192 = 1/8 for d = 1)
    const float need = 32.0f * 1.3f * (G.err + G.err0 + 0x1p-21f * (__fsqrt_rn(S) + R));
    S = 0.0f;
    float hgeo = 1.0f;
#pragma unroll
    for (int l = 0; l < DM; ++l) h[l] = fmaxf(1.5f * ext[l] / (float)nb[l], need);
    // an axis along which all points are equal adds the same number y^2 to every distance: one
    // bin of it serves, `wide` across, and the margins allow for the FP64 rounding of sums
    // with y^2 (|y| < 0.75 wide: 2^-50 wide^2)
    float ties = 0x1p-120f;
    if constexpr (DM == 2) {
        const float wide[2] = {16384.0f * h[1], 16384.0f * h[0]};
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            flat[l] = flat[l] && !flat[1 - l] && 4.0f * fabsf(mn[l]) <= wide[l];
            if (flat[l]) {
                h[l] = wide[l];
                ties = __fmaf_rn(0x1p-50f * h[l], h[l], ties);
            }
        }
    }
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        // two bins beyond the points at least, for d = 1, where the last ones go on.  A
        // grid without finite sizes has no bins here: `usable` is false for it
        K[l] = fminf(fmaxf(rintf((fmaxf(0.25f * ext[l], 2.0f * h[l]) - mn[l]) / h[l]), -4194304.0f), 4194304.0f);
        float far_ = fmaxf(fabsf(K[l]) + 1.0f, fabsf((float)nb[l] - K[l]) + 1.0f) * h[l];
        if (flat[l]) {
            K[l] = (float)(nb[l] / 2);
            far_ = fabsf(mn[l]);
        } else {
            hgeo *= h[l];
        }
        S = __fmaf_rn(far_, far_, S);
    }
    if (DM == 2 && !flat[0] && !flat[DM - 1]) hgeo = __fsqrt_rn(hgeo);
    S = (__fsqrt_rn(S) + R) * 1.0001f;
    const float ebox = 0x1p-24f * 1.01f * S, er = ebox + G.err0, e = er + G.err;
    bool usable = S < 1e18f;                           // its square is far from overflow
#pragma unroll
    for (int l = 0; l < DM; ++l) usable = usable && (flat[l] || 32.0f * (G.err + G.err0 + 0x1p-21f * S) <= h[l]);
    // the test's error, as above: rel (D_j + D_i) + fix + 16 u slack; a point is dropped when
    // D_j (1 - rel) - slack (2 + 16 u) > D_i (1 + rel) + fix.  (The floors here and in c2:
    // products of the smallest grids fall out of FP32's range)
    constexpr float u2 = 0x1p-23f, sqd = DM == 1 ? 1.0f : 1.41421357f;
    float rel, fix, wh[DM];                            // wh: half-widths times 2 + 16 u, for 2 slack + 16 u slack
    // edge[l]: the box (of a patch or a bin) is the first (bit 0) or last (bit 1) of axis l and
    // goes on for kCellBeyond bins there (d = 2): outwards `far_wh` takes the place of wh
    float far_wh[DM];
    int edge[DM];
    auto margins = [&](const float (&hw)[DM]) {
        float s = hw[0], sum = hw[0];
        if constexpr (DM == 2) {
            s = fmaxf(s, hw[1]);
            sum += hw[1];
        }
#pragma unroll
        for (int l = 0; l < DM; ++l)
            if (edge[l] != 0) sum += (float)(kCellBeyond + 1) * h[l];
        rel = u2 * ((float)(DM + 4) + R * sqd / s);
        fix = u2 * R * (2.0f * sqd * s + 4.0f * sum) + ties;
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            wh[l] = hw[l] * (2.0f + 0x1p-20f);
            far_wh[l] = (float)(kCellBeyond + 1) * h[l] * (2.0f + 0x1p-20f);
        }
    };
    if (blockIdx.y == 0 && tid == 0) {
        const float sq = DM == 1 ? 1.0f : 1.41421357f;
        const float kappa = fmaxf(0x1p-22f, e / (2.0f * hgeo));
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            G.mu[l] = mu[l];
            G.inv_h[l] = 1.0f / h[l];
            G.org[l] = 8388608.0f + K[l];
        }
        G.c1 = 2.02f * sq * kappa;
        G.c2 = 2.02f * (sq * (e / kappa) * e + (float)DM * e * e) + 0x1p-120f * (e / er);
        G.c3 = 2.02f * (float)(DM + (DM == 1 ? 12 : 15)) * 0x1p-24f;   // 12 sqrt(d) u D: 2.02 x 6 and 9 of them
        G.e = e;
        G.ebox = ebox;
        G.nb0 = nb[0];
        G.nb1 = nb[1];
        G.f0 = er / e;
    }
    // 2 slack + 16 u slack of axis l for two points whose coordinates differ by dl, on a box with
    // or without an edge
    auto slack_in = [&](float dl, int l, float acc) { return __fmaf_rn(fabsf(dl), wh[l], acc); };
    auto slack_edge = [&](float dl, int l, float acc) {
        const bool out = (edge[l] & (dl > 0.0f ? 2 : 1)) != 0;
        return __fmaf_rn(fabsf(dl), out ? far_wh[l] : wh[l], acc);
    };
    // a flat axis' bin lies at the points' own coordinate and has no width
    auto on_axis = [&](float (&c)[DM], float (&hw)[DM]) {
#pragma unroll
        for (int l = 0; l < DM; ++l)
            if (DM == 2 && flat[l]) {
                c[l] = mn[l];
                hw[l] = 0.0f;
            }
    };
    const int pnx = DM == 1 ? nb[0] / 32 : nb[0] / kPatchX, pny = DM == 1 ? 1 : nb[1] / kPatchY;
    unsigned long long* tab = p.cell_tab + G.toff;
    uint16_t* surv = s_surv[warp];
    for (int pt = blockIdx.y * kBuildWarps + warp; pt < pnx * pny; pt += gridDim.y * kBuildWarps) {
        const int px = pt % pnx, py = pt / pnx;
        // this lane's bin
        const int x = DM == 1 ? px * 32 + lane : px * kPatchX + (lane & 7), y = DM == 1 ? 0 : py * kPatchY + (lane >> 3);
        unsigned long long* out = tab + (long long)y * nb[0] + x;
        if (!usable) {
            *out = kCellScanEntry;
            continue;
        }
        // ---- points that can win somewhere in the patch
        float c[DM], hw[DM];
        c[0] = ((DM == 1 ? (float)(px * 32) + 15.5f : (float)(px * kPatchX) + 3.5f) - K[0]) * h[0];
        hw[0] = h[0] * (DM == 1 ? 16.1f : 4.1f);
        if constexpr (DM == 2) {
            c[1] = ((float)(py * kPatchY) + 1.5f - K[1]) * h[1];
            hw[1] = h[1] * 2.1f;
        }
        on_axis(c, hw);
        edge[0] = DM == 1 ? 0 : (px == 0 ? 1 : 0) | (px == pnx - 1 ? 2 : 0);
        if constexpr (DM == 2) edge[1] = (py == 0 ? 1 : 0) | (py == pny - 1 ? 2 : 0);
        bool at_edge = false;
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            if (flat[l]) edge[l] = 0;
            at_edge = at_edge || edge[l] != 0;
        }
        const int patch_edge[2] = {edge[0], DM == 2 ? edge[DM - 1] : 0};
        margins(hw);
        float bD = __int_as_float(0x7F800000);
        int bi = 0x7FFFFFFF;
        // (unrolled here and below: with few grids a warp has one patch and its SM hardly a
        // second warp, so that one point at a time costs its latency)
#pragma unroll 4
        for (int j = lane; j < N; j += 32) {
            float D = 0.0f;
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                const float t = s_g[j * DM + l] - c[l];
                D = __fmaf_rn(t, t, D);
            }
            if (D < bD) {
                bD = D;
                bi = j;
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            const float od = __shfl_xor_sync(0xFFFFFFFFu, bD, o);
            const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
            if (od < bD || (od == bD && oi < bi)) {
                bD = od;
                bi = oi;
            }
        }
        if (bi >= N) bi = 0;                        // non-finite points: nothing is dropped below
        float gb[DM];
#pragma unroll
        for (int l = 0; l < DM; ++l) gb[l] = s_g[bi * DM + l];
        const float keepD = 1.0f - rel, over = __fmaf_rn(1.0f + rel, bD, fix);
        int ns = 0;
        auto survivors = [&](auto slack_of) {
#pragma unroll 4
            for (int j0 = 0; j0 < N; j0 += 32) {
                const int j = j0 + lane;
                bool keep = false;
                if (j < N) {
                    float D = 0.0f, slack = 0.0f;
#pragma unroll
                    for (int l = 0; l < DM; ++l) {
                        const float gj = s_g[j * DM + l], t = gj - c[l];
                        D = __fmaf_rn(t, t, D);
                        slack = slack_of(gj - gb[l], l, slack);
                    }
                    keep = !(__fmaf_rn(D, keepD, -slack) > over);
                }
                const unsigned m = __ballot_sync(0xFFFFFFFFu, keep);
                if (keep) surv[ns + __popc(m & ((1u << lane) - 1u))] = (uint16_t)j;
                ns += __popc(m);
            }
        };
        if (at_edge) survivors(slack_edge);
        else survivors(slack_in);
        __syncwarp();
        // ---- this lane's bin
        c[0] = ((float)x - K[0]) * h[0];
        hw[0] = 0.5f * 1.125f * h[0];
        if constexpr (DM == 2) {
            c[1] = ((float)y - K[1]) * h[1];
            hw[1] = 0.5f * 1.125f * h[1];
        }
        on_axis(c, hw);
        edge[0] = patch_edge[0] & ((x == 0 ? 1 : 0) | (x == nb[0] - 1 ? 2 : 0));
        if constexpr (DM == 2) edge[1] = patch_edge[1] & ((y == 0 ? 1 : 0) | (y == nb[1] - 1 ? 2 : 0));
        margins(hw);
        float D0 = __int_as_float(0x7F800000), D1 = D0;
        int i0 = surv[0], i1 = surv[0];
#pragma unroll 4
        for (int t = 0; t < ns; ++t) {
            const int j = surv[t];
            float D = 0.0f;
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                const float v = s_g[j * DM + l] - c[l];
                D = __fmaf_rn(v, v, D);
            }
            const bool first = D < D0, next = D < D1;
            i1 = first ? i0 : (next ? j : i1);
            D1 = first ? D0 : (next ? D : D1);
            i0 = first ? j : i0;
            D0 = first ? D : D0;
        }
        float g0[DM], g1[DM];
#pragma unroll
        for (int l = 0; l < DM; ++l) {
            g0[l] = s_g[i0 * DM + l];
            g1[l] = s_g[i1 * DM + l];
        }
        const float rest = 1.0f - rel, o0 = __fmaf_rn(1.0f + rel, D0, fix), o1 = __fmaf_rn(1.0f + rel, D1, fix);
        auto keeps = [&](int j, auto slack_of) {
            float D = 0.0f, sl0 = 0.0f, sl1 = 0.0f;
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                const float gj = s_g[j * DM + l], v = gj - c[l];
                D = __fmaf_rn(v, v, D);
                sl0 = slack_of(gj - g0[l], l, sl0);
                sl1 = slack_of(gj - g1[l], l, sl1);
            }
            return !(__fmaf_rn(D, rest, -sl0) > o0) && !(__fmaf_rn(D, rest, -sl1) > o1);
        };
        // kept points, in order, 32 survivors at a time; a lane keeps one or two
        uint16_t list[kBuildList];
        int cnt = 0;
        auto collect = [&](auto slack_of) {
            for (int t0 = 0; t0 < ns; t0 += 32) {
                const int nt = min(32, ns - t0);
                uint32_t kept = 0;
#pragma unroll 8
                for (int t = 0; t < nt; ++t) kept |= keeps(surv[t0 + t], slack_of) ? 1u << t : 0u;
                for (; kept; kept &= kept - 1) {
                    if (cnt < kBuildList) list[cnt] = surv[t0 + __ffs((int)kept) - 1];
                    ++cnt;
                }
            }
        };
        if (at_edge) collect(slack_edge);
        else collect(slack_in);
        uint64_t ent = 0;
        for (int t = 0; t < min(cnt, kCellInline); ++t) ent |= (uint64_t)list[t] << (10 * t);
        const bool beside = DM == 2 && ((flat[0] && x != nb[0] / 2) || (flat[DM - 1] && y != nb[1] / 2));
        if (beside) {
            ent = kCellScanEntry;          // a flat axis has one bin
        } else if (cnt <= kCellInline) {
            ent |= (uint64_t)cnt << 60;
        } else if (4 * cnt > N) {
            ent = kCellScanEntry;          // a scan of the whole grid is as fast (12 against 4.6 instructions a point)
        } else {
            const unsigned long long off = atomicAdd(p.cell_cursor, (unsigned long long)cnt);
            if (pool_holds(off, (uint32_t)cnt, p.cell_pool_cap)) {
                if (cnt <= kBuildList) {
                    for (int t = 0; t < cnt; ++t) p.cell_pool[off + t] = list[t];
                } else {
                    int w = 0;
                    for (int t = 0; t < ns; ++t)
                        if (keeps(surv[t], slack_edge)) p.cell_pool[off + w++] = surv[t];
                }
                ent = off | ((uint64_t)cnt << 32) | ((uint64_t)kCellPool << 60);
            } else {
                ent = kCellScanEntry;
            }
        }
        *out = ent;
        __syncwarp();
    }
}

// Exact FP64 cell of sample m (X or Y) among the candidates of its bin, from the sample drawn
// again in its own precision: what the search knew of it would be registers that the whole
// loop carries (10^7 FP64 pairs, d = 1: 148 against 142 us).  The smallest distance that a
// search of the whole grid leaves in its entry holds for it but for FP64 pairs.
template <int DM, int MODE>
static __device__ __noinline__ int cell_recheck(const ForwardParams& p, const float* spf, const double* spd, int k,
                                                unsigned long long m, bool wantY, uint64_t e, const CellGrid& G,
                                                const unsigned char* sm)
{
    double z[DM];
    exact_sample<DM>(p, spf, spd, k, m, wantY, z);
    atomicAdd(&p.status->rechecks, 1ull);
    float a[DM];
#pragma unroll
    for (int l = 0; l < DM; ++l) a[l] = __double2float_rn(__dsub_rn(z[l], (double)G.mu[l]));
    return cell_exact<DM, MODE != 1>(G, cell_records(G, sm), a, z, e, p.cell_pool, p.g64 + G.goff * DM);
}

// The forward step.  MODE 0: FP32 samples, 1: FP64 samples (drawn in FP32 first,
// qt_cells.cuh), 2: given samples.  A work item is (layer, blockDim.x samples), one
// sample per thread; a CTA takes a contiguous run of items, so that it loads the
// two tables of a layer (170 KB at most) once or twice per launch instead of once
// per item and layer.  What bounds it: issue slots (83% busy, 580 instructions a
// pair at d = 2, most of them the draw).  2-factor workload, 10^9 pairs: 17.7 ms,
// against 142.9 ms for brute force over 1000 candidates a pair.
template <int DM, int MODE>
__global__ void __launch_bounds__(kCellThreads, 1) forward_cells_kernel(const __grid_constant__ ForwardParams p)
{
    extern __shared__ __align__(128) unsigned char dsm_c[];
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ LayerDesc s_L;
    __shared__ CellGrid s_GA, s_GB;
    __shared__ __align__(16) float s_pf[param_count(DM)];
    __shared__ __align__(16) double s_pd[param_count(DM)];
    __shared__ float s_near[kCellNearStride];
    __shared__ int s_abort;
    const int tid = threadIdx.x;
    const uint32_t bar = smem_u32(&s_bar);
    uint32_t* hist = reinterpret_cast<uint32_t*>(dsm_c + p.smem_grid_bytes);
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_proxy_async();
        s_abort = 0;
    }
    __syncthreads();
    const long long lo = p.total_items * blockIdx.x / gridDim.x, hi = p.total_items * (blockIdx.x + 1) / gridDim.x;
    uint32_t phase = 0;
    int k = -1;
    long long ibeg = 0, iend = 0;
    bool hist_live = false;
    const unsigned char* smB = dsm_c;
    auto flush = [&]() {
        const int ent = s_L.NA * s_L.NB;
        for (int e = tid; e < ent; e += (int)blockDim.x) {
            const uint32_t v = hist[e];
            if (v) count_add(p.counts, p.counts_u32, s_L.coff + e, v);
        }
    };
    for (long long item = lo; item < hi; ++item) {
        if (k < 0 || item >= iend) {
            __syncthreads();
            if (hist_live) flush();
            // the layer, then its descriptors, word by word (one round trip to L2)
            if (p.cell_ipl > 0) k = (int)(item / p.cell_ipl);
            else k = p.cell_g0;
            __syncthreads();
            for (int e = tid; e < (int)(sizeof(LayerDesc) / 4); e += (int)blockDim.x)
                reinterpret_cast<int*>(&s_L)[e] = reinterpret_cast<const int*>(p.layers + k)[e];
            for (int e = tid; e < (int)(sizeof(CellGrid) / 4); e += (int)blockDim.x) {
                reinterpret_cast<int*>(&s_GA)[e] = reinterpret_cast<const int*>(p.cells + k)[e];
                reinterpret_cast<int*>(&s_GB)[e] = reinterpret_cast<const int*>(p.cells + k + 1)[e];
            }
            if (p.source == kSampler) {
                for (int e = tid; e < param_count(DM); e += (int)blockDim.x) {
                    s_pf[e] = p.params_f[(long long)k * p.params_stride + e];
                    s_pd[e] = p.params_d[(long long)k * p.params_stride + e];
                }
                if (MODE == 1 && tid < kCellNearStride) s_near[tid] = p.cell_near[k * kCellNearStride + tid];
            }
            __syncthreads();
            if (tid == 0) {
                const uint32_t ba = cell_stage_bytes<DM>(s_GA), bb = cell_stage_bytes<DM>(s_GB);
                fence_proxy_async();
                mbar_arrive_expect_tx(bar, ba + bb);
                cell_stage<DM>(p, s_GA, smem_u32(dsm_c), bar);
                cell_stage<DM>(p, s_GB, smem_u32(dsm_c) + ba, bar);
            }
            ibeg = s_L.item_begin;
            iend = ibeg + s_L.items;
            hist_live = s_L.hist_smem != 0;
            if (hist_live)
                for (int e = tid; e < s_L.NA * s_L.NB; e += (int)blockDim.x) hist[e] = 0;
            if (!mbar_wait_bounded(bar, phase, p.spin_budget)) {
                record_error(p.status, 4 /* QT_ETIMEOUT */, 50);
                s_abort = 1;
                mbar_wait_bounded(bar, phase, kDrainUs);
            }
            phase ^= 1u;
            __syncthreads();
            if (s_abort) return;
            smB = dsm_c + cell_stage_bytes<DM>(s_GA);
        }
        const unsigned long long m = (unsigned long long)(item - ibeg) * blockDim.x + (unsigned long long)tid;
        if (m >= p.M) continue;
        // ---- the centred pair
        float a[DM], b[DM], f = 1.0f;
        if constexpr (MODE == 0) {
            float X[DM], Y[DM];
            pair_f32<DM>(s_pf, DM, p.seed, k, m, X, Y);
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                a[l] = __fsub_rn(X[l], s_GA.mu[l]);
                b[l] = __fsub_rn(Y[l], s_GB.mu[l]);
            }
        } else if constexpr (MODE == 1) {
            f = pair_near<DM>(s_near, p.seed, k, m, a, b);
        } else {
#pragma unroll
            for (int l = 0; l < DM; ++l) {
                a[l] = __double2float_rn(__dsub_rn(p.srcX[m * DM + l], (double)s_GA.mu[l]));
                b[l] = __double2float_rn(__dsub_rn(p.srcY[m * DM + l], (double)s_GB.mu[l]));
            }
        }
        // ---- both cells
        int i = 0, j = 0;
        uint64_t eA, eB;
        bool needA = false, needB = false;
        auto share = [&](const CellGrid& G) { return MODE == 1 ? __fmaf_rn(f, 1.0f - G.f0, G.f0) : 1.0f; };
        if (s_L.NA > 1) i = cell_search<DM>(s_GA, dsm_c, p.cell_pool, a, share(s_GA), eA, needA);
        if (s_L.NB > 1) j = cell_search<DM>(s_GB, smB, p.cell_pool, b, share(s_GB), eB, needB);
        if (needA) i = cell_recheck<DM, MODE>(p, s_pf, s_pd, k, m, false, eA, s_GA, dsm_c);
        if (needB) j = cell_recheck<DM, MODE>(p, s_pf, s_pd, k, m, true, eB, s_GB, smB);
        // ---- counters p^k_ij (Sec. 3.3), per-sample cells, dumps
        if ((unsigned)i >= (unsigned)s_L.NA || (unsigned)j >= (unsigned)s_L.NB) {
            record_error(p.status, 6 /* QT_EDEVICE */, 52);
            continue;
        }
        if (hist_live) atomicAdd(&hist[i * s_L.NB + j], 1u);
        else count_add(p.counts, p.counts_u32, s_L.coff + (long long)i * s_L.NB + j, 1u);
        if (MODE == 2 && p.cellsA) {
            p.cellsA[m] = i;
            p.cellsB[m] = j;
        }
        if (p.dump_count > 0 && (m % (unsigned long long)p.dump_stride) == 0ull) {
            const unsigned long long t = m / (unsigned long long)p.dump_stride;
            if (t < (unsigned long long)p.dump_count) {
                const long long row = (long long)k * p.dump_count + (long long)t;
                double z[DM];
                exact_sample<DM>(p, s_pf, s_pd, k, m, false, z);
                for (int l = 0; l < DM; ++l) p.dumpX[row * DM + l] = z[l];
                exact_sample<DM>(p, s_pf, s_pd, k, m, true, z);
                for (int l = 0; l < DM; ++l) p.dumpY[row * DM + l] = z[l];
                p.dumpI[row] = i;
                p.dumpJ[row] = j;
            }
        }
    }
    __syncthreads();
    if (hist_live) flush();
}

cudaError_t launch_build_cells(int dm, const ForwardParams& p, int num_sms, cudaStream_t st)
{
    const int ng = p.cell_g1 - p.cell_g0;
    // one patch per warp where there are few grids, about eight CTAs of eight warps
    // per SM where there are many
    const int most = dm == 1 ? 8192 / 32 / kBuildWarps : 104 * 104 / 32 / kBuildWarps + 1;
    const int slices = (8 * num_sms + ng - 1) / ng;
    dim3 grid((unsigned)ng, (unsigned)(slices < 1 ? 1 : (slices > most ? most : slices)));
    if (dm == 1) build_cells_kernel<1><<<grid, kBuildThreads, 0, st>>>(p);
    else build_cells_kernel<2><<<grid, kBuildThreads, 0, st>>>(p);
    return cudaGetLastError();
}

template <int DM, int MODE>
static cudaError_t launch_fc(const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    auto kern = forward_cells_kernel<DM, MODE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    if (e != cudaSuccess) return e;
    *bps = 1;
    long long grid = num_sms;
    if (grid > p.total_items) grid = p.total_items;
    if (grid < 1) grid = 1;
    kern<<<(unsigned)grid, (unsigned)p.tile, dyn, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_forward_cells(int dm, const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    const int mode = p.source == kArrays ? 2 : (p.prec == 1 ? 0 : 1);
#define QT_CASE(D, M) \
    if (dm == D && mode == M) return launch_fc<D, M>(p, dyn, num_sms, bps, st);
    QT_CASE(1, 0) QT_CASE(1, 1) QT_CASE(1, 2) QT_CASE(2, 0) QT_CASE(2, 1) QT_CASE(2, 2)
#undef QT_CASE
    return cudaErrorInvalidValue;
}

}  // namespace qt
