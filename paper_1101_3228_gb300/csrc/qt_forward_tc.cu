// qt_forward_tc.cu -- the tensor-core form (qt_forward_tc.cuh): the preparation of
// the FP16 operand tiles, the draw, and the dispatch of the kernels.
#include "qt_forward_tc.cuh"

namespace qt {

// FP16 operand tiles of every grid: row j of grid g (tile j/128) holds
// [g_hi (dm), g_lo (dm), g_hi (dm), cc_hi, cc_lo, 0 ...] of sigma g^ and
// sigma^2 cc (coordinates l >= d zero); padded rows carry cc_hi = 60000, more than any score of a
// sample in the FP16 range (|s| <= 1 + 16384 sqrt(10)) and finite, as the screen's
// keys need.
// Layout inside a tile: core matrices of 8 rows x 8 halves, (row block,
// K block) at ((n/8)(K/8) + k/8) * 64.
__global__ void prep_tc_tiles_kernel(const float* __restrict__ rec32, GridInfo* gi, int ngrids, int d, int dm,
                                     int rec_floats, int K, long long total_rows, __half* tiles, float* rows)
{
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= total_rows) return;
    int lo = 0, hi = ngrids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (gi[mid].tc_toff * kTcTileN <= r) lo = mid; else hi = mid - 1;
    }
    const GridInfo& G = gi[lo];
    const long long j = r - G.tc_toff * kTcTileN;
    // sigma = 2^e with sigma R <= 1
    int e = 0;
    if (G.R > 0.0f) {
        int ex;
        frexpf(G.R, &ex);   // R = f 2^ex, f in [0.5, 1)
        e = -ex;
    }
    if (j == 0) gi[lo].tc_exp = e;
    const float sg = ldexpf(1.0f, e);
    const long long tile = G.tc_toff + j / kTcTileN;
    const int n = (int)(j % kTcTileN);
    __half* t = tiles + tile * (long long)kTcTileN * K;
    auto put = [&](int k, __half v) { t[((n >> 3) * (K >> 3) + (k >> 3)) * 64 + (n & 7) * 8 + (k & 7)] = v; };
    for (int k = 0; k < K; ++k) put(k, __float2half_rn(0.0f));
    // the same point in the chunk-major FP32 records of the re-score: [chunk][dm + 1][16]
    float* row = rows + (r / kChunk) * ((dm + 1) * kChunk) + r % kChunk;
    row[0] = __int_as_float(0x7F800000);
    for (int l = 1; l <= dm; ++l) row[l * kChunk] = 0.0f;
    if (j < G.N) {
        const float* rc = rec32 + (G.roff + j) * rec_floats;
        for (int l = 0; l <= d; ++l) row[l * kChunk] = rc[l];
        for (int l = 0; l < d; ++l) {
            const float v = sg * rc[1 + l];
            const __half h = __float2half_rn(v);
            const __half lo16 = __float2half_rn(v - __half2float(h));
            put(l, h);
            put(dm + l, lo16);
            put(2 * dm + l, h);
        }
        const float c = sg * sg * rc[0];
        const __half ch = __float2half_rn(c);
        put(3 * dm, ch);
        put(3 * dm + 1, __float2half_rn(c - __half2float(ch)));
    } else {
        put(3 * dm, __float2half_rn(60000.0f));
    }
}

// First kernel of a window: one CTA of 128 threads per work item of [item_lo,
// item_hi); thread t draws row t into the item's record.
template <int DM>
__global__ void __launch_bounds__(kTcTileM) tc_draw_kernel(const __grid_constant__ ForwardParams p)
{
    const int t = threadIdx.x;
    const long long item = p.item_lo + blockIdx.x;
    const int k = tc_layer(p, item);
    const LayerDesc& L = p.layers[k];
    const unsigned long long mtile = (unsigned long long)(item - L.item_begin) * kTcTileM;
    const unsigned long long ms = mtile + (unsigned long long)t;
    draw_row<DM>(p, k, L, ms < p.M ? ms : mtile, t,
                 reinterpret_cast<float*>(p.tc_items) + (long long)blockIdx.x * TcItem<DM>::kFloats);
}

template <int DM, int KT>
static cudaError_t launch_window(const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    const long long n = p.item_hi - p.item_lo;
    if (n < 1) return cudaSuccess;
    tc_draw_kernel<DM><<<(unsigned)n, kTcTileM, 0, st>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // an item's grids apart while all of them are resident at once, and with layers of one point
    e = p.tc_one_point || 2 * n <= (long long)kTcCtas * num_sms
            ? launch_tc<DM, KT, true>(p, dyn, num_sms, bps, st)
            : launch_tc<DM, KT, false>(p, dyn, num_sms, bps, st);
    if (e != cudaSuccess) return e;
    auto certify = tc_certify_kernel<DM>;
    const int rec2 = 2 * TcItem<DM>::kFloats * 4 + p.smem_hist_entries * 4;
    e = allow_dynamic_smem(certify, rec2);
    if (e != cudaSuccess) return e;
    const long long ctas = (long long)num_sms * kCertifyCtas;
    certify<<<(unsigned)(n < ctas ? n : ctas), kTcTileM, rec2, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_tc_forward(int dm, const ForwardParams& p, int dyn, int num_sms, int* bps, cudaStream_t st)
{
    if (dm == 2) return launch_window<2, 1>(p, dyn, num_sms, bps, st);
    if (dm == 4) return launch_window<4, 1>(p, dyn, num_sms, bps, st);
    if (dm == 6) return launch_window<6, 2>(p, dyn, num_sms, bps, st);
    if (dm == 8) return launch_window<8, 2>(p, dyn, num_sms, bps, st);
    if (dm == 10) return launch_window<10, 2>(p, dyn, num_sms, bps, st);
    return cudaErrorInvalidValue;
}

}  // namespace qt
