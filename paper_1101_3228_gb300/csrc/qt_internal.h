// qt_internal.h -- structures shared by the host side of libqt and its kernels.
#pragma once
#include <cstdint>

namespace qt {

constexpr int kDMax = 16;          // largest state dimension
constexpr int kChunk = 16;         // candidates per min-tracking chunk of the FP32 screen
constexpr int kSlots = 2;          // ring slots of the streamed-grid mode

enum Form : int32_t {
    kPlainF64 = 1, kF32Recheck = 2, kTcRecheck = 3, kRouterCert = 4, kPathwise = 5,
    kCells = 6,                    // located search (d <= 2), Algorithm III and given samples
    kPathCells = 7                 // located search, Algorithm II
};
enum Source : int32_t { kSampler = 0, kArrays = 1 };

// Per-layer sampler parameters packed by the host: m[d], b[d], L[d*d], A[d*d],
// T[d*d] (read by every form) and alpha[d], beta[d] (the Euler-scheme chain of
// the path-wise form), padded to a multiple of 4 entries.
__host__ __device__ constexpr int param_stride(int d) { return (4 * d + 3 * d * d + 3) / 4 * 4; }

// Device status block, zeroed before every forward call.
struct DevStatus {
    int32_t code;                  // qt_status of the first error seen, 0 = none
    int32_t where;                 // small tag of the failing site (diagnostics)
    unsigned long long queue;      // persistent work-queue counter
    unsigned long long rechecks;   // FP64 re-evaluations
    unsigned long long candidates; // candidate distances (router form)
    unsigned long long done_items; // work items finished
    unsigned long long spare[4];   // [0]: router grid checksum; [1..3]: diagnostics
    unsigned long long cell_cursor;// located search: pool words that the tables asked for
};

// Whether a list of cnt words at offset off, both as taken from the cursor, lies in a
// pool of cap words.  The cursor counts on after the pool is full; 64 bits, because the
// words asked for can pass 2^32 (a bin whose candidates are all of 1024 points, 10816
// bins a grid: about 400 grids), and a cursor that starts again at 0 would hand out words
// that other bins refer to.
__host__ __device__ constexpr bool pool_holds(unsigned long long off, uint32_t cnt, uint32_t cap)
{
    return off + cnt <= cap;
}

// One layer pair (k, k+1) of the forward step.
struct LayerDesc {
    int32_t NA, NB;                // grid sizes N_k, N_{k+1}
    int32_t NApad, NBpad;          // sizes padded to a whole number of chunks
    int32_t gridA, gridB;          // grid indices (k, k+1): index into the per-grid tables
    int32_t segA, segB;            // streamed mode: segments per grid (0 = resident)
    long long goffA, goffB;        // point offsets into the FP64 grids
    long long roffA, roffB;        // record offsets (in records) into the prepared grids
    long long coff;                // entry offset of the count block
    long long item_begin;          // first work item of this layer
    int32_t items;                 // work items (sample tiles) of this layer
    int32_t hist_smem;             // 1 = shared-memory privatised histogram for this layer
};

// Per-grid tables written by the preparation kernel.
struct GridInfo {
    float mu[kDMax];               // centre (FP32) subtracted before the screen
    float R;                       // max norm of the centred FP32 records (rounded up)
    int32_t N, Npad;
    long long goff, roff;
    int32_t tc_exp;                // tensor-core form: operands scaled by 2^tc_exp
    int32_t tc_tiles;              // tensor-core form: 128-point operand tiles of this grid
    long long tc_toff;             // tensor-core form: first tile of this grid
};

// One grid of the located search (d <= 2): sizes and places from the host, the
// box, scales and certificate constants from build_cells_kernel.
struct alignas(16) CellGrid {
    float inv_h[2];                // bins per unit length
    float org[2];                  // 2^23 + number of the bin centred on 0
    float mu[2];                   // centre (FP32): the host's or the grid's own
    float mu0[2];                  // the host's
    float c1, c2, c3;              // certificate: 2 err(D) = f (c1 D + c2) + c3 D, 0 < f <= 1
    float e, ebox;                 // bound of a coordinate's error, and the part of it that is FP32 rounding in the box
    float f0;                      // the part of f that does not shrink with the sample's radius
    float err, err0;               // bounds of the centred samples' error per coordinate beyond FP32 rounding:
                                   // in proportion to their radius, and whatever it is (qt_near.h)
    int32_t N, nb;                 // points, bins an axis that the table has room for
    int32_t nb0, nb1;              // bins along each axis (nb1 = 1 for d = 1), nb0 nb1 <= nb^d
    long long goff;                // first point in the FP64 grids
    long long toff;                // first entry of the table
    long long roff;                // first float of the FP32 records
};

constexpr int kCellMaxN = 1024;    // points of a grid: ten bits per index
constexpr int kCellThreads = 1024; // most threads of the located-search kernels
constexpr int kCellNearStride = 20;// floats of a layer's combined FP32 parameters (d <= 2)

constexpr int kTcTileN = 128;      // grid points per tensor-core operand tile (MMA N)
constexpr int kTcTileM = 128;      // samples of a tensor-core work item (MMA M)
constexpr int kTcThreads = 128;    // tensor-core form: one warpgroup per CTA,
constexpr int kTcCtas = 4;         // four CTAs per SM
constexpr int kTcMaxSlots = 6;     // tensor-core form: most operand tiles in flight in shared memory

// Bytes of one work item's record between the kernels of the tensor-core form: the
// centred FP32 coordinates and norms ([grid][dm + 1][128]) and the chunk states
// ([grid][4][128]).
__host__ __device__ constexpr long long tc_item_cert_bytes(int dm) { return 2ll * (dm + 1) * kTcTileM * 4; }
__host__ __device__ constexpr long long tc_item_bytes(int dm) { return tc_item_cert_bytes(dm) + 2ll * 4 * kTcTileM * 4; }

// Dynamic shared memory of the tensor-core screen besides its ring of operand tiles
// (dimension class dm, K columns per operand row): the operand rows of one grid
// and the centred samples of two items.
__host__ __device__ constexpr long long tc_fixed_smem(int dm, int K)
{
    return (long long)kTcTileM * K * 2 + 2 * tc_item_cert_bytes(dm);
}

struct ForwardParams {
    // problem
    int32_t d, n;
    int32_t form;                  // Form
    int32_t source;                // Source
    int32_t prec;                  // 0 = FP64 samples, 1 = FP32 samples
    int32_t counts_u32;            // 1 = uint32 counts, 0 = int64
    unsigned long long M;          // samples per layer
    unsigned long long seed;
    long long total_items;
    int32_t tile;                  // samples per work item
    int32_t rec_floats;            // floats per FP32 record (d+1 rounded up to 4)
    int32_t rec64_doubles;         // doubles per FP64 record (d rounded up to 2)
    int32_t smem_grid_bytes;       // bytes of dynamic smem reserved for grids
    int32_t smem_hist_entries;     // u32 entries reserved for the private histogram
    int32_t seg_records;           // streamed mode: records per ring slot (multiple of kChunk)
    long long spin_budget;         // bound of every device wait in microseconds; < 0: give up at once
    int32_t pathwise_euler;        // Algorithm II: 1 = Euler-scheme chain (innovation rows scaled)
    // tables
    const LayerDesc* layers;
    const GridInfo* grids;
    const float* params_f;         // [n][param_count(d)]
    const double* params_d;        // [n][param_count(d)]
    int32_t params_stride;
    // data
    const double* g64;             // FP64 grids [sum N][d] (the exact distances)
    const float* rec32;            // FP32 records [sum Npad][rec_floats]
    const double* rec64;           // FP64 records [sum Npad][rec64_doubles]
    const double* srcX;            // Source::kArrays: samples [M][d]
    const double* srcY;
    void* counts;
    int32_t* cellsA;               // Source::kArrays: optional per-sample cells
    int32_t* cellsB;
    // dump
    long long dump_count, dump_stride;
    double* dumpX;
    double* dumpY;
    int32_t* dumpI;
    int32_t* dumpJ;
    DevStatus* status;
    // tensor-core form
    const void* tc_tiles;          // FP16 operand tiles [tiles][128][K] in the canonical K-major layout
    const float* tc_rows;          // chunk-major FP32 records [tiles * 8][dm + 1][16]
    int32_t tc_k;                  // 16 or 32
    int32_t tc_slots;              // ring slots of operand tiles in shared memory
    long long item_lo, item_hi;    // tensor-core form: work items [item_lo, item_hi) of this launch
    int32_t tc_one_point;          // tensor-core form: some layer has one point by one
    long long tc_ipl;              // tensor-core form: work items of every layer (0: one layer has them all)
    unsigned char* tc_items;       // tensor-core form: records of the window's items
    // located search (d <= 2)
    CellGrid* cells;               // [n+1]
    unsigned long long* cell_tab;  // bin entries of every grid
    float* cell_rec;               // centred FP32 points of every grid
    uint16_t* cell_pool;           // candidate lists longer than an entry
    unsigned long long* cell_cursor; // pool words asked for
    uint32_t cell_pool_cap;        // pool words
    int32_t cell_g0, cell_g1;      // grids [g0, g1) to build
    int32_t cell_recentre;         // the search may take the grids' own centres
    const float* cell_near;        // [n][kCellNearStride] combined FP32 parameters of FP64 layers
    long long cell_tile;           // path-wise form: paths per work item
    long long cell_ipl;            // work items of every layer (0: only one layer has any)
    // learned router + Elkan certificate
    const float* rt_params;        // MLP parameters, packed W1, b1, W2, b2, W3, b3
    const float* rt_linv;          // [n+1][d][d] FP32 inverse Cholesky factors (whitening)
    const int32_t* rt_bstart;      // [65] bucket starts into rt_members
    const int32_t* rt_members;     // [N] grid indices sorted by bucket
    const int32_t* rt_nb_idx;      // [n+1][N][C] neighbours of each grid point, nearest first
    const float* rt_nb_dist;       // [n+1][N][C] their distances, rounded down
    int32_t rt_C;                  // neighbours per point
    int32_t rt_N;                  // common grid size of layers >= 1
    unsigned long long rt_checksum;// checksum of the grids the router was built for
};

// Sample Lloyd: one grid size of a launch (qt_kmeans.cu).
struct KmJob {
    float* Z;                      // training draws [d][S]
    float* C;                      // centres, pairs [Npad/2][dim class][2]
    unsigned long long* sums;      // [copies][N][d + 1]: fixed-point sums, count
    unsigned long long seed;
    long long S;
    int32_t N, Npad;
    int32_t copies, pad;           // sums of CTAs taken modulo `copies`
};
// Copies of the sums: few centres have many draws each, whose additions would wait for one
// another (1e5 draws, 10 centres, d = 8: 400 us an iteration, 250 before each launch served all
// draws of four CTAs an SM at once)
__host__ __device__ constexpr int km_copies(long long N) { return N <= 64 ? 16 : 1; }
constexpr int kKmJobs = 32;        // grid sizes per launch
struct KmJobs {
    KmJob j[kKmJobs];
};

// A layer of the grids built: its base grid (neither: the origin) and first output.
struct MapLayer {
    const double* f64;             // [N][d]
    const float* f32;              // k-means centres
    long long off;
    int32_t N, pad;
};

// One layer of a tree whose backward induction runs in one launch.
struct TreeLayer {
    long long coff, goff;          // its counts and its points, from the first
    int32_t N, pad;
};

constexpr int kSwingQ = 8;         // swing option: consumption states per warp

constexpr int kRtHidden = 64;      // router MLP width
constexpr int kRtBuckets = 64;     // router classes (buckets of grid points)
__host__ __device__ constexpr int rt_param_count(int d) { return kRtHidden * d + kRtHidden + 2 * (kRtHidden * kRtHidden + kRtHidden); }

}  // namespace qt
