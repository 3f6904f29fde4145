// near_normals.cu -- test program: the FP32 stand-in of the FP64 normals
// (box_muller_near in qt_cells.cuh) against the FP64 draw of the same Philox words,
// 2^24 pairs and the extreme words.  Prints the largest error in units of 2^-20
// times the pair's radius, the largest radius, and the largest error of the radius
// itself in the same unit.
#include <cstdio>
#include <cuda_runtime.h>

#include "qt_cells.cuh"

namespace {

__device__ float g_max[3];

__device__ void put(int k, double v)
{
    atomicMax(reinterpret_cast<int*>(&g_max[k]), __float_as_int(__double2float_ru(v)));   // v >= 0
}

__device__ void check(const qt::Philox4& w)
{
    float g0, g1;
    const float rad = qt::box_muller_near(w, g0, g1);
    const double r = __dsqrt_rn(__dmul_rn(-2.0, qt::ln_f64(qt::uniform_f64(w.v[0], w.v[1]))));
    double sn, cs;
    qt::sincos2pi_f64(qt::uniform_f64(w.v[2], w.v[3]), sn, cs);
    const double unit = r * 0x1p-20;
    put(0, fmax(fabs((double)g0 - r * cs), fabs((double)g1 - r * sn)) / unit);
    put(1, r);
    put(2, fabs((double)rad - r) / unit);
}

__global__ void run()
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    check(qt::philox4x32_10(t, 0u, 3u, 0u, 0xC0FFEEu, 77u));
    // extremes: the smallest and largest uniforms, the quarters' ends, 1 - u small
    const uint32_t ends[8] = {0u, 1u << 6, 0xFFFFFFFFu, 0xFFFFFFC0u, 0x40000000u, 0x3FFFFFFFu, 0x7FFFFFFFu, 0x80000000u};
    if (t < 4096) {
        qt::Philox4 w;
        for (int q = 0; q < 4; ++q) w.v[q] = ends[(t >> (3 * q)) & 7];
        check(w);
        w.v[0] = 0xFFFFFFFFu << (t & 31);       // u0 towards 1 and down
        check(w);
        w.v[0] = 0xFFFFFFFFu >> (t & 31);       // u0 towards 0
        check(w);
    }
}

}  // namespace

int main()
{
    float h[3] = {0, 0, 0};
    if (cudaMemcpyToSymbol(g_max, h, sizeof h) != cudaSuccess) return 1;
    run<<<(1 << 24) / 256, 256>>>();
    if (cudaMemcpyFromSymbol(h, g_max, sizeof h) != cudaSuccess) return 1;
    printf("near_normals max_error %.4f max_radius %.4f max_radius_error %.4f\n", h[0], h[1], h[2]);
    return 0;
}
