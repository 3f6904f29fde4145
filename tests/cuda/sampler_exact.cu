// sampler_exact.cu -- test program: the FP32 sampler's integer constructions and
// its divide and square root without range tests (qt_sampler.cuh) against the plain
// IEEE operations they replace, for every one of the 2^23 uniforms.  Prints the
// number of words for which the uniform, the logarithm, the radius, the sine or the
// cosine differ, and the low nine bits' effect (none is allowed).
#include <cstdio>
#include <cuda_runtime.h>

#include "qt_sampler.cuh"

namespace {

__device__ float plain_ln(float u)
{
    const uint32_t bits = __float_as_uint(u);
    int e = (int)((bits >> 23) & 0xFFu) - 127;
    float f = __uint_as_float((bits & 0x007FFFFFu) | 0x3F800000u);
    if (f > 1.41421354f) {
        f = __fmul_rn(f, 0.5f);
        e += 1;
    }
    const float s = __fdiv_rn(__fsub_rn(f, 1.0f), __fadd_rn(f, 1.0f));
    const float z = __fmul_rn(s, s);
    float p = (1.0f / 11.0f);
    p = __fadd_rn(__fmul_rn(p, z), (1.0f / 9.0f));
    p = __fadd_rn(__fmul_rn(p, z), (1.0f / 7.0f));
    p = __fadd_rn(__fmul_rn(p, z), (1.0f / 5.0f));
    p = __fadd_rn(__fmul_rn(p, z), (1.0f / 3.0f));
    const float t = __fmul_rn(__fmul_rn(s, z), p);
    const float at = __fadd_rn(s, t);
    return __fadd_rn(__fmul_rn((float)e, 0.693147182f), __fadd_rn(at, at));
}

__device__ void plain_sincos(float u, float& sn, float& cs)
{
    const float v = __fmul_rn(u, 4.0f);
    const int q = (int)v;
    const float f = __fsub_rn(v, (float)q);
    float st, ct, s0, c0;
    if (f > 0.5f) {
        qt::quarter_sincos_f32(__fmul_rn(__fsub_rn(1.0f, f), 1.57079637f), st, ct);
        s0 = ct;
        c0 = st;
    } else {
        qt::quarter_sincos_f32(__fmul_rn(f, 1.57079637f), st, ct);
        s0 = st;
        c0 = ct;
    }
    sn = (q & 3) == 0 ? s0 : (q & 3) == 1 ? c0 : (q & 3) == 2 ? -s0 : -c0;
    cs = (q & 3) == 0 ? c0 : (q & 3) == 1 ? -s0 : (q & 3) == 2 ? -c0 : s0;
}

__global__ void compare(unsigned long long* bad)
{
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;   // < 2^23
    const uint32_t w = (j << 9) | (j & 511u);
    const float u = __fmul_rn((float)(2u * j + 1u), 0x1p-24f);
    const float ln = plain_ln(u), rad = __fsqrt_rn(__fmul_rn(-2.0f, ln));
    float sn, cs, s2, c2;
    plain_sincos(u, sn, cs);
    qt::sincos2pi_word(w, s2, c2);
    auto differ = [&](int k, float a, float b) {
        if (__float_as_uint(a) != __float_as_uint(b)) atomicAdd(&bad[k], 1ull);
    };
    differ(0, u, qt::uniform_f32(w));
    differ(1, ln, qt::ln_f32(u));
    differ(2, rad, qt::sqrt_mid(__fmul_rn(-2.0f, ln)));
    differ(3, sn, s2);
    differ(4, cs, c2);
}

}  // namespace

int main()
{
    unsigned long long *d, h[5] = {9, 9, 9, 9, 9};
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
    compare<<<(1 << 23) / 256, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("sampler_exact differing uniform %llu ln %llu radius %llu sin %llu cos %llu\n", h[0], h[1], h[2], h[3], h[4]);
    cudaFree(d);
    return h[0] || h[1] || h[2] || h[3] || h[4];
}
