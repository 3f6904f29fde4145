// qt_path_step.cuh -- the chain of Algorithm II (Pages & Wilbertz, arXiv:1101.3228,
// Sec. 3): the start state and one step of a path, in the order of roundings that
// qt_pathwise.cu states.  Shared by the kernels of the path-wise form.
#pragma once
#include "qt_sampler.cuh"

namespace qt {

namespace {

// Normals [lo, hi) of stream (m, k), FP32: only the Box-Muller pairs that
// overlap the range are evaluated (each Philox call yields two pairs).
template <int CNT>
__device__ __forceinline__ void normals_range_f32(uint64_t seed, int k, uint64_t m, int lo, int hi, float (&g)[CNT])
{
    const uint32_t key0 = (uint32_t)seed, key1 = (uint32_t)(seed >> 32);
    const uint32_t m0 = (uint32_t)m, m1 = (uint32_t)(m >> 32);
#pragma unroll
    for (int r = 0; r < (CNT + 3) / 4; ++r) {
        if (4 * r + 4 > lo && 4 * r < hi) {
            const Philox4 w = philox4x32_10(m0, m1, (uint32_t)k, (uint32_t)r, key0, key1);
#pragma unroll
            for (int pair = 0; pair < 2; ++pair) {
                const int q = 4 * r + 2 * pair;
                if (q + 2 > lo && q < hi) {
                    const float rad = sqrt_mid(__fmul_rn(-2.0f, ln_f32(uniform_f32(w.v[2 * pair]))));
                    float sn, cs;
                    sincos2pi_word(w.v[2 * pair + 1], sn, cs);
                    if (q < CNT) g[q] = __fmul_rn(rad, cs);
                    if (q + 1 < CNT) g[q + 1] = __fmul_rn(rad, sn);
                }
            }
        }
    }
}

template <int CNT>
__device__ __forceinline__ void normals_range_f64(uint64_t seed, int k, uint64_t m, int lo, int hi, double (&g)[CNT])
{
    const uint32_t key0 = (uint32_t)seed, key1 = (uint32_t)(seed >> 32);
    const uint32_t m0 = (uint32_t)m, m1 = (uint32_t)(m >> 32);
#pragma unroll
    for (int r = 0; r < (CNT + 1) / 2; ++r) {
        if (2 * r + 2 > lo && 2 * r < hi) {
            const Philox4 w = philox4x32_10(m0, m1, (uint32_t)k, (uint32_t)r, key0, key1);
            const double u0 = uniform_f64(w.v[0], w.v[1]);
            const double u1 = uniform_f64(w.v[2], w.v[3]);
            const double rad = __dsqrt_rn(__dmul_rn(-2.0, ln_f64(u0)));
            double sn, cs;
            sincos2pi_f64(u1, sn, cs);
            if (2 * r < CNT) g[2 * r] = __dmul_rn(rad, cs);
            if (2 * r + 1 < CNT) g[2 * r + 1] = __dmul_rn(rad, sn);
        }
    }
}

// Layer parameters as packed by the host (param_stride): m[d], b[d], L[d*d],
// A[d*d], T[d*d], alpha[d], beta[d].

// X_0 = m_0 + L_0 z (stored in X, sample precision T).
template <int DM>
__device__ __forceinline__ void path_start_f32(const float* __restrict__ P, int d, uint64_t seed, uint64_t m,
                                               float (&X)[DM])
{
    float g[2 * DM];
    normals_range_f32<2 * DM>(seed, 0, m, 0, d, g);
    const float* pm = P;
    const float* pL = P + 2 * d;
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        float acc = 0.0f;
        if (l < d) {
            acc = pm[l];
#pragma unroll
            for (int q = 0; q <= l; ++q) acc = __fadd_rn(acc, __fmul_rn(pL[l * d + q], g[q]));
        }
        X[l] = acc;
    }
}

template <int DM>
__device__ __forceinline__ void path_start_f64(const double* __restrict__ P, int d, uint64_t seed, uint64_t m,
                                               double (&X)[DM])
{
    double g[2 * DM];
    normals_range_f64<2 * DM>(seed, 0, m, 0, d, g);
    const double* pm = P;
    const double* pL = P + 2 * d;
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        double acc = 0.0;
        if (l < d) {
            acc = pm[l];
#pragma unroll
            for (int q = 0; q <= l; ++q) acc = __dadd_rn(acc, __dmul_rn(pL[l * d + q], g[q]));
        }
        X[l] = acc;
    }
}

// One step of the chain at layer k (parameters P of layer k).
template <int DM>
__device__ __forceinline__ void path_step_f32(const float* __restrict__ P, int d, bool euler, uint64_t seed, int k,
                                              uint64_t m, float (&X)[DM])
{
    float g[2 * DM];
    normals_range_f32<2 * DM>(seed, k, m, d, 2 * d, g);
    const float* pb = P + d;
    const float* pA = P + 2 * d + d * d;
    const float* pT = pA + d * d;
    const float* pal = pT + d * d;
    const float* pbe = pal + d;
    float sc[DM], Xn[DM];
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        sc[l] = 1.0f;
        if (euler && l < d) {
            const float u = __fadd_rn(pal[l], __fmul_rn(pbe[l], X[l]));
            sc[l] = __fsqrt_rn(u > 0.0f ? u : 0.0f);
        }
    }
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        float acc = 0.0f;
        if (l < d) {
            acc = pb[l];
#pragma unroll
            for (int q = 0; q < DM; ++q)
                if (q < d) acc = __fadd_rn(acc, __fmul_rn(pA[l * d + q], X[q]));
#pragma unroll
            for (int q = 0; q <= l; ++q) {
                const float t = euler ? __fmul_rn(sc[l], pT[l * d + q]) : pT[l * d + q];
                acc = __fadd_rn(acc, __fmul_rn(t, g[d + q]));
            }
        }
        Xn[l] = acc;
    }
#pragma unroll
    for (int l = 0; l < DM; ++l) X[l] = Xn[l];
}

template <int DM>
__device__ __forceinline__ void path_step_f64(const double* __restrict__ P, int d, bool euler, uint64_t seed, int k,
                                              uint64_t m, double (&X)[DM])
{
    double g[2 * DM];
    normals_range_f64<2 * DM>(seed, k, m, d, 2 * d, g);
    const double* pb = P + d;
    const double* pA = P + 2 * d + d * d;
    const double* pT = pA + d * d;
    const double* pal = pT + d * d;
    const double* pbe = pal + d;
    double sc[DM], Xn[DM];
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        sc[l] = 1.0;
        if (euler && l < d) {
            const double u = __dadd_rn(pal[l], __dmul_rn(pbe[l], X[l]));
            sc[l] = __dsqrt_rn(u > 0.0 ? u : 0.0);
        }
    }
#pragma unroll
    for (int l = 0; l < DM; ++l) {
        double acc = 0.0;
        if (l < d) {
            acc = pb[l];
#pragma unroll
            for (int q = 0; q < DM; ++q)
                if (q < d) acc = __dadd_rn(acc, __dmul_rn(pA[l * d + q], X[q]));
#pragma unroll
            for (int q = 0; q <= l; ++q) {
                const double t = euler ? __dmul_rn(sc[l], pT[l * d + q]) : pT[l * d + q];
                acc = __dadd_rn(acc, __dmul_rn(t, g[d + q]));
            }
        }
        Xn[l] = acc;
    }
#pragma unroll
    for (int l = 0; l < DM; ++l) X[l] = Xn[l];
}

template <bool F32>
struct SampleType {
    using T = double;
};
template <>
struct SampleType<true> {
    using T = float;
};

}  // namespace

}  // namespace qt
