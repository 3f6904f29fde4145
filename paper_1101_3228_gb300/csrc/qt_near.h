// qt_near.h -- host side of the FP32 stand-in of an FP64 pair draw (pair_near in
// qt_cells.cuh, d <= 2): the layer's maps, centred and combined in FP64, and the two
// bounds of its error that the located search's certificate carries.
#pragma once
#include <algorithm>
#include <cmath>

namespace qt {

// Bounds of a coordinate's error: `grows` at the largest radius (8.6), in proportion to the
// pair's radius, and `fixed` at any radius.
struct NearBound {
    double grows = 0.0, fixed = 0.0;
};

// Block `o` of a layer, as pair_near reads it: [cA (d), L (d^2), cB (d), A L (d^2),
// T (d^2)] in FP32, from the packed parameters m, b, L, A, T of the exact draw.
// Errors against the exact draw X = m + L z, Y = b + A X + T eps (FP64, every operation
// rounded), with |z_q| <= rad:
//  grows: the normals' 2^-20 rad and the coefficients' 2^-24 through the maps, and
//    2^-24 for each of the at most 2 d = 4 FMAs on the part of the partial sums that the
//    normals make up: (1 + 5/16) 2^-20 of the maps' absolute sum times rad, 1.375 2^-20 here;
//  fixed: the same roundings on the part that the constant makes up, 2^-24 |c| for the
//    constant itself and for each FMA, which do not shrink with the radius; and the FP64
//    roundings of the exact draw and of the constants here, at most 4 d + 10 = 18 of
//    2^-53 on magnitudes that may cancel in c (prices of 100 that move by 1e-9).
inline void near_layer(int d, const double* p, const float* muA, const float* muB, float* o, NearBound& A_,
                       NearBound& B_)
{
    const double *m = p, *b = p + d, *L = p + 2 * d, *A = L + d * d, *T = A + d * d;
    float *cA = o, *oL = o + d, *cB = oL + d * d, *oAL = cB + d, *oT = oAL + d * d;
    const double r = 8.6, e24 = 0x1p-24, e48 = 0x1p-48;
    for (int l = 0; l < d; ++l) {
        const double a = m[l] - (double)muA[l];
        double c = b[l] - (double)muB[l], sa = 0.0, sb = 0.0;
        double ma = std::fabs(m[l]) + std::fabs((double)muA[l]), mb = std::fabs(b[l]) + std::fabs((double)muB[l]);
        for (int q = 0; q < d; ++q) {
            c += A[l * d + q] * m[q];
            mb += std::fabs(A[l * d + q] * m[q]) + r * std::fabs(T[l * d + q]);
            double al = 0.0;
            for (int s = 0; s < d; ++s) {
                al += A[l * d + s] * L[s * d + q];
                mb += r * std::fabs(A[l * d + s] * L[s * d + q]);
            }
            oL[l * d + q] = (float)L[l * d + q];
            oAL[l * d + q] = (float)al;
            oT[l * d + q] = (float)T[l * d + q];
            sa += std::fabs(L[l * d + q]);
            sb += std::fabs(al) + std::fabs(T[l * d + q]);
        }
        ma += r * sa;
        cA[l] = (float)a;
        cB[l] = (float)c;
        A_.grows = std::max(A_.grows, 1.01 * r * sa * 0x1.6p-20);
        B_.grows = std::max(B_.grows, 1.01 * r * sb * 0x1.6p-20);
        A_.fixed = std::max(A_.fixed, 1.01 * ((d + 1) * e24 * std::fabs(a) + e48 * ma));
        B_.fixed = std::max(B_.fixed, 1.01 * ((2 * d + 1) * e24 * std::fabs(c) + e48 * mb));
    }
}

}  // namespace qt
