"""The error bounds of the located search's FP32 stand-in for FP64 pairs, on the CPU: the
library's own combination of a layer's maps (qt_near.h) is compiled for the host, the
FP32 chain of fused multiply-adds of the kernel and the FP64 draw with its roundings are
evaluated on normals disturbed by the 2^-20 of their radius that is allowed for, and

    |a~ - (X - mu_A)| <= (rad / 8.6) grows_A + fixed_A   (and the same for Y - mu_B)

must hold for every pair, at all radii, constants far from the grids' centres and
scales at which the FP64 roundings of the draw itself show.
"""
import os
import subprocess
import tempfile

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "qt_near.h"
static double urand(unsigned long long& s)
{
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return ((s >> 11) + 0.5) * 0x1p-53;
}
int main(int argc, char** argv)
{
    const int d = atoi(argv[1]);
    const double scale = atof(argv[2]), about = atof(argv[3]), off = atof(argv[4]);
    unsigned long long s = 12345;
    double worst = 0.0;
    for (int model = 0; model < 40; ++model) {
        // packed parameters m, b, L, A, T; the grids' centres `off` scales from the means
        double p[16] = {0};
        double *m = p, *b = p + d, *L = p + 2 * d, *A = L + d * d, *T = A + d * d;
        float muA[2], muB[2];
        for (int l = 0; l < d; ++l) {
            m[l] = about * (1 + 0.01 * urand(s));
            for (int q = 0; q <= l; ++q) {
                L[l * d + q] = scale * (q == l ? 0.5 + urand(s) : urand(s) - 0.5);
                T[l * d + q] = 0.3 * scale * (q == l ? 0.5 + urand(s) : urand(s) - 0.5);
            }
            for (int q = 0; q < d; ++q) A[l * d + q] = (q == l) * 0.9 + 0.1 * (urand(s) - 0.5);
        }
        for (int l = 0; l < d; ++l) {
            double am = 0;
            for (int q = 0; q < d; ++q) am += A[l * d + q] * m[q];
            b[l] = m[l] - am;
            muA[l] = (float)(m[l] + off * scale * (urand(s) - 0.5));
            muB[l] = (float)(m[l] + off * scale * (urand(s) - 0.5));
        }
        float o[20];
        qt::NearBound bA, bB;
        qt::near_layer(d, p, muA, muB, o, bA, bB);
        const float *cA = o, *oL = o + d, *cB = oL + d * d, *oAL = cB + d, *oT = oAL + d * d;
        for (int it = 0; it < 20000; ++it) {
            const double rad = std::exp(std::log(1e-8) + urand(s) * std::log(8.5e8));
            double g[4];
            float gn[4];
            for (int q = 0; q < 2 * d; ++q) {
                g[q] = rad * (2 * urand(s) - 1);
                gn[q] = (float)(g[q] + rad * 0.9999 * 0x1p-20 * (urand(s) < 0.5 ? -1 : 1));
            }
            double X[2], Y[2];
            for (int l = 0; l < d; ++l) {
                X[l] = m[l];
                for (int q = 0; q <= l; ++q) { volatile double t = L[l * d + q] * g[q]; X[l] = X[l] + t; }
            }
            for (int l = 0; l < d; ++l) {
                Y[l] = b[l];
                for (int q = 0; q < d; ++q) { volatile double t = A[l * d + q] * X[q]; Y[l] = Y[l] + t; }
                for (int q = 0; q <= l; ++q) { volatile double t = T[l * d + q] * g[d + q]; Y[l] = Y[l] + t; }
            }
            for (int l = 0; l < d; ++l) {
                float a = cA[l], y = cB[l];
                for (int q = 0; q < d; ++q) {
                    a = std::fma(oL[l * d + q], gn[q], a);
                    y = std::fma(oAL[l * d + q], gn[q], y);
                    y = std::fma(oT[l * d + q], gn[d + q], y);
                }
                const double ea = std::fabs((double)((long double)X[l] - muA[l] - a));
                const double ey = std::fabs((double)((long double)Y[l] - muB[l] - y));
                worst = std::max(worst, ea / (rad / 8.6 * bA.grows + bA.fixed));
                worst = std::max(worst, ey / (rad / 8.6 * bB.grows + bB.fixed));
            }
        }
    }
    std::printf("%.6f\n", worst);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program():
    with tempfile.TemporaryDirectory() as td:
        src, exe = os.path.join(td, "near.cpp"), os.path.join(td, "near")
        with open(src, "w") as f:
            f.write(SRC)
        subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                        os.path.join(ROOT, "paper_1101_3228_gb300", "csrc"), src, "-o", exe], check=True)
        yield exe


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("scale,about", [(1.0, 0.0), (1.0, 100.0), (1e-9, 100.0), (1e-3, -3.0), (1e4, 1.0)])
@pytest.mark.parametrize("off", [0.0, 1.0, 2000.0])
def test_stand_in_error_within_bounds(program, d, scale, about, off):
    out = subprocess.run([program, str(d), repr(scale), repr(about), repr(off)], check=True, capture_output=True,
                         text=True).stdout
    worst = float(out)
    assert 0.0 < worst <= 1.0
