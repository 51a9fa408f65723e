// Shared by the two table builders: the quadrature's panels and rows.
#pragma once

#include "sfqed_internal.h"

namespace sfq {
namespace {

constexpr int GLN = 16;
constexpr double PI = 3.14159265358979323846;

// emission: z in [-110, 8] (below: analytic tail C e^{z/3}); pair: z in [-38, 0]
constexpr double EZ_LO = -110.0, EZ_W = 0.25;
constexpr int EZ_NP = 472;
constexpr double PZ_LO = -38.0, PZ_W = 0.1;
constexpr int PZ_NP = 380;

// rows of the quadrature: the tables' chi rows, then the rate nodes
constexpr int ROW_PAIR = EM_NCHI;                               // 121
constexpr int ROW_EM_RATE = EM_NCHI + PAIR_NCHI;                // 222
constexpr int ROW_PAIR_RATE = ROW_EM_RATE + EM_NDEC * CHEB_N;   // 288
constexpr int ROWS = ROW_PAIR_RATE + PAIR_NDEC * CHEB_N;        // 343
__device__ __forceinline__ bool row_is_pair(int r) {
    return (r >= ROW_PAIR && r < ROW_EM_RATE) || r >= ROW_PAIR_RATE;
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton's method on P_16 in FP64)
__constant__ double GLX[GLN] = {
    0x1.fa92c264d787ep-1, 0x1.e39f56616f9bp-1, 0x1.bb3403514e483p-1, 0x1.82c45dda4726bp-1,
    0x1.3c5a466d5e8b8p-1, 0x1.d50259a43a772p-2, 0x1.205cae642337cp-2, 0x1.852bd6676a9f8p-4,
    -0x1.852bd6676a9f8p-4, -0x1.205cae642337cp-2, -0x1.d50259a43a772p-2, -0x1.3c5a466d5e8b8p-1,
    -0x1.82c45dda4726bp-1, -0x1.bb3403514e483p-1, -0x1.e39f56616f9bp-1, -0x1.fa92c264d787ep-1};
__constant__ double GLW[GLN] = {
    0x1.bcddab4b7c1f5p-6, 0x1.fdfb1a2c1264cp-5, 0x1.85c4ee79cc25dp-4, 0x1.fe7af2bad3875p-4,
    0x1.325f61bca3cbep-3, 0x1.5a6ebbb5a75fdp-3, 0x1.75f8c77e0c01p-3, 0x1.83feae80e4dfbp-3,
    0x1.83feae80e4dfbp-3, 0x1.75f8c77e0c01p-3, 0x1.5a6ebbb5a75fdp-3, 0x1.325f61bca3cbep-3,
    0x1.fe7af2bad3875p-4, 0x1.85c4ee79cc25dp-4, 0x1.fdfb1a2c1264cp-5, 0x1.bcddab4b7c1f5p-6};

// chi of a row
__device__ __forceinline__ double row_chi(int i) {
    if (i < ROW_PAIR) return pow(10.0, -3.0 + i / 20.0);
    if (i < ROW_EM_RATE) return pow(10.0, -2.0 + (i - ROW_PAIR) / 20.0);
    const int dec = (i - ROW_EM_RATE) / CHEB_N, k = (i - ROW_EM_RATE) % CHEB_N;
    const double lo = dec >= EM_NDEC ? -2.0 + (dec - EM_NDEC) : -3.0 + dec;
    const double s = lo + 0.5 + 0.5 * cos(PI * (k + 0.5) / CHEB_N);
    return pow(10.0, s);
}

}  // namespace
}  // namespace sfq
