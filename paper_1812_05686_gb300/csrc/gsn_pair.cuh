// Records of the FP64 response kernels that work in pairs of FP32 numbers (gsn_pair64.cu).
#pragma once
#include "gsn_internal.cuh"

namespace gsn {

// Bin integral of smooth columns: half width of the central-difference rule (2 FM + 1 bin centres)
constexpr int FM = 16;
// columns it serves: sigma in bin widths, and the gamma family's shape (d, and mu^2 / sigma^2)
constexpr double SM_SIGMA = 6.0, SM_SHAPE = 20.0;
// smallest sigma that the pairs take at all.  Gaussian, in bin widths: the eight nodes of a bin are at
// 1e-16 of the column there, and at 1e-11 of its value at 8 sigma.  Gamma family, in half widths of a tile of 32 bins: the terms of the exponent are of the
// size (half width / sigma)^2 / 2 and cancel at the column's peak
constexpr double SQ_GAUSS = 1.5, SQ_GAMMA = 1.0 / 8;
// weights outside this range (other than 0) keep the FP64 formulas: an FP32 pair would lose its low part
constexpr double PAIR_TMIN = 1e-25, PAIR_TMAX = 1e30;
// spectra enter the per-species sums as pairs of S' 2^60, so that entries down to 1e-40 keep theirs
constexpr double SPEC_SCALE = 1152921504606846976.0, SPEC_MIN = 1e-40;
// a column with more than this share of its batch's weight is evaluated in FP64 beside the pairs
constexpr float HEAVY_SHARE = 0.25f;
constexpr int SPW = 16;   // species per pass of the per-species kernel

// One fine column.
//   Gaussian           A = mu, B = 1/sigma
//   gamma              A = ln f(mu), B = d - 1, C = 1/s, mu, ln mu = lmh + lml, kc = ln d - psi(d)
//   generalized gamma  A = ln f(mu), B = kappa_1, C = (mu/s)^p, ln mu = lmh + lml
// P: quadratic coefficient of the log2 density (Gaussian, gamma); T: T_dk of the group's datasets
// (the Gaussian's times its density at the mean).
struct __align__(16) PairRec {
    double A, B, C, mu, lmh;
    float lml, Ph, Pl, pad;
    float2 kc;
    float2 T[MAXGDS];
};
static_assert(sizeof(PairRec) == 96, "three sectors");

}  // namespace gsn
