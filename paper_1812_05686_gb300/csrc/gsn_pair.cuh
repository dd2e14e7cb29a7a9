// Records of the FP64 response kernels that work in pairs of FP32 numbers (gsn_pair64.cu).
#pragma once
#include "gsn_device.cuh"

namespace gsn {

// Bin integral of smooth columns: half width of the central-difference rule (2 FM + 1 bin centres)
constexpr int FM = 16;
// columns it serves: sigma in bin widths, and the gamma family's shape (d, and mu^2 / sigma^2)
constexpr double SM_SIGMA = 6.0, SM_SHAPE = 20.0;
// Smallest sigma that the pairs take at all.  Gaussian, in bin widths: the eight nodes of a bin are off by
// 5e-20 of the bin at the column's centre, 2e-13 at 8 sigma.  Gamma family, in half widths of a tile of 32
// bins: the terms of the exponent are of the size (half width / sigma)^2 / 2 and cancel at the column's peak
constexpr double SQ_GAUSS = 1.5, SQ_GAMMA = 1.0 / 8;
// weights outside this range (other than 0) keep the FP64 formulas: an FP32 pair would lose its low part
constexpr double PAIR_TMIN = 1e-25, PAIR_TMAX = 1e30;
// spectra enter the per-species sums as pairs of S' 2^60, so that entries down to 1e-40 keep theirs
constexpr double SPEC_SCALE = 1152921504606846976.0, SPEC_MIN = 1e-40;
// a column with more than this share of its batch's weight is evaluated in FP64 beside the pairs
constexpr float HEAVY_SHARE = 0.25f;
// Stray bins: counts of 2^20 expectations or more, in the tails where a column's density leaves FP32's range
// (a tile that a band touches reaches bins 20 sigma out, 1e-87 of the peak) and w = 1 - n/mu may leave it too.
// Their expectation and their part of the adjoint take the FP64 formulas.  STRAY_RATIO: the bound on the
// difference of the high words of n and mu; STRAY_HI: high word of w = -2^20
constexpr int STRAY_RATIO = 20 << 20;
constexpr unsigned STRAY_HI = 0xC1300000u;
DEV bool is_stray(double w) { return (unsigned)__double2hiint(w) >= STRAY_HI; }
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

// FP64 bin value of one column (batches whose columns are too narrow for pairs, heavy columns, stray bins)
template <int RES>
DEV double native_value(const KArgs& a, int t, int g, int k, const double* c, int j) {
    if constexpr (RES == 0) {
        const double* ed = a.edges + tb_g_edge_off(a, g) + j;
        return ncdf_diff((ed[0] - c[F_MUH]) * c[F_A], (ed[1] - c[F_MUH]) * c[F_A]);
    } else {
        const int nb = tb_g_node_off(a, g) + j;
        const unsigned char cls = a.bclass[nb];
        if (cls == BIN_ZERO) return zerorec<double>(a, t, g, k)[Z_P0];
        const double* nd = a.ntab_d + (long long)nb * 3 * NGM_D;
        const int NG = cls == BIN_LOG ? NG_LOG_D : NG_LIN_D;
        double rho = 0.0;
        for (int n = 0; n < NG; ++n) {
            if constexpr (RES == 1) rho = fma(nd[2 * NGM_D + n], exp(fma(c[F_B], nd[NGM_D + n], fma(-c[F_C], nd[n], c[F_A]))), rho);
            else rho = fma(nd[2 * NGM_D + n], exp(fma(c[F_B], nd[NGM_D + n], c[F_A]) - exp(c[F_KAPPA] * (nd[NGM_D + n] - c[F_C]))), rho);
        }
        return rho;
    }
}

// ------------------------------------------------ arithmetic on pairs -----
// TwoSum of a running pair (sh, sl) and p, error terms collected in sl
DEV void acc_pair(float& sh, float& sl, float p, float e) {
    const float t = __fadd_rn(sh, p);
    const float bp = __fsub_rn(t, sh);
    const float er = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    sl = __fadd_rn(sl, __fadd_rn(er, e));
    sh = t;
}
// (s, l) with l brought below half an ulp of s
DEV void renorm(float& s, float& l) {
    const float t = __fadd_rn(s, l);
    l = __fsub_rn(l, __fsub_rn(t, s));
    s = t;
}
// product of two pairs: leading part p, the rest e
DEV void mul_pair(float ah, float al, float bh, float bl, float& p, float& e) {
    p = __fmul_rn(ah, bh);
    e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, fmaf(al, bh, e));
}
DEV float2 split(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}
DEV double join(float h, float l) { return (double)h + (double)l; }
// a / b to ~2^-46
DEV void div_pair(float ah, float al, float bh, float bl, float& q, float& e) {
    const float r = __frcp_rn(bh);
    q = __fmul_rn(ah, r);
    e = __fmul_rn(fmaf(-q, bl, __fadd_rn(fmaf(-q, bh, ah), al)), r);
}

// Poisson term mu - n + n ln(n / mu) of Eq. (LL) for counts and expectation that differ by less than a
// factor 1.5, without the FP64 logarithm and division (~100 FP64-pipe operations of 64 cycles): with
// e = n - mu and u = e / (n + mu),
//     term = u (e + (n + mu + e) v S),  v = u^2,  S = 1/3 + v/5 + v^2/7 + ...
// in which nothing cancels (mu - n + n ln(n / mu) loses n 2^-53 to the rounding of n / mu).  Pairs hold
// S's first five terms; the rest, v^5 (1/13 + ...) < 8e-9, is FP32.  False outside the range.  With the template
// gradients in pairs, the deviance of 8192 template toys of 2 x 1000 bins: 3.31 -> 1.12 ms.
DEV bool poisson_term(double mu, double n, float& th, float& tl) {
    const double e = n - mu, s = n + mu;
    const float2 E = split(e), A = split(s);
    if (!(fabsf(E.x) <= 0.2f * A.x) || !(A.x > 1e-30f && A.x < 1e30f)) return false;
    float uh, ul, vh, vl, p, q, yh, yl;
    div_pair(E.x, E.y, A.x, A.y, uh, ul);
    mul_pair(uh, ul, uh, ul, vh, vl);
    float R = fmaf(vh, 1.0f / 19, 1.0f / 17);
    R = fmaf(R, vh, 1.0f / 15);
    R = fmaf(R, vh, 1.0f / 13);
    constexpr double c[5] = {1.0 / 3, 1.0 / 5, 1.0 / 7, 1.0 / 9, 1.0 / 11};
    yh = R; yl = 0.f;
#pragma unroll
    for (int i = 4; i >= 0; --i) {   // y <- c_i + v y
        mul_pair(yh, yl, vh, vl, p, q);
        const float ch = (float)c[i], cl = (float)(c[i] - (double)ch);
        yh = ch; yl = cl;
        acc_pair(yh, yl, p, q);
    }
    mul_pair(yh, yl, vh, vl, p, q);
    float mh = A.x, ml = A.y;        // 2 n
    acc_pair(mh, ml, E.x, E.y);
    mul_pair(mh, ml, p, q, yh, yl);
    mh = E.x; ml = E.y;
    acc_pair(mh, ml, yh, yl);
    mul_pair(mh, ml, uh, ul, th, tl);
    return true;
}

}  // namespace gsn
