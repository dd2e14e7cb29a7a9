// FP64 response kernels on the FP32 pipes: every value is an unevaluated pair of FP32 numbers.
//
// The FP64 response was bound by the FP64 pipe, which takes 64 cycles per 32-lane operation on
// sm_103a: five (gamma) exponentials or an erfc per (bin, column) pair cost 6000-8000 cycles per warp
// in the forward and as much again in the adjoint.  An FP32 pair carries 48 bits and its operations are
// error-free sums and products (TwoSum, fused multiply-add) on the FP32 pipe, so a pair's density takes
// about 55 FP32 operations.  What stays FP64 is done once per 32 pairs (the exponent at a tile's
// reference point, the flush of the partial sums) and runs on the FP64 pipe beside them.
// Measured on 128 toys of the two-dataset workload (2 x 1200 bins, 20000 columns): forward 198.7 ->
// 3.62 ms (103 instructions per 32 pairs, issue 73%, FMA pipe 54%, FP64 pipe 44%), adjoint 186.3 -> 6.37 ms
// (165 instructions), per-species shapes of one point 72 -> 0.21 ms; 500 toys of the 900-bin Gaussian
// workload: forward 44.6 -> 0.86 ms, adjoint 49.5 -> 1.17 ms.  Errors against 64-bit references, before
// -> now: gradients of the gamma toys 3.4e-13 -> 3.2e-13, of the Gaussian toys 8.9e-15 -> 8.6e-15.
//
// Exponent.  Bins are tiled by 32; a tile has a reference point x_r.  For the gamma family the log2
// density of a column is exactly
//     E(x) = E(x_r) + g a(x) + P D(x)
//   gamma              a = x - x_r         D = ln(1 + a/x_r) - a/x_r      P = log2 e (d - 1)
//   generalized gamma  a = ln(x / x_r)     D = e^(p a) - 1 - p a          P = -log2 e (x_r / s)^p
// with g the derivative at x_r.  E(x_r) and g are FP64 (where the terms of d ln x cancel), a and D FP32
// pairs tabulated per node.  E(x_r)'s integer part goes to the result's exponent bits, so that the
// pair's terms are of the size of g a: a few 2^-48 of it is the error.  The Gaussian needs no reference
// terms: E = -(log2 e / 2) ((x - mu) / sigma)^2 from the pair x - mu.
//
// Bin integrals.  Where the density is smooth on the scale of the bins (sigma >= SM_SIGMA bin widths,
// shape >= SM_SHAPE) the integral over a bin of width h is
//     h sum_m c_m f(x_j + m h),  m = -FM..FM,
// x_j the bin's centre, c the coefficients of (delta / 2) / asinh(delta / 2) expanded in the central
// difference delta to order 2 FM.  Relative to the local value it is off by 5e-15 at 8 sigma of a Gaussian
// of 6 bins and by 1e-18 inside 6 sigma, and by 1e-18 for a gamma of shape 20 (five Gauss-Legendre
// points per bin, which it replaces, are at 1e-12 in such tails).
// The sum over columns commutes with it, so each (bin, column) pair takes ONE density value instead of
// five: the forward sums F_i = sum_k T_k f_k(x_i) over the nodes i (the bins and FM more above the
// histogram), the deviance applies c, and the adjoint reads c applied to the weights.  The nodes are
// bin centres, so this needs FM bins of the same width on either side (uniform histograms, bins in the
// linear class); other bins and narrower columns take the Gauss-Legendre nodes of the bin with the
// same evaluation (five, ten in the log-spaced bins, eight for the Gaussian), and columns below the
// SQ_* limits, where the pairs' terms would cancel or the nodes miss a Gaussian, the FP64 formulas.
// Bins that hold counts where the expectation is far below them (a million times and more) leave the
// pairs as well (is_stray).
// Classes are chosen per batch of 32 columns (the warp's) from the batch's smallest sigma.  A column
// that outweighs its batch (a mono-energetic line) is evaluated in FP64 beside the pairs: the single
// error of its pairs, 6e-15, would be the error of every bin it dominates.
#include "gsn_device.cuh"
#include "gsn_ggamma.cuh"
#include "gsn_pair.cuh"

namespace gsn {

namespace {

constexpr int PW = 8;   // warps per block of the forward

// 2^(s + lo), times the power of two whose exponent bits nb holds, as an FP32 pair; |s| < 4096
DEV void pair_exp2(float s, float lo, int nb, const float2* __restrict__ tab, float& vh, float& vl) {
    // s = n/1024 + r: the table holds 2^(i/1024), and |r| < 2^-11 leaves a cubic
    constexpr float MAGIC = 12288.0f;   // ulp 2^-10
    const float kf = __fadd_rn(s, MAGIC);
    const int bits = __float_as_int(kf);
    const float rh = __fsub_rn(s, __fsub_rn(kf, MAGIC));
    const float r = __fadd_rn(rh, lo);
    const float rl = __fsub_rn(lo, __fsub_rn(r, rh));
    const float2 T = tab[bits & 1023];
    constexpr float C1 = 0.69314718055994531f, C1L = (float)(0.69314718055994531 - (double)C1);
    constexpr float C2 = 0.24022650695910071f, C3 = 0.055504108664821580f;
    const float p = __fmul_rn(r, C1);
    float e = fmaf(r, C1, -p);
    e = fmaf(r, C1L, e);
    e = fmaf(rl, C1, e);
    e = fmaf(__fmul_rn(r, r), fmaf(r, C3, C2), e);
    const float w = __fmul_rn(T.x, p);
    const float we = fmaf(T.x, p, -w);
    const float h = __fadd_rn(T.x, w);
    float l = __fadd_rn(__fsub_rn(w, __fsub_rn(h, T.x)), we);
    l = fmaf(T.x, e, l);
    l = fmaf(T.y, p, l);
    l = __fadd_rn(l, T.y);
    const float sc = __int_as_float(((bits << 13) & 0xff800000) + nb);
    vh = h * sc;
    vl = l * sc;
}

// A column at a tile's reference point.  Gaussian: E = the mean relative to it, g unused, and the node
// pairs hold x - x_r: E(x) = P (x - mu)^2 has no terms that cancel.  Otherwise E = the fraction of
// E(x_r), whose integer part sits in the exponent bits nb, so that near the peak the pair's terms are
// of the size of g a.
struct ColTerms { float2 E, g, P; int nb; };

// Density at the node (a, D); Gaussian: (ah, al) becomes x - mu and (Dh, Dl) its square.  The exponent is
// held at a floor so that its bits do not wrap: 2^-125 of a Gaussian's peak, at most 2^-89 of the gamma
// family's (nb is at most half above the exponent at x_r).  With CUT values at the floor are 0.  The forward and
// the adjoint leave them, an instruction per value less: they enter a bin's expectation where it is above
// 2^-20 of its counts only (is_stray), as 2^-69 of the counts or less.
template <int RES, bool CUT = false>
DEV void pair_density(const ColTerms& c, float& ah, float& al, float& Dh, float& Dl, const float2* __restrict__ tab, float& vh,
                      float& vl) {
    if constexpr (RES == 0) {
        const float d = __fsub_rn(ah, c.E.x), b = __fsub_rn(d, ah);
        const float e = __fsub_rn(__fsub_rn(ah, __fsub_rn(d, b)), __fadd_rn(c.E.x, b));
        const float l = __fadd_rn(__fsub_rn(al, c.E.y), e);
        ah = __fadd_rn(d, l);
        al = __fsub_rn(l, __fsub_rn(ah, d));
        Dh = __fmul_rn(ah, ah);
        Dl = fmaf(__fadd_rn(ah, ah), al, fmaf(ah, ah, -Dh));
        float s, lo;
        mul_pair(c.P.x, c.P.y, Dh, Dl, s, lo);
        pair_exp2(fmaxf(s, -125.0f), lo, 0x3f800000, tab, vh, vl);
        if (CUT && s < -125.0f) vh = vl = 0.f;
    } else {
        float p1, e1, p2, e2;
        mul_pair(c.g.x, c.g.y, ah, al, p1, e1);
        mul_pair(c.P.x, c.P.y, Dh, Dl, p2, e2);
        const float s1 = __fadd_rn(c.E.x, p1), b1 = __fsub_rn(s1, c.E.x);
        const float t1 = __fadd_rn(__fsub_rn(c.E.x, __fsub_rn(s1, b1)), __fsub_rn(p1, b1));
        const float s2 = __fadd_rn(s1, p2), b2 = __fsub_rn(s2, s1);
        const float t2 = __fadd_rn(__fsub_rn(s1, __fsub_rn(s2, b2)), __fsub_rn(p2, b2));
        const float lo = __fadd_rn(__fadd_rn(c.E.y, __fadd_rn(e1, e2)), __fadd_rn(t1, t2));
        pair_exp2(fmaxf(s2, -90.0f), lo, c.nb, tab, vh, vl);
        if (CUT && s2 < -90.0f) vh = vl = 0.f;
    }
}

// e^q - 1 - q to full relative precision
DEV double gg_Q_d(double q) {
    if (fabs(q) > 0.5) return expm1(q) - q;
    // Horner over q^k / (k + 2)!, k = 13..0
    constexpr double c[14] = {1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320, 1.0 / 362880,
                              1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0, 1.0 / 87178291200.0,
                              1.0 / 1307674368000.0};
    double v = c[13];
#pragma unroll
    for (int i = 12; i >= 0; --i) v = fma(v, q, c[i]);
    return v * q * q;
}

// reference point of a tile: x_r, ln x_r = lx + lxl, 1 / x_r
struct TileRef { double x, lx, ix, lxl; };
DEV TileRef tile_ref(const KArgs& a, int g, int tile) {
    const double* r = a.tref + 4LL * (a.tb->g_tile_off[g] + tile);
    return {r[0], r[1], r[2], r[3]};
}

// E(x_r) in log2 units: integer part to the exponent bits, fraction as a pair
DEV void set_exponent(ColTerms& o, double E) {
    const double n = fmin(fmax(rint(E), -30.0), 30.0);
    o.nb = 0x3f800000 + ((int)n << 23);
    o.E = split(E - n);
}

// exponent terms of one column at a tile's reference point; gamma family: dl = ln(x_r / mu), for the
// generalized gamma y = (x_r / s)^p as well
template <int RES>
DEV ColTerms column_terms(const PairRec& c, const TileRef& t, double p, double& dl, double& y) {
    constexpr double L2 = 1.4426950408889634074;
    ColTerms o;
    o.P = make_float2(c.Ph, c.Pl);
    if constexpr (RES == 0) {
        o.E = split(c.A - t.x);
        o.g = make_float2(0.f, 0.f);
        o.nb = 0;
    } else {
        dl = (t.lx - c.lmh) + (t.lxl - (double)c.lml);
        if constexpr (RES == 1) {
            set_exponent(o, L2 * fma(c.B, dl, fma(-c.C, t.x - c.mu, c.A)));
            o.g = split(L2 * fma(c.B, t.ix, -c.C));
        } else {
            // ln f(mu) + kappa_1 L - A Q(p L), the derivative kappa_1 - p A (e^(pL) - 1)
            const double q = p * dl, Q = gg_Q_d(q);
            set_exponent(o, L2 * fma(c.B, dl, fma(-c.C, Q, c.A)));
            o.g = split(L2 * fma(-p * c.C, q + Q, c.B));
            y = c.C * (1.0 + (q + Q));
            o.P = split(-L2 * y);
        }
    }
    return o;
}

template <int RES> DEV double toy_power(const KArgs& a, int t, int g) {
    if constexpr (RES == 2) {
        const int q = tb_g_resp(a, g, 5);
        return q >= 0 ? a.params[(long long)t * a.params_stride + q] * tb_g_rscale(a, g, 5) : 1.0;
    } else {
        return 1.0;
    }
}

// class of a batch of columns: 2 smooth, 1 quadrature nodes in pairs, 0 FP64 formulas
DEV int batch_class(const KArgs& a, int g, const float4& bs) {
    return bs.w >= a.tb->g_smin[g] ? 2 : bs.z >= a.tb->g_qmin[g] ? 1 : 0;
}

// FP64 density of one column at a bin centre (a, D as tabulated) of a tile
template <int RES>
DEV double centre_density(const PairRec& c, const TileRef& t, double p, double a, double D) {
    if constexpr (RES == 0) {
        const double z = ((t.x - c.A) + a) * c.B;
        return exp(-0.5 * z * z) * (c.B * INV_SQRT2PI);
    } else {
        const double L0 = (t.lx - c.lmh) + (t.lxl - (double)c.lml);
        if constexpr (RES == 1) return exp(fma(c.B, L0 + fma(a, t.ix, D), fma(-c.C, (t.x - c.mu) + a, c.A)));
        const double L = L0 + a;
        return exp(fma(c.B, L, fma(-c.C, gg_Q_d(p * L), c.A)));
    }
}

// W-weighted sums of one bin of one column in FP64: value rho, and by response the derivative sums
// u[] (Gaussian, gamma: U1, U2; generalized gamma: the four node sums, then W at the bin at zero)
template <int RES>
DEV double native_sums(const KArgs& a, int t, int g, int k, const double* c, int j, double W, double* u) {
    const double* ed = a.edges + tb_g_edge_off(a, g) + j;
    double rho = 0.0;
    if constexpr (RES == 0) {
        const double z0 = (ed[0] - c[F_MUH]) * c[F_A], z1 = (ed[1] - c[F_MUH]) * c[F_A];
        rho = ncdf_diff(z0, z1);
        const double p0 = exp(-0.5 * z0 * z0) * INV_SQRT2PI, p1 = exp(-0.5 * z1 * z1) * INV_SQRT2PI;
        u[0] = fma(W, -(p1 - p0), u[0]);
        u[1] = fma(W, -(z1 * p1 - z0 * p0), u[1]);
    } else {
        const int nb = tb_g_node_off(a, g) + j;
        const unsigned char cl = a.bclass[nb];
        if (cl == BIN_ZERO) {
            const double* zr = zerorec<double>(a, t, g, k);
            rho = zr[Z_P0];
            if constexpr (RES == 1) { u[0] = fma(W, zr[Z_P0D], u[0]); u[1] = fma(W, zr[Z_P0S], u[1]); }
            else u[4] += W;
            return rho;
        }
        const double* nd = a.ntab_d + (long long)nb * 3 * NGM_D;
        const int NG = cl == BIN_LOG ? NG_LOG_D : NG_LIN_D;
        double s1 = 0.0, s2 = 0.0, s3 = 0.0;
        for (int n = 0; n < NG; ++n) {
            if constexpr (RES == 1) {
                const double fw = nd[2 * NGM_D + n] * exp(fma(c[F_B], nd[NGM_D + n], fma(-c[F_C], nd[n], c[F_A])));
                rho += fw; s1 = fma(fw, nd[NGM_D + n] - c[F_KAPPA], s1); s2 = fma(fw, nd[n] - c[F_MUH], s2);
            } else {
                const double l = nd[NGM_D + n] - c[F_C], y = exp(c[F_KAPPA] * l);
                const double fw = nd[2 * NGM_D + n] * exp(fma(c[F_B], nd[NGM_D + n], c[F_A]) - y);
                rho += fw; s1 = fma(fw, l, s1); s2 = fma(fw, y, s2); s3 = fma(fw * y, l, s3);
            }
        }
        if constexpr (RES == 1) { u[0] = fma(W, s1, u[0]); u[1] = fma(W, s2, u[1]); }
        else { u[0] = fma(W, rho, u[0]); u[1] = fma(W, s1, u[1]); u[2] = fma(W, s2, u[2]); u[3] = fma(W, s3, u[3]); }
    }
    return rho;
}

DEV void load_table(const KArgs& a, float2* tab) {
    const float4* src = reinterpret_cast<const float4*>(a.ex2tab);
    float4* dst = reinterpret_cast<float4*>(tab);
    for (int i = threadIdx.x; i < 512; i += blockDim.x) dst[i] = src[i];
}

}  // namespace

// ------------------------------------------------------------- forward -----
// lanes <-> the 32 bins (nodes) of a tile; the warp walks the batches of 32 columns whose band
// reaches it.  Each lane turns one column of the batch into its exponent terms (FP64, once per
// tile), the warp then reads the columns from shared memory one by one.
//   q[0] = (E, g)   q[1] = (P, nb, -)   q[2..] = T of two datasets each
template <int NDS> struct FwdRec { float4 q[2 + (NDS + 1) / 2]; };

template <int RES, int NDS>
__global__ void __launch_bounds__(PW * 32, 2) k_forward_p(KArgs a) {
    constexpr int NU = RES == 0 ? 4 : 5;   // quadrature nodes in flight (8; 5 or 10 per bin)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* tab = reinterpret_cast<float2*>(smem_raw);
    FwdRec<NDS>* srec_all = reinterpret_cast<FwdRec<NDS>*>(smem_raw + 8192);
    float2* sq_all = reinterpret_cast<float2*>(smem_raw + 8192 + sizeof(FwdRec<NDS>) * PW * 32);
    load_table(a, tab);
    __syncthreads();
    const int split_i = blockIdx.y;
    const int t = blockIdx.z / a.G, g = blockIdx.z % a.G;
    if (!tb_g_active(a, g)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FwdRec<NDS>* srec = srec_all + warp * 32;
    float2* sq = sq_all + warp * (NGM_D * 3 * 32) + lane;   // [node][a, D, w][lane]
    int wlo, whi;
    toy_window_union(a, t, g, wlo, whi);
    if (whi <= wlo) return;
    const int J = tb_g_bins(a, g), ju = a.tb->g_ju[g];
    const int flo = max(wlo, ju) - FM, fhi = whi > ju ? whi + FM : flo;   // nodes (none unless some bin >= ju)
    const int tile = blockIdx.x * PW + warp, j0 = tile * 32, j = j0 + lane;
    const bool tM = j0 < whi && j0 + 32 > wlo;                 // bins of the window in the tile
    const bool tF = fhi > flo && j0 < fhi && j0 + 32 > flo;    // nodes
    if (!tM && !tF) return;
    const bool vM = j >= wlo && j < whi, vF = fhi > flo && j >= flo && j < fhi;
    const bool lowbins = j0 < ju && tM && wlo < ju;             // bins that smooth columns integrate by nodes
    const TileRef tr = tile_ref(a, g, tile);
    const double pw = toy_power<RES>(a, t, g);
    const double* ed = a.edges + tb_g_edge_off(a, g);
    const double h = a.tb->g_h[g];   // bin width of the uniform part
    // energies the tile covers: its bins in the window, and the cells of its nodes
    float xlo, xhi;
    {
        const int b0 = max(j0, wlo), b1 = min(min(j0 + 32, whi), J);
        const int n0 = max(j0, flo), n1 = min(j0 + 32, fhi);
        xlo = INFINITY; xhi = -INFINITY;
        if (tM) { xlo = (float)ed[b0]; xhi = (float)ed[b1]; }
        if (tF) {
            const double e0 = n0 <= J ? ed[n0] : ed[J] + (n0 - J) * h, e1 = n1 <= J ? ed[n1] : ed[J] + (n1 - J) * h;
            xlo = fminf(xlo, (float)e0);
            xhi = fmaxf(xhi, (float)e1);
        }
    }
    const float xlow = (float)ed[min(min(ju, j0 + 32), J)];    // their upper edge in the tile
    float ah = 0.f, al = 0.f, Dh = 0.f, Dl = 0.f;
    if (vF) {
        const float4 s = a.snode[a.tb->g_snode_off[g] + j];
        ah = s.x; al = s.y; Dh = s.z; Dl = s.w;
        if constexpr (RES == 2) { const float2 q = split(gg_Q_d(pw * join(ah, al))); Dh = q.x; Dl = q.y; }
    }
    const bool zero = RES >= 1 && tb_g_zero(a, g) && j0 == 0 && tM && wlo == 0;   // lane 0 holds the bin at zero
    const int nbat = a.nbat;
    const float4* bsum = a.batsum + ((long long)t * a.G + g) * nbat;
    const PairRec* prec = a.pairbuf + ((long long)t * a.G + g) * nbat * 32;
    const unsigned* heavy = a.heavy + ((long long)t * a.G + g) * nbat;
    double Fd[NDS] = {}, Md[NDS] = {};
    int nq = -1;   // nodes staged for the tile's bins (-1: not yet)
    long long npairs = 0;
    // the split takes every nsplit-th batch: a tile's band is a contiguous range of batches, which
    // contiguous splits would leave to a few warps
    for (int b0 = split_i; b0 < nbat; b0 += 32 * a.nsplit) {
        float4 bs = make_float4(INFINITY, -INFINITY, 0.f, 0.f);
        if (b0 + lane * a.nsplit < nbat) bs = bsum[b0 + lane * a.nsplit];
        unsigned hits = __ballot_sync(0xffffffffu, !(bs.y < xlo || bs.x > xhi));
        const int cls_l = batch_class(a, g, bs);
        while (hits) {
            const int bl = __ffs(hits) - 1;
            hits &= hits - 1;
            const int cls = __shfl_sync(0xffffffffu, cls_l, bl);
            const int b = b0 + bl * a.nsplit;
            if (cls == 0) {
                if (!tM) continue;
                for (int k = b * 32; k < min(a.K, b * 32 + 32); ++k) {
                    const double* c = colrec<double>(a, t, g, k);
                    if (c[F_XMAX] < (double)xlo || c[F_XMIN] > (double)xhi) continue;
                    ++npairs;
                    if (!vM) continue;
                    const double v = native_value<RES>(a, t, g, k, c, j);
#pragma unroll
                    for (int dd = 0; dd < NDS; ++dd) Md[dd] = fma(v, c[F_TN0 + dd], Md[dd]);
                }
                __syncwarp();
                continue;
            }
            const bool smooth = cls == 2;
            const bool low = lowbins && __shfl_sync(0xffffffffu, bs.x, bl) <= xlow;   // its band reaches them
            if (smooth && !tF && !low) continue;
            if (!smooth && !tM) continue;
            npairs += 32;
            const unsigned hm = heavy[b];
            for (unsigned m = hm; m; m &= m - 1) {
                const int k = b * 32 + __ffs(m) - 1;
                const double* c = colrec<double>(a, t, g, k);
                double v = 0.0, w = 0.0;
                if (smooth && vF) v = centre_density<RES>(prec[k], tr, pw, join(ah, al), RES == 0 ? 0.0 : join(Dh, Dl));
                if (vM && (!smooth || (low && j < ju))) w = native_value<RES>(a, t, g, k, c, j);
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) { Fd[dd] = fma(v, c[F_TN0 + dd], Fd[dd]); Md[dd] = fma(w, c[F_TN0 + dd], Md[dd]); }
            }
            {
                PairRec c = prec[b * 32 + lane];
                if (hm >> lane & 1) {
#pragma unroll
                    for (int dd = 0; dd < MAXGDS; ++dd) c.T[dd] = make_float2(0.f, 0.f);
                }
                double dl, y;
                const ColTerms o = column_terms<RES>(c, tr, pw, dl, y);
                FwdRec<NDS>& r = srec[lane];
                r.q[0] = make_float4(o.E.x, o.E.y, o.g.x, o.g.y);
                r.q[1] = make_float4(o.P.x, o.P.y, __int_as_float(o.nb), 0.f);
#pragma unroll
                for (int dd = 0; dd < NDS; dd += 2)
                    r.q[2 + dd / 2] = make_float4(c.T[dd].x, c.T[dd].y, dd + 1 < NDS ? c.T[dd + 1].x : 0.f, dd + 1 < NDS ? c.T[dd + 1].y : 0.f);
            }
            __syncwarp();
            float sh[4][NDS] = {}, sl[4][NDS] = {};
            auto terms = [&](const FwdRec<NDS>& r) {
                return ColTerms{make_float2(r.q[0].x, r.q[0].y), make_float2(r.q[0].z, r.q[0].w), make_float2(r.q[1].x, r.q[1].y),
                                __float_as_int(r.q[1].z)};
            };
            auto add = [&](const FwdRec<NDS>& r, float vh, float vl, float* ah4, float* al4) {
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) {
                    const float4 T = r.q[2 + dd / 2];
                    float p, e;
                    mul_pair(vh, vl, dd & 1 ? T.z : T.x, dd & 1 ? T.w : T.y, p, e);
                    acc_pair(ah4[dd], al4[dd], p, e);
                }
            };
            if (smooth && tF) {
                // four interleaved sums: independent chains, and the collected error terms of eight
                // columns each stay small against the next (their own rounding is what the sum loses)
                for (int c4 = 0; c4 < 32; c4 += 4) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const FwdRec<NDS> r = srec[c4 + u];
                        float xh = ah, xl = al, yh = Dh, yl = Dl, vh, vl;
                        pair_density<RES>(terms(r), xh, xl, yh, yl, tab, vh, vl);
                        add(r, vh, vl, sh[u], sl[u]);
                    }
                }
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) renorm(sh[u][dd], sl[u][dd]);
                    acc_pair(sh[0][dd], sl[0][dd], sh[1][dd], sl[1][dd]);
                    acc_pair(sh[2][dd], sl[2][dd], sh[3][dd], sl[3][dd]);
                    acc_pair(sh[0][dd], sl[0][dd], sh[2][dd], sl[2][dd]);
                    Fd[dd] += join(sh[0][dd], sl[0][dd]);
                    sh[0][dd] = sl[0][dd] = 0.f;
                }
            }
            // bins below ju take quadrature nodes for every column that reaches them
            if (!smooth || low) {
                const bool use = vM && (!smooth || j < ju);
                if (nq < 0) {
                    // nodes of the lane's bin, once per tile
                    const int nb = tb_g_node_off(a, g) + min(j, J - 1);
                    const int mine = vM ? (int)a.qn[nb] : 0;
                    nq = __reduce_max_sync(0xffffffffu, mine);
                    nq = (nq + NU - 1) / NU * NU;
                    for (int n = 0; n < nq; ++n) {
                        const float2* q = reinterpret_cast<const float2*>(a.qnode) + ((long long)nb * NGM_D + n) * 3;
                        float2 qa = make_float2(0.f, 0.f), qd = qa, qw = qa;
                        if (n < mine) { qa = q[0]; qd = q[1]; qw = q[2]; }
                        if constexpr (RES == 2) qd = split(gg_Q_d(pw * join(qa.x, qa.y)));
                        sq[(n * 3) * 32] = qa; sq[(n * 3 + 1) * 32] = qd; sq[(n * 3 + 2) * 32] = qw;
                    }
                }
                for (int ci = 0; ci < 32; ++ci) {
                    const FwdRec<NDS> r = srec[ci];
                    const ColTerms c = terms(r);
                    float uh = 0.f, ul = 0.f;
                    for (int n0 = 0; n0 < nq; n0 += NU) {
#pragma unroll
                        for (int n = n0; n < n0 + NU; ++n) {   // independent evaluations
                            float2 qa = sq[(n * 3) * 32], qd = sq[(n * 3 + 1) * 32];
                            const float2 qw = sq[(n * 3 + 2) * 32];
                            float vh, vl, p, e;
                            pair_density<RES>(c, qa.x, qa.y, qd.x, qd.y, tab, vh, vl);
                            mul_pair(vh, vl, qw.x, qw.y, p, e);
                            acc_pair(uh, ul, p, e);
                        }
                    }
                    if (zero && lane == 0) {
                        const int k = b * 32 + ci;
                        const float2 z = k < a.K ? split(zerorec<double>(a, t, g, k)[Z_P0]) : make_float2(0.f, 0.f);
                        uh = z.x; ul = z.y;
                    }
                    add(r, uh, ul, sh[0], sl[0]);
                    if ((ci & 7) == 7) {
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) {
                            if (use) Md[dd] += join(sh[0][dd], sl[0][dd]);
                            sh[0][dd] = sl[0][dd] = 0.f;
                        }
                    }
                }
            }
            __syncwarp();
        }
    }
    if (a.work) {
        const unsigned m = __ballot_sync(0xffffffffu, vM);
        if (lane == 0) atomicAdd(&a.work[K_FORWARD], (unsigned long long)npairs * __popc(m));
    }
    const int nds = tb_g_nds(a, g);
#pragma unroll
    for (int dd = 0; dd < NDS; ++dd) {
        if (dd >= nds) break;
        const int d = tb_g_ds(a, g, dd);
        if (vM) a.mubuf[((long long)t * a.nsplit + split_i) * a.total_bins + tb_ds_off(a, d) + j] = Md[dd];
        if (vF) a.fbuf[((long long)t * a.nsplit + split_i) * a.fext + tb_ds_off(a, d) + d * FM + j] = Fd[dd];
    }
}

// ------------------------------------------------ filtered weights for the adjoint -----
// wf_i = sum_m c_m h_(i - m) w_(i - m) over the bins >= ju (h: bin widths, equal up to rounding): the
// transpose of the bin integral of the smooth columns, as FP32 pairs, without the stray bins (grid: toys x
// blocks of nodes)
__global__ void __launch_bounds__(256) k_wfilter(KArgs a) {
    const int t = blockIdx.x, n = blockIdx.y * 256 + threadIdx.x;
    if (n >= a.fext) return;
    int lo = 0, hi = a.D - 1;
    while (lo < hi) { const int m = (lo + hi + 1) >> 1; if (tb_ds_off(a, m) + m * FM <= n) lo = m; else hi = m - 1; }
    const int d = lo, i = n - (tb_ds_off(a, d) + d * FM), g = tb_ds_group(a, d);
    const int J = tb_ds_bins(a, d), ju = a.tb->g_ju[g];
    const double* ed = a.edges + tb_g_edge_off(a, g);
    double v = 0.0;
    if (tb_ds_resp(a, d) && ju < J) {
        const double* w = reinterpret_cast<const double*>(a.wbuf) + (long long)t * a.total_bins + tb_ds_off(a, d);
        for (int m = -FM; m <= FM; ++m) {
            const int j = i - m;
            if (j >= ju && j < J) {
                const double wj = w[j];
                v = fma(a.conv[m < 0 ? -m : m] * (is_stray(wj) ? 0.0 : wj), ed[j + 1] - ed[j], v);
            }
        }
    }
    a.wfbuf[(long long)t * a.fext + n] = split(v);
}

// ------------------------------------------------------------ backward -----
// lanes <-> the 32 columns of a batch; the warp walks the tiles of its band and accumulates, per
// dataset, the weighted moments sum w f {1, a, D} (and a^2, a D for the free power), which tile by
// tile give the sums of the per-column derivatives in FP64.  The tile's nodes (offsets and filtered
// weights, or quadrature nodes times bin weights) are staged in shared memory 32 at a time.
template <int RES, int NDS>
__global__ void __launch_bounds__(256, 2) k_backward_p(KArgs a) {
    constexpr int NM = RES == 2 ? 5 : 3, NA = NDS + NM - 1;
    constexpr int NV = 1 + (NDS + 1) / 2;    // float4 per staged node
    const int task = blockIdx.x, g = blockIdx.y, t = blockIdx.z;
    if (!tb_g_active(a, g)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int W = a.bw_warps;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float2* tab = reinterpret_cast<float2*>(smem_raw);
    float4* sn = reinterpret_cast<float4*>(smem_raw + 8192) + warp * 32 * NV;
    double* su = reinterpret_cast<double*>(smem_raw + 8192 + sizeof(float4) * 32 * NV * W);   // [NDS][W*32]
    double* sresp = su + NDS * W * 32;                                                        // [W][NRESP]
    // flags of the toy's deviance blocks (read beside the table, used where the tiles begin)
    const double* dflag = a.devpart + (long long)t * a.dev_chunks * (2 + a.ntpl) + 1;
    const double flag0 = lane < a.dev_chunks ? dflag[lane * (2 + a.ntpl)] : 0.0;
    load_table(a, tab);
    __syncthreads();
    const int cbw = task / a.bw_bsplit, bsp = task % a.bw_bsplit;
    const int b = cbw * W + warp, kbase = cbw * W * 32, k = b * 32 + lane;
    const bool kval = k < a.K;
    const int nds = tb_g_nds(a, g);
    const int J = tb_g_bins(a, g), ju = a.tb->g_ju[g];
    const double* ed = a.edges + tb_g_edge_off(a, g);
    const double* prm = a.params + (long long)t * a.params_stride;
    const int nbase = tb_g_node_off(a, g);
    const double h = a.tb->g_h[g];
    int wlo, whi;
    toy_window_union(a, t, g, wlo, whi);
    double U0[NDS] = {}, u[5] = {};   // w-weighted values; derivative sums (native_sums)
    float Uh[NDS] = {}, Ul[NDS] = {}, Sh[3] = {}, Sl[3] = {};
    const double* c = colrec<double>(a, t, g, kval ? k : a.K - 1);   // read where needed, not kept in registers
    long long nvisit = 0;
    if (b < a.nbat && whi > wlo) {
        const float4 bs = a.batsum[((long long)t * a.G + g) * a.nbat + b];
        const int cls = batch_class(a, g, bs);
        const int flo = max(wlo, ju) - FM, fhi = cls == 2 && whi > ju ? whi + FM : flo;
        // bins (and nodes above the histogram) inside the band
        int ja, jb;
        {
            int lo = 0, hi = J;
            while (lo < hi) { const int m = (lo + hi) >> 1; if (ed[m + 1] <= (double)bs.x) lo = m + 1; else hi = m; }
            ja = lo;
            lo = 0; hi = J;
            while (lo < hi) { const int m = (lo + hi) >> 1; if (ed[m] < (double)bs.y) lo = m + 1; else hi = m; }
            jb = lo;   // one past
            if (fhi > J && (double)bs.y > ed[J]) jb = J + (int)fmin((double)FM, ceil(((double)bs.y - ed[J]) / h));
        }
        const int rlo = fhi > flo ? min(wlo, flo) : wlo, rhi = max(whi, fhi > flo ? fhi : whi);
        ja = max(ja, rlo); jb = min(jb, rhi);
        if (jb > ja) {
            int flags = (int)flag0;
            for (int q = lane + 32; q < a.dev_chunks; q += 32) flags |= (int)dflag[q * (2 + a.ntpl)];
            const bool stray_toy = __any_sync(0xffffffffu, flags & 4);   // the deviance found stray bins
            const int t0 = ja >> 5, t1 = ((jb - 1) >> 5) + 1, ch = (t1 - t0 + a.bw_bsplit - 1) / a.bw_bsplit;
            const int ta = t0 + bsp * ch, tb = min(t1, ta + ch);
            const double pw = toy_power<RES>(a, t, g);
            const PairRec& pc = a.pairbuf[((long long)t * a.G + g) * a.nbat * 32 + k];
            float2 Tk[NDS];
#pragma unroll
            for (int dd = 0; dd < NDS; ++dd) Tk[dd] = pc.T[dd];
            const double Nn = RES == 0 ? c[F_A] * INV_SQRT2PI : 1.0;
            // weights of bin j (those of stray bins, the others, or both), and their sum over the datasets
            // with a column's T
            auto weights = [&](int j, double* wj, double& Wj, const double* cc, bool plain, bool stray) {
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) {
                    const double w = dd < nds ? reinterpret_cast<const double*>(a.wbuf)[(long long)t * a.total_bins +
                                                                                        tb_ds_off(a, tb_g_ds(a, g, dd)) + j] : 0.0;
                    wj[dd] = (is_stray(w) ? stray : plain) ? w : 0.0;
                    Wj = fma(wj[dd], cc[F_TN0 + dd], Wj);
                }
            };
            // columns that outweigh their batch, in FP64 with lanes <-> nodes and bins
            const unsigned hm = cls == 0 ? 0u : a.heavy[((long long)t * a.G + g) * a.nbat + b];
            for (unsigned m = hm; m; m &= m - 1) {
                const int src = __ffs(m) - 1, kk = b * 32 + src;
                const double* cc = colrec<double>(a, t, g, kk);
                const PairRec& pk = a.pairbuf[((long long)t * a.G + g) * a.nbat * 32 + kk];
                double hU[NDS] = {}, hu[5] = {};
                for (int tile = ta; tile < tb; ++tile) {
                    const int i = tile * 32 + lane, lo = max(ja, tile * 32), hi = min(jb, tile * 32 + 32);
                    const TileRef tr = tile_ref(a, g, tile);
                    if (cls == 2 && i >= max(lo, flo) && i < min(hi, fhi)) {
                        const float4 s = a.snode[a.tb->g_snode_off[g] + i];
                        const double da = join(s.x, s.y), D = RES == 1 ? join(s.z, s.w) : 0.0;
                        const double f = centre_density<RES>(pk, tr, pw, da, D);
                        double W = 0.0;
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd)
                            if (dd < nds) {
                                const int d = tb_g_ds(a, g, dd);
                                const float2 w2 = a.wfbuf[(long long)t * a.fext + tb_ds_off(a, d) + d * FM + i];
                                const double w = join(w2.x, w2.y);
                                hU[dd] = fma(w, f, hU[dd]);
                                W = fma(w, cc[F_TN0 + dd], W);
                            }
                        const double Wf = W * f;
                        if constexpr (RES == 0) {
                            const double z = ((tr.x - pk.A) + da) * pk.B;
                            hu[0] = fma(Wf, z, hu[0]); hu[1] = fma(Wf, fma(z, z, -1.0), hu[1]);
                        } else if constexpr (RES == 1) {
                            const double L = (tr.lx - pk.lmh) + (tr.lxl - (double)pk.lml) + fma(da, tr.ix, D);
                            hu[0] = fma(Wf, L + join(pk.kc.x, pk.kc.y), hu[0]); hu[1] = fma(Wf, (tr.x - pk.mu) + da, hu[1]);
                        } else {
                            const double l = (tr.lx - cc[F_C]) + da, y = exp(pw * l);
                            hu[0] += Wf; hu[1] = fma(Wf, l, hu[1]); hu[2] = fma(Wf, y, hu[2]); hu[3] = fma(Wf * y, l, hu[3]);
                        }
                    }
                    if (i >= max(lo, wlo) && i < min(min(hi, whi), cls == 2 ? ju : J)) {
                        double wj[NDS], Wj = 0.0;
                        weights(i, wj, Wj, cc, true, false);
                        const double rho = native_sums<RES>(a, t, g, kk, cc, i, Wj, hu);
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) hU[dd] = fma(wj[dd], rho, hU[dd]);
                    }
                }
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) { const double v = warp_sum<double>(hU[dd]); if (lane == src) U0[dd] = v; }
#pragma unroll
                for (int i = 0; i < (RES == 2 ? 5 : 2); ++i) { const double v = warp_sum<double>(hu[i]); if (lane == src) u[i] = v; }
            }
            const bool mine = !(hm >> lane & 1);   // the lane's column takes the pairs' sums
            // FP64 formulas, bin by bin: the band's bins of columns that the pairs do not take, and the tiles'
            // stray bins for the columns that entered their expectation (stray_sum)
            if (cls == 0 || stray_toy)
                for (int tile = ta; tile < tb; ++tile) {
                    const int mlo = max(max(ja, tile * 32), wlo), mhi = min(min(min(jb, tile * 32 + 32), whi), J);
                    const int a0 = stray_toy ? max(tile * 32, wlo) : mlo, a1 = stray_toy ? min(min(tile * 32 + 32, whi), J) : mhi;
                    const bool reach = stray_toy && !(c[F_XMAX] < (double)(float)ed[a0] || c[F_XMIN] > (double)(float)ed[a1]);
                    for (int j = a0; j < a1; ++j) {
                        const bool plain = cls == 0 && j >= mlo && j < mhi;
                        nvisit += plain;
                        double wj[NDS], Wj = 0.0;
                        weights(j, wj, Wj, c, plain, reach);
                        bool any = false;
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) any = any || wj[dd] != 0.0;
                        if (!any) continue;
                        const double rho = native_sums<RES>(a, t, g, kval ? k : a.K - 1, c, j, Wj, u);
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) U0[dd] = fma(wj[dd], rho, U0[dd]);
                    }
                }
            for (int tile = cls == 0 ? tb : ta; tile < tb; ++tile) {
                const int lo = max(ja, tile * 32), hi = min(jb, tile * 32 + 32);   // the band's bins in the tile
                const int mlo = max(lo, wlo), mhi = min(min(hi, whi), J);
                const TileRef tr = tile_ref(a, g, tile);
                double dl = 0.0, y = 0.0;
                const ColTerms ct = column_terms<RES>(pc, tr, pw, dl, y);
                // sums of the tile: w_d f per dataset, then W f a, W f D (a^2, a D) with W = sum_d w_d T_d
                // (one dataset: its own weight, T applied at the end).  Eight nodes at a time: the
                // collected error terms stay small against the next ones
                float mh[NA], ml[NA];
#pragma unroll
                for (int i = 0; i < NA; ++i) mh[i] = ml[i] = 0.f;
                auto nodes = [&](int n0, int n1) {
                    for (int n8 = n0; n8 < n1; n8 += 8) {
                        float qh[NA], ql[NA];
#pragma unroll
                        for (int i = 0; i < NA; ++i) qh[i] = ql[i] = 0.f;
                        const int n9 = min(n8 + 8, n1);
#pragma unroll 2
                        for (int n = n8; n < n9; ++n) {
                            float4 s = sn[n * NV];
                            float vh, vl, Wh = 0.f, Wl = 0.f, p, e, p1, e1;
                            pair_density<RES>(ct, s.x, s.y, s.z, s.w, tab, vh, vl);
#pragma unroll
                            for (int dd = 0; dd < NDS; ++dd) {
                                const float4 w4 = sn[n * NV + 1 + dd / 2];
                                const float wh = dd & 1 ? w4.z : w4.x, wl = dd & 1 ? w4.w : w4.y;
                                mul_pair(vh, vl, wh, wl, p, e);
                                acc_pair(qh[dd], ql[dd], p, e);
                                if constexpr (NDS > 1) {
                                    mul_pair(wh, wl, Tk[dd].x, Tk[dd].y, p1, e1);
                                    if (dd == 0) { Wh = p1; Wl = e1; } else acc_pair(Wh, Wl, p1, e1);
                                }
                            }
                            if constexpr (NDS > 1) mul_pair(vh, vl, Wh, Wl, p, e);
                            mul_pair(p, e, s.x, s.y, p1, e1);
                            acc_pair(qh[NDS], ql[NDS], p1, e1);
                            if constexpr (RES == 2) {
                                float p2, e2;
                                mul_pair(p1, e1, s.x, s.y, p2, e2);
                                acc_pair(qh[NDS + 2], ql[NDS + 2], p2, e2);
                                mul_pair(p1, e1, s.z, s.w, p2, e2);
                                acc_pair(qh[NDS + 3], ql[NDS + 3], p2, e2);
                            }
                            mul_pair(p, e, s.z, s.w, p1, e1);
                            acc_pair(qh[NDS + 1], ql[NDS + 1], p1, e1);
                        }
#pragma unroll
                        for (int i = 0; i < NA; ++i) { renorm(qh[i], ql[i]); acc_pair(mh[i], ml[i], qh[i], ql[i]); }
                    }
                };
                if (cls == 2) {
                    const int n0 = max(lo, flo), n1 = min(hi, fhi);
                    if (n1 > n0) {
                        const int i = tile * 32 + lane;
                        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                        float2 wv[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                        if (i >= n0 && i < n1) {
                            s = a.snode[a.tb->g_snode_off[g] + i];
                            if constexpr (RES == 2) { const float2 q = split(gg_Q_d(pw * join(s.x, s.y))); s.z = q.x; s.w = q.y; }
#pragma unroll
                            for (int dd = 0; dd < NDS; ++dd)
                                if (dd < nds) {
                                    const int d = tb_g_ds(a, g, dd);
                                    wv[dd] = a.wfbuf[(long long)t * a.fext + tb_ds_off(a, d) + d * FM + i];
                                }
                        }
                        __syncwarp();
                        sn[lane * NV] = s;
                        sn[lane * NV + 1] = make_float4(wv[0].x, wv[0].y, wv[1].x, wv[1].y);
                        if constexpr (NDS > 2) sn[lane * NV + 2] = make_float4(wv[2].x, wv[2].y, wv[3].x, wv[3].y);
                        __syncwarp();
                        nodes(n0 - tile * 32, n1 - tile * 32);
                        nvisit += n1 - n0;
                    }
                }
                const int qhi = cls == 2 ? min(mhi, ju) : mhi;
                if (qhi > mlo) {
                    // quadrature nodes of the bins [mlo, qhi)
                    const int nbin = qhi - mlo;
                    const int nqm = __reduce_max_sync(0xffffffffu, lane < nbin ? (int)a.qn[nbase + mlo + lane] : 0);
                    for (int i0 = 0; i0 < nbin * nqm; i0 += 32) {
                        const int i = i0 + lane, jj = mlo + (nqm ? i / nqm : 0), n = nqm ? i % nqm : 0;
                        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                        float2 wv[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                        if (jj < qhi && n < (int)a.qn[nbase + jj]) {
                            const float2* q = reinterpret_cast<const float2*>(a.qnode) + ((long long)(nbase + jj) * NGM_D + n) * 3;
                            const float2 qa = q[0], qw = q[2];
                            float2 qd = q[1];
                            if constexpr (RES == 2) qd = split(gg_Q_d(pw * join(qa.x, qa.y)));
                            s = make_float4(qa.x, qa.y, qd.x, qd.y);
                            const double wt = join(qw.x, qw.y);
#pragma unroll
                            for (int dd = 0; dd < NDS; ++dd)
                                if (dd < nds)
                                {
                                    const double w = reinterpret_cast<const double*>(a.wbuf)[(long long)t * a.total_bins +
                                                                                             tb_ds_off(a, tb_g_ds(a, g, dd)) + jj];
                                    wv[dd] = split(is_stray(w) ? 0.0 : wt * w);
                                }
                        }
                        __syncwarp();
                        sn[lane * NV] = s;
                        sn[lane * NV + 1] = make_float4(wv[0].x, wv[0].y, wv[1].x, wv[1].y);
                        if constexpr (NDS > 2) sn[lane * NV + 2] = make_float4(wv[2].x, wv[2].y, wv[3].x, wv[3].y);
                        __syncwarp();
                        nodes(0, min(32, nbin * nqm - i0));
                    }
                    nvisit += nbin;
                    if (RES >= 1 && mlo == 0 && tb_g_zero(a, g) && mine) {
                        double wj[NDS], Wj = 0.0;
                        weights(0, wj, Wj, c, true, false);
                        const double rho = native_sums<RES>(a, t, g, kval ? k : a.K - 1, c, 0, Wj, u);
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) U0[dd] = fma(wj[dd], rho, U0[dd]);
                    }
                }
                // the tile's moments, datasets weighted by their T, to the column's sums (pairs: an FP64
                // operation costs 64 cycles per warp)
                float Mh[NM] = {}, Ml[NM] = {};
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) {
                    acc_pair(Uh[dd], Ul[dd], mh[dd], ml[dd]);
                    float p, e;
                    mul_pair(mh[dd], ml[dd], Tk[dd].x, Tk[dd].y, p, e);
                    acc_pair(Mh[0], Ml[0], p, e);
                }
#pragma unroll
                for (int i = 1; i < NM; ++i) {
                    if constexpr (NDS == 1) mul_pair(mh[i], ml[i], Tk[0].x, Tk[0].y, Mh[i], Ml[i]);
                    else { Mh[i] = mh[NDS - 1 + i]; Ml[i] = ml[NDS - 1 + i]; }
                }
                // sums s += k m of pairs
                auto fold = [&](int s, float2 k, int m) {
                    float p, e;
                    mul_pair(k.x, k.y, Mh[m], Ml[m], p, e);
                    acc_pair(Sh[s], Sl[s], p, e);
                };
                if constexpr (RES == 0) {
#pragma unroll
                    for (int i = 0; i < NM; ++i) acc_pair(Sh[i], Sl[i], Mh[i], Ml[i]);
                } else if constexpr (RES == 1) {
                    // sum W f (ln x - kappa), ln x - kappa = D + a / x_r + dl + kc, and sum W f (x - mu)
                    const float2 d2 = split(dl);
                    float kh = pc.kc.x, kl = pc.kc.y;
                    acc_pair(kh, kl, d2.x, d2.y);
                    acc_pair(Sh[0], Sl[0], Mh[2], Ml[2]);
                    fold(0, split(tr.ix), 1);
                    fold(0, make_float2(kh, kl), 0);
                    acc_pair(Sh[1], Sl[1], Mh[1], Ml[1]);
                    fold(1, split(tr.x - pc.mu), 0);
                } else {
                    const double M[5] = {join(Mh[0], Ml[0]), join(Mh[1], Ml[1]), join(Mh[2], Ml[2]), join(Mh[3], Ml[3]), join(Mh[4], Ml[4])};
                    const double l = tr.lx - c[F_C], yb = M[0] + pw * M[1] + M[2];
                    if (mine) {
                        u[0] += M[0];
                        u[1] += fma(l, M[0], M[1]);
                        u[2] = fma(y, yb, u[2]);
                        u[3] = fma(y, fma(l, yb, M[1] + pw * M[3] + M[4]), u[3]);
                    }
                }
                // every eight tiles the pairs' sums go to the column's FP64 sums (class 0 and the heavy columns have
                // theirs there): a pair that is never renormalised loses bits as the square of its terms
                if (((tile - ta) & 7) == 7 || tile + 1 == tb) {
                    if (mine) {
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) U0[dd] = fma(Nn, join(Uh[dd], Ul[dd]), U0[dd]);
                        if constexpr (RES == 0) {
                            u[0] = fma(c[F_A], join(Sh[1], Sl[1]), u[0]);
                            u[1] += fma(c[F_A] * c[F_A], join(Sh[2], Sl[2]), -join(Sh[0], Sl[0]));
                        } else if constexpr (RES == 1) {
                            u[0] += join(Sh[0], Sl[0]);
                            u[1] += join(Sh[1], Sl[1]);
                        }
                    }
#pragma unroll
                    for (int dd = 0; dd < NDS; ++dd) Uh[dd] = Ul[dd] = 0.f;
#pragma unroll
                    for (int i = 0; i < 3; ++i) Sh[i] = Sl[i] = 0.f;
                }
            }
        }
    }
    if (a.work) {
        const unsigned m = __ballot_sync(0xffffffffu, kval);
        if (lane == 0 && nvisit > 0) atomicAdd(&a.work[K_BACKWARD], (unsigned long long)nvisit * __popc(m));
    }
    // chain rule per column, as in the FP64 kernel
    const double LY = prm[tb_g_resp(a, g, 0)] * tb_g_rscale(a, g, 0);
    const double rb = prm[tb_g_resp(a, g, 3)] * tb_g_rscale(a, g, 3), rc = prm[tb_g_resp(a, g, 4)] * tb_g_rscale(a, g, 4);
    double r[NRESP] = {};
    if (kval) {
        const double mu = c[F_MUH];
        double g_mu, g_var;
        if constexpr (RES == 2) {
            const double* g2 = a.colbuf2 + (((long long)t * a.G + g) * a.K + k) * NFG;
            double gm = 0.0, gv = 0.0, gp = 0.0;
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                gm = fma(g2[FG_MU + i], u[i], gm);
                gv = fma(g2[FG_VAR + i], u[i], gv);
                gp = fma(g2[FG_P + i], u[i], gp);
            }
            g_mu = gm; g_var = gv;
            r[5] = gp;
        } else if constexpr (RES == 0) {
            g_mu = u[0] * c[F_A];
            g_var = 0.5 * u[1] * c[F_A] * c[F_A];
        } else {
            const double d = mu * c[F_C], s = 1.0 / c[F_C], var = d * s * s;
            const double gd = u[0], gs = u[1] * c[F_C] * c[F_C];
            g_mu = gd * (2.0 * d / mu) - gs * (s / mu);
            g_var = -gd * (d / var) + gs / mu;
        }
        const double g_mt = g_mu + g_var * (rb + 2.0 * rc * mu);
        r[0] = g_mt * (mu / LY);
        r[1] = g_mt * LY * c[F_DEQ];
        r[2] = g_var;
        r[3] = g_var * mu;
        r[4] = g_var * mu * mu;
    }
#pragma unroll
    for (int i = 0; i < NRESP; ++i) {
        const double v = warp_sum<double>(r[i]);
        if (lane == 0) sresp[warp * NRESP + i] = v;
    }
#pragma unroll
    for (int dd = 0; dd < NDS; ++dd) su[dd * W * 32 + warp * 32 + lane] = kval ? U0[dd] : 0.0;
    __syncthreads();
    double* part = a.partbuf + (((long long)t * a.G + g) * a.nbtask + task) * a.NPART;
    if (threadIdx.x < NRESP) {
        double s = 0.0;
        for (int w = 0; w < W; ++w) s += sresp[w * NRESP + threadIdx.x];
        part[threadIdx.x] = s;
    }
    // rates: S'^T u over the block's columns, a warp per (dataset, species), lanes on the columns
    const int ncol = min(W * 32, a.K - kbase);
    for (int i = warp; i < MAXGDS * a.S; i += W) {
        const int dd = i / a.S, s = i % a.S;
        double v = 0.0;
        if (dd < NDS && dd < nds && a.ft.sp_kind[s] < 2 && a.rfac[tb_g_ds(a, g, dd) * a.S + s] != 0.0) {
            const double* Srow = a.Sd + (long long)s * a.K + kbase;
            for (int cc = lane; cc < ncol; cc += 32) v = fma(Srow[cc], su[dd * W * 32 + cc], v);
            v = warp_sum<double>(v);
        }
        if (lane == 0) part[NRESP + i] = v;
    }
}

// ---------------------------------------------------- per-species path -----
// M[g][s][j] = sum_k R_jk S'_sk: as the forward, with up to SPW species' spectra in the place of the
// T_dk.  Lanes <-> the 32 bins of a tile; the grid's z takes (toy, species pass, batch split).  Two
// passes over the batches (smooth columns at the bin centres, the others and the low bins by
// quadrature) keep one set of sums in registers; k_species_reduce adds the splits and applies the bin
// integral of the smooth part.
constexpr int SPB = 4;   // warps per block

template <int RES>
__global__ void __launch_bounds__(SPB * 32, 4) k_species_p(KArgs a) {
    constexpr int NU = RES == 0 ? 4 : 5;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* tab = reinterpret_cast<float2*>(smem_raw);
    load_table(a, tab);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4* srec = reinterpret_cast<float4*>(smem_raw + 8192) + warp * 64;                            // [32][2]
    float4* ssp = reinterpret_cast<float4*>(smem_raw + 8192 + SPB * 1024) + warp * (32 * SPW / 2);    // [32][SPW / 2]
    float2* sq = reinterpret_cast<float2*>(smem_raw + 8192 + SPB * (1024 + 32 * SPW * 8)) + warp * (NGM_D * 3 * 32) + lane;
    const int g = blockIdx.y, nchunk = (a.sp_count + SPW - 1) / SPW;
    const int split_i = blockIdx.z % a.sp_nsplit, chunk = blockIdx.z / a.sp_nsplit % nchunk, t = blockIdx.z / a.sp_nsplit / nchunk;
    if (!tb_g_active(a, g)) return;
    const int J = tb_g_bins(a, g), ju = a.tb->g_ju[g];
    const int flo = ju - FM, fhi = ju < J ? J + FM : flo;
    const int tile = blockIdx.x * SPB + warp, j0 = tile * 32, j = j0 + lane;
    const bool tM = j0 < J, tF = fhi > flo && j0 < fhi && j0 + 32 > flo;
    if (!tM && !tF) return;
    const bool vM = j < J, vF = fhi > flo && j >= flo && j < fhi;
    const bool lowbins = j0 < ju && tM;
    const TileRef tr = tile_ref(a, g, tile);
    const double pw = toy_power<RES>(a, t, g), h = a.tb->g_h[g];
    const double* ed = a.edges + tb_g_edge_off(a, g);
    auto edge = [&](int i) { return (float)(i <= J ? ed[i] : ed[J] + (i - J) * h); };
    const float xlo = edge(j0), xhi = edge(tF ? max(min(j0 + 32, fhi), min(j0 + 32, J)) : min(j0 + 32, J)), xlow = edge(min(min(ju, j0 + 32), J));
    float ah = 0.f, al = 0.f, Dh = 0.f, Dl = 0.f;
    if (vF) {
        const float4 s = a.snode[a.tb->g_snode_off[g] + j];
        ah = s.x; al = s.y; Dh = s.z; Dl = s.w;
        if constexpr (RES == 2) { const float2 q = split(gg_Q_d(pw * join(ah, al))); Dh = q.x; Dl = q.y; }
    }
    const bool zero = RES >= 1 && tb_g_zero(a, g) && j0 == 0;
    const float4* bsum = a.batsum + ((long long)t * a.G + g) * a.nbat;
    const PairRec* prec = a.pairbuf + ((long long)t * a.G + g) * a.nbat * 32;
    const int s0 = a.sp_first + chunk * SPW, Spad = (a.S + SPW - 1) / SPW * SPW;
    // [t][g][split][species][centres, bins][Jmax + FM]
    double* out = a.sp_part + (((long long)t * a.G + g) * a.sp_nsplit + split_i) * a.S * 2 * (a.Jmax + FM);
    int nq = -1;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        if (pass == 0 ? !tF : !tM) continue;
        double acc[SPW];
#pragma unroll
        for (int i = 0; i < SPW; ++i) acc[i] = 0.0;
        for (int b0 = split_i; b0 < a.nbat; b0 += 32 * a.sp_nsplit) {
            float4 bs = make_float4(INFINITY, -INFINITY, 0.f, 0.f);
            if (b0 + lane * a.sp_nsplit < a.nbat) bs = bsum[b0 + lane * a.sp_nsplit];
            const int cls_l = batch_class(a, g, bs);
            const bool want = pass == 0 ? cls_l == 2 : (cls_l != 2 || (lowbins && bs.x <= xlow));
            unsigned hits = __ballot_sync(0xffffffffu, want && !(bs.y < xlo || bs.x > xhi));
            while (hits) {
                const int bl = __ffs(hits) - 1;
                hits &= hits - 1;
                const int cls = __shfl_sync(0xffffffffu, cls_l, bl), b = b0 + bl * a.sp_nsplit;
                if (cls == 0) {
                    for (int k = b * 32; k < min(a.K, b * 32 + 32); ++k) {
                        const double* c = colrec<double>(a, t, g, k);
                        if (c[F_XMAX] < (double)xlo || c[F_XMIN] > (double)xhi) continue;
                        if (!vM) continue;
                        const double v = native_value<RES>(a, t, g, k, c, j) * SPEC_SCALE;
#pragma unroll
                        for (int i = 0; i < SPW; ++i)
                            if (s0 + i < a.S) acc[i] = fma(v, a.Sd[(long long)(s0 + i) * a.K + k], acc[i]);
                    }
                    __syncwarp();
                    continue;
                }
                for (unsigned m = a.sp_heavy[b]; m; m &= m - 1) {   // lines, in FP64 (their S' is 0 in the table)
                    const int k = b * 32 + __ffs(m) - 1;
                    double v = 0.0;
                    if (pass == 0) v = centre_density<RES>(prec[k], tr, pw, join(ah, al), RES == 0 ? 0.0 : join(Dh, Dl));
                    else if (vM && (cls != 2 || j < ju)) v = native_value<RES>(a, t, g, k, colrec<double>(a, t, g, k), j);
                    v *= SPEC_SCALE;
#pragma unroll
                    for (int i = 0; i < SPW; ++i)
                        if (s0 + i < a.S) acc[i] = fma(v, a.Sd[(long long)(s0 + i) * a.K + k], acc[i]);
                }
                {
                    double dl, y;
                    const ColTerms o = column_terms<RES>(prec[b * 32 + lane], tr, pw, dl, y);
                    srec[lane * 2] = make_float4(o.E.x, o.E.y, o.g.x, o.g.y);
                    srec[lane * 2 + 1] = make_float4(o.P.x, o.P.y, __int_as_float(o.nb), 0.f);
                    const float4* src = reinterpret_cast<const float4*>(a.Sp) + ((long long)b * 32 * Spad + s0) / 2;
                    for (int i = lane; i < 32 * SPW / 2; i += 32) ssp[i] = src[(long long)(i / (SPW / 2)) * (Spad / 2) + i % (SPW / 2)];
                    if constexpr (RES == 0) {   // the Gaussian's norm goes to the spectra
                        __syncwarp();
                        const float2 nn = split(prec[b * 32 + lane].B * INV_SQRT2PI);
#pragma unroll
                        for (int i = 0; i < SPW / 2; ++i) {
                            const float4 q = ssp[lane * (SPW / 2) + i];
                            float4 o2;
                            mul_pair(q.x, q.y, nn.x, nn.y, o2.x, o2.y);
                            mul_pair(q.z, q.w, nn.x, nn.y, o2.z, o2.w);
                            ssp[lane * (SPW / 2) + i] = o2;
                        }
                    }
                }
                __syncwarp();
                float sh[SPW], sl[SPW];
#pragma unroll
                for (int i = 0; i < SPW; ++i) sh[i] = sl[i] = 0.f;
                auto terms = [&](int ci) {
                    const float4 q0 = srec[ci * 2], q1 = srec[ci * 2 + 1];
                    return ColTerms{make_float2(q0.x, q0.y), make_float2(q0.z, q0.w), make_float2(q1.x, q1.y), __float_as_int(q1.z)};
                };
                auto add = [&](int ci, float vh, float vl) {
#pragma unroll
                    for (int i = 0; i < SPW / 2; ++i) {
                        const float4 q = ssp[ci * (SPW / 2) + i];
                        float p, e;
                        mul_pair(vh, vl, q.x, q.y, p, e);
                        acc_pair(sh[2 * i], sl[2 * i], p, e);
                        mul_pair(vh, vl, q.z, q.w, p, e);
                        acc_pair(sh[2 * i + 1], sl[2 * i + 1], p, e);
                    }
                };
                if (pass == 0) {
                    for (int ci = 0; ci < 32; ++ci) {
                        float xh = ah, xl = al, yh = Dh, yl = Dl, vh, vl;
                        pair_density<RES, true>(terms(ci), xh, xl, yh, yl, tab, vh, vl);
                        add(ci, vh, vl);
                    }
                } else {
                    if (nq < 0) {
                        const int nb = tb_g_node_off(a, g) + min(j, J - 1);
                        const int mine = vM ? (int)a.qn[nb] : 0;
                        nq = (__reduce_max_sync(0xffffffffu, mine) + NU - 1) / NU * NU;
                        for (int n = 0; n < nq; ++n) {
                            const float2* q = reinterpret_cast<const float2*>(a.qnode) + ((long long)nb * NGM_D + n) * 3;
                            float2 qa = make_float2(0.f, 0.f), qd = qa, qw = qa;
                            if (n < mine) { qa = q[0]; qd = q[1]; qw = q[2]; }
                            if constexpr (RES == 2) qd = split(gg_Q_d(pw * join(qa.x, qa.y)));
                            sq[(n * 3) * 32] = qa; sq[(n * 3 + 1) * 32] = qd; sq[(n * 3 + 2) * 32] = qw;
                        }
                    }
                    for (int ci = 0; ci < 32; ++ci) {
                        const ColTerms c = terms(ci);
                        float uh = 0.f, ul = 0.f;
                        for (int n0 = 0; n0 < nq; n0 += NU) {
#pragma unroll
                            for (int n = n0; n < n0 + NU; ++n) {
                                float2 qa = sq[(n * 3) * 32], qd = sq[(n * 3 + 1) * 32];
                                const float2 qw = sq[(n * 3 + 2) * 32];
                                float vh, vl, p, e;
                                pair_density<RES, true>(c, qa.x, qa.y, qd.x, qd.y, tab, vh, vl);
                                mul_pair(vh, vl, qw.x, qw.y, p, e);
                                acc_pair(uh, ul, p, e);
                            }
                        }
                        if (zero && lane == 0) {
                            const int k = b * 32 + ci;
                            const float2 z = k < a.K ? split(zerorec<double>(a, t, g, k)[Z_P0]) : make_float2(0.f, 0.f);
                            uh = z.x; ul = z.y;
                        }
                        add(ci, uh, ul);
                    }
                }
                if (pass == 0 || cls != 2 || j < ju) {
#pragma unroll
                    for (int i = 0; i < SPW; ++i) acc[i] += join(sh[i], sl[i]);
                }
                __syncwarp();
            }
        }
        if (pass == 0 ? vF : vM) {
#pragma unroll
            for (int i = 0; i < SPW; ++i)
                if (s0 + i < a.S) out[((long long)(s0 + i) * 2 + pass) * (a.Jmax + FM) + j] = acc[i];
        }
    }
}

// grid (strips of 256 bins, groups x species, toys)
__global__ void __launch_bounds__(256) k_species_reduce(KArgs a) {
    const int g = blockIdx.y / a.sp_count, s = a.sp_first + blockIdx.y % a.sp_count, t = blockIdx.z;
    if (!tb_g_active(a, g)) return;
    __shared__ double fs[256 + 2 * FM];
    const int J = tb_g_bins(a, g), ju = a.tb->g_ju[g], Jp = a.Jmax + FM;
    const int j0 = blockIdx.x * 256, j = j0 + threadIdx.x;
    if (j0 >= J) return;
    const long long step = (long long)a.S * 2 * Jp;
    const double* row = a.sp_part + (((long long)t * a.G + g) * a.sp_nsplit) * step + (long long)s * 2 * Jp;
    if (ju < J) {
        for (int i = threadIdx.x; i < 256 + 2 * FM; i += 256) {
            const int n = j0 - FM + i;
            double v = 0.0;
            if (n >= ju - FM && n < J + FM)
                for (int q = 0; q < a.sp_nsplit; ++q) v += row[q * step + n];
            fs[i] = v;
        }
        __syncthreads();
    }
    if (j >= J) return;
    double v = 0.0;
    for (int q = 0; q < a.sp_nsplit; ++q) v += row[q * step + Jp + j];
    if (j >= ju) {
        const double* f = fs + threadIdx.x + FM;
        if (f[0] != 0.0) {
            const double* ed = a.edges + tb_g_edge_off(a, g);
            double w = 0.0;
#pragma unroll
            for (int m = FM; m > 0; --m) w = fma(a.conv[m], f[-m] + f[m], w);
            v = fma(fma(a.conv[0], f[0], w), ed[j + 1] - ed[j], v);
        }
    }
    a.Mbuf[(long long)t * a.mstride + ((long long)g * a.S + s) * a.Jmax + j] = v * (1.0 / SPEC_SCALE);
}

// ------------------------------------------------------------ launchers ----
namespace {

// dynamic shared memory above 48 KB: asked for before every launch
template <class K>
cudaError_t allow_smem(K kernel, size_t bytes) {
    return bytes > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) : cudaSuccess;
}

template <int RES, int NDS>
cudaError_t launch_fp(const KArgs& a, cudaStream_t st) {
    const size_t sm = 8192 + (sizeof(FwdRec<NDS>) * 32 + sizeof(float2) * NGM_D * 3 * 32) * PW;
    cudaError_t e = allow_smem(k_forward_p<RES, NDS>, sm);
    if (e != cudaSuccess) return e;
    k_forward_p<RES, NDS><<<dim3(a.ntile, a.nsplit, a.T * a.G), PW * 32, sm, st>>>(a);
    return cudaGetLastError();
}
template <int RES, int NDS>
cudaError_t launch_bp(const KArgs& a, cudaStream_t st) {
    const int W = a.bw_warps;
    const size_t sm = 8192 + sizeof(float4) * 32 * (1 + (NDS + 1) / 2) * W + sizeof(double) * (NDS * W * 32 + W * NRESP);
    cudaError_t e = allow_smem(k_backward_p<RES, NDS>, sm);
    if (e != cudaSuccess) return e;
    k_backward_p<RES, NDS><<<dim3(a.nbtask, a.G, a.T), W * 32, sm, st>>>(a);
    return cudaGetLastError();
}
template <int RES>
cudaError_t fwd_nds(const KArgs& a, cudaStream_t st) {
    return a.max_nds <= 1 ? launch_fp<RES, 1>(a, st) : a.max_nds == 2 ? launch_fp<RES, 2>(a, st) : launch_fp<RES, 4>(a, st);
}
template <int RES>
cudaError_t bwd_nds(const KArgs& a, cudaStream_t st) {
    return a.max_nds <= 1 ? launch_bp<RES, 1>(a, st) : a.max_nds == 2 ? launch_bp<RES, 2>(a, st) : launch_bp<RES, 4>(a, st);
}

}  // namespace

cudaError_t launch_forward_pair(const KArgs& a, cudaStream_t st) {
    return a.res == 0 ? fwd_nds<0>(a, st) : a.res == 1 ? fwd_nds<1>(a, st) : fwd_nds<2>(a, st);
}

cudaError_t launch_backward_pair(const KArgs& a, cudaStream_t st) {
    k_wfilter<<<dim3(a.T, (a.fext + 255) / 256), 256, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return a.res == 0 ? bwd_nds<0>(a, st) : a.res == 1 ? bwd_nds<1>(a, st) : bwd_nds<2>(a, st);
}

cudaError_t launch_species_pair(const KArgs& a, cudaStream_t st) {
    const int nchunk = (a.sp_count + SPW - 1) / SPW;
    const size_t sm = 8192 + SPB * (1024 + 32 * SPW * 8 + sizeof(float2) * NGM_D * 3 * 32);
    const int ntile = (a.Jmax + FM + 31) / 32;
    const dim3 grid((ntile + SPB - 1) / SPB, a.G, a.T * nchunk * a.sp_nsplit);
    cudaError_t e;
    if (a.res == 0) { if ((e = allow_smem(k_species_p<0>, sm))) return e; k_species_p<0><<<grid, SPB * 32, sm, st>>>(a); }
    else if (a.res == 1) { if ((e = allow_smem(k_species_p<1>, sm))) return e; k_species_p<1><<<grid, SPB * 32, sm, st>>>(a); }
    else { if ((e = allow_smem(k_species_p<2>, sm))) return e; k_species_p<2><<<grid, SPB * 32, sm, st>>>(a); }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_species_reduce<<<dim3((a.Jmax + 255) / 256, a.G * a.sp_count, a.T), 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace gsn
