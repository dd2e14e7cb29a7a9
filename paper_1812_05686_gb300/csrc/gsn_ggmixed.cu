// Mixed-precision kernels of the free-power generalized gamma on linear bins (3-node rule), two bins per
// packed FP32 instruction (fma / add / mul .rn.f32x2).
//
// The general per-node kernels read every column (forward) or bin (adjoint) from global memory inside
// their inner loop and evaluated one pair per instruction: 258 and 289 cycles per 32 pairs where the
// arithmetic needs about 60.  Here the records (forward) and the bins' node tables with their side-node
// terms (adjoint) are staged in shared memory, lanes hold two bins (forward: j and j + 32, two of the
// general kernel's tiles) or take two bins of the batch at a time (adjoint), and the value is
// straight-line code where every lane's ln(1+t) and e^q - 1 - q are in their series' ranges (|q| <= 1/2,
// or 2 with the doublings); elsewhere, and in bins of the general node table, one pair at a time as before.  Every operation, the
// order of every sum and the columns that each 32-bin tile takes are those of the general kernels.
// 1024 toys of 2 x 1200 bins x 20000 columns: forward 36.9 -> 14.4 ms, adjoint 38.1 -> 17.6 ms.
#include "gsn_device.cuh"
#include "gsn_ggamma.cuh"

#include <type_traits>

namespace gsn {

// Resident blocks per SM and pairs in flight: four blocks (64 registers, 50-280 bytes spilled) without
// unrolling ran best: 16.8 / 17.6 ms against 17.3 / 18.7 with three, 17.1 / 19.0 with three and two in
// flight, 17.3 / 17.4 with five (forward / adjoint).
#ifndef GSN_GGF_MINBLOCKS
#define GSN_GGF_MINBLOCKS 4
#endif
#ifndef GSN_GGB_MINBLOCKS
#define GSN_GGB_MINBLOCKS 4
#endif
#ifndef GSN_GGF_UNROLL
#define GSN_GGF_UNROLL 1
#endif
#ifndef GSN_GGB_UNROLL
#define GSN_GGB_UNROLL 1
#endif
constexpr int GGF_UNROLL = GSN_GGF_UNROLL, GGB_UNROLL = GSN_GGB_UNROLL;

namespace {

DEV float2 f2(float x) { return make_float2(x, x); }
DEV float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
DEV float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
DEV float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
DEV float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
DEV float2 ex2f2(float2 x) { return make_float2(ex2f(x.x), ex2f(x.y)); }

// ln(1 + t) as log1pmx2_f gives it for t in [-1/2, 1] (D(t) + t, D by its series)
DEV float2 ln1p2(float2 t) {
    const float2 x = add2(f2(2.0f), t);
    float2 r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(x.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(x.y));
    r = fma2(fma2(neg2(x), r, f2(1.0f)), r, r);
    const float2 u = mul2(t, r);
    const float2 v = mul2(u, u);
    float2 p = fma2(v, f2(1.0f / 15.0f), f2(1.0f / 13.0f));
    p = fma2(p, v, f2(1.0f / 11.0f));
    p = fma2(p, v, f2(1.0f / 9.0f));
    p = fma2(p, v, f2(1.0f / 7.0f));
    p = fma2(p, v, f2(1.0f / 5.0f));
    p = fma2(p, v, f2(1.0f / 3.0f));
    const float2 D = fma2(mul2(add2(u, u), v), p, mul2(neg2(t), u));
    return add2(D, t);
}
// Q = e^q - 1 - q and e1 = e^q - 1 as gg_q2f gives them for |q| <= 1/2
DEV float2 q2series2(float2 q, float2& e1) {
    float2 s = fma2(q, f2(1.0f / 3628800), f2(1.0f / 362880));
    s = fma2(s, q, f2(1.0f / 40320));
    s = fma2(s, q, f2(1.0f / 5040));
    s = fma2(s, q, f2(1.0f / 720));
    s = fma2(s, q, f2(1.0f / 120));
    s = fma2(s, q, f2(1.0f / 24));
    s = fma2(s, q, f2(1.0f / 6));
    s = fma2(s, q, f2(0.5f));
    const float2 h = mul2(q, q), Q = mul2(h, s);
    e1 = add2(q, Q);
    return Q;
}
// the same for |q| <= 2: beyond 1/2 the series at q / 4 and two doublings
DEV float2 q2mid2(float2 q, float2& e1) {
    float2 es, E;
    const float2 Qs = q2series2(q, es);
    float2 Q = q2series2(mul2(q, f2(0.25f)), E);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        Q = fma2(E, E, add2(Q, Q));
        E = fma2(E, E, add2(E, E));
    }
    const bool sx = fabsf(q.x) <= 0.5f, sy = fabsf(q.y) <= 0.5f;
    e1 = make_float2(sx ? es.x : E.x, sy ? es.y : E.y);
    return make_float2(sx ? Qs.x : Q.x, sy ? Qs.y : Q.y);
}
template <bool MID> DEV float2 q2(float2 q, float2& e1) { return MID ? q2mid2(q, e1) : q2series2(q, e1); }
// x in [x0, x1], mean in [m0, m1] (all > 0): ln(1 + t) and q = p ln(x/mu) within the series' ranges for
// every one of them (a margin covers the roundings of t and q)
// 2: |q| <= 1/2 for all, 1: |q| <= 2, 0: not all within the ranges
DEV int in_series(float x0, float x1, float m0, float m1, float p) {
    const float ta = (x0 - m1) / m1, tb = (x1 - m0) / m0;   // smallest and largest t
    if (!(ta >= -0.49f && tb <= 0.98f)) return 0;
    const float q = p * fmaxf(log1pf(tb), -log1pf(ta));
    return q <= 0.49f ? 2 : q <= 1.95f ? 1 : 0;
}
DEV bool in_ln(float2 t) { return t.x >= -0.5f && t.x <= 1.0f && t.y >= -0.5f && t.y <= 1.0f; }
DEV bool in_q(float2 q, float m) { return fabsf(q.x) <= m && fabsf(q.y) <= m; }

}  // namespace

// ------------------------------------------------------------- forward -----
struct GGRec { float4 q0, q1, q2; };   // (mu_hi, mu_lo, A, A_p) (kappa_1, p, TN0, TN1) (TN2, TN3, -, -)

template <int NDS>
__global__ void __launch_bounds__(FWD_WARPS * 32, GSN_GGF_MINBLOCKS) k_forward_gg(KArgs a) {
    __shared__ GGRec srec[FWD_WARPS][32];
    const int split = blockIdx.y;
    const int t = blockIdx.z / a.G, g = blockIdx.z % a.G;
    if (!tb_g_active(a, g)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int wlo, whi;
    toy_window_union(a, t, g, wlo, whi);
    const int jw = (blockIdx.x * FWD_WARPS + warp) * 64;   // two tiles of 32 bins
    bool use[2], valid[2];
    float xlo[2], xhi[2], xc_[2], lam[2][3], wt[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j0 = jw + 32 * h, j = j0 + lane;
        use[h] = j0 < whi && j0 + 32 > wlo;
        valid[h] = use[h] && j >= wlo && j < whi;
        const int jr = min(max(j, wlo), max(whi - 1, wlo));
        const int nb = tb_g_node_off(a, g) + min(jr, tb_g_bins(a, g) - 1);
        if (use[h]) use[h] = !__any_sync(0xffffffffu, a.bclass[nb] != BIN_LIN);  // low tiles: k_forward_gg_low
        xlo[h] = INFINITY; xhi[h] = -INFINITY;
        if (use[h]) {
            xlo[h] = (float)a.edges[tb_g_edge_off(a, g) + max(j0, wlo)];
            xhi[h] = (float)a.edges[tb_g_edge_off(a, g) + min(j0 + 31, whi - 1) + 1];
        }
        const float* nodes = a.ntab_f + (long long)nb * 3 * NGM_F;
        xc_[h] = a.xc_f[nb];
#pragma unroll
        for (int n = 0; n < 3; ++n) { lam[h][n] = nodes[NGM_F + n]; wt[h][n] = valid[h] ? nodes[2 * NGM_F + n] : 0.f; }
    }
    if (!use[0] && !use[1]) return;
    const int q5 = tb_g_resp(a, g, 5);
    const float pw = (float)(a.params[(long long)t * a.params_stride + q5] * tb_g_rscale(a, g, 5));
    const float xmin = fminf(xlo[0], xlo[1]), xmax = fmaxf(xhi[0], xhi[1]);   // the used tiles' edges
    const GGSides sa = gg_sides(pw, lam[0]), sb = gg_sides(pw, lam[1]);
    const float2 xc = make_float2(xc_[0], xc_[1]), lam1 = make_float2(lam[0][1], lam[1][1]);
    const float2 dl0 = make_float2(sa.dlam0, sb.dlam0), dl2 = make_float2(sa.dlam2, sb.dlam2);
    const float2 Q0 = make_float2(sa.Q0, sb.Q0), Q2 = make_float2(sa.Q2, sb.Q2);
    const float2 E0 = make_float2(sa.E0, sb.E0), E2 = make_float2(sa.E2, sb.E2);
    const float2 w0 = make_float2(wt[0][0], wt[1][0]), w1 = make_float2(wt[0][1], wt[1][1]), w2 = make_float2(wt[0][2], wt[1][2]);
    const int kchunk = (a.K + a.nsplit - 1) / a.nsplit;
    const int k_beg = split * kchunk, k_end = min(a.K, k_beg + kchunk);
    const float* blk = reinterpret_cast<const float*>(a.blkbuf) + ((long long)t * a.G + g) * a.nblk * 2;
    const float4* rec = reinterpret_cast<const float4*>(colrec<float>(a, t, g, 0));
    double accd[2][NDS] = {};
    int ncol[2] = {0, 0};
    for (int b = k_beg / COLBLK; b * COLBLK < k_end; ++b) {
        bool hb[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) hb[h] = use[h] && !(blk[2 * b + 1] < xlo[h] || blk[2 * b] > xhi[h]);
        if (!hb[0] && !hb[1]) continue;
        float2 acc[NDS] = {};
        float s[2][NDS] = {}, cc[2][NDS] = {};
        const int kb = max(b * COLBLK, k_beg), ke = min((b + 1) * COLBLK, k_end);
        float4 r0, r1, r2, r3;
        auto load = [&](int k, int lim) {
            r2 = make_float4(INFINITY, -INFINITY, 0.f, 0.f);
            r0 = r1 = r3 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < lim) { const float4* p = rec + (long long)k * 4; r0 = p[0]; r1 = p[1]; r2 = p[2]; r3 = p[3]; }
        };
        // groups of columns that end where k is a multiple of 32: the sums are folded there
        int k0 = kb, k1 = min(ke, (kb | 31) + 1);
        load(k0 + lane, k1);
        for (; k0 < ke;) {
            const unsigned mA = __ballot_sync(0xffffffffu, hb[0] && !(r2.y < xlo[0] || r2.x > xhi[0]));
            const unsigned mB = __ballot_sync(0xffffffffu, hb[1] && !(r2.y < xlo[1] || r2.x > xhi[1]));
            const int rg = in_series(xmin, xmax, r0.x, r0.x, r1.z);
            const unsigned mF = __ballot_sync(0xffffffffu, rg == 2), mM = __ballot_sync(0xffffffffu, rg >= 1);
            __syncwarp();
            srec[warp][lane] = {r0, make_float4(r1.x, r1.z, r2.z, r2.w), make_float4(r3.x, r3.y, 0.f, 0.f)};
            __syncwarp();
            const int n0 = k1 - k0, last = n0 - 1;
            const bool endA = ((k1 - 1) & 31) == 31 && (mA >> last & 1), endB = ((k1 - 1) & 31) == 31 && (mB >> last & 1);
            k0 = k1;
            k1 = min(ke, k0 + 32);
            load(k0 + lane, k1);
            ncol[0] += __popc(mA); ncol[1] += __popc(mB);
            // straight-line value: every lane within the series' ranges
            auto value = [&](const GGRec& c, auto mid) -> float2 {
                const float2 Dx = add2(add2(xc, f2(-c.q0.x)), f2(-c.q0.y));
                const float2 L1 = add2(ln1p2(mul2(Dx, f2(c.q0.z))), lam1);
                float2 e1;
                const float2 Q = q2<decltype(mid)::value>(mul2(f2(c.q1.y), L1), e1);
                const float2 Ql = fma2(e1, E0, add2(Q, Q0)), Qr = fma2(e1, E2, add2(Q, Q2));
                const float2 nAp = f2(-c.q0.w), Kp = f2(c.q1.x);
                const float2 vl = ex2f2(fma2(nAp, Ql, mul2(Kp, add2(L1, dl0))));
                const float2 vc = ex2f2(fma2(nAp, Q, mul2(Kp, L1)));
                const float2 vr = ex2f2(fma2(nAp, Qr, mul2(Kp, add2(L1, dl2))));
                return fma2(w0, vl, fma2(w1, vc, mul2(w2, vr)));
            };
            // any arguments: a vote on the lanes' own, then one bin at a time
            auto general = [&](const GGRec& c) -> float2 {
                {
                    const float2 tt = mul2(add2(add2(xc, f2(-c.q0.x)), f2(-c.q0.y)), f2(c.q0.z));
                    if (__all_sync(0xffffffffu, in_ln(tt)) &&
                        __all_sync(0xffffffffu, in_q(mul2(f2(c.q1.y), add2(ln1p2(tt), lam1)), 2.0f)))
                        return value(c, std::true_type());
                }
                float v[2];
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const float Dx = ((h ? xc.y : xc.x) - c.q0.x) - c.q0.y;
                    float Lc;
                    log1pmx2_f(Dx * c.q0.z, Lc);
                    const float L1 = Lc + (h ? lam1.y : lam1.x);
                    float e1;
                    const float Q = gg_q2f(c.q1.y * L1, e1);
                    const float Ql = fmaf(e1, h ? E0.y : E0.x, Q + (h ? Q0.y : Q0.x)), Qr = fmaf(e1, h ? E2.y : E2.x, Q + (h ? Q2.y : Q2.x));
                    const float vl = ex2f(fmaf(-c.q0.w, Ql, c.q1.x * (L1 + (h ? dl0.y : dl0.x))));
                    const float vc = ex2f(fmaf(-c.q0.w, Q, c.q1.x * L1));
                    const float vr = ex2f(fmaf(-c.q0.w, Qr, c.q1.x * (L1 + (h ? dl2.y : dl2.x))));
                    const float r = fmaf(h ? w0.y : w0.x, vl, fmaf(h ? w1.y : w1.x, vc, (h ? w2.y : w2.x) * vr));
                    if (h) v[1] = r; else v[0] = r;
                }
                return make_float2(v[0], v[1]);
            };
            auto tn = [&](const GGRec& c, int dd) { return dd == 0 ? c.q1.z : dd == 1 ? c.q1.w : dd == 2 ? c.q2.x : c.q2.y; };
            if ((mA & mB & mM) == 0xffffffffu) {
                auto dense = [&](auto mid) {
#pragma unroll GGF_UNROLL
                    for (int ci = 0; ci < 32; ++ci) {
                        const GGRec c = srec[warp][ci];
                        const float2 v = value(c, mid);
#pragma unroll
                        for (int dd = 0; dd < NDS; ++dd) acc[dd] = fma2(v, f2(tn(c, dd)), acc[dd]);
                    }
                };
                if (mF == 0xffffffffu) dense(std::false_type()); else dense(std::true_type());
            } else {
                for (unsigned m = mA | mB; m; m &= m - 1) {
                    const int ci = __ffs(m) - 1;
                    const GGRec c = srec[warp][ci];
                    const float2 v = mF >> ci & 1 ? value(c, std::false_type()) : general(c);
                    const bool hA = mA >> ci & 1, hB = mB >> ci & 1;
#pragma unroll
                    for (int dd = 0; dd < NDS; ++dd) {
                        const float T = tn(c, dd);
                        if (hA) acc[dd].x = fmaf(v.x, T, acc[dd].x);
                        if (hB) acc[dd].y = fmaf(v.y, T, acc[dd].y);
                    }
                }
            }
#pragma unroll
            for (int dd = 0; dd < NDS; ++dd) {
                if (endA) { two_sum_acc(s[0][dd], cc[0][dd], acc[dd].x); acc[dd].x = 0.f; }
                if (endB) { two_sum_acc(s[1][dd], cc[1][dd], acc[dd].y); acc[dd].y = 0.f; }
            }
        }
#pragma unroll
        for (int dd = 0; dd < NDS; ++dd) {
            two_sum_acc(s[0][dd], cc[0][dd], acc[dd].x);
            two_sum_acc(s[1][dd], cc[1][dd], acc[dd].y);
            accd[0][dd] += (double)s[0][dd] + (double)cc[0][dd];
            accd[1][dd] += (double)s[1][dd] + (double)cc[1][dd];
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (a.work) {
            const unsigned m = __ballot_sync(0xffffffffu, use[h] && valid[h]);
            if (lane == 0) atomicAdd(&a.work[K_FORWARD], (unsigned long long)ncol[h] * __popc(m));
        }
        if (!use[h] || !valid[h]) continue;
        double* out = a.mubuf + ((long long)t * a.nsplit + split) * a.total_bins + jw + 32 * h + lane;
#pragma unroll
        for (int dd = 0; dd < NDS; ++dd)
            if (dd < tb_g_nds(a, g)) out[tb_ds_off(a, tb_g_ds(a, g, dd))] = accd[h][dd];
    }
}

// ------------------------------------------------------------ backward -----
// lanes <-> columns.  Staged per pair of bins (2p, 2p + 1) of a batch of 32, both bins of every quantity:
//   xc, lam1 | dlam0, dlam2 | w0, w1 | w2, Q0 | E0, Q2 | E2, w_d0 | w_d1, w_d2 | w_d3, -
constexpr int GGB_V = 8;   // float4 per pair

template <int NDS>
__global__ void __launch_bounds__(256, GSN_GGB_MINBLOCKS) k_backward_gg(KArgs a) {
    const int task = blockIdx.x, g = blockIdx.y, t = blockIdx.z;
    if (!tb_g_active(a, g)) return;
    const int W = a.bw_warps;
    const int cbw = task / a.bw_bsplit, bsp = task % a.bw_bsplit;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kbase = cbw * W * 32;
    const int k = kbase + warp * 32 + lane;
    const bool kval = k < a.K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* sb = reinterpret_cast<float4*>(smem_raw) + warp * 16 * GGB_V;
    float* su = reinterpret_cast<float*>(smem_raw + sizeof(float4) * 16 * GGB_V * W);                       // [NDS][W*32]
    double* sresp = reinterpret_cast<double*>(smem_raw + sizeof(float4) * 16 * GGB_V * W + sizeof(float) * MAXGDS * W * 32);
    const int nds = tb_g_nds(a, g);
    const int J = tb_g_bins(a, g);
    const double* ed = a.edges + tb_g_edge_off(a, g);
    int wlo, whi;
    toy_window_union(a, t, g, wlo, whi);
    float c[NFP];
    {
        const float4* cr = reinterpret_cast<const float4*>(colrec<float>(a, t, g, kval ? k : a.K - 1));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = cr[i];
            c[4 * i] = v.x; c[4 * i + 1] = v.y; c[4 * i + 2] = v.z; c[4 * i + 3] = v.w;
        }
    }
    const float xmn = warp_min<float>(kval ? c[F_XMIN] : INFINITY);
    const float xmx = warp_max<float>(kval ? c[F_XMAX] : -INFINITY);
    int ja = 0, jb = -1;
    if (xmx >= xmn) {
        int lo = 0, hi = J;
        while (lo < hi) { const int m = (lo + hi) >> 1; if (ed[m + 1] <= (double)xmn) lo = m + 1; else hi = m; }
        ja = lo;
        lo = 0; hi = J;
        while (lo < hi) { const int m = (lo + hi) >> 1; if (ed[m] < (double)xmx) lo = m + 1; else hi = m; }
        jb = lo - 1;
        ja = max(ja, wlo); jb = min(jb, whi - 1);
        const int len = jb - ja + 1;
        if (len > 0) {
            const int ch = (len + a.bw_bsplit - 1) / a.bw_bsplit;
            const int na = ja + bsp * ch;
            jb = min(jb, na + ch - 1);
            ja = na;
        }
    }
    const float* wv[NDS];
#pragma unroll
    for (int dd = 0; dd < NDS; ++dd)
        wv[dd] = reinterpret_cast<const float*>(a.wbuf) + (long long)t * a.total_bins + tb_ds_off(a, tb_g_ds(a, g, dd < nds ? dd : 0));
    const int nbase = tb_g_node_off(a, g), jlin = tb_g_jlin(a, g);
    const float mumin = warp_min<float>(kval ? c[F_MUH] : INFINITY), mumax = warp_max<float>(kval ? c[F_MUH] : 0.f);
    const float p = c[F_KAPPA], A = c[F_A], Ap = c[F_B], Kp = c[F_C];
    const float nmuh = -c[F_MUH], nmul = -c[F_MUL];
    float T[NDS];
#pragma unroll
    for (int dd = 0; dd < NDS; ++dd) T[dd] = c[F_TN0 + dd];
    float Gs[4] = {0.f, 0.f, 0.f, 0.f}, Gc[4] = {0.f, 0.f, 0.f, 0.f}, U0[NDS] = {}, U0c[NDS] = {}, Z0 = 0.f;
    for (int jj0 = ja; jj0 <= jb; jj0 += 32) {
        const int nbat = min(32, jb - jj0 + 1);
        // stage the batch: one bin per lane (the last one again after an odd count)
        __syncwarp();
        {
            const int jj = min(jj0 + lane, jb);
            float v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = 0.f;
            if (a.bclass[nbase + jj] == BIN_LIN) {
                const float* nd = a.ntab_f + (long long)(nbase + jj) * 3 * NGM_F;
                v[0] = a.xc_f[nbase + jj];
                v[1] = nd[NGM_F + 1];
                v[2] = nd[NGM_F] - nd[NGM_F + 1];
                v[3] = nd[NGM_F + 2] - nd[NGM_F + 1];
                v[4] = nd[2 * NGM_F]; v[5] = nd[2 * NGM_F + 1]; v[6] = nd[2 * NGM_F + 2];
                v[7] = gg_q2f(p * v[2], v[8]);
                v[9] = gg_q2f(p * v[3], v[10]);
            }
            {
#pragma unroll
                for (int dd = 0; dd < NDS; ++dd) v[11 + dd] = dd < nds ? wv[dd][jj] : 0.f;
            }
            float* o = reinterpret_cast<float*>(sb + (lane >> 1) * GGB_V) + (lane & 1);
#pragma unroll
            for (int i = 0; i < 11 + NDS; ++i) o[2 * i] = v[i];
        }
        __syncwarp();
        float bG[4] = {0.f, 0.f, 0.f, 0.f}, bU[NDS] = {};
        auto accumulate = [&](const float* w, float rho, float s1, float s2, float s3, bool zero) {
            float Wj = w[0] * T[0];
#pragma unroll
            for (int dd = 1; dd < NDS; ++dd) Wj = fmaf(w[dd], T[dd], Wj);
            if (zero) {
                Z0 += Wj;
            } else {
                bG[0] = fmaf(Wj, rho, bG[0]); bG[1] = fmaf(Wj, s1, bG[1]);
                bG[2] = fmaf(Wj, s2, bG[2]); bG[3] = fmaf(Wj, s3, bG[3]);
            }
#pragma unroll
            for (int dd = 0; dd < NDS; ++dd) bU[dd] = fmaf(w[dd], rho, bU[dd]);
        };
        // one bin at a time: bins of the general node table, arguments outside the series' ranges
        auto single = [&](int i) {
            const float* S = reinterpret_cast<const float*>(sb + (i >> 1) * GGB_V) + (i & 1);
            const int j = jj0 + i;
            float w[NDS];
#pragma unroll
            for (int dd = 0; dd < NDS; ++dd) w[dd] = S[2 * (11 + dd)];
            const unsigned char cls = a.bclass[nbase + j];
            float rho = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
            if (cls == BIN_ZERO) {
                rho = zerorec<float>(a, t, g, kval ? k : a.K - 1)[Z_P0];
            } else {
                const float* nd = a.ntab_f + (long long)(nbase + j) * 3 * NGM_F;
                const float Dx = (a.xc_f[nbase + j] + nmuh) + nmul;
                float Lc;
                log1pmx2_f(Dx * A, Lc);
                if (cls == BIN_LIN) {
                    const float L1 = Lc + nd[NGM_F + 1];
                    float e1;
                    const float Qc = gg_q2f(p * L1, e1);
                    const float Ln[3] = {L1 + S[4], L1, L1 + S[6]};
                    const float Qn[3] = {fmaf(e1, S[16], Qc + S[14]), Qc, fmaf(e1, S[20], Qc + S[18])};
                    const float En[3] = {fmaf(e1, S[16], e1 + S[16]), e1, fmaf(e1, S[20], e1 + S[20])};
#pragma unroll
                    for (int n = 0; n < 3; ++n) {
                        const float fw = nd[2 * NGM_F + n] * ex2f(fmaf(-Ap, Qn[n], Kp * Ln[n]));
                        rho += fw; s1 = fmaf(fw, Ln[n], s1); s2 = fmaf(fw, Qn[n], s2); s3 = fmaf(fw * En[n], Ln[n], s3);
                    }
                } else {
                    for (int n = 0; n < NG_LOG_F; ++n) {
                        const float L = Lc + nd[NGM_F + n];
                        float e1;
                        const float Q = gg_q2f(p * L, e1);
                        const float fw = nd[2 * NGM_F + n] * ex2f(fmaf(-Ap, Q, Kp * L));
                        rho += fw; s1 = fmaf(fw, L, s1); s2 = fmaf(fw, Q, s2); s3 = fmaf(fw * e1, L, s3);
                    }
                }
            }
            accumulate(w, rho, s1, s2, s3, cls == BIN_ZERO);
        };
        // two bins at once, straight-line
        auto both = [&](const float4* P, bool second, auto mid) {
            const float4 X0 = P[0], X1 = P[1], X2 = P[2], X3 = P[3], X4 = P[4], X5 = P[5];
            const float2 Dx = add2(add2(make_float2(X0.x, X0.y), f2(nmuh)), f2(nmul));
            const float2 L1 = add2(ln1p2(mul2(Dx, f2(A))), make_float2(X0.z, X0.w));
            float2 e1;
            const float2 Qc = q2<decltype(mid)::value>(mul2(f2(p), L1), e1);
            const float2 Q0 = make_float2(X3.z, X3.w), E0 = make_float2(X4.x, X4.y), Q2 = make_float2(X4.z, X4.w),
                         E2 = make_float2(X5.x, X5.y);
            const float2 La = add2(L1, make_float2(X1.x, X1.y)), Lb = add2(L1, make_float2(X1.z, X1.w));
            const float2 Qa = fma2(e1, E0, add2(Qc, Q0)), Qb = fma2(e1, E2, add2(Qc, Q2));
            const float2 Ea = fma2(e1, E0, add2(e1, E0)), Eb = fma2(e1, E2, add2(e1, E2));
            const float2 nAp = f2(-Ap), Kv = f2(Kp);
            const float2 xa = ex2f2(fma2(nAp, Qa, mul2(Kv, La)));
            const float2 xm = ex2f2(fma2(nAp, Qc, mul2(Kv, L1)));
            const float2 xb = ex2f2(fma2(nAp, Qb, mul2(Kv, Lb)));
            const float2 w0 = make_float2(X2.x, X2.y), w1 = make_float2(X2.z, X2.w), w2 = make_float2(X3.x, X3.y);
            const float2 fa = mul2(w0, xa), fm = mul2(w1, xm), fb = mul2(w2, xb);
            const float2 rho = add2(add2(fa, fm), fb);
            const float2 s1 = fma2(fb, Lb, fma2(fm, L1, mul2(fa, La)));
            const float2 s2 = fma2(fb, Qb, fma2(fm, Qc, mul2(fa, Qa)));
            const float2 s3 = fma2(mul2(fb, Eb), Lb, fma2(mul2(fm, e1), L1, mul2(mul2(fa, Ea), La)));
            const float4 X6 = NDS > 1 ? P[6] : X5, X7 = NDS > 3 ? P[7] : X5;
            const float wa[4] = {X5.z, X6.x, X6.z, X7.x}, wb[4] = {X5.w, X6.y, X6.w, X7.y};
            accumulate(wa, rho.x, s1.x, s2.x, s3.x, false);
            if (second) accumulate(wb, rho.y, s1.y, s2.y, s3.y, false);
        };
        const bool linear = jj0 >= jlin;   // every bin of the batch
        const int rg = linear ? in_series((float)ed[jj0], (float)ed[jj0 + nbat], mumin, mumax, p) : 0;
        if (rg) {
            auto dense = [&](auto mid) {
#pragma unroll GGB_UNROLL
                for (int i = 0; i + 1 < nbat; i += 2) both(sb + (i >> 1) * GGB_V, true, mid);
                if (nbat & 1) both(sb + (nbat >> 1) * GGB_V, false, mid);   // its second bin is the copy staged beside it
            };
            if (rg == 2) dense(std::false_type()); else dense(std::true_type());
        } else {
            // part of the batch outside: a vote per pair of bins, then one bin at a time
#pragma unroll 1
            for (int i = 0; i < nbat; i += 2) {
                const float4* P = sb + (i >> 1) * GGB_V;
                const float4 X0 = P[0];
                const float2 tt = mul2(add2(add2(make_float2(X0.x, X0.y), f2(nmuh)), f2(nmul)), f2(A));
                const bool second = i + 1 < nbat;
                if (jj0 + i >= jlin && __all_sync(0xffffffffu, in_ln(tt)) &&
                    __all_sync(0xffffffffu, in_q(mul2(f2(p), add2(ln1p2(tt), make_float2(X0.z, X0.w))), 2.0f))) {
                    both(P, second, std::true_type());
                } else {
                    single(i);
                    if (second) single(i + 1);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) two_sum_acc(Gs[i], Gc[i], bG[i]);
#pragma unroll
        for (int dd = 0; dd < NDS; ++dd) two_sum_acc(U0[dd], U0c[dd], bU[dd]);
    }
    if (a.work) {
        const unsigned m = __ballot_sync(0xffffffffu, kval);
        if (lane == 0 && jb >= ja) atomicAdd(&a.work[K_BACKWARD], (unsigned long long)(jb - ja + 1) * __popc(m));
    }
    // chain rule per column: FP64 combination of the compensated sums with the FP64 coefficients
    const double* prm = a.params + (long long)t * a.params_stride;
    const double LY = prm[tb_g_resp(a, g, 0)] * tb_g_rscale(a, g, 0);
    const double rb = prm[tb_g_resp(a, g, 3)] * tb_g_rscale(a, g, 3), rc = prm[tb_g_resp(a, g, 4)] * tb_g_rscale(a, g, 4);
    float r[NRESP] = {};
    if (kval) {
        const float mu = c[F_MUH] + c[F_MUL];
        const double* g2 = a.colbuf2 + (((long long)t * a.G + g) * a.K + k) * NFG;
        const double U[5] = {(double)Gs[0] + (double)Gc[0], (double)Gs[1] + (double)Gc[1], (double)Gs[2] + (double)Gc[2],
                             (double)Gs[3] + (double)Gc[3], (double)Z0};
        double gm = 0.0, gv = 0.0, gp = 0.0;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            gm = fma(g2[FG_MU + i], U[i], gm);
            gv = fma(g2[FG_VAR + i], U[i], gv);
            gp = fma(g2[FG_P + i], U[i], gp);
        }
        const float g_mu = (float)gm, g_var = (float)gv;
        r[5] = (float)gp;
        const float g_mt = g_mu + g_var * ((float)rb + 2.0f * (float)rc * mu);
        r[0] = g_mt * (mu / (float)LY);
        r[1] = g_mt * (float)LY * c[F_DEQ];
        r[2] = g_var;
        r[3] = g_var * mu;
        r[4] = g_var * mu * mu;
    }
#pragma unroll
    for (int i = 0; i < NRESP; ++i) {
        const float v = warp_sum_comp(r[i], 0.f);
        if (lane == 0) sresp[warp * NRESP + i] = (double)v;
    }
#pragma unroll
    for (int dd = 0; dd < MAXGDS; ++dd)
        su[dd * W * 32 + warp * 32 + lane] = kval && dd < NDS ? (U0[dd < NDS ? dd : 0] + U0c[dd < NDS ? dd : 0]) * c[F_N] : 0.f;
    __syncthreads();
    double* part = a.partbuf + (((long long)t * a.G + g) * a.nbtask + task) * a.NPART;
    if (threadIdx.x < NRESP) {
        double s = 0.0;
        for (int w = 0; w < W; ++w) s += sresp[w * NRESP + threadIdx.x];
        part[threadIdx.x] = s;
    }
    const int ncol = min(W * 32, a.K - kbase);
    for (int i = threadIdx.x; i < MAXGDS * a.S; i += blockDim.x) {
        const int dd = i / a.S, s = i % a.S;
        double v = 0.0;
        if (dd < nds && a.ft.sp_kind[s] < 2 && a.rfac[tb_g_ds(a, g, dd) * a.S + s] != 0.0) {
            const float* Srow = a.Sf + (long long)s * a.K + kbase;
            float acc = 0.f, cmp = 0.f, part32 = 0.f;
            for (int cc = 0; cc < ncol; ++cc) {
                part32 = fmaf(Srow[cc], su[dd * W * 32 + cc], part32);
                if ((cc & 31) == 31) { two_sum_acc(acc, cmp, part32); part32 = 0.f; }
            }
            two_sum_acc(acc, cmp, part32);
            v = (double)(acc + cmp);
        }
        part[NRESP + i] = v;
    }
}

// ------------------------------------------------------------ launchers ----
cudaError_t launch_forward_gg(const KArgs& a, cudaStream_t st) {
    const dim3 grid((a.Jmax + FWD_WARPS * 64 - 1) / (FWD_WARPS * 64), a.nsplit, a.T * a.G);
    if (a.max_nds <= 1) k_forward_gg<1><<<grid, FWD_WARPS * 32, 0, st>>>(a);
    else if (a.max_nds == 2) k_forward_gg<2><<<grid, FWD_WARPS * 32, 0, st>>>(a);
    else k_forward_gg<4><<<grid, FWD_WARPS * 32, 0, st>>>(a);
    return cudaGetLastError();
}
cudaError_t launch_backward_gg(const KArgs& a, cudaStream_t st) {
    const dim3 grid(a.nbtask, a.G, a.T);
    const int W = a.bw_warps;
    const size_t sm = sizeof(float4) * 16 * GGB_V * W + sizeof(float) * MAXGDS * W * 32 + sizeof(double) * W * NRESP;
    if (a.max_nds <= 1) k_backward_gg<1><<<grid, W * 32, sm, st>>>(a);
    else if (a.max_nds == 2) k_backward_gg<2><<<grid, W * 32, sm, st>>>(a);
    else k_backward_gg<4><<<grid, W * 32, sm, st>>>(a);
    return cudaGetLastError();
}

}  // namespace gsn
