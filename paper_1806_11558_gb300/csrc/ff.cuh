// ff.cuh -- double-float ("float-float") arithmetic for far-field kernel
// evaluations.
//
// On GB300 the FP64 pipe issues 2 DFMA per SM per clock against 128 FFMA, so
// the batched ACA (Sec. 2.3), whose entries are far-field (admissible blocks,
// well-separated panels), evaluates the 7x7 quadrature sum with pairs of
// floats carrying about 48 significant bits:
//   * Knuth's TwoSum and the FMA-based TwoProduct (Dekker's exact product)
//     give the rounding errors of a + b and a * b exactly;
//   * the reciprocal square root starts from the hardware estimate rsqrtf and
//     takes one step of second order whose residual 1 - r y0^2 is formed from
//     exact products, so the result is accurate to ~1e-14 relative;
//   * sums of positive terms carry their low parts separately and are
//     normalised once at the end.
// Differences of points are taken relative to the panel centroids, so the
// representation error of a coordinate is relative to the panel size, not to
// the distance from the origin; that also holds for neighbouring panels, so
// the regular near-field entries (non-touching pairs of dense leaves) use the
// same evaluation.
#pragma once

#include "hm_internal.cuh"

namespace hm {

// s + e == a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// s + e == a + b exactly, valid when |a| >= |b|
__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

// p + e == a * b exactly
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// (h, l) of a double: h = nearest float, l = nearest float of the remainder
__device__ __forceinline__ void split_double(double x, float &h, float &l) {
    h = __double2float_rn(x);
    l = __double2float_rn(x - (double)h);
}

// Float panel record of the regular entries (rows of the float panel table PF,
// component-major like the FP64 one).  The 7 points of the rule are the
// centroid c and two orbits of three, c + u_k and c + rho u_k (k = 0, 1, 2),
// with u_k = s (V_k - c) for the vertices V_k, u_0 + u_1 + u_2 = 0 and a
// constant rho, so the record holds c and the u_k instead of seven points:
//   [0, 9)   c as three floats (h, l and the rest): x, y, z of each
//   [9, 27)  u_0, u_1, u_2: (h x, y, z, l x, y, z) of each
//   [27, 33) |u_k|^2 (h, l);  [33, 39) rho^2 |u_k|^2 (h, l)
//   [39] max_k |u_k|, rounded up
//   [40] wa_hi, [41] wa_lo : |T| / sqrt(4 pi)
//   [42, 45) vertex indices (int bits)
constexpr int PF_ROWS = 45;
constexpr int PF_CH = 0, PF_CL = 3, PF_CM = 6, PF_U = 9, PF_N = 27, PF_N2 = 33, PF_RAD = 39, PF_WA = 40, PF_VID = 42;
// sqrt(4 pi)
constexpr double SQRT_4PI = 3.5449077018110320545963349666822903655950989122447742564276155;

// A float pair h + l (|l| <= ulp(h) / 2 when normalised).
struct __align__(8) FF {
    float h, l;
};

__device__ __forceinline__ FF ff_from(double x) {
    FF r;
    split_double(x, r.h, r.l);
    return r;
}
__device__ __forceinline__ double ff_to(FF a) { return (double)a.h + (double)a.l; }

// a * b, normalised, to ~2^-47 relative
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
    float ph, pe;
    two_prod(a.h, b.h, ph, pe);
    pe = __fmaf_rn(a.h, b.l, pe);
    pe = __fmaf_rn(a.l, b.h, pe);
    FF r;
    fast_two_sum(ph, pe, r.h, r.l);
    return r;
}

// (hs, lo) -= b * c: the high parts subtract exactly (TwoSum) and every
// rounding error goes to lo, so a chain of these followed by one
// fast_two_sum(hs, lo) is accurate to ~2^-48 of the largest term
__device__ __forceinline__ void ff_sub_prod(float &hs, float &lo, FF b, FF c) {
    float ph, pe;
    two_prod(b.h, c.h, ph, pe);
    pe = __fmaf_rn(b.h, c.l, pe);
    pe = __fmaf_rn(b.l, c.h, pe);
    float s, e;
    two_sum(hs, -ph, s, e);
    hs = s;
    lo = __fadd_rn(lo, __fsub_rn(e, pe));
}

// (ch + cl)(xh + xl) as an unnormalised pair
__device__ __forceinline__ void ff_scale(float ch, float cl, float xh, float xl, float &ph, float &pl) {
    two_prod(ch, xh, ph, pl);
    pl = __fmaf_rn(ch, xl, pl);
    pl = __fmaf_rn(cl, xh, pl);
}

// a . b of two vectors of float pairs as an unnormalised pair, to ~2^-48 |a||b|
__device__ __forceinline__ void ff_dot3(const float (&ah)[3], const float (&al)[3], const float (&bh)[3],
                                        const float (&bl)[3], float &h, float &l) {
    float ph[3], pl[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        two_prod(ah[d], bh[d], ph[d], pl[d]);
        pl[d] = __fmaf_rn(ah[d], bl[d], pl[d]);
        pl[d] = __fmaf_rn(al[d], bh[d], pl[d]);
    }
    float t, u, v;
    two_sum(ph[0], ph[1], t, u);
    two_sum(t, ph[2], h, v);
    l = __fadd_rn(__fadd_rn(__fadd_rn(pl[0], pl[1]), __fadd_rn(pl[2], u)), v);
}

// -(a + b) of two pairs
__device__ __forceinline__ void ff_neg_sum(float ah, float al, float bh, float bl, float &h, float &l) {
    float t, e;
    two_sum(ah, bh, t, e);
    h = -t;
    l = -__fadd_rn(e, __fadd_rn(al, bl));
}

// the hardware estimate of 1 / sqrt(x) (2^-22.9 relative) without the
// denormal handling of rsqrtf: callers keep x a normal number
__device__ __forceinline__ float rsqrt_estimate(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 1 / sqrt(t + l): estimate y0 and its relative correction (y0 + y0 c / 2
// with c = d + 3/4 d^2, d = 1 - (t + l) y0^2 from exact products): ~2^-47
__device__ __forceinline__ void inv_sqrt_ff(float t, float l, float &y0, float &c) {
    y0 = rsqrt_estimate(t);
    const float g = __fmul_rn(t, y0);
    float ge = __fmaf_rn(t, y0, -g);
    ge = __fmaf_rn(l, y0, ge);
    float d = __fmaf_rn(-g, y0, 1.0f);
    d = __fmaf_rn(-ge, y0, d);
    c = __fmaf_rn(__fmul_rn(0.75f, d), d, d);
}

// A sum of inverse distances of one weight: s + lo2 / 2 (lo2 collects twice
// the rounding errors of s and the corrections).  FIRST: s may be smaller than
// the new term (the second term of a sum); otherwise s >= y0 by the distance
// ratio of at most 2 that the caller checks.
template <bool FIRST> __device__ __forceinline__ void add_inv(float t, float l, float &s, float &lo2) {
    float y0, c, v, e;
    inv_sqrt_ff(t, l, y0, c);
    if (FIRST) two_sum(s, y0, v, e);
    else fast_two_sum(s, y0, v, e);
    s = v;
    lo2 = __fmaf_rn(2.0f, e, __fmaf_rn(y0, c, lo2));
}

// c_R - c_C as float pairs: the hi and lo differences are exact (TwoSum) and
// only their combination rounds, so neighbouring panels (|D| ~ panel size)
// keep full relative accuracy
__device__ __forceinline__ void centroid_diff(const float *__restrict__ R, int rs, const float *__restrict__ C, int cs,
                                              float (&Dh)[3], float (&Dl)[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        float s, e, t, f, u, g;
        two_sum(R[(PF_CH + d) * rs], -C[(PF_CH + d) * cs], s, e);
        two_sum(R[(PF_CL + d) * rs], -C[(PF_CL + d) * cs], t, f);
        two_sum(e, t, u, g);
        float sh, sl;
        two_sum(s, u, sh, sl);
        g = __fadd_rn(g, __fadd_rn(f, __fsub_rn(R[(PF_CM + d) * rs], C[(PF_CM + d) * cs])));
        fast_two_sum(sh, __fadd_rn(sl, g), Dh[d], Dl[d]);
    }
}

// times (|T_R| / sqrt(4 pi)) (|T_C| / sqrt(4 pi))
__device__ __forceinline__ void entry_scale(float ah, float al, const float *__restrict__ R, int rs,
                                            const float *__restrict__ C, int cs, float &eh, float &el) {
    float wh, wl;
    ff_scale(R[PF_WA * rs], R[(PF_WA + 1) * rs], C[PF_WA * cs], C[(PF_WA + 1) * cs], wh, wl);
    ff_scale(ah, al, wh, wl, eh, el);
}

// The entry from the differences of the 49 pairs of points, each formed to
// 2^-48 of itself whatever the distance: for panels too near (or coordinates
// too small or large) for the sums of regular_entry_ff2 below.
__device__ __noinline__ static FF regular_entry_near(const float *__restrict__ R, int rs, const float *__restrict__ C,
                                                     int cs, const QuadParams &qp) {
    float Dh[3], Dl[3];
    centroid_diff(R, rs, C, cs, Dh, Dl);
    float acc_h = 0.0f, acc_l = 0.0f;
#pragma unroll 1
    for (int p = 0; p < NQ; ++p) {
        // X_p = D + a_p
        float Xh[3], Xl[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            float ah = 0.0f, al = 0.0f;
            if (p > 0) {
                const int k = (p - 1) % 3;
                ah = R[(PF_U + 6 * k + d) * rs];
                al = R[(PF_U + 6 * k + 3 + d) * rs];
                if (p > 3) ff_scale(qp.rho[0], qp.rho[1], ah, al, ah, al);
            }
            float s, e;
            two_sum(Dh[d], ah, s, e);
            e = __fadd_rn(e, __fadd_rn(Dl[d], al));
            fast_two_sum(s, e, Xh[d], Xl[d]);
        }
        float sp_h = 0.0f, sp_l = 0.0f;
#pragma unroll 1
        for (int q = 0; q < NQ; ++q) {
            // r^2 = |X_p - b_q|^2
            float ph[3], pl[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                float bh = 0.0f, bl = 0.0f;
                if (q > 0) {
                    const int k = (q - 1) % 3;
                    bh = C[(PF_U + 6 * k + d) * cs];
                    bl = C[(PF_U + 6 * k + 3 + d) * cs];
                    if (q > 3) ff_scale(qp.rho[0], qp.rho[1], bh, bl, bh, bl);
                }
                float s, e;
                two_sum(Xh[d], -bh, s, e);
                e = __fadd_rn(e, __fsub_rn(Xl[d], bl));
                two_prod(s, s, ph[d], pl[d]);
                pl[d] = __fmaf_rn(__fmul_rn(2.0f, s), e, pl[d]);
            }
            float t1, u1, t2, u2;
            two_sum(ph[0], ph[1], t1, u1);
            two_sum(t1, ph[2], t2, u2);
            const float r2l = __fadd_rn(__fadd_rn(__fadd_rn(pl[0], pl[1]), __fadd_rn(pl[2], u1)), u2);
            // 1 / sqrt(r2): estimate + one Newton step with an exact residual
            const float y0 = rsqrtf(t2);
            float yh, yl;
            two_prod(y0, y0, yh, yl);
            float mh, ml;
            two_prod(t2, yh, mh, ml);
            ml = __fmaf_rn(t2, yl, ml);
            ml = __fmaf_rn(r2l, yh, ml);
            float del = __fsub_rn(__fsub_rn(1.0f, mh), ml);
            del = __fmaf_rn(__fmul_rn(0.75f, del), del, del);
            const float corr = __fmul_rn(__fmul_rn(0.5f, y0), del);
            // sp += w_q (y0 + corr)
            float qh, ql;
            ff_scale(qp.w_h[q], qp.w_l[q], y0, corr, qh, ql);
            float s, e;
            two_sum(sp_h, qh, s, e);
            sp_h = s;
            sp_l = __fadd_rn(sp_l, __fadd_rn(e, ql));
        }
        // acc += w_p sp
        float sh, sl;
        fast_two_sum(sp_h, sp_l, sh, sl);
        float qh, ql;
        ff_scale(qp.w_h[p], qp.w_l[p], sh, sl, qh, ql);
        float s, e;
        two_sum(acc_h, qh, s, e);
        acc_h = s;
        acc_l = __fadd_rn(acc_l, __fadd_rn(e, ql));
    }
    float ah, al;
    fast_two_sum(acc_h, acc_l, ah, al);
    FF r;
    entry_scale(ah, al, R, rs, C, cs, r.h, r.l);
    return r;
}

// Regular entry a_ij = |Ti||Tj|/(4 pi) sum_p sum_q w_p w_q / |x_p - y_q| for
// panel records R (row, test) and C (column, trial); element k of a record at
// R[k * rs].  Returns the float pair (eh, el), not normalised.
//
// The squared distances come from the orbits of the rule: with the centroid
// difference D and the scaled vertex offsets u_k (row) and w_l (column),
//   |D + o u_k - o' w_l|^2 = P_k(o) + Q_l(o') + o o' G_kl,   o, o' in {0, 1, rho},
//   P_k(o) = |D|^2 + o 2 D.u_k + o^2 |u_k|^2,  Q_l(o') = -o' 2 D.w_l + o'^2 |w_l|^2,
//   G_kl = -2 u_k.w_l,
// where the |u_k|^2 stand in the record and the third of each triple of dot
// products is minus the sum of the other two: 10 additions per pair of points
// instead of three differences, their squares and sums (52 operations).  The
// inverse roots of one weight w_p w_q are summed before the weight is applied
// (6 weights instead of 49).  The high parts add without loss (FastTwoSum:
// the terms are ordered by size, see the check below), the low parts with one
// rounding each, so r^2 carries ~2^-48 |D|^2.  The arithmetic pipe is the bound:
// about 1,850 operations per entry against 4,200 with the 49 differences.
// Measured on a sphere of 655,220 panels (leaves of 80 rows, eps 1e-6): near
// field 153 -> 95 ms, ACA 381 -> 265 ms.  Against the sum in 80-bit arithmetic
// (separations of 3 to 300 radii): 3e-15 rms, where the differences with a
// first-order root gave 7e-15.
//
// Valid where the panels are well apart, |D| >= 3 (max |u| + max |w|): the
// distances then lie in [2/3, 4/3] |D|, so 2^-48 |D|^2 is also a small error
// of the smallest r^2, |Q| < P, and two inverse distances outweigh a third.
// Other pairs (a few per row of the near field) take regular_entry_near, as
// do distances whose squares leave the range where the low parts are normal.
__device__ __forceinline__ void regular_entry_ff2(const float *__restrict__ R, int rs, const float *__restrict__ C,
                                                  int cs, const QuadParams &qp, float &eh_out, float &el_out) {
    float Dh[3], Dl[3];
    centroid_diff(R, rs, C, cs, Dh, Dl);
    float R0h, R0l;
    ff_dot3(Dh, Dl, Dh, Dl, R0h, R0l);
    const float rad = __fadd_rn(R[PF_RAD * rs], C[PF_RAD * cs]);
    if (!(R0h >= 9.0f * rad * rad && R0h > 1e-18f && R0h < 1e30f)) {
        const FF e = regular_entry_near(R, rs, C, cs, qp);
        eh_out = e.h;
        el_out = e.l;
        return;
    }
    // w' = -2 w; Q_l for both orbits
    float wh[2][3], wl[2][3], Qh[6], Ql[6];
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            wh[l][d] = __fmul_rn(-2.0f, C[(PF_U + 6 * l + d) * cs]);
            wl[l][d] = __fmul_rn(-2.0f, C[(PF_U + 6 * l + 3 + d) * cs]);
        }
    {
        float bh[3], bl[3];
        ff_dot3(Dh, Dl, wh[0], wl[0], bh[0], bl[0]);
        ff_dot3(Dh, Dl, wh[1], wl[1], bh[1], bl[1]);
        ff_neg_sum(bh[0], bl[0], bh[1], bl[1], bh[2], bl[2]);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            float e, th, tl;
            two_sum(C[(PF_N + 2 * l) * cs], bh[l], Qh[l], e);
            Ql[l] = __fadd_rn(e, __fadd_rn(C[(PF_N + 2 * l + 1) * cs], bl[l]));
            ff_scale(qp.rho[0], qp.rho[1], bh[l], bl[l], th, tl);
            two_sum(C[(PF_N2 + 2 * l) * cs], th, Qh[3 + l], e);
            Ql[3 + l] = __fadd_rn(e, __fadd_rn(C[(PF_N2 + 2 * l + 1) * cs], tl));
        }
    }
    // sums of the inverse distances by weight: centroid with the orbits 1 and
    // 2 (s01, s02), within and between the orbits (s11, s12, s22)
    float s00, c00, s01 = 0.0f, l01 = 0.0f, s02 = 0.0f, l02 = 0.0f;
    float s11 = 0.0f, l11 = 0.0f, s12 = 0.0f, l12 = 0.0f, s22 = 0.0f, l22 = 0.0f;
    inv_sqrt_ff(R0h, R0l, s00, c00);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        float t, e;
        fast_two_sum(R0h, Qh[l], t, e);
        add_inv<true>(t, __fadd_rn(e, __fadd_rn(R0l, Ql[l])), s01, l01);
        fast_two_sum(R0h, Qh[3 + l], t, e);
        add_inv<true>(t, __fadd_rn(e, __fadd_rn(R0l, Ql[3 + l])), s02, l02);
    }
    // D' = 2 D
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        Dh[d] = __fmul_rn(2.0f, Dh[d]);
        Dl[d] = __fmul_rn(2.0f, Dl[d]);
    }
    // the loop over the row's vertices stays rolled: its body is ~450
    // operations, and one copy of it keeps the instruction cache warm
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const float *U = R + (PF_U + 6 * k) * rs, *N = R + (PF_N + 2 * k) * rs, *N2 = R + (PF_N2 + 2 * k) * rs;
        float uh[3], ul[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            uh[d] = U[d * rs];
            ul[d] = U[(3 + d) * rs];
        }
        float P1h, P1l, P2h, P2l;
        {
            float ah, al, t, e, f, th, tl;
            ff_dot3(Dh, Dl, uh, ul, ah, al);
            fast_two_sum(R0h, ah, t, e);
            fast_two_sum(t, N[0], P1h, f);
            P1l = __fadd_rn(__fadd_rn(e, f), __fadd_rn(R0l, __fadd_rn(al, N[rs])));
            ff_scale(qp.rho[0], qp.rho[1], ah, al, th, tl);
            fast_two_sum(R0h, th, t, e);
            fast_two_sum(t, N2[0], P2h, f);
            P2l = __fadd_rn(__fadd_rn(e, f), __fadd_rn(R0l, __fadd_rn(tl, N2[rs])));
        }
        add_inv<false>(P1h, P1l, s01, l01);
        add_inv<false>(P2h, P2l, s02, l02);
        float Gh[3], Gl[3];
        ff_dot3(uh, ul, wh[0], wl[0], Gh[0], Gl[0]);
        ff_dot3(uh, ul, wh[1], wl[1], Gh[1], Gl[1]);
        ff_neg_sum(Gh[0], Gl[0], Gh[1], Gl[1], Gh[2], Gl[2]);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            float g1h, g1l, g2h, g2l, t, v, e, f;
            ff_scale(qp.rho[0], qp.rho[1], Gh[l], Gl[l], g1h, g1l);
            ff_scale(qp.rho[2], qp.rho[3], Gh[l], Gl[l], g2h, g2l);
            fast_two_sum(P1h, Qh[l], v, e);
            fast_two_sum(v, Gh[l], t, f);
            e = __fadd_rn(__fadd_rn(__fadd_rn(P1l, Ql[l]), __fadd_rn(e, Gl[l])), f);
            if (l == 1) add_inv<true>(t, e, s11, l11);
            else add_inv<false>(t, e, s11, l11);
            fast_two_sum(P1h, Qh[3 + l], v, e);
            fast_two_sum(v, g1h, t, f);
            e = __fadd_rn(__fadd_rn(__fadd_rn(P1l, Ql[3 + l]), __fadd_rn(e, g1l)), f);
            add_inv<false>(t, e, s12, l12);
            fast_two_sum(P2h, Qh[l], v, e);
            fast_two_sum(v, g1h, t, f);
            e = __fadd_rn(__fadd_rn(__fadd_rn(P2l, Ql[l]), __fadd_rn(e, g1l)), f);
            if (l == 0) add_inv<true>(t, e, s12, l12);
            else add_inv<false>(t, e, s12, l12);
            fast_two_sum(P2h, Qh[3 + l], v, e);
            fast_two_sum(v, g2h, t, f);
            e = __fadd_rn(__fadd_rn(__fadd_rn(P2l, Ql[3 + l]), __fadd_rn(e, g2l)), f);
            if (l == 1) add_inv<true>(t, e, s22, l22);
            else add_inv<false>(t, e, s22, l22);
        }
    }
    // weighted sum of the six classes
    const float sv[6] = {s00, s01, s02, s11, s12, s22};
    const float lv[6] = {__fmul_rn(s00, c00), l01, l02, l11, l12, l22};
    float acc_h = 0.0f, acc_l = 0.0f;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        float h, l, ph, pl, t, e;
        fast_two_sum(sv[c], __fmul_rn(0.5f, lv[c]), h, l);
        ff_scale(qp.cw[2 * c], qp.cw[2 * c + 1], h, l, ph, pl);
        two_sum(acc_h, ph, t, e);
        acc_h = t;
        acc_l = __fadd_rn(acc_l, __fadd_rn(e, pl));
    }
    float ah, al;
    fast_two_sum(acc_h, acc_l, ah, al);
    entry_scale(ah, al, R, rs, C, cs, eh_out, el_out);
}

__device__ __forceinline__ double regular_entry_ff(const float *__restrict__ R, int rs, const float *__restrict__ C,
                                                   int cs, const QuadParams &qp) {
    float eh, el;
    regular_entry_ff2(R, rs, C, cs, qp, eh, el);
    return (double)eh + (double)el;
}

}  // namespace hm
