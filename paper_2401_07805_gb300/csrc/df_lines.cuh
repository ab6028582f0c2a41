// Sweeps of the double-float operators along one line of Q = P + 1 points, in double-float arithmetic (dfloat.cuh).
//
// Support points (Gauss-Lobatto) and quadrature points (Gauss-Legendre) are symmetric about 1/2.  Q = 3: the middle points
// coincide, the outer values are three-term dot products, and the transposed sweep takes the even and the odd part of the
// outer points with three multiplications (3/10, 4/10 and tau = sqrt(3/20), the distance of the outer Gauss points from
// 1/2).  Q = 4: even and odd parts are transformed apart (the even-odd decomposition of tensor-product elements).  FP32
// instructions per line of 3 results: 62 (values), 61 (derivatives), against 93 for three 3-term dot products, with a
// third of their shared-memory loads, since one thread forms a whole line.
//
//   val   y_q = sum_a S[q][a] u_a           valT  o_a = sum_q S[q][a] f_q
//   der   d_q = sum_r D[q][r] y_r           derT  o_r = sum_q D[q][r] t_q,   D = (collocation derivative) / DSCALE:
// the derivative at the Gauss points up to the factor DSCALE (1 / (2 tau) for Q = 3, where D holds the integers
// -3, 4, -1 / -1, 0, 1 / 1, -4, 3; 1 for Q = 4); the factor and 1/h are part of the cached coefficients.
#pragma once

#include "dfloat.cuh"

namespace evap {

constexpr float dfk_hi(double v) { return (float)v; }
constexpr float dfk_lo(double v) { return (float)(v - (double)(float)v); }
#define EVAP_DFK(v) (dfl{dfk_hi(v), dfk_lo(v)})

// a + b without the closing normalization (|lo| may reach a few ulp(hi)): for sums that are added further
__device__ __forceinline__ dfl df_addl(dfl a, dfl b) {
    dfl s = two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return s;
}
__device__ __forceinline__ dfl df_twice(dfl a) { return {a.hi + a.hi, a.lo + a.lo}; }
__device__ __forceinline__ dfl df_half(dfl a) { return {0.5f * a.hi, 0.5f * a.lo}; }

// Which sums are normalized: results stored for the next sweep (df_addo) and, for Q = 3, sums multiplied next (df_addi) and the
// gradients; sums that are added further are not.  Errors against 64 bits relative to point-wise dot products, geometric
// means (velocity rows / divergence row / adjoint g_x / g_u0 / g_phi over 100 to 2242 drawn Q2 cases, g_phi 1.004 +- 0.005; pressure
// term alone, 34):
//   outer values as u_1 + 3/10 C -+ tau dm with C = u_0 - 2 u_1 + u_2, the transposed middle as s + f_1 - 2 (3/10 s),
//     even part and gradients unnormalized    0.98 / 1.03 / 0.99 / 1.00 / 1.05 / 1.12          (48^3 Q2 apply 218 us, adjoint 561)
//   this arrangement                          0.92 / 0.91 / 0.90 / 0.89 / 1.00 / 0.77          (216 us, 550)
// 64^3 Q2 apply with the first arrangement (us): both of df_addo and df_addi normalized 552, one of them 540, none 529.
// Q = 4 normalizes the stored results only (45^3 Q3: 576 -> 544 us; 0.91 / 0.97 / 0.92 / 0.92 / 0.95 / 0.99).
__device__ __forceinline__ dfl df_addo(dfl a, dfl b) { return df_add(a, b); }
__device__ __forceinline__ dfl df_addi(dfl a, dfl b) { return df_add(a, b); }

template <int Q>
struct DfLine;

template <>
struct DfLine<3> {
    static constexpr double TAU = 0.5 * 0.7745966692414833770358531;  // sqrt(3/5) / 2
    static constexpr double DSCALE = 1.0 / (2.0 * TAU);
    static __device__ __forceinline__ dfl dot3(const dfl u[3], dfl c0, dfl c1, dfl c2) {
        dfl s = df_prod(c0, u[0]);
        df_fma(s, c1, u[1]);
        df_fma(s, c2, u[2]);
        return df_norm(s);
    }
    static __device__ __forceinline__ void val(const dfl u[3], dfl y[3]) {
        constexpr double a0 = 0.3 + TAU, a2 = 0.3 - TAU;
        y[0] = dot3(u, EVAP_DFK(a0), EVAP_DFK(0.4), EVAP_DFK(a2));
        y[1] = u[1];
        y[2] = dot3(u, EVAP_DFK(a2), EVAP_DFK(0.4), EVAP_DFK(a0));
    }
    template <bool FINAL>  // FINAL: the results are converted next
    static __device__ __forceinline__ void valT(const dfl f[3], dfl o[3]) {
        const dfl s = df_addi(f[0], f[2]), d = df_addi(f[0], df_neg(f[2]));
        const dfl p = df_mul(s, EVAP_DFK(0.3)), r = df_mul(d, EVAP_DFK(TAU));
        const dfl p2 = df_mul(s, EVAP_DFK(0.4));  // (not s - 2 p: that doubles the rounding of p)
        o[0] = FINAL ? df_addl(p, r) : df_addo(p, r);
        o[1] = FINAL ? df_addl(f[1], p2) : df_addo(f[1], p2);
        o[2] = FINAL ? df_addl(p, df_neg(r)) : df_addo(p, df_neg(r));
    }
    static __device__ __forceinline__ void der(const dfl y[3], dfl d[3]) {
        const dfl A = df_addl(y[1], df_neg(y[0])), B = df_addl(y[2], df_neg(y[1]));
        const dfl D = df_addl(A, df_neg(B));
        d[0] = df_add(D, df_twice(A));
        d[1] = df_add(A, B);
        d[2] = df_add(df_twice(B), df_neg(D));
    }
    static __device__ __forceinline__ void derT(const dfl t[3], dfl o[3]) {
        const dfl a = df_addl(t[0], df_neg(t[2]));
        o[0] = df_neg(df_addl(df_addl(t[1], df_twice(t[0])), a));
        o[1] = df_twice(df_twice(a));
        o[2] = df_addl(df_addl(t[1], df_twice(t[2])), df_neg(a));
    }
};

template <>
struct DfLine<4> {
    static constexpr double DSCALE = 1.0;
    // even parts: sum over a pair of symmetric points; odd parts: difference.  A row q of S acts on the even part
    // (e0, e1) as e1 / 2 + al (e0 - e1) (its entries sum to 1) and on the odd part (o0, o1) by (ga, de).
    static constexpr CtBasis<3> B = make_ct_basis<3>();
    static constexpr double al(int q) { return 0.5 * (B.S[q][0] + B.S[q][3]); }
    static constexpr double ga(int q) { return 0.5 * (B.S[q][0] - B.S[q][3]); }
    static constexpr double de(int q) { return 0.5 * (B.S[q][1] - B.S[q][2]); }
    // a row q of the derivative: eta (e0 - e1) from the even part (its entries sum to 0), (xa, xb) on the odd part
    static constexpr double eta(int q) { return 0.5 * (B.Dc[q][0] + B.Dc[q][3]); }
    static constexpr double xa(int q) { return 0.5 * (B.Dc[q][0] - B.Dc[q][3]); }
    static constexpr double xb(int q) { return 0.5 * (B.Dc[q][1] - B.Dc[q][2]); }
    static __device__ __forceinline__ dfl dot2(dfl c0, dfl v0, dfl c1, dfl v1) {
        dfl s = df_prod(c0, v0);
        df_fma(s, c1, v1);
        return s;
    }
    template <int q>
    static __device__ __forceinline__ void val_pair(dfl e1h, dfl f, dfl o0, dfl o1, dfl y[4]) {
        constexpr double a_ = al(q), g_ = ga(q), d_ = de(q);
        dfl E = e1h;
        df_fma(E, EVAP_DFK(a_), f);
        const dfl O = dot2(EVAP_DFK(g_), o0, EVAP_DFK(d_), o1);
        y[q] = df_addo(E, O);
        y[3 - q] = df_addo(E, df_neg(O));
    }
    static __device__ __forceinline__ void val(const dfl u[4], dfl y[4]) {
        const dfl e0 = df_addl(u[0], u[3]), e1 = df_addl(u[1], u[2]);
        const dfl o0 = df_addl(u[0], df_neg(u[3])), o1 = df_addl(u[1], df_neg(u[2]));
        const dfl f = df_addl(e0, df_neg(e1));
        val_pair<0>(df_half(e1), f, o0, o1, y);
        val_pair<1>(df_half(e1), f, o0, o1, y);
    }
    template <bool FINAL>
    static __device__ __forceinline__ void valT(const dfl t[4], dfl o[4]) {
        const dfl s0 = df_addl(t[0], t[3]), s1 = df_addl(t[1], t[2]);
        const dfl d0 = df_addl(t[0], df_neg(t[3])), d1 = df_addl(t[1], df_neg(t[2]));
        constexpr double a0 = al(0), a1 = al(1), g0 = ga(0), g1 = ga(1), e0 = de(0), e1 = de(1);
        const dfl ev = dot2(EVAP_DFK(a0), s0, EVAP_DFK(a1), s1);               // even result of the outer pair
        const dfl ei = df_addl(df_half(df_addl(s0, s1)), df_neg(ev));           // and of the inner one
        const dfl od = dot2(EVAP_DFK(g0), d0, EVAP_DFK(g1), d1), oi = dot2(EVAP_DFK(e0), d0, EVAP_DFK(e1), d1);
        o[0] = FINAL ? df_addl(ev, od) : df_addo(ev, od);
        o[3] = FINAL ? df_addl(ev, df_neg(od)) : df_addo(ev, df_neg(od));
        o[1] = FINAL ? df_addl(ei, oi) : df_addo(ei, oi);
        o[2] = FINAL ? df_addl(ei, df_neg(oi)) : df_addo(ei, df_neg(oi));
    }
    static __device__ __forceinline__ void der(const dfl y[4], dfl d[4]) {
        const dfl o0 = df_addl(y[0], df_neg(y[3])), o1 = df_addl(y[1], df_neg(y[2]));
        const dfl f = df_addl(df_addl(y[0], y[3]), df_neg(df_addl(y[1], y[2])));
        constexpr double h0 = eta(0), h1 = eta(1), a0 = xa(0), a1 = xa(1), b0 = xb(0), b1 = xb(1);
        const dfl v0 = df_mul(EVAP_DFK(h0), f), v1 = df_mul(EVAP_DFK(h1), f);
        const dfl w0 = dot2(EVAP_DFK(a0), o0, EVAP_DFK(b0), o1), w1 = dot2(EVAP_DFK(a1), o0, EVAP_DFK(b1), o1);
        d[0] = df_addl(w0, v0);
        d[3] = df_addl(w0, df_neg(v0));
        d[1] = df_addl(w1, v1);
        d[2] = df_addl(w1, df_neg(v1));
    }
    static __device__ __forceinline__ void derT(const dfl t[4], dfl o[4]) {
        const dfl s0 = df_addl(t[0], t[3]), s1 = df_addl(t[1], t[2]);  // act on the odd part
        const dfl d0 = df_addl(t[0], df_neg(t[3])), d1 = df_addl(t[1], df_neg(t[2]));
        constexpr double h0 = eta(0), h1 = eta(1), a0 = xa(0), a1 = xa(1), b0 = xb(0), b1 = xb(1);
        const dfl ev = dot2(EVAP_DFK(h0), d0, EVAP_DFK(h1), d1);  // even result, + on the outer and - on the inner pair
        const dfl oo = dot2(EVAP_DFK(a0), s0, EVAP_DFK(a1), s1), oi = dot2(EVAP_DFK(b0), s0, EVAP_DFK(b1), s1);
        o[0] = df_addl(ev, oo);
        o[3] = df_addl(ev, df_neg(oo));
        o[1] = df_addl(df_neg(ev), oi);
        o[2] = df_neg(df_addl(ev, oi));
    }
};

// kappa = DSCALE / h: physical gradient = kappa (D y)
inline double df_kappa(const MeshArgs<double>& m) {
    return (m.P == 2 ? DfLine<3>::DSCALE : DfLine<4>::DSCALE) * m.inv_h;
}

// Line `l` (of Q^2) of direction DIR (0 x, 1 y, 2 z) in a cell's Q^3 points, x fastest: first point and stride.
template <int Q, int DIR>
struct LineAt {
    static constexpr int stride = DIR == 0 ? 1 : (DIR == 1 ? Q : Q * Q);
    static __device__ __forceinline__ int first(int l) {
        return DIR == 0 ? Q * l : (DIR == 1 ? l % Q + Q * Q * (l / Q) : l);
    }
};
template <int Q, int DIR>
__device__ __forceinline__ void ld_line(const dfl* cell, int l, dfl v[Q]) {
    const int p0 = LineAt<Q, DIR>::first(l);
#pragma unroll
    for (int k = 0; k < Q; ++k) v[k] = cell[p0 + k * LineAt<Q, DIR>::stride];
}
template <int Q, int DIR>
__device__ __forceinline__ void st_line(dfl* cell, int l, const dfl v[Q]) {
    const int p0 = LineAt<Q, DIR>::first(l);
#pragma unroll
    for (int k = 0; k < Q; ++k) cell[p0 + k * LineAt<Q, DIR>::stride] = v[k];
}

}  // namespace evap
