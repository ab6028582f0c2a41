// Adjoint of the momentum apply, FP64-accurate.  The u0 terms and the material coefficients come from the
// quadrature-point cache of set_fields (the double-float pairs the forward apply uses, so g_x is its transpose to
// rounding); the chain-rule factors that depend only on phi and mdot (H'(d) d'(phi), its phi-derivative, the normal,
// 1/|grad phi|, c_1 delta, ...) come from the adjoint table that set_fields fills in FP64 for the interface cells.
//
// L = w . A(phi, u0) x + w_p . (B x - g(phi, mdot))  (velocity block and divergence row of Eq. weakNavierStokes).
// Per quadrature point with W the weight, (X, G) values/gradients of x, (Om, OmG) of w, (U, GU) of u0, pi of w_p:
//   dL/dX_d     = W rho (c_m Om_d + newton sum_c Om_c GU_cd)
//   dL/dG_db    = W rho Om_d U_b + 2 W mu (sym(OmG)_db - z delta_db (n . OmG n)) + W pi delta_db
//   dL/dU_b     = W rho sum_c Om_c G_cb,           dL/dGU_cd = newton W rho Om_c X_d
//   dL/drho     = W Om . (c_m X + G U + newton GU X),  dL/dmu = 2 W OmG : eps_mod(X)
//   dL/dn       = -2 W mu z tr(G) (OmG + OmG^T) n,  dL/dv_dil = -W pi
//   chain rule through Eqs. (heaviside), (rhoEff), (muEff), (normal_vector), (delta), (evaporDil):
//     drho/dH = -rho^2 (1/rho_l - 1/rho_g), dmu/dH = mu_l - mu_g, dH/dphi = H'(d) d'(phi),
//     d delta/dphi = (H''(d) d'(phi)^2 + H'(d) d''(phi)) |grad phi|, d delta/d grad phi = H'(d) d'(phi) n,
//     dn/d grad phi = (I - n n^T)/|grad phi|; the zone gate is piecewise constant.
// The value/gradient sensitivities are tested like the forward operator (S^T and Dc^T sweeps); the Q1 sensitivities
// are integrated against the level-set shape functions N_j and grad N_j (Q1 on the level-set mesh: the velocity
// cell subdivided n_sub times per direction).
#include <algorithm>

#include "async_copy.cuh"
#include "df_lines.cuh"
#include "physics.cuh"

namespace evap {

// g_x = w on the Dirichlet DoFs and 0 elsewhere, g_u0 = g_phi = g_mdot = 0: a warp walks whole x-lines of nodes, so the
// line's position is split once per warp.
__global__ void __launch_bounds__(256) k_adjoint_init(int M, int64_t Nu, int64_t Np, unsigned faces,
                                                      const double* __restrict__ w, double* gx, double* gu,
                                                      double* gphi, double* gm) {
    const int lines = 3 * M * M;
    const int wpb = blockDim.x / 32, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int line = blockIdx.x * wpb + warp; line < lines; line += gridDim.x * wpb) {
        const int c = line / (M * M), rem = line - c * M * M, gz = rem / M, gy = rem - gz * M;
        const bool cyz = ((faces & 4u) && gy == 0) || ((faces & 8u) && gy == M - 1) || ((faces & 16u) && gz == 0) ||
                         ((faces & 32u) && gz == M - 1);
        const int64_t off = c * Nu + (int64_t)M * (gy + (int64_t)M * gz);
        for (int i = lane; i < M; i += 32) {
            if (gx)
                gx[off + i] = cyz || ((faces & 1u) && i == 0) || ((faces & 2u) && i == M - 1) ? w[off + i] : 0.0;
            if (gu) gu[off + i] = 0.0;
        }
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Np; i += stride) {
        if (gphi) gphi[i] = 0.0;
        if (gm) gm[i] = 0.0;
    }
}

// K = n_sub + 1: level-set shape functions per direction on a velocity cell (Q1 on its n_sub sub-intervals).
// The interpolation of x and w, the value / gradient sensitivities and their testing run in double-float arithmetic
// (dfloat.cuh) on the FP32 pipe, with the coefficients of the double-float cache (the pairs of the FP64 values the
// forward apply uses); so do the material-law sensitivities of the interface-zone points, with the factors of the
// adjoint table.  The level-set test sweeps run in FP64, in the table cells only.
// Layout: as the forward apply (momentum_df.cu), sweeps by lines (df_lines.cuh; the 6 Q^2 lines of the six fields x and
// w, two rounds over a cell's Q^3 threads) and the sensitivities by one thread per quadrature point, which overwrites
// its own point's values and gradients with them.  Only the threads of table cells run the interface-zone work and the
// level-set sweeps.  At most 48 KB of shared memory per block, so no launch needs a function attribute.
// Measured at 48^3 Q2 (us; one point per thread with Q-term dot products 779): cells per block / blocks per SM 4 / 5 550 (96
// registers); 2 / 10 564; 4 / 4 586; 3 / 6 589.  On a subdivided level set (n_sub = 2; 947 before): 4 / 5 599; 4 / 4 and 3 / 6 591;
// 2 / 10 605.  Q3 at 32^3 (859 before; one cell, more exceed 48 KB): 1, 4, 6 and 8 blocks per SM 519, 9 543.  ncu at 64^3: issue
// 59 %, FP64 pipe 61 % (conversions).
// Normalization as in the forward apply: the value sensitivities that start the test sums and the last transposed sweep (converted
// to FP64 next) are left unnormalized.
#ifndef EVAP_ADJ_CB2
#define EVAP_ADJ_CB2 4
#endif
#ifndef EVAP_ADJ_MINB2
#define EVAP_ADJ_MINB2 5
#endif
#ifndef EVAP_ADJ_CB3
#define EVAP_ADJ_CB3 1
#endif
#ifndef EVAP_ADJ_MINB3
#define EVAP_ADJ_MINB3 6
#endif

// slots of a cell in shared memory (pairs of Q^3 points): 0..5 X, Om (then the value sensitivities of x and u0), 6..23
// the gradients 6 + 3 f + d of field f (then the gradient sensitivities of x and u0), 24..38 the cached coefficients
// 0..13 and 17 (then the tests along y and z, 12 slots); then the level-set sensitivities, 5 doubles per point
constexpr int ADJ_SLOTS = 24, ADJ_COEF = 15;
template <int P, int CB>
constexpr size_t adj_smem() {
    return sizeof(float2) * CB * (ADJ_SLOTS + ADJ_COEF + 5) * (P + 1) * (P + 1) * (P + 1);
}

template <int P, int CB, int K, int MINB>
__global__ void __launch_bounds__(CB*(P + 1) * (P + 1) * (P + 1), MINB)
    k_adjoint(MeshArgs<double> m, Basis<double> bas, dfl rho_liq, dfl rho_gas,
              const int8_t* __restrict__ code, const int32_t* __restrict__ tindex, const float2* __restrict__ adjt,
              const float2* __restrict__ qcd, const double* __restrict__ w,
              const double* __restrict__ wp, const double* __restrict__ x, double* gx, double* gu, double* gphi,
              double* gm, int colour) {
    constexpr int Q = P + 1, NQ = Q * Q * Q, NL = Q * Q;
    using Ln = DfLine<Q>;
    static_assert(K * Q * Q <= NQ && K * K * K <= NQ, "one thread per entry of each level-set test sweep");
    __shared__ double sNL[Q][K], sDL[Q][K];
    __shared__ double q1a[CB][5][K * Q * Q], q1b[CB][5][K * K * Q];  // level-set test sweeps (FP64)
    extern __shared__ float2 smem_adj[];
    constexpr int CELL = (ADJ_SLOTS + ADJ_COEF + 5) * NQ;
    const int tid = threadIdx.x;
    const int lc = tid / NQ, t = tid % NQ;
    dfl* const cb = reinterpret_cast<dfl*>(smem_adj) + lc * CELL;
    int cx, cy, cz;
    const bool active = colour_cell32(blockIdx.x * CB + lc, m.n, colour, cx, cy, cz);
    const int64_t cell = cx + (int64_t)m.n * (cy + (int64_t)m.n * cz);
    const bool plain = colour >= 0;  // a colour pass: no other cell of the launch touches this cell's nodes
    {  // each thread fetches (and later reads) only its own point's coefficients: 0..3, 13, 17, newton 4..12
        dfl* myq = cb + ADJ_SLOTS * NQ + t;
        const float2* src = qcd + cell * QC_K * NQ + t;
#pragma unroll
        for (int k = 0; k < ADJ_COEF; ++k)
            if (k < 4 || k > 12 || m.newton) cp_async8(myq + k * NQ, src + (k == 14 ? 17 : k) * NQ);
    }
    cp_async_commit();
    if (tid < K * Q) {
        sNL[tid / K][tid % K] = bas.NL[tid / K][tid % K];
        sDL[tid / K][tid % K] = bas.DL[tid / K][tid % K];
    }
    const int n = m.n, M = m.M;
    const int64_t m1 = n + 1;     // pressure nodes per axis (w_p)
    const int64_t ml = m.nl + 1;  // level-set nodes per axis
    const bool tcell = code[cell] == CELL_TABLE;
    // this thread's lines: line l of the fields f0, f0 + Q, ...; its z-line's offset in a component, and which of its nodes
    // are constrained (bit k)
    const int f0 = t / NL, l = t % NL;
    const int64_t zst = (int64_t)M * M;
    int64_t zoff;
    unsigned zcons;
    {
        const int gxi = P * cx + l % Q, gyi = P * cy + l / Q, gz0 = P * cz;
        const unsigned fc = m.faces;
        zcons = ((fc & 1u) && gxi == 0) || ((fc & 2u) && gxi == M - 1) || ((fc & 4u) && gyi == 0) ||
                        ((fc & 8u) && gyi == M - 1)
                    ? (1u << Q) - 1u
                    : 0u;
        if ((fc & 16u) && gz0 == 0) zcons |= 1u;
        if ((fc & 32u) && gz0 + P == M - 1) zcons |= 1u << P;
        zoff = gxi + (int64_t)M * gyi + zst * gz0;
    }
    // w_p interpolated to the points along x, y (z: by the point's thread), in FP64: 2 operations per sweep, not 14 per point
    __shared__ double p0[CB][8], px[CB][4 * Q], py[CB][2 * Q * Q];
    auto lerp = [&](double u, double v, int q) -> double { return fma(bas.t[q], v - u, u); };  // at Gauss point q
    if (wp && t < 8) p0[lc][t] = wp[(cx + (t & 1)) + m1 * ((cy + ((t >> 1) & 1)) + m1 * (cz + (t >> 2)))];
    // values at the points: the lines along z (from memory), y and x, then the derivatives along the three directions
    for (int f = f0; f < 6; f += Q) {
        const double* src = (f < 3 ? x : w) + (f < 3 ? f : f - 3) * m.Nu + zoff;
        dfl u[Q], v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) u[k] = (zcons >> k) & 1u ? dfl{0.f, 0.f} : df_from_double(src[k * zst]);
        Ln::val(u, v);
        st_line<Q, 2>(cb + (6 + f) * NQ, l, v);
    }
    __syncthreads();
    for (int f = f0; f < 6; f += Q) {
        dfl u[Q], v[Q];
        ld_line<Q, 1>(cb + (6 + f) * NQ, l, u);
        Ln::val(u, v);
        st_line<Q, 1>(cb + (12 + f) * NQ, l, v);
    }
    if (wp && t < 4 * Q) px[lc][t] = lerp(p0[lc][2 * (t / Q)], p0[lc][2 * (t / Q) + 1], t % Q);  // [qx][jb][jc]
    __syncthreads();
    for (int f = f0; f < 6; f += Q) {
        dfl u[Q], v[Q];
        ld_line<Q, 0>(cb + (12 + f) * NQ, l, u);
        Ln::val(u, v);
        st_line<Q, 0>(cb + f * NQ, l, v);
    }
    if (wp && t < 2 * NL) {  // [qx][qy][jc]
        const int q = t % Q, r = (t / Q) % Q, jc = t / NL;
        py[lc][t] = lerp(px[lc][q + Q * (2 * jc)], px[lc][q + Q * (2 * jc + 1)], r);
    }
    __syncthreads();
    for (int f = f0; f < 6; f += Q) {
        dfl u[Q], v[Q];
        ld_line<Q, 0>(cb + f * NQ, l, u);
        Ln::der(u, v);
        st_line<Q, 0>(cb + (6 + 3 * f) * NQ, l, v);
        ld_line<Q, 1>(cb + f * NQ, l, u);
        Ln::der(u, v);
        st_line<Q, 1>(cb + (7 + 3 * f) * NQ, l, v);
        ld_line<Q, 2>(cb + f * NQ, l, u);
        Ln::der(u, v);
        st_line<Q, 2>(cb + (8 + 3 * f) * NQ, l, v);
    }
    __syncthreads();
    double dphi = 0.0, dg[3] = {0, 0, 0}, dm = 0.0;
    {
        // values and gradients of x (X, G) and w (Om, OmG) at this thread's point, in units of kappa, read where they
        // are used: the sensitivities are formed in an order that lets them replace their inputs
        const dfl* pt = cb + t;
        auto X = [pt](int k) { return pt[k * NQ]; };
        auto Om = [pt](int k) { return pt[(3 + k) * NQ]; };
        auto G = [pt](int k, int d) { return pt[(6 + 3 * k + d) * NQ]; };
        auto OmG = [pt](int k, int d) { return pt[(15 + 3 * k + d) * NQ]; };
        cp_async_wait_all();
        const dfl* qp = cb + ADJ_SLOTS * NQ + t;
        const dfl Wk = qp[14 * NQ];  // kappa W
        // this point's entries of the adjoint table (table cells only; k_fill_table)
        const float2* ap = tcell ? adjt + (int64_t)tindex[cell] * ADJ_K * NQ + t : nullptr;
        const dfl rho = tcell ? ld_df(ap + ADJ_RHO * NQ) : (code[cell] == CELL_LIQUID ? rho_liq : rho_gas);
        const dfl wr = df_mul(Wk, rho);
        // the phi / mdot sensitivities and the normal are needed only in the interface zone (or with the correction
        // applied everywhere), which lies in table cells; elsewhere H is 0 or 1 and its derivatives vanish
        const bool full = tcell && (ap[ADJ_ZONE * NQ].x != 0.f || (m.stress != 0 && m.corr_zone != 0));
        const dfl wm = qp[13 * NQ];
        const dfl pid = wp ? df_from_double(lerp(py[lc][t % NL], py[lc][t % NL + NL], t / NL)) : dfl{0.f, 0.f};  // w_p here
        const dfl Wkpi = df_mul(Wk, pid);
        dfl corr{0.f, 0.f};
        if (full) {  // material-law sensitivities (interface-zone points only), double-float arithmetic
            const dfl nv[3] = {ld_df(ap + (ADJ_N + 0) * NQ), ld_df(ap + (ADJ_N + 1) * NQ), ld_df(ap + (ADJ_N + 2) * NQ)};
            const bool zg = ap[ADJ_ZG * NQ].x != 0.f;
            const dfl tr = df_add(df_add(G(0, 0), G(1, 1)), G(2, 2));
            // OmG n, OmG^T n and n . OmG n
            dfl on[3], otn[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                dfl u = df_prod(OmG(i, 0), nv[0]), v = df_prod(OmG(0, i), nv[0]);
#pragma unroll
                for (int j = 1; j < 3; ++j) {
                    df_fma(u, OmG(i, j), nv[j]);
                    df_fma(v, OmG(j, i), nv[j]);
                }
                on[i] = df_norm(u);
                otn[i] = df_norm(v);
            }
            dfl nOn = df_prod(nv[0], on[0]);
            df_fma(nOn, nv[1], on[1]);
            df_fma(nOn, nv[2], on[2]);
            nOn = df_norm(nOn);
            if (zg) corr = df_mul(wm, nOn);  // the corrected strain's term of g_x
            // dL/drho = W Om . (c_m X + G u0 + newton grad u0 X) = (1/rho) sum_k Om_k (cached W rho terms)_k
            dfl sr{0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                dfl f = df_prod(qp[0], X(k));
#pragma unroll
                for (int b2 = 0; b2 < 3; ++b2) df_fma(f, qp[(1 + b2) * NQ], G(k, b2));
                if (m.newton) {
#pragma unroll
                    for (int d = 0; d < 3; ++d) df_fma(f, qp[(4 + 3 * k + d) * NQ], X(d));
                }
                if (k == 0)
                    sr = df_prod(Om(0), df_norm(f));
                else
                    df_fma(sr, Om(k), df_norm(f));
            }
            const dfl dL_drho = df_mul(ld_df(ap + ADJ_IRHO * NQ), df_norm(sr));
            // dL/dmu = 2 W (OmG : sym G - z tr(G) n . OmG n)
            dfl smu = df_prod(OmG(0, 0), G(0, 0));
            df_fma(smu, OmG(1, 1), G(1, 1));
            df_fma(smu, OmG(2, 2), G(2, 2));
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int l = k + 1; l < 3; ++l)
                    df_fma(smu, df_add(OmG(k, l), OmG(l, k)), df_scale2(df_add(G(k, l), G(l, k)), 0.5f));
            if (zg) df_fma(smu, df_neg(tr), nOn);
            const dfl dL_dmu = df_mul(df_scale2(Wk, 2.0f), df_norm(smu));  // (/ kappa)
            // dL/dn = -2 W mu z tr(G) (OmG + OmG^T) n; its part normal to n drops out (dn/dgrad phi)
            dfl dLdn[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
            if (zg) {
                const dfl wtr = df_neg(df_mul(wm, tr));
#pragma unroll
                for (int i = 0; i < 3; ++i) dLdn[i] = df_mul(wtr, df_add(on[i], otn[i]));
            }
            dfl dp = df_prod(dL_drho, ld_df(ap + ADJ_CRHO * NQ));
            df_fma(dp, dL_dmu, ld_df(ap + ADJ_CMU * NQ));
            dfl pn = df_prod(dLdn[0], nv[0]);
            df_fma(pn, dLdn[1], nv[1]);
            df_fma(pn, dLdn[2], nv[2]);
            pn = df_neg(df_norm(pn));
            const dfl ign = ld_df(ap + ADJ_IGN * NQ);
            dfl dgv[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                dfl u = dLdn[i];
                df_fma(u, pn, nv[i]);
                dgv[i] = df_mul(df_norm(u), ign);
            }
            if (wp) {  // through v_dil = mdot c_1 delta (Eq. evaporDil), dL/dv_dil = -W pi
                const dfl dLdv = df_neg(Wkpi);  // (times kappa)
                dm = df_to_double(df_mul(dLdv, ld_df(ap + ADJ_KD1 * NQ)));
                df_fma(dp, dLdv, ld_df(ap + ADJ_KD2 * NQ));
                const dfl k3 = df_mul(dLdv, ld_df(ap + ADJ_KD3 * NQ));
#pragma unroll
                for (int i = 0; i < 3; ++i) dgv[i] = df_add(dgv[i], df_mul(k3, nv[i]));
            }
            dphi = df_to_double(df_norm(dp));
#pragma unroll
            for (int i = 0; i < 3; ++i) dg[i] = df_to_double(dgv[i]);
        }
        // value / gradient sensitivities of the velocity block and of B^T w_p, over the point's own entries: with X and
        // Om in registers, those of u0 from G (3..5), of x (0..2), the gradients of x from OmG (over G), then of u0
        const dfl xq[3] = {X(0), X(1), X(2)}, om[3] = {Om(0), Om(1), Om(2)};
        dfl* const out = cb + t;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            dfl u = df_prod(om[0], G(0, d));
            df_fma(u, om[1], G(1, d));
            df_fma(u, om[2], G(2, d));
            out[(3 + d) * NQ] = df_mul(wr, df_norm(u));
            dfl v = df_prod(qp[0], om[d]);
            if (m.newton) {
#pragma unroll
                for (int k = 0; k < 3; ++k) df_fma(v, om[k], qp[(4 + 3 * k + d) * NQ]);
            }
            out[d * NQ] = v;
        }
        const dfl hwm = df_scale2(wm, 0.5f);
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                dfl g = df_prod(om[d], qp[(1 + e) * NQ]);
                df_fma(g, hwm, df_add(OmG(d, e), OmG(e, d)));
                dfl r = df_norm(g);
                if (d == e) {
                    r = df_add(r, Wkpi);
                    if (full) r = df_sub(r, corr);
                }
                out[(6 + 3 * d + e) * NQ] = r;
            }
        if (m.newton) {
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
                for (int e = 0; e < 3; ++e) out[(15 + 3 * d + e) * NQ] = df_mul(wr, df_mul(om[d], xq[e]));
        }
    }
    double* const lsv = reinterpret_cast<double*>(cb + (ADJ_SLOTS + ADJ_COEF) * NQ);  // [5][point]
    if (tcell) {
        lsv[t] = dphi;
        lsv[NQ + t] = dg[0];
        lsv[2 * NQ + t] = dg[1];
        lsv[3 * NQ + t] = dg[2];
        lsv[4 * NQ + t] = dm;
    }
    __syncthreads();
    // test with gradients: the lines along y and z into the coefficients' slots (u0: only with the Newton term)
    const int gfields = m.newton ? 6 : 3;
    for (int f = f0; f < gfields; f += Q) {
        dfl u[Q], v[Q];
        ld_line<Q, 1>(cb + (7 + 3 * f) * NQ, l, u);
        Ln::derT(u, v);
        st_line<Q, 1>(cb + (ADJ_SLOTS + f) * NQ, l, v);
        ld_line<Q, 2>(cb + (8 + 3 * f) * NQ, l, u);
        Ln::derT(u, v);
        st_line<Q, 2>(cb + (ADJ_SLOTS + 6 + f) * NQ, l, v);
    }
    // level-set sensitivities: g_phi[j] = sum_q N_j dL/dphi + grad N_j . dL/dgrad phi, g_mdot[j] = sum_q N_j
    // dL/dmdot with the level-set shape functions N_j of the cell (K per direction), by three sweeps; field f:
    // 0 dL/dphi, 1..3 dL/dgrad phi (x, y, z), 4 dL/dmdot.  Along direction d the 1D factor is the reference
    // derivative DL for field 1 + d, NL otherwise.  x-sweep: [jx][qy][qz].
    if (tcell && t < K * Q * Q) {
        const int jx = t % K, qy = (t / K) % Q, qz = (t / K) / Q;
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            double sacc = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q)
                sacc += (f == 1 ? sDL[q][jx] : sNL[q][jx]) * lsv[f * NQ + q + Q * (qy + Q * qz)];
            q1a[lc][f][t] = sacc;
        }
    }
    __syncthreads();
    for (int f = f0; f < 6; f += Q) {  // x: values + the three tests, and their value sweep
        dfl u[Q], v[Q], s[Q];
        ld_line<Q, 0>(cb + f * NQ, l, s);
        if (f < 3 || m.newton) {
            ld_line<Q, 0>(cb + (6 + 3 * f) * NQ, l, u);
            Ln::derT(u, v);
            ld_line<Q, 0>(cb + (ADJ_SLOTS + f) * NQ, l, u);
#pragma unroll
            for (int k = 0; k < Q; ++k) s[k] = df_addl(df_addl(s[k], v[k]), u[k]);
            ld_line<Q, 0>(cb + (ADJ_SLOTS + 6 + f) * NQ, l, u);
#pragma unroll
            for (int k = 0; k < Q; ++k) s[k] = df_add(s[k], u[k]);
        }
        Ln::template valT<false>(s, v);
        st_line<Q, 0>(cb + f * NQ, l, v);
    }
    if (tcell && t < K * K * Q) {  // y-sweep: [jx][jy][qz]
        const int jx = t % K, jy = (t / K) % K, qz = t / (K * K);
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            double sacc = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q)
                sacc += (f == 2 ? sDL[q][jy] : sNL[q][jy]) * q1a[lc][f][jx + K * (q + Q * qz)];
            q1b[lc][f][t] = sacc;
        }
    }
    __syncthreads();
    if (active && tcell && t < K * K * K) {  // z-sweep and scatter of level-set node (jx, jy, jz) of a table cell
        const int jx = t % K, jy = (t / K) % K, jz = t / (K * K);
        double r[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            double sacc = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) sacc += (f == 3 ? sDL[q][jz] : sNL[q][jz]) * q1b[lc][f][jx + K * (jy + K * q)];
            r[f] = sacc;
        }
        const int ks = K - 1;  // n_sub
        const int64_t nd = (ks * cx + jx) + ml * ((ks * cy + jy) + ml * (ks * cz + jz));
        if (gphi) acc_add(&gphi[nd], r[0] + m.inv_h * (r[1] + r[2] + r[3]), plain);
        if (gm) acc_add(&gm[nd], r[4], plain);
    }
    for (int f = f0; f < 6; f += Q) {
        dfl u[Q], v[Q];
        ld_line<Q, 1>(cb + f * NQ, l, u);
        Ln::template valT<false>(u, v);
        st_line<Q, 1>(cb + f * NQ, l, v);
    }
    __syncthreads();
    if (!active) return;
    for (int f = f0; f < 6; f += Q) {  // z, and the scatter
        double* const out = f < 3 ? gx : gu;
        if (!out) continue;
        double* dst = out + (f < 3 ? f : f - 3) * m.Nu + zoff;
        const unsigned cons = f < 3 ? zcons : 0u;
        dfl u[Q], v[Q];
        ld_line<Q, 2>(cb + f * NQ, l, u);
        Ln::template valT<true>(u, v);
#pragma unroll
        for (int k = 0; k < Q; ++k)
            if (!((cons >> k) & 1u)) acc_add(&dst[k * zst], df_to_double(v[k]), plain);
    }
}

int launch_adjoint(evap_mesh* h, const double* w, const double* wp, const double* x, double* gx, double* gu,
                   double* gphi, double* gm, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    const unsigned gi = (unsigned)std::min<int64_t>((3 * (int64_t)m.M * m.M + 7) / 8, 152 * 16);
    k_adjoint_init<<<gi, 256, 0, s>>>(m.M, m.Nu, m.Nphi, m.faces, w, gx, gu, gphi, gm);
    EVAP_CHECK_LAUNCH("adjoint_init");
    const float2* qcd = reinterpret_cast<const float2*>(h->qcdf);
    const dfl rho_liq = df_from_double(m.rho_H1), rho_gas = df_from_double(m.rho_H0);  // rho outside table cells
    const int c0 = h->deterministic ? 0 : -1, c1 = h->deterministic ? 8 : 0;  // colour passes, or one atomic pass
    auto run = [&](auto kern, int CB, int threads, size_t dyn) -> int {
        for (int colour = c0; colour < std::max(c1, c0 + 1); ++colour) {
            const int64_t cells = colour_cells(m.n, colour);
            if (cells == 0) continue;
            kern<<<(unsigned)((cells + CB - 1) / CB), threads, dyn, s>>>(m, h->b, rho_liq, rho_gas, h->cell_code,
                                                                       h->table_index, h->adj_table, qcd, w, wp, x,
                                                                       gx, gu, gphi, gm, colour);
            EVAP_CHECK_LAUNCH("adjoint");
        }
        return EVAP_OK;
    };
    if (m.P == 2) {
        constexpr int CB = EVAP_ADJ_CB2, MB = EVAP_ADJ_MINB2;
        return m.nsub == 1 ? run(k_adjoint<2, CB, 2, MB>, CB, CB * 27, adj_smem<2, CB>())
                           : run(k_adjoint<2, CB, 3, MB>, CB, CB * 27, adj_smem<2, CB>());
    }
    constexpr int CB = EVAP_ADJ_CB3, MB = EVAP_ADJ_MINB3;
    return m.nsub == 1 ? run(k_adjoint<3, CB, 2, MB>, CB, CB * 64, adj_smem<3, CB>())
                       : run(k_adjoint<3, CB, 3, MB>, CB, CB * 64, adj_smem<3, CB>());
}

}  // namespace evap
