// FP64-accurate momentum apply in double-float arithmetic: the velocity block of Eq. weakNavierStokes linearized
// about u0 (App. D) with the corrected stress of Eq. modified_viscous_stress, the divergence row of Eq. continuity and,
// for the velocity-pressure apply, the pressure term -(div v, p), y = sum_i R_i^T A_i R_i x (Sec. 2.5), with every
// sweep, flux and test evaluated on hi + lo pairs of FP32 numbers (dfloat.cuh):
//   gather   x, u0 at the (P+1)^3 nodes (Dirichlet nodes of x read as 0), converted to double-float
//   values   3 sweeps of the 1D matrix S[q][a] = l_a(t_q) per component            -> x_c at the Gauss points
//   grads    collocation derivative Dc at the Gauss points along each direction     -> d_b x_c
//   flux     F_c  = W rho (c_m x_c + u0 . grad x_c + newton (grad u0 x)_c)
//            T_cb = 2 W mu (eps_cb - tr(eps) (z n)_c (z n)_b),  eps = sym grad x
//   test     w_c = F_c + sum_b Dc^T T_cb, then 3 transposed sweeps S^T            -> nodal contributions
//   scatter  atomic FP64 add into y (constrained rows hold y = x, written by the init kernel)
//
// Why: on GB300 the FP64 pipe (~1.2 TFLOP/s measured) bounds the plain FP64 apply two orders of magnitude below the
// HBM roof, while the FP32 pipe issues ~60x as many FMAs.  A double-float multiply-add costs ~12 FP32 instructions, so
// the same Gauss sums at ~48-bit precision (relative rounding ~4e-15 per operation, below the 1e-12 parity bar by
// two orders of magnitude) leave the FP64 pipe with only the conversions of the nodal values (x in, y out).
//
// Layout: CB cells per block with Q^3 threads each.  In a sweep a thread owns one line of Q points of one component
// (Q^2 lines x 3 components: every thread for Q = 3, 48 of 64 for Q = 4) and forms its Q results in registers with the
// line transforms of df_lines.cuh, so a sweep costs Q shared loads and Q stores per thread; the fluxes are
// formed by one thread per quadrature point.  The first sweep (z) gathers its lines from memory and the last one (z)
// scatters its own, both as rows of x-consecutive nodes.  The lines of the test along y and z overlay the coefficient
// slots, which the fluxes have read by then.
// What bounds it: FP32 issue (the additions of the error-free transformations).
//
// The quadrature-point coefficients are the pairs of k_qp_coeffs (qcdf, [cell][QC_K][nq] float2), 8 bytes per
// coefficient as in FP64, with the factor kappa = DSCALE / h of the derivative in the slots that multiply one (1..3,
// 17) and kappa^2 in the viscous one (13).  Each thread copies its point's coefficients into shared memory with
// cp.async at the start, so that their HBM latency is hidden behind the interpolation sweeps.  The correction term is
// skipped at points where its gate z n is zero (outside the interface zone), and the Newton terms on Picard meshes.
#include <algorithm>

#include "async_copy.cuh"
#include "df_lines.cuh"
#include "physics.cuh"

namespace evap {

// slots of a cell in shared memory (pairs of Q^3 points): 0..2 X (then F), 3..11 G_kd at 3 + 3 k + d (then the six
// stress entries at 3.., the divergence row at 9), 12.. the coefficients (then the tests along y and z, 6 slots)
constexpr int DF_SLOTS = 12;
template <int P, int CB>
constexpr size_t df_smem() {
    return sizeof(float2) * CB * (DF_SLOTS + QC_K) * (P + 1) * (P + 1) * (P + 1);
}
// slot of the symmetric stress entry (k, l)
__device__ __forceinline__ constexpr int t_slot(int k, int l) {
    return 3 + (k <= l ? (k * (5 - k)) / 2 + l : (l * (5 - l)) / 2 + k);
}

// Cells per block and blocks per SM (a register cap).  Measured at 64^3 Q2 with the divergence row (us per apply; one
// point per thread with Q-term dot products: 673): CB 1 / 28 blocks 503 (a block is one warp), 495 with the sweeps
// ordered by warp barriers (128^3: 3610 -> 3518), 489 with three-term dots (3499); 2 / 16 526; 4 / 8 510; 5 / 6 552; 7 / 4 592; 8 / 4
// 581; 13 / 2 757 (these with 503).
// Q3 at 45^3 (701 before): 2 and 4 cells 544, 1 cell 579.  ncu at 64^3: 1843 warp instructions per cell, issue 82 % active, FP64
// pipe 68 % (conversions).
#ifndef EVAP_DF_CB2
#define EVAP_DF_CB2 1
#endif
#ifndef EVAP_DF_MINB2
#define EVAP_DF_MINB2 28
#endif
#ifndef EVAP_DF_CB3
#define EVAP_DF_CB3 2
#endif
#ifndef EVAP_DF_MINB3
#define EVAP_DF_MINB3 4
#endif

// The pressure space at the 1D Gauss points: shape values as pairs, and the points in FP64.
struct Q1Basis {
    dfl N1[MAXQ][2];
    double t[MAXQ];
};

template <int P, int CB, bool PRES, int MINB, bool DET>
__global__ void __launch_bounds__(CB*(P + 1) * (P + 1) * (P + 1), MINB)
    k_momentum_df(MeshArgs<double> m, const __grid_constant__ Q1Basis bas, const float2* __restrict__ qc, const double* __restrict__ x,
                  double* __restrict__ y, double* __restrict__ yp, const double* __restrict__ pin, int colour) {
    constexpr int Q = P + 1, NQ = Q * Q * Q, NL = Q * Q, TASKS = 3 * NL;
    using Ln = DfLine<Q>;
    auto sync = [] {  // a block of one warp needs no block barrier
        if (CB * NQ <= 32) __syncwarp();
        else __syncthreads();
    };
    __shared__ dfl sN1[Q][2];
    __shared__ dfl q1a[CB][2 * Q * Q], q1b[CB][4 * Q];
    // the pressure at the cell's corners, then interpolated along x and y (z: by the point's thread), in FP64: 2 FP64
    // operations per sweep instead of 14 per point (672 -> 562 us at 64^3, the call with its initialization 608, 584 with the line
    // transforms as they are; the pressure interpolated in double-float arithmetic 531, but with a larger error of the pressure term)
    __shared__ double p0[PRES ? CB : 1][8], px[PRES ? CB : 1][4 * Q], py[PRES ? CB : 1][2 * Q * Q];
    auto lerp = [&](double u, double v, int q) -> double { return fma(bas.t[q], v - u, u); };  // at Gauss point q
    extern __shared__ float2 smem_df[];
    dfl* const sb = reinterpret_cast<dfl*>(smem_df);  // [cell][slot][point]
    constexpr int CELL = (DF_SLOTS + QC_K) * NQ;
    const int tid = threadIdx.x;
    const int n = m.n, M = m.M;
    const unsigned cell0 = blockIdx.x * CB;
    constexpr bool plain = DET;  // a colour pass: no other cell of the launch touches this cell's nodes
    // ---- point view: cell lc, point t = (a, b, c)
    const int lc = tid / NQ, t = tid % NQ;
    int cx, cy, cz;
    const bool active = colour_cell32(cell0 + lc, n, DET ? colour : -1, cx, cy, cz);
    dfl* const cb = sb + lc * CELL;
    {
        const int64_t cell = cx + (int64_t)n * (cy + (int64_t)n * cz);
        float2* myq = reinterpret_cast<float2*>(cb + DF_SLOTS * NQ + t);
        // each thread fetches (and later reads) only its own point's coefficients
        const float2* src = qc + cell * QC_K * NQ + t;
#pragma unroll
        for (int k = 0; k < QC_K; ++k)
            if (m.newton || k < 4 || k > 12) cp_async8(myq + k * NQ, src + k * NQ);
        cp_async_commit();
    }
    if (tid < 2 * Q) sN1[tid / 2][tid % 2] = bas.N1[tid / 2][tid % 2];
    // ---- line view: cell ll, component f, line l
    const int ll = Q == 3 ? lc : tid / TASKS, task = Q == 3 ? t : tid % TASKS;
    const int f = task / NL, l = task % NL;
    int lx = cx, ly = cy, lz = cz;
    bool lact = active;  // the line's cell exists (a block's missing cells repeat the last one and scatter nothing)
    if (Q != 3) lact = colour_cell32(cell0 + ll, n, DET ? colour : -1, lx, ly, lz);
    const bool line = Q == 3 || ll < CB;  // this thread owns a line
    dfl* const lb = sb + (line ? ll : 0) * CELL;
    // the z-line of nodes this thread gathers and scatters, and which of them are free
    const int gx = P * lx + l % Q, gy = P * ly + l / Q, gz0 = P * lz;
    const int64_t zst = (int64_t)M * M;
    const int64_t gidx = (int64_t)f * m.Nu + gx + (int64_t)M * gy + zst * gz0;
    unsigned cons = 0;  // bit k: node k is constrained
    if (line) {
        const unsigned fc = m.faces;
        const bool cxy = ((fc & 1u) && gx == 0) || ((fc & 2u) && gx == M - 1) || ((fc & 4u) && gy == 0) ||
                         ((fc & 8u) && gy == M - 1);
        cons = cxy ? (1u << Q) - 1u : 0u;
        if ((fc & 16u) && gz0 == 0) cons |= 1u;
        if ((fc & 32u) && gz0 + P == M - 1) cons |= 1u << P;
        dfl u[Q], v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) u[k] = (cons >> k) & 1u ? dfl{0.f, 0.f} : df_from_double(x[gidx + k * zst]);
        Ln::val(u, v);
        st_line<Q, 2>(lb + (3 + f) * NQ, l, v);
    }
    if (PRES && tid < CB * 8) {
        const int c2 = tid / 8, o = tid % 8;
        int ex, ey, ez;
        colour_cell32(cell0 + c2, n, DET ? colour : -1, ex, ey, ez);
        const int64_t m1 = n + 1;
        p0[c2][o] = pin[(ex + (o & 1)) + m1 * ((ey + ((o >> 1) & 1)) + m1 * (ez + (o >> 2)))];
    }
    sync();
    if (PRES && tid < CB * 4 * Q) {  // [qx][jb][jc]
        const int c2 = tid / (4 * Q), o = tid % (4 * Q), q = o % Q, r = o / Q;
        px[c2][o] = lerp(p0[c2][2 * r], p0[c2][2 * r + 1], q);
    }
    if (line) {
        dfl u[Q], v[Q];
        ld_line<Q, 1>(lb + (3 + f) * NQ, l, u);
        Ln::val(u, v);
        st_line<Q, 1>(lb + (6 + f) * NQ, l, v);
    }
    sync();
    if (PRES && tid < CB * 2 * Q * Q) {  // [qx][qy][jc]
        const int c2 = tid / (2 * Q * Q), o = tid % (2 * Q * Q), q = o % Q, r = (o / Q) % Q, jc = o / (Q * Q);
        py[c2][o] = lerp(px[c2][q + Q * (2 * jc)], px[c2][q + Q * (2 * jc + 1)], r);
    }
    if (line) {  // x: the values at the points, and their derivative along x
        dfl u[Q], v[Q];
        ld_line<Q, 0>(lb + (6 + f) * NQ, l, u);
        Ln::val(u, v);
        st_line<Q, 0>(lb + f * NQ, l, v);
    }
    sync();
    if (line) {
        dfl u[Q], v[Q];
        ld_line<Q, 0>(lb + f * NQ, l, u);
        Ln::der(u, v);
        st_line<Q, 0>(lb + (3 + 3 * f) * NQ, l, v);
        ld_line<Q, 1>(lb + f * NQ, l, u);
        Ln::der(u, v);
        st_line<Q, 1>(lb + (4 + 3 * f) * NQ, l, v);
        ld_line<Q, 2>(lb + f * NQ, l, u);
        Ln::der(u, v);
        st_line<Q, 2>(lb + (5 + 3 * f) * NQ, l, v);
    }
    sync();
    // quadrature-point fluxes from the cached coefficients; a thread reads and overwrites its own point's entries only
    {
        dfl X[3], G[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            X[k] = cb[k * NQ + t];
#pragma unroll
            for (int d = 0; d < 3; ++d) G[k][d] = cb[(3 + 3 * k + d) * NQ + t];
        }
        cp_async_wait_all();
        const dfl* q = cb + DF_SLOTS * NQ + t;
        const dfl c0 = q[0];
        const dfl cu[3] = {q[NQ], q[2 * NQ], q[3 * NQ]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dfl v = df_prod(c0, X[k]);
#pragma unroll
            for (int d = 0; d < 3; ++d) df_fma(v, cu[d], G[k][d]);
            if (m.newton) {
#pragma unroll
                for (int d = 0; d < 3; ++d) df_fma(v, q[(4 + 3 * k + d) * NQ], X[d]);
            }
            cb[k * NQ + t] = v;  // only starts a new accumulation: left unnormalized
        }
        const dfl c13 = q[13 * NQ];
        const dfl tr = df_add(df_add(G[0][0], G[1][1]), G[2][2]);
        const dfl hm = df_scale2(c13, 0.5f);
        const dfl nz[3] = {q[14 * NQ], q[15 * NQ], q[16 * NQ]};
        const bool corr = (nz[0].hi != 0.f) || (nz[1].hi != 0.f) || (nz[2].hi != 0.f);
        const dfl sm = corr ? df_mul(c13, tr) : dfl{0.f, 0.f};
        const dfl rw = q[17 * NQ];  // kappa W
        dfl wp{0.f, 0.f};
        if constexpr (PRES) wp = df_mul(rw, df_from_double(lerp(py[lc][t % NL], py[lc][t % NL + NL], t / NL)));
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int e = k; e < 3; ++e) {  // symmetric: 6 distinct entries
                dfl v = k == e ? df_mul(c13, G[k][k]) : df_mul(hm, df_add(G[k][e], G[e][k]));
                if (corr) {
                    dfl w = v;
                    df_fma(w, df_neg(sm), df_mul(nz[k], nz[e]));
                    v = df_norm(w);
                }
                if (PRES && k == e) v = df_sub(v, wp);
                cb[t_slot(k, e) * NQ + t] = v;
            }
        if (yp) {
            dfl r = df_prod(rw, tr);
            const dfl src = q[18 * NQ];
            const dfl s2 = two_sum(r.hi, -src.hi);
            r.hi = s2.hi;
            r.lo = __fadd_rn(r.lo, __fsub_rn(s2.lo, src.lo));
            cb[9 * NQ + t] = df_norm(r);
        }
    }
    sync();
    // test with gradients: the lines along y and z into the coefficients' slots
    if (line) {
        dfl u[Q], v[Q];
        ld_line<Q, 1>(lb + t_slot(f, 1) * NQ, l, u);
        Ln::derT(u, v);
        st_line<Q, 1>(lb + (DF_SLOTS + f) * NQ, l, v);
        ld_line<Q, 2>(lb + t_slot(f, 2) * NQ, l, u);
        Ln::derT(u, v);
        st_line<Q, 2>(lb + (DF_SLOTS + 3 + f) * NQ, l, v);
    }
    // divergence row, Q1 test functions: sum_q N1_j(q) r_q by three sweeps, whose outputs fill the first warps
    if (yp && tid < CB * 2 * Q * Q) {  // x-sweep: [jx][qy][qz]
        const int c2 = tid / (2 * Q * Q), o = tid % (2 * Q * Q);
        const dfl* r = sb + c2 * CELL + 9 * NQ + Q * (o >> 1);
        dfl s = df_prod(sN1[0][o & 1], r[0]);
#pragma unroll
        for (int qq = 1; qq < Q; ++qq) df_fma(s, sN1[qq][o & 1], r[qq]);
        q1a[c2][o] = df_norm(s);
    }
    sync();
    if (line) {  // x: F + the three tests, and its value sweep
        dfl u[Q], v[Q], w[Q];
        ld_line<Q, 0>(lb + t_slot(f, 0) * NQ, l, u);
        Ln::derT(u, v);
        ld_line<Q, 0>(lb + f * NQ, l, w);
        ld_line<Q, 0>(lb + (DF_SLOTS + f) * NQ, l, u);
#pragma unroll
        for (int k = 0; k < Q; ++k) w[k] = df_addl(df_addl(w[k], v[k]), u[k]);
        ld_line<Q, 0>(lb + (DF_SLOTS + 3 + f) * NQ, l, u);
#pragma unroll
        for (int k = 0; k < Q; ++k) w[k] = df_add(w[k], u[k]);
        Ln::template valT<false>(w, v);
        st_line<Q, 0>(lb + f * NQ, l, v);
    }
    if (yp && tid < CB * 4 * Q) {  // y-sweep: [jx][jy][qz]
        const int c2 = tid / (4 * Q), o = tid % (4 * Q), jx = o & 1, jy = (o >> 1) & 1, qz = o >> 2;
        dfl s = df_prod(sN1[0][jy], q1a[c2][jx + 2 * (0 + Q * qz)]);
#pragma unroll
        for (int qq = 1; qq < Q; ++qq) df_fma(s, sN1[qq][jy], q1a[c2][jx + 2 * (qq + Q * qz)]);
        q1b[c2][o] = df_norm(s);
    }
    sync();
    if (line) {
        dfl u[Q], v[Q];
        ld_line<Q, 1>(lb + f * NQ, l, u);
        Ln::template valT<false>(u, v);
        st_line<Q, 1>(lb + f * NQ, l, v);
    }
    if (yp && tid < CB * 8) {  // z-sweep: Q1 node (jx, jy, jz)
        const int c2 = tid / 8, o = tid % 8, jx = o & 1, jy = (o >> 1) & 1, jz = o >> 2;
        int ex, ey, ez;
        if (colour_cell32(cell0 + c2, n, DET ? colour : -1, ex, ey, ez)) {
            dfl s = df_prod(sN1[0][jz], q1b[c2][jx + 2 * (jy + 2 * 0)]);
#pragma unroll
            for (int qq = 1; qq < Q; ++qq) df_fma(s, sN1[qq][jz], q1b[c2][jx + 2 * (jy + 2 * qq)]);
            const int64_t m1 = n + 1;
            acc_add(&yp[(ex + jx) + m1 * ((ey + jy) + m1 * (ez + jz))], df_to_double(df_norm(s)), plain);
        }
    }
    sync();
    if (line && lact) {  // z, and the scatter of the line's free nodes
        dfl u[Q], v[Q];
        ld_line<Q, 2>(lb + f * NQ, l, u);
        Ln::template valT<true>(u, v);
#pragma unroll
        for (int k = 0; k < Q; ++k)
            if (!((cons >> k) & 1u)) acc_add(&y[gidx + k * zst], df_to_double(v[k]), plain);
    }
}

// y = A x (+ y_p = B x - g, + the pressure term when p is given); the init kernel has written y = x on the Dirichlet
// DoFs (faces of m) and zeros elsewhere.
int launch_momentum_df(evap_mesh* h, const MeshArgs<double>& m, const double* x, double* y, double* yp,
                       const double* p, cudaStream_t s) {
    Q1Basis b{};
    for (int q = 0; q < h->b.Q; ++q) {
        b.t[q] = h->b.t[q];
        for (int j = 0; j < 2; ++j) b.N1[q][j] = df_from_double(h->b.N1[q][j]);
    }
    const float2* qc = reinterpret_cast<const float2*>(h->qcdf);
    const int c0 = h->deterministic ? 0 : -1, c1 = h->deterministic ? 8 : 0;  // colour passes, or one atomic pass
    // at most 48 KB of shared memory per block, so no launch needs a function attribute
    auto run = [&](auto kern, int CB, int threads, size_t dyn) -> int {
        for (int colour = c0; colour < std::max(c1, c0 + 1); ++colour) {
            const int64_t cells = colour_cells(m.n, colour);
            if (cells == 0) continue;
            const unsigned grid = (unsigned)((cells + CB - 1) / CB);
            kern<<<grid, threads, dyn, s>>>(m, b, qc, x, y, yp, p, colour);
            EVAP_CHECK_LAUNCH("momentum_df");
        }
        return EVAP_OK;
    };
    const bool det = h->deterministic;
    if (m.P == 2) {
        constexpr int CB = EVAP_DF_CB2, MINB = EVAP_DF_MINB2;
        constexpr size_t dyn = df_smem<2, CB>();
        return p ? run(det ? k_momentum_df<2, CB, true, MINB, true> : k_momentum_df<2, CB, true, MINB, false>, CB,
                       CB * 27, dyn)
                 : run(det ? k_momentum_df<2, CB, false, MINB, true> : k_momentum_df<2, CB, false, MINB, false>, CB,
                       CB * 27, dyn);
    }
    constexpr int CB = EVAP_DF_CB3, MINB = EVAP_DF_MINB3;
    constexpr size_t dyn = df_smem<3, CB>();
    return p ? run(det ? k_momentum_df<3, CB, true, MINB, true> : k_momentum_df<3, CB, true, MINB, false>, CB, CB * 64,
                   dyn)
             : run(det ? k_momentum_df<3, CB, false, MINB, true> : k_momentum_df<3, CB, false, MINB, false>, CB,
                   CB * 64, dyn);
}

}  // namespace evap
