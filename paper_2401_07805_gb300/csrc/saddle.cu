// Velocity-pressure coupling of Eq. (weakNavierStokes) with the Q1 pressure of Sec. 2.5 (k_p = 1), FP64:
//   pressure gradient of the preconditioner   t = v + B^T p   (the saddle-point apply folds its pressure term -(div v, p)
//                                       into the momentum kernel's stress flux)
//   continuity right-hand side         g_j = sum_q W N1_j v_dil                           (Eq. continuity, evaporDil)
//   saddle-point apply                 [y; y_p] = [A x - B^T p; B x]
// with B the divergence row of the momentum apply (velocity Gauss rule, Dirichlet entries of x read as 0) and
// Dirichlet-constrained velocity rows left to the momentum apply (identity), so B^T p vanishes there.
#include "dfloat.cuh"
#include "physics.cuh"

namespace evap {

// t = v + B^T p with the gradient in FP32.  B_c[j][v] = prod_d F^c_d[j_d][v_d] is a tensor product of 1D integrals (as in
// schur.cu: g1 = the integral of N1_J l_V' along c, a1 = that of N1_J l_V along the other two, both exact with the
// velocity Gauss rule), and a velocity node meets at most 3 pressure nodes per direction.  So one thread per velocity node
// sums its 3 x 3 x 3 neighbours separably (x, then y, then z) and adds v: no scatter, no intermediate vector.  Measured at
// 64^3 Q2 (us): 63; a quadrature kernel with its scatter, memset and addition took 109 + 4 + 28.
// The 1D row of velocity node V: its first pressure node I0 and the factors of I0, I0 + 1, I0 + 2 (0 where there is none).
__device__ __forceinline__ int gradient_row(const float (&a1)[2][MAXQ], const float (&g1)[2][MAXQ], int P, int n, int V,
                                            float (&a)[3], float (&g)[3]) {
    const int e = V / P, b = V - e * P;  // cell and local node; b = 0: a vertex, shared with cell e - 1
    a[0] = a[1] = a[2] = g[0] = g[1] = g[2] = 0.f;
    if (b != 0) {  // inside cell e: pressure nodes e, e + 1
        a[0] = a1[0][b]; a[1] = a1[1][b];
        g[0] = g1[0][b]; g[1] = g1[1][b];
        return e;
    }
    // vertex e: node e - 1 and e from cell e - 1 (local node P), e and e + 1 from cell e (local node 0)
    if (e > 0) {
        a[0] = a1[0][P]; a[1] = a1[1][P];
        g[0] = g1[0][P]; g[1] = g1[1][P];
    }
    if (e < n) {
        a[1] += a1[0][0]; a[2] = a1[1][0];
        g[1] += g1[0][0]; g[2] = g1[1][0];
    }
    return e - 1;
}
__global__ void __launch_bounds__(128) k_add_gradient(int n, int P, int M, int64_t Nu, unsigned faces, CouplingTables tab,
                                                      const float* __restrict__ p, const double* __restrict__ v,
                                                      double* __restrict__ t) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
    if (x >= M || y >= M) return;
    const int64_t node = x + (int64_t)M * (y + (int64_t)M * z);
    float acc[3] = {0.f, 0.f, 0.f};
    if (!constrained_node(x, y, z, M, faces)) {
        float ax[3], gx[3], ay[3], gy[3], az[3], gz[3];
        const int ix = gradient_row(tab.a, tab.g, P, n, x, ax, gx), iy = gradient_row(tab.a, tab.g, P, n, y, ay, gy),
                  iz = gradient_row(tab.a, tab.g, P, n, z, az, gz);
        const int m1 = n + 1;
#pragma unroll
        for (int kz = 0; kz < 3; ++kz) {
            if (az[kz] == 0.f && gz[kz] == 0.f) continue;
            float r0 = 0.f, r1 = 0.f, r2 = 0.f;
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                if (ay[ky] == 0.f && gy[ky] == 0.f) continue;
                const float* row = p + ix + (int64_t)m1 * ((iy + ky) + (int64_t)m1 * (iz + kz));
                float sa = 0.f, sg = 0.f;
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    if (ax[kx] == 0.f && gx[kx] == 0.f) continue;  // (also keeps the reads inside the lattice)
                    const float q = row[kx];
                    sa = fmaf(ax[kx], q, sa);
                    sg = fmaf(gx[kx], q, sg);
                }
                r0 = fmaf(ay[ky], sg, r0);
                r1 = fmaf(gy[ky], sa, r1);
                r2 = fmaf(ay[ky], sa, r2);
            }
            acc[0] = fmaf(az[kz], r0, acc[0]);
            acc[1] = fmaf(az[kz], r1, acc[1]);
            acc[2] = fmaf(gz[kz], r2, acc[2]);
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) t[c * Nu + node] = v[c * Nu + node] + (double)acc[c];
}

// g_j += sum_q N1_j(x_q) (W v_dil)_q over the cell's velocity Gauss points, from the cached coefficient slot 18.
template <int P>
__global__ void __launch_bounds__(128) k_continuity_rhs(MeshArgs<double> m, Basis<double> bas,
                                                        const float2* __restrict__ qc, double* __restrict__ g) {
    constexpr int Q = P + 1, NQ = Q * Q * Q;
    const int64_t cell = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (cell >= m.ncell) return;
    const int n = m.n;
    const int cx = (int)(cell % n), cy = (int)((cell / n) % n), cz = (int)(cell / ((int64_t)n * n));
    const float2* v = qc + cell * QC_K * NQ + 18 * NQ;
    double out[8] = {};
    for (int t = 0; t < NQ; ++t) {
        const int a = t % Q, b = (t / Q) % Q, c = t / (Q * Q);
        const double vt = df_to_double(ld_df(v + t));
#pragma unroll
        for (int j = 0; j < 8; ++j)
            out[j] += bas.N1[a][j & 1] * bas.N1[b][(j >> 1) & 1] * bas.N1[c][j >> 2] * vt;
    }
    const int64_t m1 = n + 1;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        atomicAdd(&g[(cx + (j & 1)) + m1 * ((cy + ((j >> 1) & 1)) + m1 * (cz + (j >> 2)))], out[j]);
}

// f += sum_q W rho c_m N_i (u_c + g_c / c_m) at the velocity Gauss points (the BDF1 inertia load of the old velocity
// plus the body force), from the cached coefficient slot 0 (W rho c_m); Dirichlet entries of u are read as 0 and the
// constrained rows of f are left untouched (zero).
template <int P, int CB>
__global__ void __launch_bounds__(CB*(P + 1) * (P + 1) * (P + 1))
    k_mass_load(MeshArgs<double> m, Basis<double> bas, const float2* __restrict__ qc, const double* __restrict__ u,
                double g0, double g1, double g2, double* __restrict__ f) {
    constexpr int Q = P + 1, NQ = Q * Q * Q;
    __shared__ double sS[Q][Q];
    __shared__ double buf[2][3][CB][NQ];
    const int tid = threadIdx.x;
    const int lc = tid / NQ, t = tid % NQ;
    const int64_t cell = (int64_t)blockIdx.x * CB + lc;
    const bool active = cell < m.ncell;
    if (tid < Q * Q) sS[tid / Q][tid % Q] = bas.S[tid / Q][tid % Q];
    const int a = t % Q, b = (t / Q) % Q, c = t / (Q * Q);
    const int n = m.n, M = m.M;
    int64_t gidx = 0;
    bool cons = false;
    if (active) {
        const int cx = (int)(cell % n), cy = (int)((cell / n) % n), cz = (int)(cell / ((int64_t)n * n));
        const int gx = P * cx + a, gy = P * cy + b, gz = P * cz + c;
        gidx = gx + (int64_t)M * (gy + (int64_t)M * gz);
        cons = constrained_node(gx, gy, gz, M, m.faces);
#pragma unroll
        for (int k = 0; k < 3; ++k) buf[0][k][lc][t] = cons ? 0.0 : u[k * m.Nu + gidx];
    }
    __syncthreads();
    if (active)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double v = 0.0;
#pragma unroll
            for (int r = 0; r < Q; ++r) v += sS[a][r] * buf[0][k][lc][r + Q * (b + Q * c)];
            buf[1][k][lc][t] = v;
        }
    __syncthreads();
    if (active)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double v = 0.0;
#pragma unroll
            for (int r = 0; r < Q; ++r) v += sS[b][r] * buf[1][k][lc][a + Q * (r + Q * c)];
            buf[0][k][lc][t] = v;
        }
    __syncthreads();
    if (active) {
        const double cf0 = df_to_double(ld_df(qc + cell * QC_K * NQ + t));  // W rho c_m
        const double gc[3] = {g0 / m.c_mass, g1 / m.c_mass, g2 / m.c_mass};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double v = 0.0;
#pragma unroll
            for (int r = 0; r < Q; ++r) v += sS[c][r] * buf[0][k][lc][a + Q * (b + Q * r)];
            buf[1][k][lc][t] = cf0 * (v + gc[k]);
        }
    }
    __syncthreads();
    // test with N_i: transposed sweeps z, y, x
    if (active)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) v += sS[q][c] * buf[1][k][lc][a + Q * (b + Q * q)];
            buf[0][k][lc][t] = v;
        }
    __syncthreads();
    if (active)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) v += sS[q][b] * buf[0][k][lc][a + Q * (q + Q * c)];
            buf[1][k][lc][t] = v;
        }
    __syncthreads();
    if (!active || cons) return;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) v += sS[q][a] * buf[1][k][lc][q + Q * (b + Q * c)];
        atomicAdd(&f[k * m.Nu + gidx], v);
    }
}

int launch_mass_load(evap_mesh* h, const double* u, const double g[3], double* f, cudaStream_t st) {
    const MeshArgs<double>& m = h->m;
    EVAP_CUDA(cudaMemsetAsync(f, 0, 3 * m.Nu * sizeof(double), st));
    if (m.P == 2) {
        constexpr int CB = 8;
        k_mass_load<2, CB><<<(unsigned)((m.ncell + CB - 1) / CB), CB * 27, 0, st>>>(m, h->b, (const float2*)h->qcdf, u, g[0], g[1],
                                                                                   g[2], f);
    } else {
        constexpr int CB = 4;
        k_mass_load<3, CB><<<(unsigned)((m.ncell + CB - 1) / CB), CB * 64, 0, st>>>(m, h->b, (const float2*)h->qcdf, u, g[0], g[1],
                                                                                   g[2], f);
    }
    EVAP_CHECK_LAUNCH("mass_load");
    return EVAP_OK;
}

__global__ void k_add_vec(double* __restrict__ y, const double* __restrict__ g, int64_t N) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        y[i] += g[i];
}

int launch_add_gradient(evap_mesh* h, const float* p, const double* v, double* t, cudaStream_t st) {
    const MeshArgs<double>& m = h->m;
    const CouplingTables tab = coupling_tables(h);
    const dim3 grid((unsigned)((m.M + 31) / 32), (unsigned)((m.M + 3) / 4), (unsigned)m.M);
    k_add_gradient<<<grid, dim3(32, 4), 0, st>>>(m.n, m.P, m.M, m.Nu, m.faces, tab, p, v, t);
    EVAP_CHECK_LAUNCH("add_gradient");
    return EVAP_OK;
}

// z = S~^(-1) r, S~ = B diag(A)^(-1) B^T (a SIMPLE-type approximation of the Schur complement B A^(-1) B^T: it keeps
// the discrete B, so the pressure nodes of open faces are treated like every other node): at most cg_iters iterations
// of the FP32 single-launch CG on the assembled stencil (schur.cu), or |r| <= EVAP_SADDLE_SCHUR_RTOL |r0| (an inexact
// solve: the outer method is flexible).
#ifndef EVAP_SADDLE_SCHUR_RTOL
#define EVAP_SADDLE_SCHUR_RTOL 1e-6
#endif
int schur_apply(evap_mesh* h, const double* r, double* z, int cg_iters, cudaStream_t st) {
    return schur_solve(h, r, z, EVAP_SADDLE_SCHUR_RTOL, cg_iters, nullptr, st);
}

// g (the continuity right-hand side of the current fields), computed once per set_fields into h->cont_rhs.
int continuity_rhs(evap_mesh* h, const double** g, cudaStream_t st) {
    const MeshArgs<double>& m = h->m;
    if (!h->cont_rhs) EVAP_CUDA(cudaMalloc(&h->cont_rhs, m.Np * sizeof(double)));
    if (!h->cont_valid) {
        EVAP_CUDA(cudaMemsetAsync(h->cont_rhs, 0, m.Np * sizeof(double), st));
        const unsigned grid = (unsigned)blocks_for(m.ncell, 128, 1LL << 40);
        if (m.P == 2)
            k_continuity_rhs<2><<<grid, 128, 0, st>>>(m, h->b, (const float2*)h->qcdf, h->cont_rhs);
        else
            k_continuity_rhs<3><<<grid, 128, 0, st>>>(m, h->b, (const float2*)h->qcdf, h->cont_rhs);
        EVAP_CHECK_LAUNCH("continuity_rhs");
        h->cont_valid = true;
    }
    *g = h->cont_rhs;
    return EVAP_OK;
}

// [y; y_p] = [A x - B^T p; B x]: the momentum apply with the pressure term folded into its stress flux (whose
// divergence row is B x - g), followed by + g.
int launch_saddle_apply(evap_mesh* h, const double* x, const double* p, double* y, double* yp, cudaStream_t st,
                        bool lifted) {
    const double* g = nullptr;
    int rc = continuity_rhs(h, &g, st);
    if (rc) return rc;
    if ((rc = launch_momentum<double>(h, x, y, yp, st, true, p, lifted))) return rc;
    k_add_vec<<<blocks_for(h->m.Np, 256, 152 * 8), 256, 0, st>>>(yp, g, h->m.Np);
    EVAP_CHECK_LAUNCH("saddle_add_g");
    return EVAP_OK;
}

}  // namespace evap
