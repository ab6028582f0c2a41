// Surface-tension force of Eq. (surfaceTension) as the right-hand side of the momentum equation, FP64:
//   b_(i,c) = sum_q W_q N_i(x_q) alpha kappa_h(x_q) n_c(x_q) delta(x_q) rho(x_q) c_rho,
//   c_rho = (rho_g - rho_l) / (rho_l rho_g ln(rho_g / rho_l))  (the density-scaled delta, same section),
// kappa_h and n_h the caller's Q1 curvature and normal fields on the level-set mesh (normalized at the point:
// n_h / |n_h|, zero where |n_h| <= 1e-4), delta (Eq. delta) and the reciprocal rho (Eq. rhoEff) from the level set at
// the point.  One thread
// per velocity quadrature point; the test with the Q_p shape functions runs as three transposed 1D sweeps
// (z, y, x) through shared memory.  Dirichlet-constrained entries stay zero.  Cells outside the interface zone are
// skipped (one cell in eight is not, on four drops at 64^3), delta and rho come from the material-law table: 3156 us at
// 64^3 Q2 when every cell evaluated its interpolants and the material law, now 270.
#include <cmath>
#include <cstring>
#include <limits>

#include "physics.cuh"

namespace evap {

template <int P, int CB>
__global__ void __launch_bounds__(CB*(P + 1) * (P + 1) * (P + 1))
    k_surface_tension(MeshArgs<double> m, Basis<double> bas, const int8_t* __restrict__ code,
                      const int32_t* __restrict__ tindex, const double* __restrict__ table,
                      const double* __restrict__ nf, const double* __restrict__ kappa, unsigned kappa_hi, double alpha_crho,
                      double* __restrict__ out) {
    constexpr int Q = P + 1, NQ = Q * Q * Q;
    __shared__ double sS[Q][Q];
    __shared__ double buf[2][CB][3][NQ];
    const int tid = threadIdx.x;
    const int lc = tid / NQ, t = tid % NQ;
    const int64_t cell = (int64_t)blockIdx.x * CB + lc;
    const int a = t % Q, b = (t / Q) % Q, c = t / (Q * Q);
    const int n = m.n;
    int cx = 0, cy = 0, cz = 0;
    // delta vanishes in cells without a point of the interface zone: their contribution is zero unless the caller's
    // factor or fields are not finite there, or the product of factor and curvature may not be (kappa_hi: launch)
    bool active = cell < m.ncell;
    if (active) {
        cx = (int)(cell % n);
        cy = (int)((cell / n) % n);
        cz = (int)(cell / ((int64_t)n * n));
        const int ns = m.nsub, ml = m.nl + 1, K = ns + 1;
        bool need = code[cell] == CELL_TABLE;
        for (int j = t; j < K * K * K && !need; j += NQ) {
            const int64_t node = (ns * cx + j % K) + (int64_t)ml * ((ns * cy + (j / K) % K) + (int64_t)ml * (ns * cz + j / (K * K)));
            need = !(((unsigned)__double2hiint(kappa[node]) & 0x7fffffffu) < kappa_hi && isfinite(nf[node]) && isfinite(nf[m.Nphi + node]) &&
                     isfinite(nf[2 * m.Nphi + node]));
        }
        active = need;
    }
    __shared__ int run[CB];
    if (tid < CB) run[tid] = 0;
    __syncthreads();
    if (active) run[lc] = 1;
    if (!__syncthreads_or(active)) return;
    active = run[lc] != 0;
    if (tid < Q * Q) sS[tid / Q][tid % Q] = bas.S[tid / Q][tid % Q];
    if (active) {
        // level-set-space fields at the point: the Q1 interpolants of the level-set cell containing it, with one set of
        // weights
        double loc[3] = {bas.t[a], bas.t[b], bas.t[c]};
        int sub[3] = {cx, cy, cz};
        if (m.nsub > 1) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double s = loc[d] * m.nsub;
                const int k = min(max((int)floor(s), 0), m.nsub - 1);
                sub[d] = m.nsub * sub[d] + k;
                loc[d] = s - k;
            }
        }
        const int64_t ml = m.nl + 1, base = sub[0] + ml * (sub[1] + ml * sub[2]);
        const double wx[2] = {1.0 - loc[0], loc[0]}, wy[2] = {1.0 - loc[1], loc[1]}, wz[2] = {1.0 - loc[2], loc[2]};
        double kq = 0.0, nh[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int jc = 0; jc < 2; ++jc)
#pragma unroll
            for (int jb = 0; jb < 2; ++jb) {
                const double wyz = wy[jb] * wz[jc];
                const int64_t r = base + ml * (jb + ml * jc);
                kq += wyz * (wx[0] * kappa[r] + wx[1] * kappa[r + 1]);
#pragma unroll
                for (int d = 0; d < 3; ++d) nh[d] += wyz * (wx[0] * nf[d * m.Nphi + r] + wx[1] * nf[d * m.Nphi + r + 1]);
            }
        // delta and rho of the point from the material-law table of set_fields (outside the zone delta is 0)
        const double* tb = table + (int64_t)max(tindex[cell], 0) * TAB_K * NQ + t;
        const double dr = code[cell] == CELL_TABLE ? tb[6 * NQ] * tb[0] : 0.0;
        const double W = bas.w[a] * bas.w[b] * bas.w[c] * m.vol_w;
        const double nn = sqrt(nh[0] * nh[0] + nh[1] * nh[1] + nh[2] * nh[2]);
        const double s = nn > NODAL_NORMAL_TINY ? W * alpha_crho * kq * dr / nn : 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) buf[0][lc][d][t] = s * nh[d];
    }
    __syncthreads();
    // test with N_i = l_a(x) l_b(y) l_c(z): transposed sweeps z, y, x
    if (active)
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) v += sS[q][c] * buf[0][lc][f][a + Q * (b + Q * q)];
            buf[1][lc][f][t] = v;
        }
    __syncthreads();
    if (active)
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) v += sS[q][b] * buf[1][lc][f][a + Q * (q + Q * c)];
            buf[0][lc][f][t] = v;
        }
    __syncthreads();
    if (!active) return;
    const int M = m.M;
    const int gx = P * cx + a, gy = P * cy + b, gz = P * cz + c;
    const unsigned fc = m.faces;
    const bool cons = ((fc & 1u) && gx == 0) || ((fc & 2u) && gx == M - 1) || ((fc & 4u) && gy == 0) ||
                      ((fc & 8u) && gy == M - 1) || ((fc & 16u) && gz == 0) || ((fc & 32u) && gz == M - 1);
    if (cons) return;
    const int64_t gidx = gx + (int64_t)M * (gy + (int64_t)M * gz);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) v += sS[q][a] * buf[0][lc][f][q + Q * (b + Q * c)];
        atomicAdd(&out[f * m.Nu + gidx], v);
    }
}

int launch_surface_tension(evap_mesh* h, const double* nf, const double* kappa, double alpha, double* out,
                           cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    const double rl = m.rho_l, rg = m.rho_g;
    const double crho = (rg - rl) / (rl * rg * std::log(rg / rl));
    // high word from which on a curvature is not finite or its product with the factor may overflow; 0, every curvature, for
    // a factor that is not finite
    const double fac = std::fabs(alpha * crho);
    unsigned kappa_hi = 0;
    if (std::isfinite(fac)) {
        const double most = fac > 1.0 ? std::numeric_limits<double>::max() / fac : std::numeric_limits<double>::infinity();
        uint64_t bits;
        std::memcpy(&bits, &most, sizeof(bits));
        kappa_hi = (unsigned)(bits >> 32);
    }
    EVAP_CUDA(cudaMemsetAsync(out, 0, 3 * m.Nu * sizeof(double), s));
    if (m.P == 2) {
        constexpr int CB = 8;
        k_surface_tension<2, CB><<<(unsigned)((m.ncell + CB - 1) / CB), CB * 27, 0, s>>>(m, h->b, h->cell_code, h->table_index, h->table, nf, kappa,
                                                                                        kappa_hi, alpha * crho, out);
    } else {
        constexpr int CB = 4;
        k_surface_tension<3, CB><<<(unsigned)((m.ncell + CB - 1) / CB), CB * 64, 0, s>>>(m, h->b, h->cell_code, h->table_index, h->table, nf, kappa,
                                                                                        kappa_hi, alpha * crho, out);
    }
    EVAP_CHECK_LAUNCH("surface_tension");
    return EVAP_OK;
}

}  // namespace evap
