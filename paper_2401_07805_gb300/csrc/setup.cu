// evap_set_fields work: field preparation, FP64 quadrature-point coefficient table of the interface cells, and
// the level-set transport velocity with closest-point projection (App. C).
#include <cmath>

#include "df_lines.cuh"
#include "physics.cuh"

namespace evap {

template <typename T>
__global__ void k_fill(T* p, int64_t n, T v) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

__global__ void k_to_float(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

template <typename T>
int launch_fill(T* p, int64_t n, T v, cudaStream_t s) {
    k_fill<T><<<blocks_for(n, 256), 256, 0, s>>>(p, n, v);
    EVAP_CHECK_LAUNCH("fill");
    return EVAP_OK;
}
template int launch_fill<double>(double*, int64_t, double, cudaStream_t);
template int launch_fill<float>(float*, int64_t, float, cudaStream_t);

int launch_to_float(const double* a, float* b, int64_t n, cudaStream_t s) {
    k_to_float<<<blocks_for(n, 256), 256, 0, s>>>(a, b, n);
    EVAP_CHECK_LAUNCH("to_float");
    return EVAP_OK;
}

// b = (float)a and c = (hi, lo) of a
__global__ void k_to_float_df(const double* __restrict__ a, float* __restrict__ b, float2* __restrict__ c, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = a[i];
        const float hi = (float)v;
        b[i] = hi;
        c[i] = make_float2(hi, (float)(v - (double)hi));
    }
}

int refresh_ugamma_copies(evap_mesh* h, cudaStream_t s) {
    const int64_t n = 3 * h->m.Nphi;
    k_to_float_df<<<blocks_for(n, 256), 256, 0, s>>>(h->ugamma, h->ugamma32, (float2*)h->ugammadf, n);
    EVAP_CHECK_LAUNCH("ugamma_copies");
    return EVAP_OK;
}

// phi clamped to [-1, 1]; FP32 copies of phi and u.
__global__ void k_prepare(double* phi, float* phi32, const double* __restrict__ u, float* __restrict__ u32,
                          int64_t Np, int64_t Nu3) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Np; i += stride) {
        double v = phi[i];
        v = v > 1.0 ? 1.0 : (v < -1.0 ? -1.0 : v);
        phi[i] = v;
        phi32[i] = (float)v;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Nu3; i += stride) u32[i] = (float)u[i];
}

// Cell classification: all quadrature points liquid (H = 1), all gas (H = 0), or a table cell (interface zone,
// mixed phases, or correction applied everywhere).  Table cells get a slot by an atomic counter.
__global__ void k_classify(MeshArgs<double> m, Basis<double> b, const double* __restrict__ phi, int8_t* code,
                           int32_t* tindex, int32_t* counter) {
    const int64_t cell = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (cell >= m.ncell) return;
    const int n = m.n;
    const int cx = (int)(cell % n), cy = (int)((cell / n) % n), cz = (int)(cell / ((int64_t)n * n));
    bool all_liq = true, all_gas = true;
    // the interpolant lies between the cell's nodal values: away from the zone's edges these decide (most cells)
    constexpr double EDGE = PHI_BAND + 1e-12;  // more than the rounding of an interpolated value
    bool liq = true, gas = true;
    {
        const int k = m.nsub, ml = m.nl + 1;
        const double* f = phi + k * cx + (int64_t)ml * (k * cy + (int64_t)ml * (k * cz));
        for (int c = 0; c <= k; ++c)
            for (int bb = 0; bb <= k; ++bb)
                for (int a = 0; a <= k; ++a) {
                    const double v = f[a + ml * (bb + (int64_t)ml * c)];
                    liq = liq && v >= EDGE;
                    gas = gas && v <= -EDGE;
                }
    }
    if (liq || gas) {
        all_liq = liq;
        all_gas = gas;
    } else {
        for (int qz = 0; qz < b.Q && (all_liq || all_gas); ++qz)
            for (int qy = 0; qy < b.Q; ++qy)
                for (int qx = 0; qx < b.Q && (all_liq || all_gas); ++qx) {
                    double v, g[3];
                    ls_at(phi, m, cx, cy, cz, b.t[qx], b.t[qy], b.t[qz], v, g);
                    all_liq = all_liq && (v >= PHI_BAND);
                    all_gas = all_gas && (v <= -PHI_BAND);
                }
    }
    const bool everywhere = m.stress != 0 && m.corr_zone != 0;
    int8_t c = (!everywhere && all_liq) ? CELL_LIQUID : ((!everywhere && all_gas) ? CELL_GAS : CELL_TABLE);
    code[cell] = c;
    tindex[cell] = c == CELL_TABLE ? atomicAdd(counter, 1) : -1;
}

// Table entries at one quadrature point of a table cell: rho, mu, z n (z = correction gate), v_dil (Eq. evaporDil
// with the sign of App. A), delta.
//
// The FP64 pipe bounds it: one location and one set of weights for phi, its gradient and mdot, the logarithm, sine and
// cosine shared by the table and the adjoint's factors, one reciprocal for the normal.  The density jump multiplies the
// rounding of phi and H by up to the density ratio, so these keep their order of operations.  Measured at 64^3 (31.7 k
// table cells): 728 -> 486 us (an interpolation per field and every function evaluated twice before).
__global__ void k_fill_table(MeshArgs<double> m, Basis<double> b, const double* __restrict__ phi,
                             const double* __restrict__ mdot, const int8_t* __restrict__ code,
                             const int32_t* __restrict__ tindex, double kdmu, double kdk, double* table,
                             float* table32, float2* adj) {
    const unsigned nq = b.Q * b.Q * b.Q;
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const unsigned cell = (unsigned)(gid / nq);
    if (cell >= m.ncell || code[cell] != CELL_TABLE) return;
    const unsigned q = (unsigned)(gid - (int64_t)cell * nq);
    const unsigned Q = b.Q, qx = q % Q, qy = (q / Q) % Q, qz = q / (Q * Q);
    const unsigned n = m.n, row = cell / n;
    int ci[3] = {(int)(cell - row * n), (int)(row % n), (int)(row / n)};
    double loc[3] = {b.t[qx], b.t[qy], b.t[qz]};
    double ih = m.inv_h;
    if (m.nsub > 1) {  // the level-set cell holding the point (the upper one on a face)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double s = loc[a] * m.nsub;
            int c = (int)floor(s);
            c = c < 0 ? 0 : (c > m.nsub - 1 ? m.nsub - 1 : c);
            ci[a] = m.nsub * ci[a] + c;
            loc[a] = s - c;
        }
        ih *= m.nsub;
    }
    const int64_t m1 = m.nl + 1, base = ci[0] + m1 * (ci[1] + m1 * ci[2]);
    // the same weighted sums over the 8 nodes as ls_at, with their products formed once
    double ph = 0.0, g[3] = {0.0, 0.0, 0.0}, md = 0.0;
    {
        const double wx[2] = {1.0 - loc[0], loc[0]}, wy[2] = {1.0 - loc[1], loc[1]}, wz[2] = {1.0 - loc[2], loc[2]};
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int bb = 0; bb < 2; ++bb)
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const int64_t r = base + a + m1 * (bb + m1 * c);
                    const double v = phi[r], w = wx[a] * wy[bb] * wz[c];
                    ph += w * v;
                    md += w * mdot[r];
                    g[0] += (a ? wy[bb] : -wy[bb]) * wz[c] * v;
                    g[1] += (bb ? wx[a] : -wx[a]) * wz[c] * v;
                    g[2] += wx[a] * wy[bb] * (c ? v : -v);
                }
        g[0] *= ih;
        g[1] *= ih;
        g[2] *= ih;
    }
    // material law (Eqs. heaviside, rhoEff, muEff, normal_vector, delta) and
    // the derivatives of H: H'(d) d'(phi) and H''(d) d'(phi)^2 + H'(d) d''(phi)
    const bool zone = fabs(ph) < PHI_BAND;
    double H = ph >= PHI_BAND ? 1.0 : 0.0, dHdd = 0.0, d2 = 0.0;
    if (zone) {
        // (H in this very order: the reciprocal density multiplies its rounding by the density ratio)
        const double d = m.eps * log((1.0 + ph) / (1.0 - ph));
        double sn, cs;
        sincos(PI * d / (3.0 * m.eps), &sn, &cs);
        H = 0.5 + d / (6.0 * m.eps) + sn / (2.0 * PI);
        const double io = 1.0 / (1.0 - ph * ph);  // d'(phi) = 2 eps io, d''(phi) = 4 eps phi io^2
        const double h1 = (1.0 + cs) * (1.0 / 6.0), h2 = sn * (-PI / 18.0);  // eps H'(d), eps^2 H''(d)
        dHdd = 2.0 * h1 * io;
        d2 = 4.0 * (io * io) * (h2 + h1 * ph);
    }
    const double irl = 1.0 / m.rho_l, irg = 1.0 / m.rho_g;
    const double irho = H / m.rho_l + (1.0 - H) / m.rho_g, rho = 1.0 / irho;
    const double mu = H * m.mu_l + (1.0 - H) * m.mu_g;
    const double gn = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    const bool dir = gn * m.h > GRAD_TINY;
    const double ign = dir ? 1.0 / gn : 0.0;
    const double nv[3] = {dir ? g[0] * ign : 0.0, dir ? g[1] * ign : 0.0, dir ? g[2] * ign : 0.0};
    const double z = correction_on(m, zone) ? 1.0 : 0.0, kdil = irg - irl;  // c_1
    const double delta = zone ? dHdd * gn : 0.0;
    const double vals[TAB_K] = {rho, mu, z * nv[0], z * nv[1], z * nv[2], md * kdil * delta, delta};
    const int64_t tb = (int64_t)tindex[cell] * TAB_K * nq + q;
#pragma unroll
    for (int k = 0; k < TAB_K; ++k) {
        table[tb + (int64_t)k * nq] = vals[k];
        table32[tb + (int64_t)k * nq] = (float)vals[k];
    }
    // (the adjoint's weight is kappa W: kdmu = kappa (mu_l - mu_g), kdk = kdil / kappa)
    double av[ADJ_K];
    av[ADJ_CRHO] = -rho * rho * (irl - irg) * dHdd;
    av[ADJ_CMU] = kdmu * dHdd;
    av[ADJ_N + 0] = nv[0];
    av[ADJ_N + 1] = nv[1];
    av[ADJ_N + 2] = nv[2];
    av[ADJ_ZG] = z;
    av[ADJ_IGN] = ign;
    av[ADJ_KD1] = kdk * delta;
    av[ADJ_KD2] = md * kdk * d2 * gn;
    av[ADJ_KD3] = md * kdk * dHdd;
    av[ADJ_IRHO] = irho;
    av[ADJ_RHO] = rho;
    av[ADJ_ZONE] = zone ? 1.0 : 0.0;
    const int64_t abase = (int64_t)tindex[cell] * ADJ_K * nq + q;
#pragma unroll
    for (int k = 0; k < ADJ_K; ++k) {
        const dfl v = df_from_double(av[k]);
        adj[abase + (int64_t)k * nq] = make_float2(v.hi, v.lo);
    }
}

int launch_setup_coefficients(evap_mesh* h, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    k_prepare<<<blocks_for(3 * m.Nu, 256), 256, 0, s>>>(h->phi, h->phi32, h->u, h->u32, m.Nphi, 3 * m.Nu);
    EVAP_CHECK_LAUNCH("prepare");
    EVAP_CUDA(cudaMemsetAsync(h->table_count, 0, sizeof(int32_t), s));
    k_classify<<<blocks_for(m.ncell, 128, 1LL << 40), 128, 0, s>>>(m, h->b, h->phi, h->cell_code, h->table_index,
                                                                   h->table_count);
    EVAP_CHECK_LAUNCH("classify");
    int32_t count = 0;
    EVAP_CUDA(cudaMemcpyAsync(&count, h->table_count, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    EVAP_CUDA(cudaStreamSynchronize(s));
    const int nq = h->b.Q * h->b.Q * h->b.Q;
    if (count > h->table_cap) {
        if (h->table) cudaFree(h->table);
        if (h->table32) cudaFree(h->table32);
        if (h->adj_table) cudaFree(h->adj_table);
        h->table = nullptr;
        h->table32 = nullptr;
        h->adj_table = nullptr;
        h->table_cap = 0;
        const int64_t cap = count + count / 8 + 16;
        EVAP_CUDA(cudaMalloc(&h->table, cap * TAB_K * nq * sizeof(double)));
        EVAP_CUDA(cudaMalloc(&h->table32, cap * TAB_K * nq * sizeof(float)));
        EVAP_CUDA(cudaMalloc(&h->adj_table, cap * ADJ_K * nq * sizeof(float2)));
        h->table_cap = cap;
    }
    if (count > 0) {
        const int64_t total = m.ncell * nq;
        const double kdil = dilation_coefficient(m);
        k_fill_table<<<blocks_for(total, 256, 1LL << 40), 256, 0, s>>>(m, h->b, h->phi, h->mdot, h->cell_code,
                                                                       h->table_index, df_kappa(m) * (m.mu_l - m.mu_g),
                                                                       kdil / df_kappa(m), h->table, h->table32,
                                                                       h->adj_table);
        EVAP_CHECK_LAUNCH("fill_table");
    }
    return EVAP_OK;
}

// ------------------------------------------------------------------------------------------ transport velocity
// Point evaluation in cell units s = y / h of the level-set mesh (m: the level-set view of the mesh, ls_args):
// cell = clamp(floor(s), 0, n - 1), trilinear phi; the Q_p velocity from the velocity cell located the same way at
// s / n_sub (nu cells per axis).
struct PointEval {
    const double* phi;
    const double* u;
    MeshArgs<double> m;
    int nu;           // velocity cells per axis
    double inv_sub;   // 1 / n_sub
    double gl[MAXQ];  // Gauss-Lobatto support points of the velocity element

    __device__ void velocity(const double s_ls[3], double out[3]) const {
        int k[3];
        double xi[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double s = s_ls[a] * inv_sub;
            int c = (int)floor(s);
            c = c < 0 ? 0 : (c > nu - 1 ? nu - 1 : c);
            k[a] = c;
            xi[a] = s - c;
        }
        const int P = m.P, Q = P + 1;
        double l[3][MAXQ];
        for (int d = 0; d < 3; ++d)
            for (int a = 0; a < Q; ++a) {
                double v = 1.0;
                for (int j = 0; j < Q; ++j)
                    if (j != a) v *= (xi[d] - gl[j]) / (gl[a] - gl[j]);
                l[d][a] = v;
            }
        out[0] = out[1] = out[2] = 0.0;
        for (int c = 0; c < Q; ++c)
            for (int b = 0; b < Q; ++b)
                for (int a = 0; a < Q; ++a) {
                    const int64_t node = (int64_t)(P * k[0] + a) +
                                         (int64_t)m.M * ((int64_t)(P * k[1] + b) + (int64_t)m.M * (P * k[2] + c));
                    const double wgt = l[0][a] * l[1][b] * l[2][c];
                    out[0] += wgt * u[node];
                    out[1] += wgt * u[m.Nu + node];
                    out[2] += wgt * u[2 * m.Nu + node];
                }
    }
};

constexpr double PHI_CLAMP = 1.0 - 0x1p-40;
constexpr int CPP_NORMAL_STEPS = 20;  // projection of the node
constexpr int CPP_TRIAL_STEPS = 6;    // projection of a trial point of the tangential step
constexpr int CPP_BACKTRACK = 6;
constexpr double CPP_STALL = 1e-12;   // an accepted step shortening |y - x| by less than this fraction ends it

__device__ __forceinline__ double clampd(double v, double lo, double hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ double dist3(const double a[3], const double b[3]) {
    const double d0 = a[0] - b[0], d1 = a[1] - b[1], d2 = a[2] - b[2];
    return sqrt(d0 * d0 + d1 * d1 + d2 * d2);
}

enum : int { TRIAL_RUN = 0, TRIAL_FAIL, TRIAL_OK, TRIAL_IDLE };  // a trial point's projection

// Closest point of x on d(phi_h) = d_t with the backtracked tangential step (App. C), written as a state machine
// in which every trip of the loop makes exactly one point evaluation of phi_h and grad phi_h: the projection of the
// node (phase 0, at most CPP_NORMAL_STEPS normal steps) and the projection of a trial point y - omega t (phase 2, at
// most CPP_TRIAL_STEPS normal steps, omega = 1, 1/2, ..., 1/2^(CPP_BACKTRACK-1)); the tangential direction at a new y
// takes the normal of the evaluation that ended the projection there.  The sequence of updates of a node is: project x
// (normal steps y <- y - (d(y) - d*) / |grad d(y)| n(y) until |d(y) - d*| <= tol h); then repeat up to kmax times:
// tangential part t of y - x at y; for omega = 1, 1/2, ...: project y - omega t; accept the first trial point that
// reached the isocontour and is strictly closer to x; stop when none is, when the accepted step is <= tol or shortens
// |y - x| by <= CPP_STALL of it.  Not converged: the first projection failed or kmax outer iterations ran without a
// stop.
struct CppLane {
    int b = -1;  // band entry, -1 none
    int phase = 0, steps = 0, k = 0, bt = 0, ev = 0, trips = 0;
    int st = TRIAL_IDLE;
    double x[3], y[3], yn[3], tp[3];
    double nv[3], nrm = 0.0, dn = 0.0;  // of the trial point that ended last: unit normal, |grad phi|, distance to x
    double dist = 0.0, dist_prev = 0.0;
};

// Cell and local coordinate of s in [0, n] (cell units, n <= 2^11): clamp(floor(s), 0, n - 1) and s - cell, with the
// difference as the only FP64 instruction: the floor of a non-negative double is its bits with the fraction masked off, and its integer value
// the leading mantissa bits.  (Any other s, a NaN for one, still gives a cell of the mesh.)
__device__ __forceinline__ void locate_in_range(double s, int n, int& k, double& xi) {
    const int hi = __double2hiint(s);
    const int e = min((hi >> 20) - 1023, 20);
    const bool frac = e < 0;  // s < 1
    const int sh = frac ? 0 : e;
    const int fl = frac ? 0 : (hi & ~(0xFFFFF >> sh));
    const int c = frac ? 0 : (((hi & 0xFFFFF) | 0x100000) >> (20 - sh));
    k = min(c, n - 1);
    xi = s - (c > n - 1 ? (double)(n - 1) : __hiloint2double(fl, 0));
}

// v clamped to [0, hi]: in the interior the high words alone decide (hi > 0)
__device__ __forceinline__ double clamp_range(double v, double hi) {
    if ((unsigned)__double2hiint(v) < (unsigned)__double2hiint(hi)) return v;
    return clampd(v, 0.0, hi);
}

// phi_h and grad phi_h (physical units) at s (cell units) by successive linear interpolation along x, y, z
// (the trilinear Q1 interpolant of Sec. 2.5; fewer FP64 operations than the weighted sum over the 8 nodes).
__device__ __forceinline__ void q1_lerp(const PointEval& e, const double s[3], double& val, double g[3]) {
    int k[3];
    double t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) locate_in_range(s[a], e.m.n, k[a], t[a]);
    const int64_t m1 = e.m.n + 1;
    const double* f = e.phi + k[0] + m1 * (k[1] + m1 * k[2]);
    double ex[2][2], dx[2][2];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const double v0 = f[m1 * (b + m1 * c)], v1 = f[1 + m1 * (b + m1 * c)];
            dx[c][b] = v1 - v0;
            ex[c][b] = fma(t[0], dx[c][b], v0);
        }
    double exy[2], dxy[2], dyx[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        dyx[c] = ex[c][1] - ex[c][0];
        exy[c] = fma(t[1], dyx[c], ex[c][0]);
        dxy[c] = fma(t[1], dx[c][1] - dx[c][0], dx[c][0]);
    }
    const double dz = exy[1] - exy[0];
    val = fma(t[2], dz, exy[0]);
    g[0] = fma(t[2], dxy[1] - dxy[0], dxy[0]) * e.m.inv_h;
    g[1] = fma(t[2], dyx[1] - dyx[0], dyx[0]) * e.m.inv_h;
    g[2] = dz * e.m.inv_h;
}

// Unit normal of phi_h at lattice node (i, j, k), point-located in the cell clamp(node, 0, n - 1): the point is a corner
// of that cell, so the gradient is the difference along each of its three edges there (the trilinear formula with
// weights 0 and 1, in which only these terms are nonzero); zero where |grad phi| h <= GRAD_TINY.
__device__ __forceinline__ void node_normal(const PointEval& e, int i, int j, int k, double nx[3]) {
    const MeshArgs<double>& m = e.m;
    const int64_t m1 = m.n + 1;
    const int ic = min(i, m.n - 1), jc = min(j, m.n - 1), kc = min(k, m.n - 1);
    const double* f = e.phi;
    const double g[3] = {(f[ic + 1 + m1 * (j + m1 * k)] - f[ic + m1 * (j + m1 * k)]) * m.inv_h,
                         (f[i + m1 * (jc + 1 + m1 * k)] - f[i + m1 * (jc + m1 * k)]) * m.inv_h,
                         (f[i + m1 * (j + m1 * (kc + 1))] - f[i + m1 * (j + m1 * kc)]) * m.inv_h};
    const double nrm = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    nx[0] = nx[1] = nx[2] = 0.0;
    if (nrm * m.h > GRAD_TINY) { nx[0] = g[0] / nrm; nx[1] = g[1] / nrm; nx[2] = g[2] / nrm; }
}

// Transport velocity at Q1 node (i, j, k) from the fluid velocity uv of the point it takes:
// u_Gamma = uv + mdot/rho_* n(x), n(x) the point-located normal at the node.
__device__ __forceinline__ void transport_store(const PointEval& e, const double* __restrict__ mdot, int64_t node, int i,
                                                int j, int k, const double uv[3], double rho_t,
                                                double* __restrict__ ug) {
    double nx[3];
    node_normal(e, i, j, k, nx);
    const double c = mdot[node] / rho_t;
    ug[node] = uv[0] + c * nx[0];
    ug[e.m.Nphi + node] = uv[1] + c * nx[1];
    ug[2 * e.m.Nphi + node] = uv[2] + c * nx[2];
}

__device__ __forceinline__ bool in_projection_band(int variant, double phx) {
    return variant == 2 ? (-PHI_GAS_BAND < phx) && (phx < PHI_BAND) : (-PHI_BAND < phx) && (phx < PHI_GAS_BAND);
}

// Pass 1, one thread per Q1 node: variant 1 (Eq. transport_vel_local_continuous) and the nodes of variants 2/3
// outside the projection band (y = x) are finished here; band nodes are appended to a list for pass 2, so that
// the iterating nodes fill whole warps.
__global__ void k_transport_direct(PointEval e, const double* __restrict__ mdot, double* __restrict__ ug,
                                   int32_t* __restrict__ flags, int32_t* __restrict__ band, int32_t* band_count) {
    const MeshArgs<double>& m = e.m;
    const int64_t node = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (node >= m.Nphi) return;
    const double phx = e.phi[node];
    flags[node] = 0;
    if (m.variant != 1 && in_projection_band(m.variant, phx)) {
        band[atomicAdd(band_count, 1)] = (int32_t)node;
        return;
    }
    const unsigned m1 = (unsigned)m.n + 1u, nd = (unsigned)node, t = nd / m1;  // N_phi < 2^31 (band entries are int32)
    const int i = (int)(nd - t * m1), k = (int)(t / m1), j = (int)(t - (unsigned)k * m1);
    double uv[3];
    if (m.nsub == 1 || m.nsub == m.P) {  // the node is a velocity node
        const int st = m.nsub == 1 ? m.P : 1;
        const int64_t vn = (int64_t)(st * i) + (int64_t)m.M * ((int64_t)(st * j) + (int64_t)m.M * (st * k));
        uv[0] = e.u[vn];
        uv[1] = e.u[m.Nu + vn];
        uv[2] = e.u[2 * m.Nu + vn];
    } else {
        const double y[3] = {(double)i, (double)j, (double)k};
        e.velocity(y, uv);
    }
    const double rho_t = m.variant == 1 ? material(phx, 0.0, 0.0, 0.0, m).rho : (m.variant == 2 ? m.rho_l : m.rho_g);
    transport_store(e, mdot, node, i, j, k, uv, rho_t, ug);
}

// Pass 2, persistent, one warp per block: closest points of the band nodes on the liquid (variant 2) or gas (variant 3)
// end of the zone, y of band entry b to band_y[3 b], the convergence flag to flags[node].  band_count[1] hands out the
// entries.
//
// What bounds it: a warp's FP64 instruction occupies its scheduler's FP64 unit for 64 cycles however few lanes are
// active, so the pass costs (trips of the slowest lane) x (~200 instructions) x 64 cycles on every scheduler, and a node
// makes 20 to 500 trips (mean 97, on four drops at 64^3).  Hence (a) a lane whose node is done takes the next band
// entry; (b) when the list is exhausted the warp's remaining nodes are spread over its idle lanes, G = 2, 4 or 8 lanes
// per node, which project the trial points of the next G backtracking lengths at once: the first accepted one in
// the order of the lengths is taken, so the points are the ones of the serial iteration bit for bit, and the longest
// chains (many rejected lengths per outer iteration) shrink several times; (c) the tangential direction reuses the
// evaluation that ended the projection; (d) point location and clamping run on the integer units.
// The evaluations counted are those of the serial iteration (one per trip, one per tangential direction).
__global__ void __launch_bounds__(32) k_transport_band(PointEval e, double tol, int kmax, const int32_t* __restrict__ band,
                                                       int32_t* band_count, double* __restrict__ band_y,
                                                       int32_t* __restrict__ flags, unsigned long long* flag_count,
                                                       unsigned long long* evals) {
    const MeshArgs<double>& m = e.m;
    constexpr unsigned FULL = 0xffffffffu;
    const int count = band_count[0];
    const int m1 = m.n + 1;
    const double d_t = m.variant == 2 ? 3.0 * m.eps : -3.0 * m.eps;
    const double eps = m.eps, h = m.h, nn = (double)m.n;
    const int lane = threadIdx.x;
    int G = 1, sub = 0;  // lanes per node (warp-uniform), this lane's place in its group
    CppLane L;
    auto take = [&]() {
        L.b = atomicAdd(&band_count[1], 1);
        if (L.b >= count) {
            L.b = -1;
            return;
        }
        const int64_t node = band[L.b];
        L.x[0] = (double)(node % m1);
        L.x[1] = (double)((node / m1) % m1);
        L.x[2] = (double)(node / ((int64_t)m1 * m1));
        L.y[0] = L.x[0]; L.y[1] = L.x[1]; L.y[2] = L.x[2];
        L.phase = 0;
        L.steps = 0;
        L.trips = 0;
        L.ev = 0;
    };
    // the group's node is done (called by all of its lanes); lanes look for the next entry while they work alone
    auto finish = [&](bool converged) {
        if (sub == 0) {
            band_y[3 * (int64_t)L.b + 0] = L.y[0];
            band_y[3 * (int64_t)L.b + 1] = L.y[1];
            band_y[3 * (int64_t)L.b + 2] = L.y[2];
            flags[band[L.b]] = converged ? 0 : 1;
            if (!converged) atomicAdd(flag_count, 1ULL);
            atomicAdd(evals, (unsigned long long)L.trips);
        }
        L.b = -1;
        if (G == 1) take();
    };
    // this lane's trial point y - 2^-bt t
    auto start_trial = [&](int bt) {
        L.bt = bt;
        L.steps = 0;
        L.ev = 0;
        L.st = bt < CPP_BACKTRACK ? TRIAL_RUN : TRIAL_IDLE;
        const double omega = __hiloint2double((1023 - bt) << 20, 0);
#pragma unroll
        for (int a = 0; a < 3; ++a) L.yn[a] = clamp_range(L.y[a] - omega * L.tp[a], nn);
    };
    // the lanes of a warp that start with a node: all, or an even share of a short list
    if (lane < (count + (int)gridDim.x - 1) / (int)gridDim.x) take();
    const double c_step = 1.0 / (2.0 * eps * h);  // step (cell units) = r / (|grad d| h), |grad d| = 2 eps |g| / (1 - ph^2)
    const double tol_h = tol * h;
    for (;;) {
        const unsigned act = __ballot_sync(FULL, L.b >= 0);
        if (!act) break;
        if (act != FULL && G < 8) {  // the list is exhausted: more lanes per node as soon as the nodes left allow it
            const unsigned leaders = G == 1 ? FULL : (G == 2 ? 0x55555555u : 0x11111111u);
            const unsigned lead = act & leaders;
            const int na = __popc(lead);
            const int Gn = na <= 4 ? 8 : (na <= 8 ? 4 : (na <= 16 ? 2 : 1));
            if (Gn > G) {  // node j -> lanes j Gn ... j Gn + Gn - 1; its running trials keep their places
                const int j = lane / Gn, s2 = lane % Gn;
                const bool has = j < na;
                const int src = (has ? (int)__fns(lead, 0, j + 1) : lane) + (has && s2 < G ? s2 : 0);
                CppLane N;
                N.b = __shfl_sync(FULL, L.b, src);
                N.phase = __shfl_sync(FULL, L.phase, src);
                N.steps = __shfl_sync(FULL, L.steps, src);
                N.k = __shfl_sync(FULL, L.k, src);
                N.bt = __shfl_sync(FULL, L.bt, src);
                N.ev = __shfl_sync(FULL, L.ev, src);
                N.trips = __shfl_sync(FULL, L.trips, src);
                N.st = __shfl_sync(FULL, L.st, src);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    N.x[a] = __shfl_sync(FULL, L.x[a], src);
                    N.y[a] = __shfl_sync(FULL, L.y[a], src);
                    N.yn[a] = __shfl_sync(FULL, L.yn[a], src);
                    N.tp[a] = __shfl_sync(FULL, L.tp[a], src);
                    N.nv[a] = __shfl_sync(FULL, L.nv[a], src);
                }
                N.dist = __shfl_sync(FULL, L.dist, src);
                N.dist_prev = __shfl_sync(FULL, L.dist_prev, src);
                N.dn = __shfl_sync(FULL, L.dn, src);
                N.nrm = __shfl_sync(FULL, L.nrm, src);
                L = N;
                if (!has) L.b = -1;
                if (has && s2 >= G && L.phase == 2) start_trial(L.bt + s2);  // src is the leader: its bt is the base
                G = Gn;
                sub = s2;
            }
        }
        // one point evaluation per running lane, and its normal step
        bool on = false, ended = false;
        double nrm = 0.0, nv[3] = {0.0, 0.0, 0.0};
        const bool trial = L.phase == 2;
        if (L.b >= 0 && (!trial || L.st == TRIAL_RUN)) {
            ++L.ev;
            double p[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) p[a] = trial ? L.yn[a] : L.y[a];
            double ph, g[3];
            q1_lerp(e, p, ph, g);
            ph = clampd(ph, -PHI_CLAMP, PHI_CLAMP);
            const double r = eps * log((1.0 + ph) / (1.0 - ph)) - d_t;
            nrm = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
            const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
#pragma unroll
            for (int a = 0; a < 3; ++a) nv[a] = g[a] * inv;
            on = fabs(r) <= tol_h;
            if (!on && L.steps < (trial ? CPP_TRIAL_STEPS : CPP_NORMAL_STEPS) && nrm > 0.0) {
                const double step = r * (1.0 - ph * ph) * inv * c_step;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    p[a] = clamp_range(p[a] - step * nv[a], nn);
                    if (trial) L.yn[a] = p[a];
                    else L.y[a] = p[a];
                }
                ++L.steps;
            } else {
                ended = true;
            }
        }
        __syncwarp();
        if (!__any_sync(FULL, ended)) continue;
        // a projection ended in some lane: its distance and normal, kept until the group decides
        bool tangent = false;
        if (ended) {
            L.nrm = nrm;
#pragma unroll
            for (int a = 0; a < 3; ++a) L.nv[a] = nv[a];
            if (trial) {
                L.dn = dist3(L.yn, L.x);
                L.st = on && L.dn < L.dist ? TRIAL_OK : TRIAL_FAIL;
            }
        }
        // the group's trials in the order of their lengths: the first that did not fail decides
        const int base = lane - sub;
        const unsigned gm = (1u << G) - 1u;
        const bool in2 = L.b >= 0 && trial;
        const unsigned failed = (__ballot_sync(FULL, in2 && (L.st == TRIAL_FAIL || L.st == TRIAL_IDLE)) >> base) & gm;
        const unsigned okay = (__ballot_sync(FULL, in2 && L.st == TRIAL_OK) >> base) & gm;
        const int first = __ffs(~failed) - 1;
        const bool accept = in2 && first < G && ((okay >> first) & 1u);
        const bool none = in2 && first >= G;
        if (G == 1) {
            if (accept || none) L.trips += L.ev;
        } else if (__any_sync(FULL, accept || none)) {
            // the accepted point with its distance and normal to all lanes of the group; the evaluations up to it
            int ev = (accept && sub <= first) || none ? L.ev : 0;
            for (int o = 1; o < G; o <<= 1) ev += __shfl_xor_sync(FULL, ev, o);
            const int src = accept ? base + first : lane;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                L.yn[a] = __shfl_sync(FULL, L.yn[a], src);
                L.nv[a] = __shfl_sync(FULL, L.nv[a], src);
            }
            L.dn = __shfl_sync(FULL, L.dn, src);
            L.nrm = __shfl_sync(FULL, L.nrm, src);
            if (accept || none) L.trips += ev;
        }
        if (ended && !trial) {  // projection of the node
            L.trips += L.ev;
            if (on) {
                L.dist = dist3(L.y, L.x);
                L.k = 0;
                if (kmax <= 0) finish(false);
                else tangent = true;
            } else {
                finish(false);
            }
        } else if (accept) {
            L.dist = L.dn;
            const double step = dist3(L.yn, L.y);
            const double gain = L.dist_prev - L.dist;
            L.y[0] = L.yn[0]; L.y[1] = L.yn[1]; L.y[2] = L.yn[2];
            if (step <= tol || gain <= CPP_STALL * L.dist) finish(true);
            else if (++L.k == kmax) finish(false);
            else tangent = true;
        } else if (none) {
            if (L.bt - sub + G >= CPP_BACKTRACK) finish(true);  // no shorter point on the isocontour
            else start_trial(L.bt + G);
        }
        if (tangent) {  // tangential part of y - x at y, first trial points
            ++L.trips;
            const double n0 = L.nv[0], n1 = L.nv[1], n2 = L.nv[2];
            L.tp[0] = L.tp[1] = L.tp[2] = 0.0;
            if (L.nrm > 0.0) {
                const bool alt = fabs(n0) > 0.9;  // v = e_y instead of e_x
                const double vn = alt ? n1 : n0;
                double t0[3] = {(alt ? 0.0 : 1.0) - vn * n0, (alt ? 1.0 : 0.0) - vn * n1, -vn * n2};
                const double t0n = sqrt(t0[0] * t0[0] + t0[1] * t0[1] + t0[2] * t0[2]);
                if (t0n > 0.0) {
                    const double it = 1.0 / t0n;
                    t0[0] *= it; t0[1] *= it; t0[2] *= it;
                }
                const double t1[3] = {n1 * t0[2] - n2 * t0[1], n2 * t0[0] - n0 * t0[2], n0 * t0[1] - n1 * t0[0]};
                const double dl[3] = {L.y[0] - L.x[0], L.y[1] - L.x[1], L.y[2] - L.x[2]};
                const double a0 = dl[0] * t0[0] + dl[1] * t0[1] + dl[2] * t0[2];
                const double a1 = dl[0] * t1[0] + dl[1] * t1[1] + dl[2] * t1[2];
#pragma unroll
                for (int a = 0; a < 3; ++a) L.tp[a] = a0 * t0[a] + a1 * t1[a];
            }
            L.dist_prev = L.dist;
            L.phase = 2;
            start_trial(sub);
        }
        __syncwarp();
    }
}

// Pass 3, one thread per band entry: u_Gamma at the band nodes from their closest points.
__global__ void k_transport_band_finish(PointEval e, const double* __restrict__ mdot, const int32_t* __restrict__ band,
                                        const int32_t* __restrict__ band_count, const double* __restrict__ band_y,
                                        double* __restrict__ ug) {
    const int count = band_count[0];
    const double rho_t = e.m.variant == 2 ? e.m.rho_l : e.m.rho_g;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < count; b += gridDim.x * blockDim.x) {
        const double y[3] = {band_y[3 * (int64_t)b], band_y[3 * (int64_t)b + 1], band_y[3 * (int64_t)b + 2]};
        const unsigned m1 = (unsigned)e.m.n + 1u, nd = (unsigned)band[b], t = nd / m1;
        const int i = (int)(nd - t * m1), k = (int)(t / m1), j = (int)(t - (unsigned)k * m1);
        double uv[3];
        e.velocity(y, uv);
        transport_store(e, mdot, band[b], i, j, k, uv, rho_t, ug);
    }
}

// Points whose velocity the last pass took, y [3][N_phi] (physical coordinates, component-major): the node itself,
// then (second kernel) the closest point of every band node.
__global__ void k_node_points(int n, int64_t Np, double h, double* __restrict__ y) {
    const int m1 = n + 1;
    for (int64_t node = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; node < Np;
         node += (int64_t)gridDim.x * blockDim.x) {
        y[node] = h * (double)(node % m1);
        y[Np + node] = h * (double)((node / m1) % m1);
        y[2 * Np + node] = h * (double)(node / ((int64_t)m1 * m1));
    }
}

__global__ void k_band_points(const int32_t* __restrict__ band, const int32_t* __restrict__ band_count,
                              const double* __restrict__ band_y, double h, int64_t Np, double* __restrict__ y) {
    const int count = band_count[0];
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < count; b += gridDim.x * blockDim.x) {
        const int64_t node = band[b];
#pragma unroll
        for (int a = 0; a < 3; ++a) y[a * Np + node] = h * band_y[3 * (int64_t)b + a];
    }
}

int launch_closest_points(evap_mesh* h, double* y, cudaStream_t s) {
    const MeshArgs<double> m = ls_args<double>(h);
    k_node_points<<<blocks_for(m.Nphi, 256), 256, 0, s>>>(m.n, m.Nphi, m.h, y);
    EVAP_CHECK_LAUNCH("node_points");
    if (m.variant != 1) {
        k_band_points<<<blocks_for(m.Nphi, 256), 256, 0, s>>>(h->band_list, h->band_count, h->band_y, m.h, m.Nphi, y);
        EVAP_CHECK_LAUNCH("band_points");
    }
    return EVAP_OK;
}

constexpr int CPP_WARPS = 6 * 152;  // 6 one-warp blocks per SM
int launch_transport_velocity(evap_mesh* h, cudaStream_t s, const double* phi) {
    PointEval e;
    e.phi = phi ? phi : h->phi;
    e.u = h->u;
    e.m = ls_args<double>(h);
    e.nu = h->m.n;
    e.inv_sub = 1.0 / h->m.nsub;
    const int P = h->m.P;
    if (P == 2) {
        e.gl[0] = 0.0; e.gl[1] = 0.5; e.gl[2] = 1.0; e.gl[3] = 0.0;
    } else {
        const double r = 0.5 / std::sqrt(5.0);
        e.gl[0] = 0.0; e.gl[1] = 0.5 - r; e.gl[2] = 0.5 + r; e.gl[3] = 1.0;
    }
    EVAP_CUDA(cudaMemsetAsync(h->flag_count, 0, sizeof(unsigned long long), s));
    EVAP_CUDA(cudaMemsetAsync(h->band_count, 0, 2 * sizeof(int32_t), s));
    EVAP_CUDA(cudaMemsetAsync(h->cpp_evals, 0, sizeof(unsigned long long), s));
    k_transport_direct<<<blocks_for(h->m.Nphi, 128, 1LL << 40), 128, 0, s>>>(e, h->mdot, h->ugamma, h->cpp_flags,
                                                                            h->band_list, h->band_count);
    EVAP_CHECK_LAUNCH("transport_direct");
    if (h->m.variant != 1) {
        // Persistent pass of at most 6 warps per SM, each with an even share of a shorter list.  Measured (us per
        // transport pass; sphere 33^3 with 13 k band nodes / four drops 64^3, 41 k / slab 64^3, 38 k / deformed 128^3,
        // 181 k / sphere 48^3 with n_sub = 2, 198 k): 3 warps 1256 / 2588 / 304 / 7958 / 9117; 4 1231 / 2152 / 260 /
        // 6336 / 7253; 6 1047 / 1960 / 267 / 5523 / 6334; 8 1156 / 2003 / 245 / 5518 / 6301; 16 1472 / 2639 / 292 /
        // 5801 / 6581.  Before the lane groups (one lane per node to the end): 2970 / 3559 / 477 / 9290 / 9139.
        int32_t count = 0;
        EVAP_CUDA(cudaMemcpyAsync(&count, h->band_count, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        EVAP_CUDA(cudaStreamSynchronize(s));
        const int grid = (int)std::min<int64_t>(std::max<int64_t>(count, 1), CPP_WARPS);
        k_transport_band<<<grid, 32, 0, s>>>(e, h->prm.cpp_tol, h->prm.cpp_kmax, h->band_list, h->band_count,
                                             h->band_y, h->cpp_flags, h->flag_count, h->cpp_evals);
        EVAP_CHECK_LAUNCH("transport_band");
        k_transport_band_finish<<<blocks_for(h->m.Nphi, 128, 152 * 16), 128, 0, s>>>(e, h->mdot, h->band_list,
                                                                                      h->band_count, h->band_y,
                                                                                      h->ugamma);
        EVAP_CHECK_LAUNCH("transport_band_finish");
    }
    return refresh_ugamma_copies(h, s);
}

}  // namespace evap
