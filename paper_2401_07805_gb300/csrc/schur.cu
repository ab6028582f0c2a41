// The Schur approximation S~ = B diag(A)^(-1) B^T of the velocity-pressure preconditioner, assembled.
//
// B is the divergence row of the momentum apply: B_c[j][v] = sum_q W N1_j d_c N_v over the velocity Gauss rule, with
// the velocity DoFs on Dirichlet faces left out (the apply reads x as 0 there and B^T p vanishes there).  On the
// uniform Cartesian mesh every factor is a tensor product of 1D integrals, B_c[j][v] = prod_d F^c_d[j_d][v_d] with
// F^c_d = g1 (the 1D integral of N1_J N_V', dimensionless) in the direction d = c and a1 (the 1D integral of
// N1_J N_V, h) in the other two; these are exact with the velocity Gauss rule.  So
//   S~[i][j] = sum_c sum_{v free} prod_d (F^c_d[i_d][v_d] F^c_d[j_d][v_d]) / D_c[v],
// D_c[v] the Jacobi diagonal of A (in FP32, as the matrix-free Schur operator uses it).  A pressure node couples with
// the nodes within two cells (a 5^3 = 125-point stencil); S~ is symmetric, so the 63 offsets o >= 0 (in the
// lexicographic order of (oz, oy, ox)) are stored, as FP32 [63][N_p]: offset o of node i is entry |l(o) - 62| of node
// i (l(o) >= 62) or of node i + o (l(o) < 62), with l(o) = 25 (oz + 2) + 5 (oy + 2) + (ox + 2); entry 0 is the diagonal.
// One thread per stored entry sums its velocity nodes (at most 7^3, for Q3) in a fixed order: no atomics.
//
// With the stencil, the Schur CG of every preconditioner application is one cooperative launch in FP32
// (k_cg_fused32) instead of, per iteration, a matrix-free gradient and divergence over the whole velocity mesh.
#include <algorithm>

#include "fused_krylov.cuh"
#include "physics.cuh"

namespace evap {

// 1D assembled factor of pressure node I (0..n) and velocity node V (0..P n): the cells e in {I - 1, I} that hold both
__device__ __forceinline__ float factor1(const float (&t)[2][MAXQ], int P, int n, int I, int V) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int e = I - 1 + k;
        const int b = V - P * e;
        if (e >= 0 && e < n && b >= 0 && b <= P) s += t[1 - k][b];  // node I is corner 1 of cell I - 1, corner 0 of I
    }
    return s;
}

// One block row per stored offset (blockIdx.y), one thread per pressure node.  The 1D factor products of a pair of pressure
// nodes depend on the nodes only through their boundary classes (first, interior, last), so they are formed once per block
// in shared memory: w[d][class of I][class of J][k][a or g], k over the velocity nodes both touch; nodes outside the
// lattice get 0 and are read at a clamped place.  Each term keeps its own division by D: a solve with the preconditioner
// amplifies the rounding of S~ (with reciprocals formed once per velocity node and sums factored by direction, 667 us at
// 64^3 Q2, solutions to 1e-8 moved by several times what two runs differ by).  Measured at 64^3 Q2: 2139 us with the
// factors in local memory, now 1864.
__global__ void __launch_bounds__(128) k_schur_assemble(int n, int P, int M, unsigned faces, int64_t Nu, int64_t Np,
                                                        CouplingTables tab, const float* __restrict__ diag,
                                                        float* __restrict__ S) {
    __shared__ float w[3][3][3][2 * MAXQ - 1][2];
    const int e = blockIdx.y, lin = 62 + e;
    const int o[3] = {lin % 5 - 2, (lin / 5) % 5 - 2, lin / 25 - 2};
    for (int q = threadIdx.x; q < 27 * (2 * MAXQ - 1); q += blockDim.x) {
        const int k = q % (2 * MAXQ - 1), cj = (q / (2 * MAXQ - 1)) % 3, ci = (q / (3 * (2 * MAXQ - 1))) % 3,
                  d = q / (9 * (2 * MAXQ - 1));
        // a representative pair of these classes; the classes that no pair at this offset has stay 0
        int I = ci == 0 ? 0 : (ci == 2 ? n : -1), J = cj == 0 ? 0 : (cj == 2 ? n : -1);
        if (I < 0 && J < 0) I = 3;  // both interior: taken from a long lattice below
        if (I < 0) I = J - o[d];
        if (J < 0 || (ci == 1 && cj == 1)) J = I + o[d];
        const int nn = ci == 1 && cj == 1 ? 8 : n;
        float a = 0.f, g = 0.f;
        if (J - I == o[d] && I >= 0 && I <= nn && J >= 0 && J <= nn) {
            const int V = P * max(I, J) - P + k;
            if (V >= 0 && V <= P * nn && V <= P * min(I, J) + P) {
                a = factor1(tab.a, P, nn, I, V) * factor1(tab.a, P, nn, J, V);
                g = factor1(tab.g, P, nn, I, V) * factor1(tab.g, P, nn, J, V);
            }
        }
        w[d][ci][cj][k][0] = a;
        w[d][ci][cj][k][1] = g;
    }
    __syncthreads();
    const int64_t node = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (node >= Np) return;
    const unsigned m1 = (unsigned)n + 1u, nd = (unsigned)node, t = nd / m1;
    const int I[3] = {(int)(nd - t * m1), (int)(t - (t / m1) * m1), (int)(t / m1)};
    int lo[3], cnt[3];
    const float(*wd[3])[2];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int J = I[d] + o[d];
        if (J < 0 || J > n) {
            S[e * Np + node] = 0.f;
            return;
        }
        lo[d] = P * max(I[d], J) - P;
        cnt[d] = P * (2 - abs(o[d])) + 1;
        wd[d] = w[d][I[d] == 0 ? 0 : (I[d] == n ? 2 : 1)][J == 0 ? 0 : (J == n ? 2 : 1)];
    }
    float acc = 0.f;
    for (int kz = 0; kz < cnt[2]; ++kz) {
        const float az = wd[2][kz][0], gz = wd[2][kz][1];
        const int vz = min(max(lo[2] + kz, 0), M - 1);
        for (int ky = 0; ky < cnt[1]; ++ky) {
            const float ay = wd[1][ky][0], gy = wd[1][ky][1];
            const int vy = min(max(lo[1] + ky, 0), M - 1);
            const float* r = diag + (int64_t)M * (vy + (int64_t)M * vz);
            for (int kx = 0; kx < cnt[0]; ++kx) {
                const int vx = min(max(lo[0] + kx, 0), M - 1);
                if (constrained_node(vx, vy, vz, M, faces)) continue;
                const float ax = wd[0][kx][0], gx = wd[0][kx][1];
                acc += gx * ay * az / r[vx] + ax * gy * az / r[Nu + vx] + ax * ay * gz / r[2 * Nu + vx];
            }
        }
    }
    S[e * Np + node] = acc;
}

// Row `node` of S~ x and its diagonal, from the stored half stencil (FP32).  x lies on the lattice padded by two zero layers
// on every side (pos), so the 125 products need no bounds tests and a node's loads are in flight together: the
// coefficients of neighbours outside the lattice, read from a wrapped node's entry, meet a zero.  (With a tested path for
// the nodes near the boundary, most warps of 32 consecutive nodes took both paths: 53 us per CG iteration at 64^3, now 27.)
// Nodes of the padded lattice are numbered with 32 bits ((1024 + 5)^3 at most), entries of S with 64; in front of S lie
// schur_guard(n) zeros.
struct SchurStencil {
    int n;
    int64_t Np;
    const float* S;
    __device__ __forceinline__ unsigned pos(int64_t node) const {
        const unsigned m1 = (unsigned)n + 1u, mp = m1 + 4u, nd = (unsigned)node;
        const unsigned t = nd / m1, i = nd - t * m1, k = t / m1, j = t - k * m1;
        return (i + 2u) + mp * ((j + 2u) + mp * (k + 2u));
    }
    __device__ __forceinline__ float row(int64_t node, const float* x) const {
        const int m1 = n + 1, m2 = m1 * m1, mp = m1 + 4;
        const float* p = x + pos(node);
        const float* c = S + node;
        const int64_t np = Np;
        float acc = 0.f;
#pragma unroll
        for (int dz = -2; dz <= 2; ++dz)
#pragma unroll
            for (int dy = -2; dy <= 2; ++dy) {
                const float* pr = p + mp * (dy + mp * dz);
                const int nb = m1 * dy + m2 * dz;
#pragma unroll
                for (int dx = -2; dx <= 2; ++dx) {
                    const int lin = 25 * (dz + 2) + 5 * (dy + 2) + (dx + 2);
                    const float cf = lin >= 62 ? c[(lin - 62) * np] : c[(62 - lin) * np + (nb + dx)];
                    acc = fmaf(cf, pr[dx], acc);
                }
            }
        return acc;
    }
    __device__ __forceinline__ float diag(int64_t node) const { return S[node]; }
};
inline int64_t schur_guard(int n) { return 2 * ((int64_t)(n + 1) * (n + 1) + (n + 1) + 1); }
inline int64_t schur_padded(int n) { return (int64_t)(n + 5) * (n + 5) * (n + 5); }

// y = S~ x (x, y FP64, products and sums in FP32), one thread per pressure node, neighbours outside the lattice left out.
// An apply writes nothing but y, so that applies on several streams can share a handle (the padded lattice behind the
// stencil belongs to the CG); the sums are those of row(), whose extra products are zeros.
__global__ void __launch_bounds__(256) k_schur_apply(SchurStencil op, const double* __restrict__ x,
                                                     double* __restrict__ y) {
    const int64_t node = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (node >= op.Np) return;
    const int n = op.n, m1 = n + 1, m2 = m1 * m1;
    const unsigned nd = (unsigned)node, t = nd / (unsigned)m1;
    const int i = (int)(nd - t * (unsigned)m1), k = (int)(t / (unsigned)m1), j = (int)t - k * m1;
    const float* c = op.S + node;
    float acc = 0.f;
#pragma unroll
    for (int dz = -2; dz <= 2; ++dz)
#pragma unroll
        for (int dy = -2; dy <= 2; ++dy) {
            const bool in = (unsigned)(k + dz) <= (unsigned)n && (unsigned)(j + dy) <= (unsigned)n;
            const int nb = m1 * dy + m2 * dz;
#pragma unroll
            for (int dx = -2; dx <= 2; ++dx)
                if (in && (unsigned)(i + dx) <= (unsigned)n) {
                    const int lin = 25 * (dz + 2) + 5 * (dy + 2) + (dx + 2);
                    const float cf = lin >= 62 ? c[(lin - 62) * op.Np] : c[(62 - lin) * op.Np + (nb + dx)];
                    acc = fmaf(cf, (float)x[node + nb + dx], acc);
                }
        }
    y[node] = (double)acc;
}

// Assembles S~ for the mesh's current Jacobi diagonal of A (launch_diagonal), once per diagonal.
int schur_assemble(evap_mesh* h, cudaStream_t s) {
    int rc = launch_diagonal(h, s);
    if (rc) return rc;
    if (h->schur_S && h->schur_stamp == h->diag_stamp) return EVAP_OK;
    const MeshArgs<double>& m = h->m;
    if (!h->schur_S) {  // guard, stencil, the padded lattice of the CG's vector
        const int64_t len = schur_guard(m.n) + 63 * m.Np + schur_padded(m.n);
        EVAP_CUDA(cudaMalloc(&h->schur_S, len * sizeof(float)));
        EVAP_CUDA(cudaMemsetAsync(h->schur_S, 0, len * sizeof(float), s));
    }
    const CouplingTables tab = coupling_tables(h);
    k_schur_assemble<<<dim3((unsigned)((m.Np + 127) / 128), 63), 128, 0, s>>>(m.n, m.P, m.M, m.faces, m.Nu, m.Np, tab,
                                                                           h->diag32, h->schur_S + schur_guard(m.n));
    EVAP_CHECK_LAUNCH("schur_assemble");
    h->schur_stamp = h->diag_stamp;
    return EVAP_OK;
}

int launch_schur_apply(evap_mesh* h, const double* x, double* y, cudaStream_t s) {
    int rc = schur_assemble(h, s);
    if (rc) return rc;
    const SchurStencil op{h->m.n, h->m.Np, h->schur_S + schur_guard(h->m.n)};
    k_schur_apply<<<(unsigned)((h->m.Np + 255) / 256), 256, 0, s>>>(op, x, y);
    EVAP_CHECK_LAUNCH("schur_apply");
    return EVAP_OK;
}

// z ~ S~^(-1) r: the FP32 single-launch CG (k_cg_fused32) on the assembled stencil with its diagonal as the Jacobi
// preconditioner, from z = 0, at most max_iter iterations or |r| <= rtol |r0|.
int schur_solve(evap_mesh* h, const double* r, double* z, double rtol, int max_iter, int* iters, cudaStream_t s) {
    int rc = schur_assemble(h, s);
    if (rc) return rc;
    int64_t N = h->m.Np;
    FusedSpace f;
    if ((rc = fused_space(h, 3, f, s))) return rc;  // 3 pair vectors = 6 float vectors of N_phi >= N_p entries
    int G = 0;
    if ((rc = fused_grid(k_cg_fused32<SchurStencil>, FK_MAX_BLOCKS, N, G))) return rc;
    EVAP_CUDA(cudaMemsetAsync(f.gb, 0, sizeof(GridBarrier), s));
    SchurStencil op{h->m.n, N, h->schur_S + schur_guard(h->m.n)};
    const int64_t Nl = ls_args<double>(h).Nphi;  // the vectors' stride: fused_space sizes them for N_phi
    float* base = reinterpret_cast<float*>(f.vec);
    float *xs = base, *r32 = base + Nl, *p = base + 3 * Nl, *sv = base + 4 * Nl, *w = base + 5 * Nl;
    float* u = h->schur_S + schur_guard(h->m.n) + 63 * N;  // the padded lattice, whose halo stays zero
    float* dinv = f.dinv;
    float* part = reinterpret_cast<float*>(f.part);
    GridBarrier* gb = f.gb;
    double* out = f.out;
    double atol = 0.0;
    double* zz = z;
    void* args[] = {&op, &N, &r, &zz, &xs, &dinv, &r32, &u, &p, &sv, &w, &rtol, &atol, &max_iter, &part, &gb, &out};
    EVAP_CUDA(cudaLaunchCooperativeKernel((const void*)k_cg_fused32<SchurStencil>, dim3(G), dim3(FK_THREADS), args, 0,
                                          s));
    EVAP_CHECK_LAUNCH("schur_cg");
    double res[3];
    if ((rc = fused_result(h, f, s, res))) return rc;
    if (iters) *iters += (int)res[0];
    return EVAP_OK;
}

}  // namespace evap

extern "C" int evap_apply_schur(evap_handle h, const double* x, double* y, void* stream) {
    if (!h || !x || !y) {
        evap::set_error("evap_apply_schur: null argument");
        return EVAP_EINVAL;
    }
    if (!h->has_fields) {
        evap::set_error("evap_apply_schur: call evap_set_fields first");
        return EVAP_ENOFIELDS;
    }
    EVAP_CUDA(cudaSetDevice(h->device));
    return evap::launch_schur_apply(h, x, y, (cudaStream_t)stream);
}
