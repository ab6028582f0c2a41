// Tensor-product mass preconditioner of the FP32 inner solve of the momentum system.
//
// The velocity block is dominated by its inertia term rho c_m M (at dt = 1e-4 the viscous and convective parts are
// below 1 % of it), and on the uniform mesh the Q_p mass matrix is a Kronecker product M = Mx (x) My (x) Mz of the 1D
// Q_p mass matrices.  The preconditioner is
//     P = Sigma (Mx (x) My (x) Mz)^(-1) Sigma,   Sigma = diag( sqrt( diag(M) / diag(A) ) )
// on the free (unconstrained) velocity DoFs and the identity on the Dirichlet ones: the Jacobi diagonal of A sets
// the local density and viscous scale, the Kronecker inverse removes the mass matrix's own conditioning.  Within a
// phase P A ~ I; the density jump across the interface leaves a bounded cluster of outliers.  (Measured with the
// assembled operator of the four-sphere workload: GMRES(16) to 1e-10 needed 47 / 63 / 71 iterations with Jacobi
// and 9 / 18 / 19 with P on 12^3 / 20^3 / 28^3 cells.)
//
// The free DoFs of a face-constrained box form a tensor product of per-axis ranges, so M^(-1) on them is three
// sweeps of banded 1D solves (bandwidth p): one block per tile of 32 lines, staged through shared memory so that
// global loads and stores stay coalesced for every axis; each lane of the
// first warp solves one line with the LU factors of its axis (factorized once on the host in FP64, no pivoting: the
// 1D mass matrix is symmetric positive definite).
#include <cmath>
#include <vector>

#include "physics.cuh"

namespace evap {

constexpr int TP_LANES = 32;     // lines per tile (one solving warp)
constexpr int TP_THREADS = 128;  // threads of a block: all load and store the tile, the first warp solves
constexpr int TP_STEP = 8;       // line entries per step of the recurrences

// Factors of one free node i in shared memory: f[0..P-1] = L[i][i-1-k], then b[0..P-1] = U[i][i+1+k] / U[i][i] and
// b[P] = 1 / U[i][i], each padded to a vector.
template <int P>
struct TpShape {
    static constexpr int FW = P == 2 ? 2 : 4, BW = 4;  // entries per node, forward and backward
};
template <typename T, int N>
struct alignas(sizeof(T) * N <= 16 ? sizeof(T) * N : 16) TpVec {
    T v[N];
};
template <typename T, int P>
__device__ __forceinline__ void tp_solve_line(const T* __restrict__ ff, const T* __restrict__ fb, int Mf,
                                              T* __restrict__ col, int stride) {
    using FV = TpVec<T, TpShape<P>::FW>;
    using BV = TpVec<T, TpShape<P>::BW>;
    // The last P values of each recurrence stay in registers (win[0] the nearest) and enter last, so that a step waits on
    // one FMA only (the backward factors are scaled by the pivot for this); TP_STEP entries and their factors are loaded
    // together, as vectors, ahead of the step's chain: 9 instructions per entry both ways.  The factors are zero where a
    // neighbour falls outside the line.
    T win[P];
    auto chain = [&](const T* f, T v) -> T {
#pragma unroll
        for (int k = P - 1; k >= 0; --k) v -= f[k] * win[k];
#pragma unroll
        for (int k = P - 1; k > 0; --k) win[k] = win[k - 1];
        win[0] = v;
        return v;
    };
#pragma unroll
    for (int k = 0; k < P; ++k) win[k] = T(0);
    const FV* f = reinterpret_cast<const FV*>(ff);
    T* c = col;
    int left = Mf;
    for (; left >= TP_STEP; left -= TP_STEP, f += TP_STEP, c += TP_STEP * stride) {  // forward: L y = d (unit lower)
        T v[TP_STEP];
        FV w[TP_STEP];
#pragma unroll
        for (int e = 0; e < TP_STEP; ++e) {
            v[e] = c[e * stride];
            w[e] = f[e];
        }
#pragma unroll
        for (int e = 0; e < TP_STEP; ++e) c[e * stride] = chain(w[e].v, v[e]);
    }
    for (; left > 0; --left, ++f, c += stride) *c = chain(f->v, *c);
#pragma unroll
    for (int k = 0; k < P; ++k) win[k] = T(0);
    const BV* g = reinterpret_cast<const BV*>(fb) + (Mf - 1);
    c = col + (Mf - 1) * stride;
    left = Mf;
    for (; left >= TP_STEP; left -= TP_STEP, g -= TP_STEP, c -= TP_STEP * stride) {  // backward: U x = y
        T v[TP_STEP];
        BV w[TP_STEP];
#pragma unroll
        for (int e = 0; e < TP_STEP; ++e) {
            w[e] = g[-e];
            v[e] = c[-e * stride] * w[e].v[P];
        }
#pragma unroll
        for (int e = 0; e < TP_STEP; ++e) c[-e * stride] = chain(w[e].v, v[e]);
    }
    for (; left > 0; --left, --g, c -= stride) *c = chain(g->v, *c * g->v[P]);
}

// One sweep along AXIS for all three components (v enters scaled by sc).  MODE 0: t = M_axis^(-1) (Sigma sc v);
// MODE 1: t = M_axis^(-1) t; MODE 2: z = Sigma M_axis^(-1) t on the free DoFs, z = sc v on the Dirichlet ones, and
// w = (Dirichlet ? z : 0) (the initialization of the operator apply that follows).  One block per tile of TP_LANES
// lines; lines whose transverse position is constrained are all-Dirichlet and are solved only as a copy in MODE 2.
// A tile of x-lines is one contiguous run of memory; a tile of y- or z-lines is rows of 32 neighbouring lines.  What
// bounds the sweep is memory once enough loads are in flight: every thread issues LD independent ones at a time, and
// blocks of 128 threads let all tiles of a 64^3 sweep be resident at once.  Measured at 64^3 Q2 FP32 (us, x / y / z
// sweep, ncu): 68 / 28 / 35 with 256 threads and one load in flight per thread, the chain of a step two and three
// operations long.
template <typename T, int P, int AXIS, int MODE>
__global__ void __launch_bounds__(TP_THREADS) k_tp_sweep(int M, int64_t Nu, unsigned faces, const T* __restrict__ fac_all,
                                                     int lo, int hi, const T* __restrict__ sigma,
                                                     const T* __restrict__ v, T sc, T* __restrict__ t,
                                                     T* __restrict__ z, T* __restrict__ w) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int FW = TpShape<P>::FW, BW = TpShape<P>::BW, LD = 8, TS = TP_LANES + 1;
    const int Mf = hi - lo + 1;
    T* const fb = reinterpret_cast<T*>(smem_raw);  // [Mf][BW], first: its rows and those of ff are aligned vectors
    T* const ff = fb + Mf * BW;                     // [Mf][FW]
    T* const tile = ff + Mf * FW;                   // [M][TS]
    const int tid = threadIdx.x;
    for (int i = tid; i < Mf; i += TP_THREADS) {
#pragma unroll
        for (int k = 0; k < P; ++k) {
            ff[i * FW + k] = fac_all[k * Mf + i];
            fb[i * BW + k] = fac_all[(P + k) * Mf + i];
        }
        fb[i * BW + P] = fac_all[2 * P * Mf + i];
    }
    // tile -> (component, first line); line l of the tile has transverse coordinates (ta, tb) and base address
    const int M2 = M * M;
    int comp, first, nlines;  // first line id of the tile within the component, its lines
    if (AXIS == 1) {  // y-lines (id x + M z): 32 consecutive x at fixed (z, component)
        const int tiles_x = (M + TP_LANES - 1) / TP_LANES, b = (int)blockIdx.x;
        comp = b / (tiles_x * M);
        const int r = b - comp * tiles_x * M, zz = r / tiles_x, tx = r - zz * tiles_x;
        first = zz * M + tx * TP_LANES;
        nlines = min(TP_LANES, M - tx * TP_LANES);
    } else {  // x-lines (id y + M z) or z-lines (id x + M y): 32 consecutive ids per component
        const int tiles = (M2 + TP_LANES - 1) / TP_LANES;
        comp = (int)blockIdx.x / tiles;
        first = ((int)blockIdx.x - comp * tiles) * TP_LANES;
        nlines = min(TP_LANES, M2 - first);
    }
    // per-line constraint flag (lines on a Dirichlet face of a transverse direction)
    __shared__ int s_cons[TP_LANES];
    if (tid < TP_LANES) {
        const int id = first + tid, tb = id / M, ta = id - tb * M;
        s_cons[tid] = AXIS == 0 ? constrained_node(1, ta, tb, M, faces & ~3u)
                                : (AXIS == 1 ? constrained_node(ta, 1, tb, M, faces & ~12u)
                                             : constrained_node(ta, tb, 1, M, faces & ~48u));
    }
    __syncthreads();
    // Addresses: line l of a tile of x-lines starts at base + l M, line `lane` of a tile of y-lines at x + M^2 z = (first +
    // lane) + (M^2 - M) z and of z-lines at x + M y.  Loads past a range are clamped into it, not skipped, so that LD of
    // them are in flight per thread.
    const int lane = tid % 32, warp = tid / 32;
    constexpr int WARPS = TP_THREADS / 32;
    const int ln = AXIS == 0 ? 0 : min(lane, nlines - 1);
    const int64_t base = (int64_t)comp * Nu + (AXIS == 0 ? (int64_t)first * M
                                                         : first + ln + (AXIS == 1 ? (int64_t)(first / M) * (M2 - M) : 0));
    const int64_t es = AXIS == 1 ? M : M2;
    if (AXIS == 0) {  // a warp loads 2 lines, 4 entries per lane of each
        for (int l0 = 2 * warp; l0 < nlines; l0 += 2 * WARPS)
            for (int e0 = lane; e0 < Mf; e0 += 128) {
                T x[2][4], g[2][4];
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int64_t a = base + min(l0 + q, nlines - 1) * M + lo + min(e0 + 32 * k, Mf - 1);
                        x[q][k] = MODE == 0 ? v[a] : t[a];
                        g[q][k] = MODE == 0 ? sigma[a] : T(1);
                    }
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (e0 + 32 * k < Mf && l0 + q < nlines)
                            tile[(e0 + 32 * k) * TS + l0 + q] = MODE == 0 ? sc * x[q][k] * g[q][k] : x[q][k];
            }
    } else {
        const T* src = t + base + lo * es;
        for (int e0 = warp; e0 < Mf; e0 += LD * WARPS) {
            T x[LD];
#pragma unroll
            for (int k = 0; k < LD; ++k) x[k] = src[min(e0 + k * WARPS, Mf - 1) * es];
#pragma unroll
            for (int k = 0; k < LD; ++k)
                if (e0 + k * WARPS < Mf) tile[(e0 + k * WARPS) * TS + lane] = x[k];
        }
    }
    __syncthreads();
    if (tid < nlines && !s_cons[tid]) tp_solve_line<T, P>(ff, fb, Mf, tile + tid, TP_LANES + 1);
    __syncthreads();
    if (AXIS == 0) {
        for (int l = warp; l < nlines; l += WARPS) {
            if (s_cons[l]) continue;
            T* dst = t + base + (int64_t)l * M + lo;
            for (int e = lane; e < Mf; e += 32) dst[e] = tile[e * TS + l];
        }
    } else if (MODE < 2) {
        if (lane < nlines && !s_cons[lane]) {
            T* dst = t + base + lo * es;
#pragma unroll 4
            for (int e = warp; e < Mf; e += WARPS) dst[e * es] = tile[e * TS + lane];
        }
    } else {  // every node of the tile's lines: free -> Sigma t, Dirichlet -> sc v; w = Dirichlet ? z : 0
        const bool cl = s_cons[ln] != 0;
        for (int e0 = warp; e0 < M; e0 += LD * WARPS) {
            T sv[LD];
#pragma unroll
            for (int k = 0; k < LD; ++k) {
                const int e = min(e0 + k * WARPS, M - 1);
                sv[k] = (cl || e < lo || e > hi ? v : sigma)[base + e * es];
            }
#pragma unroll
            for (int k = 0; k < LD; ++k) {
                const int e = e0 + k * WARPS;
                if (e >= M || lane >= nlines) continue;
                const bool dir = cl || e < lo || e > hi;
                const T zz = dir ? sc * sv[k] : sv[k] * tile[(e - lo) * TS + lane];
                z[base + e * es] = zz;
                if (w) w[base + e * es] = dir ? zz : T(0);
            }
        }
    }
}

// Sigma = sqrt(diag(M) / diag(A)) on the free DoFs (1 on the Dirichlet ones); md: the 1D mass diagonal [M].
template <typename T>
__global__ void k_tp_sigma(int M, int64_t Nu, unsigned faces, const double* __restrict__ md,
                           const T* __restrict__ diag, T* __restrict__ sigma) {
    const int64_t N = 3 * Nu;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t node = i % Nu;
        const int x = (int)(node % M), y = (int)((node / M) % M), zc = (int)(node / ((int64_t)M * M));
        sigma[i] = constrained_node(x, y, zc, M, faces) ? T(1) : (T)sqrt(md[x] * md[y] * md[zc] / (double)diag[i]);
    }
}

// Host: the 1D Q_p mass matrix (consistent, (p+1)-point Gauss) of n cells of width h, its diagonal, and the banded
// LU factors of its restriction to [lo, hi].
static void mass_1d(const Basis<double>& b, int n, double h, std::vector<double>& Mg) {
    const int P = b.P, M = P * n + 1;
    Mg.assign((size_t)M * M, 0.0);
    for (int c = 0; c < n; ++c)
        for (int a = 0; a <= P; ++a)
            for (int bb = 0; bb <= P; ++bb) {
                double s = 0.0;
                for (int q = 0; q <= P; ++q) s += b.w[q] * b.S[q][a] * b.S[q][bb];
                Mg[(size_t)(P * c + a) * M + (P * c + bb)] += h * s;
            }
}

static void factor_band(const std::vector<double>& Mg, int M, int P, int lo, int hi, std::vector<double>& out) {
    const int Mf = hi - lo + 1;
    std::vector<double> A((size_t)Mf * Mf);
    for (int i = 0; i < Mf; ++i)
        for (int j = 0; j < Mf; ++j) A[(size_t)i * Mf + j] = Mg[(size_t)(lo + i) * M + (lo + j)];
    for (int j = 0; j < Mf; ++j)
        for (int i = j + 1; i <= std::min(j + P, Mf - 1); ++i) {
            const double l = A[(size_t)i * Mf + j] / A[(size_t)j * Mf + j];
            A[(size_t)i * Mf + j] = l;
            for (int c = j + 1; c <= std::min(j + P, Mf - 1); ++c) A[(size_t)i * Mf + c] -= l * A[(size_t)j * Mf + c];
        }
    out.assign((size_t)(2 * P + 1) * Mf, 0.0);
    for (int i = 0; i < Mf; ++i) {
        for (int k = 0; k < P; ++k) {
            if (i - 1 - k >= 0) out[(size_t)k * Mf + i] = A[(size_t)i * Mf + (i - 1 - k)];
            if (i + 1 + k < Mf) out[(size_t)(P + k) * Mf + i] = A[(size_t)i * Mf + (i + 1 + k)] / A[(size_t)i * Mf + i];
        }
        out[(size_t)2 * P * Mf + i] = 1.0 / A[(size_t)i * Mf + i];
    }
}

// Factors of the three axes (FP64 and FP32 copies, then the 1D mass diagonal in FP64): they depend on the mesh
// and its Dirichlet faces only, so they are built and uploaded once per mesh (on the stream, waited for).  Sigma follows
// the Jacobi diagonal: the FP32 scale after every new diagonal, the FP64 one only when an FP64 solve asks for it;
// both are enqueued on the stream without a host synchronization.
int tensor_prec_setup(evap_mesh* h, bool fp64, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    const int P = m.P, M = m.M;
    const int64_t N = 3 * m.Nu;
    if (!h->tp_fac) {
        std::vector<double> Mg;
        mass_1d(h->b, m.n, m.h, Mg);
        std::vector<double> all;
        for (int a = 0; a < 3; ++a) {
            const int lo = (m.faces & (1u << (2 * a))) ? 1 : 0;
            const int hi = (m.faces & (1u << (2 * a + 1))) ? M - 2 : M - 1;
            h->tp_lo[a] = lo;
            h->tp_hi[a] = hi;
            h->tp_off[a] = (int64_t)all.size();
            std::vector<double> f;
            factor_band(Mg, M, P, lo, hi, f);
            all.insert(all.end(), f.begin(), f.end());
        }
        const size_t nf = all.size();
        for (int i = 0; i < M; ++i) all.push_back(Mg[(size_t)i * M + i]);
        // device layout (bytes): factors FP64 [nf], mass diagonal FP64 [M], factors FP32 [nf]
        const size_t bytes = (nf + M) * sizeof(double) + nf * sizeof(float);
        EVAP_CUDA(cudaMalloc(&h->tp_fac, bytes));
        std::vector<float> f32(all.begin(), all.begin() + nf);
        double* fac64 = (double*)h->tp_fac;
        EVAP_CUDA(cudaMemcpyAsync(fac64, all.data(), all.size() * sizeof(double), cudaMemcpyHostToDevice, s));
        EVAP_CUDA(cudaMemcpyAsync(fac64 + nf + M, f32.data(), nf * sizeof(float), cudaMemcpyHostToDevice, s));
        EVAP_CUDA(cudaStreamSynchronize(s));  // the host copies end here
        h->tp_nf = (int64_t)nf;
    }
    const double* md = (const double*)h->tp_fac + h->tp_nf;
    if (!h->tp_valid) {
        if (!h->tp_sigma) EVAP_CUDA(cudaMalloc(&h->tp_sigma, N * sizeof(float)));
        k_tp_sigma<float><<<blocks_for(N, 256), 256, 0, s>>>(M, m.Nu, m.faces, md, h->diag32, h->tp_sigma);
        EVAP_CHECK_LAUNCH("tp_sigma");
        h->tp_valid = true;
        h->tp64_valid = false;
    }
    if (fp64 && !h->tp64_valid) {
        if (!h->tp_sigma64) EVAP_CUDA(cudaMalloc(&h->tp_sigma64, N * sizeof(double)));
        k_tp_sigma<double><<<blocks_for(N, 256), 256, 0, s>>>(M, m.Nu, m.faces, md, h->diag, h->tp_sigma64);
        EVAP_CHECK_LAUNCH("tp_sigma");
        h->tp64_valid = true;
    }
    return EVAP_OK;
}

template <typename T, int P, int AXIS, int MODE>
static int tp_launch(evap_mesh* h, const T* v, T sc, T* t, T* z, T* w, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    const int M = m.M;
    const int lo = h->tp_lo[AXIS], hi = h->tp_hi[AXIS], Mf = hi - lo + 1;
    const size_t smem = ((size_t)(TpShape<P>::FW + TpShape<P>::BW) * Mf + (size_t)M * (TP_LANES + 1)) * sizeof(T);
    if (smem > 48 * 1024)
        EVAP_CUDA(cudaFuncSetAttribute(k_tp_sweep<T, P, AXIS, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
    const double* fac64 = (const double*)h->tp_fac;
    const T* fac = sizeof(T) == 8 ? (const T*)fac64 : (const T*)(const void*)((const float*)(fac64 + h->tp_nf + M));
    const T* sigma = sizeof(T) == 8 ? (const T*)h->tp_sigma64 : (const T*)h->tp_sigma;
    const int64_t M2 = (int64_t)M * M;
    const int64_t blocks = AXIS == 1 ? 3 * (int64_t)((M + TP_LANES - 1) / TP_LANES) * M
                                     : 3 * ((M2 + TP_LANES - 1) / TP_LANES);
    k_tp_sweep<T, P, AXIS, MODE><<<(unsigned)blocks, TP_THREADS, smem, s>>>(M, m.Nu, m.faces, fac + h->tp_off[AXIS],
                                                                         lo, hi, sigma, v, sc, t, z, w);
    EVAP_CHECK_LAUNCH("tp_sweep");
    return EVAP_OK;
}

// z = P (sc v) (and w = Dirichlet ? z : 0 when w is given); t: scratch [3 N_u]; z must not alias v or t.
template <typename T>
int tensor_prec_apply(evap_mesh* h, const T* v, T sc, T* t, T* z, T* w, cudaStream_t s) {
    int rc;
    if (h->m.P == 2) {
        if ((rc = tp_launch<T, 2, 0, 0>(h, v, sc, t, z, w, s))) return rc;
        if ((rc = tp_launch<T, 2, 1, 1>(h, v, sc, t, z, w, s))) return rc;
        return tp_launch<T, 2, 2, 2>(h, v, sc, t, z, w, s);
    }
    if ((rc = tp_launch<T, 3, 0, 0>(h, v, sc, t, z, w, s))) return rc;
    if ((rc = tp_launch<T, 3, 1, 1>(h, v, sc, t, z, w, s))) return rc;
    return tp_launch<T, 3, 2, 2>(h, v, sc, t, z, w, s);
}
template int tensor_prec_apply<float>(evap_mesh*, const float*, float, float*, float*, float*, cudaStream_t);
template int tensor_prec_apply<double>(evap_mesh*, const double*, double, double*, double*, double*, cudaStream_t);

}  // namespace evap
