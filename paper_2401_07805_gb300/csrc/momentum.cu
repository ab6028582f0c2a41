// Momentum apply y = A x (velocity block of Eq. weakNavierStokes linearized about u0, App. D) with the divergence row
// y_p = B x - g (Eq. continuity with the dilation rate of Eq. evaporDil): the pieces shared by its implementations.
//   k_momentum_init   y = x on the Dirichlet DoFs, 0 elsewhere (the scatter of the applies adds the free rows)
//   k_qp_coeffs       the quadrature-point coefficients of the operator (W rho c_m, W rho u0, W rho grad u0, 2 W mu,
//                     z n, W, W v_dil, some with powers of kappa), evaluated once per set_fields and stored as
//                     double-float pairs and, for the u0 terms, in FP32 (the FP32 apply of momentum32.cu): on GB300 the
//                     arithmetic, not HBM, bounds these operators, and the material law and the u0 interpolation
//                     would otherwise be recomputed by every apply
//   launch_momentum   dispatch: FP64 -> double-float kernel, FP32 -> line kernel; the lifting variant (all columns)
#include "df_lines.cuh"
#include "physics.cuh"

namespace evap {

// y = x on Dirichlet DoFs, 0 elsewhere; y_p = 0.  Each warp walks whole x-lines (component c, gy, gz) of M nodes,
// so the line's position is split once per warp and the lanes only test their own gx.
template <typename T>
__global__ void __launch_bounds__(256) k_momentum_init(int M, int64_t Nu, unsigned faces, const T* __restrict__ x,
                                                       T* __restrict__ y, T* __restrict__ yp, int64_t Np) {
    const int lines = 3 * M * M;
    const int wpb = blockDim.x / 32, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int line = blockIdx.x * wpb + warp; line < lines; line += gridDim.x * wpb) {
        const int c = line / (M * M), rem = line - c * M * M, gz = rem / M, gy = rem - gz * M;
        const bool cyz = ((faces & 4u) && gy == 0) || ((faces & 8u) && gy == M - 1) || ((faces & 16u) && gz == 0) ||
                         ((faces & 32u) && gz == M - 1);
        const int64_t off = c * Nu + (int64_t)M * (gy + (int64_t)M * gz);
        for (int gx = lane; gx < M; gx += 32) {
            const bool cons = cyz || ((faces & 1u) && gx == 0) || ((faces & 2u) && gx == M - 1);
            y[off + gx] = cons ? x[off + gx] : T(0);
        }
    }
    if (yp) {
        const int64_t stride = (int64_t)gridDim.x * blockDim.x;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Np; i += stride) yp[i] = T(0);
    }
}

// Quadrature-point coefficients of the momentum operator, evaluated once per set_fields from u0 and the material-law table,
// as double-float pairs (layout [cell][QC_K][nq]):
//   0: W rho c_m   1..3: kappa W rho u0_b   4..12: newton W rho d_d u0_c (index 4 + 3c + d)   13: kappa^2 2 W mu
//   14..16: z n_b (correction gate times normal)   17: kappa W   18: W v_dil
// W = w_qx w_qy w_qz h^3, kappa = DSCALE / h the factor between a gradient and the derivative sweeps (df_lines.cuh).  The
// FP64-accurate apply and the adjoint read the pairs as they stand; the Jacobi diagonal, the mass load and the continuity
// right-hand side read the few slots they need (the two FP64 loads thus take their factors to ~48 bits, as every consumer).  Slots 1..12 are also stored in FP32 for the FP32 apply (there W rho u0 / h:
// that kernel takes reference gradients), in its 32-cell block layout
// qc32[((blk * QC32_K + k) * NQ + pt) * 32 + lane], cell 32 blk + lane (lexicographic).
// Every factor that does not depend on u0 is formed in FP64 and rounded once to a pair (a power of kappa applied to a pair
// would round it twice: the divergence row at Q2 then had 1.03 times the error against 64 bits).
// u0 is interpolated by lines (df_lines.cuh).  The weights and, outside table cells, W rho and 2 W mu take the same NQ
// values in every cell: tabulated on the host, so that the FP64 pipe converts u0 and the table cells' entries only.  A
// block takes CB cells of one 32-cell block, and writes their FP32 entries through shared memory in runs of CB floats.
// Measured at 64^3 Q2 (us): 1374 -> 372 (point-wise dot products, an FP64 copy of every coefficient beside the pairs, 1.1
// GB, and scattered FP32 stores before); the writes alone take 210 at the HBM rate.
template <int NQ>
struct QpTables {
    float2 wk[NQ], wr[2][NQ], wkr[2][NQ], wm[2][NQ];  // kappa W; W rho, kappa W rho and kappa^2 2 W mu of gas (0), liquid (1)
};
template <int P, int CB>
__global__ void __launch_bounds__(CB*(P + 1) * (P + 1) * (P + 1))
    k_qp_coeffs(MeshArgs<double> m, Basis<double> bas, QpTables<(P + 1) * (P + 1) * (P + 1)> tabs, dfl cm_df,
                double kappa, double kappa2, dfl ik, const int8_t* __restrict__ code, const int32_t* __restrict__ tindex,
                const double* __restrict__ table, const double* __restrict__ u0, float2* __restrict__ qcdf,
                float* __restrict__ qc32) {
    constexpr int Q = P + 1, NQ = Q * Q * Q, NL = Q * Q, TASKS = 3 * NL;
    static_assert(32 % CB == 0, "a block's cells lie in one 32-cell block");
    using Ln = DfLine<Q>;
    __shared__ dfl buf[CB][12][NQ];  // slots: 0..2 U, 3 + 3 k + d the derivatives (in units of kappa)
    __shared__ float2 swk[NQ], swr[2][NQ], swkr[2][NQ], swm[2][NQ];
    const int tid = threadIdx.x;
    const int lc = tid / NQ, t = tid % NQ;
    const unsigned cell0 = blockIdx.x * CB;
    int cx, cy, cz;
    const bool active = colour_cell32(cell0 + lc, m.n, -1, cx, cy, cz);
    for (int i = tid; i < NQ; i += CB * NQ) {
        swk[i] = tabs.wk[i];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            swr[k][i] = tabs.wr[k][i];
            swkr[k][i] = tabs.wkr[k][i];
            swm[k][i] = tabs.wm[k][i];
        }
    }
    const int M = m.M;
    const int64_t zst = (int64_t)M * M;
    for (int k0 = t; k0 < TASKS; k0 += NQ) {
        const int f = k0 / NL, l = k0 % NL;
        const double* src = u0 + f * m.Nu + (P * cx + l % Q) + (int64_t)M * (P * cy + l / Q) + zst * (P * cz);
        dfl u[Q], v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) u[k] = df_from_double(src[k * zst]);
        Ln::val(u, v);
        st_line<Q, 2>(buf[lc][3 + f], l, v);
    }
    __syncthreads();
    for (int k0 = t; k0 < TASKS; k0 += NQ) {
        const int f = k0 / NL, l = k0 % NL;
        dfl u[Q], v[Q];
        ld_line<Q, 1>(buf[lc][3 + f], l, u);
        Ln::val(u, v);
        st_line<Q, 1>(buf[lc][6 + f], l, v);
    }
    __syncthreads();
    for (int k0 = t; k0 < TASKS; k0 += NQ) {
        const int f = k0 / NL, l = k0 % NL;
        dfl u[Q], v[Q];
        ld_line<Q, 0>(buf[lc][6 + f], l, u);
        Ln::val(u, v);
        st_line<Q, 0>(buf[lc][f], l, v);
    }
    __syncthreads();
    for (int k0 = t; k0 < TASKS; k0 += NQ) {
        const int f = k0 / NL, l = k0 % NL;
        dfl u[Q], v[Q];
        ld_line<Q, 0>(buf[lc][f], l, u);
        Ln::der(u, v);
        st_line<Q, 0>(buf[lc][3 + 3 * f], l, v);
        ld_line<Q, 1>(buf[lc][f], l, u);
        Ln::der(u, v);
        st_line<Q, 1>(buf[lc][4 + 3 * f], l, v);
        ld_line<Q, 2>(buf[lc][f], l, u);
        Ln::der(u, v);
        st_line<Q, 2>(buf[lc][5 + 3 * f], l, v);
    }
    __syncthreads();
    const unsigned cell = cell0 + lc;
    float f32[QC32_K];
    {
        dfl wr, wk, wm, nz[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}}, wv{0.f, 0.f};
        const int8_t cc = active ? code[cell] : (int8_t)CELL_GAS;
        if (cc == CELL_TABLE) {
            const double* tb = table + (int64_t)tindex[cell] * TAB_K * NQ + t;
            const double Wd = bas.w[t % Q] * bas.w[(t / Q) % Q] * bas.w[t / NL] * m.vol_w;
            const double wrd = Wd * tb[0];
            wr = df_from_double(wrd);
            wk = df_from_double(kappa * wrd);
            wm = df_from_double(kappa2 * (2.0 * Wd * tb[NQ]));
#pragma unroll
            for (int d = 0; d < 3; ++d) nz[d] = df_from_double(tb[(2 + d) * NQ]);
            wv = df_from_double(Wd * tb[5 * NQ]);
        } else {
            const int liq = cc == CELL_LIQUID ? 1 : 0;
            wr = ld_df(&swr[liq][t]);
            wk = ld_df(&swkr[liq][t]);
            wm = ld_df(&swm[liq][t]);
        }
        float2* dst = qcdf + (int64_t)cell * QC_K * NQ + t;
        auto put = [&](int k, dfl v) {
            if (active) dst[k * NQ] = make_float2(v.hi, v.lo);
        };
        put(0, df_mul(wr, cm_df));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const dfl v = df_mul(wk, buf[lc][k][t]);
            put(1 + k, v);
            f32[k] = df_mul(v, ik).hi;
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const dfl v = m.newton ? df_mul(wk, df_norm(buf[lc][3 + k][t])) : dfl{0.f, 0.f};
            put(4 + k, v);
            f32[3 + k] = v.hi;
        }
        put(13, wm);
#pragma unroll
        for (int d = 0; d < 3; ++d) put(14 + d, nz[d]);
        put(17, ld_df(&swk[t]));
        put(18, wv);
    }
    __syncthreads();
    float* const st = reinterpret_cast<float*>(buf);  // [k][point][cell]
#pragma unroll
    for (int k = 0; k < QC32_K; ++k) st[(k * NQ + t) * CB + lc] = f32[k];
    __syncthreads();
    float* const dst32 = qc32 + (int64_t)(cell0 >> 5) * QC32_K * NQ * 32 + (cell0 & 31u);
    const int live = min(CB, (int)(m.ncell - (int64_t)cell0));
    for (int i = tid; i < QC32_K * NQ * CB; i += CB * NQ)
        if (i % CB < live) dst32[(int64_t)(i / CB) * 32 + i % CB] = st[i];
}

template <int P, int CB>
static void run_qp_coeffs(evap_mesh* h, cudaStream_t s) {
    constexpr int Q = P + 1, NQ = Q * Q * Q;
    const MeshArgs<double>& m = h->m;
    const double kd = df_kappa(m);
    QpTables<NQ> tabs;
    auto pair = [](double v) {
        const dfl d = df_from_double(v);
        return make_float2(d.hi, d.lo);
    };
    for (int q = 0; q < NQ; ++q) {
        const double W = h->b.w[q % Q] * h->b.w[(q / Q) % Q] * h->b.w[q / (Q * Q)] * m.vol_w;
        tabs.wk[q] = pair(kd * W);
        for (int k = 0; k < 2; ++k) {
            const double wr = W * (k ? m.rho_H1 : m.rho_H0);
            tabs.wr[k][q] = pair(wr);
            tabs.wkr[k][q] = pair(kd * wr);
            tabs.wm[k][q] = pair(kd * kd * 2.0 * W * (k ? m.mu_H1 : m.mu_H0));
        }
    }
    k_qp_coeffs<P, CB><<<(unsigned)((m.ncell + CB - 1) / CB), CB * NQ, 0, s>>>(
        m, h->b, tabs, df_from_double(m.c_mass), kd, kd * kd, df_from_double(m.inv_h / kd), h->cell_code, h->table_index,
        h->table, h->u, (float2*)h->qcdf, h->qc32);
}

int launch_qp_coeffs(evap_mesh* h, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    const int nq = h->b.Q * h->b.Q * h->b.Q;
    const int64_t need = m.ncell * QC_K * nq;
    if (h->qcdf_len < 2 * need) {
        if (h->qcdf) cudaFree(h->qcdf);
        h->qcdf = nullptr;
        h->qcdf_len = 0;
        EVAP_CUDA(cudaMalloc(&h->qcdf, 2 * need * sizeof(float)));
        h->qcdf_len = 2 * need;
    }
    const int64_t need32 = (m.ncell + 31) / 32 * QC32_K * nq * 32;
    if (h->qc32_len < need32) {
        if (h->qc32) cudaFree(h->qc32);
        h->qc32 = nullptr;
        h->qc32_len = 0;
        EVAP_CUDA(cudaMalloc(&h->qc32, need32 * sizeof(float)));
        h->qc32_len = need32;
    }
    if (m.P == 2)
        run_qp_coeffs<2, 8>(h, s);
    else
        run_qp_coeffs<3, 4>(h, s);
    EVAP_CHECK_LAUNCH("qp_coeffs");
    return EVAP_OK;
}

// dst = src on the DoFs of the Dirichlet faces, one warp per x-line as k_momentum_init.
__global__ void __launch_bounds__(256) k_constrained_copy(int M, int64_t Nu, unsigned faces,
                                                          const double* __restrict__ src, double* __restrict__ dst) {
    const int lines = 3 * M * M;
    const int wpb = blockDim.x / 32, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int line = blockIdx.x * wpb + warp; line < lines; line += gridDim.x * wpb) {
        const int c = line / (M * M), rem = line - c * M * M, gz = rem / M, gy = rem - gz * M;
        const bool cyz = ((faces & 4u) && gy == 0) || ((faces & 8u) && gy == M - 1) || ((faces & 16u) && gz == 0) ||
                         ((faces & 32u) && gz == M - 1);
        const int64_t off = c * Nu + (int64_t)M * (gy + (int64_t)M * gz);
        for (int gx = lane; gx < M; gx += 32)
            if (cyz || ((faces & 1u) && gx == 0) || ((faces & 2u) && gx == M - 1)) dst[off + gx] = src[off + gx];
    }
}

// *flag = 1 if src is nonzero on a Dirichlet DoF.
__global__ void __launch_bounds__(256) k_constrained_nonzero(int M, int64_t Nu, unsigned faces,
                                                             const double* __restrict__ src, unsigned* flag) {
    const int lines = 3 * M * M;
    const int wpb = blockDim.x / 32, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    bool any = false;
    for (int line = blockIdx.x * wpb + warp; line < lines; line += gridDim.x * wpb) {
        const int c = line / (M * M), rem = line - c * M * M, gz = rem / M, gy = rem - gz * M;
        const bool cyz = ((faces & 4u) && gy == 0) || ((faces & 8u) && gy == M - 1) || ((faces & 16u) && gz == 0) ||
                         ((faces & 32u) && gz == M - 1);
        const int64_t off = c * Nu + (int64_t)M * (gy + (int64_t)M * gz);
        for (int gx = lane; gx < M; gx += 32)
            if ((cyz || ((faces & 1u) && gx == 0) || ((faces & 2u) && gx == M - 1)) && src[off + gx] != 0.0) any = true;
    }
    if (__any_sync(0xffffffffu, any) && lane == 0) atomicOr(flag, 1u);
}

static unsigned constrained_grid(const MeshArgs<double>& m) {
    const int64_t lines = 3 * (int64_t)m.M * m.M;
    return (unsigned)std::min<int64_t>((lines + 7) / 8, 152 * 16);
}

int launch_constrained_copy(evap_mesh* h, const double* src, double* dst, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    if (!m.faces) return EVAP_OK;
    k_constrained_copy<<<constrained_grid(m), 256, 0, s>>>(m.M, m.Nu, m.faces, src, dst);
    EVAP_CHECK_LAUNCH("constrained_copy");
    return EVAP_OK;
}

int constrained_nonzero(evap_mesh* h, const double* src, bool* any, cudaStream_t s) {
    const MeshArgs<double>& m = h->m;
    *any = false;
    if (!m.faces) return EVAP_OK;
    // the input-check counter doubles as the flag (it is only read right after its own reduction)
    if (!h->nonfinite) EVAP_CUDA(cudaMalloc(&h->nonfinite, sizeof(unsigned long long)));
    unsigned* flag = reinterpret_cast<unsigned*>(h->nonfinite);
    EVAP_CUDA(cudaMemsetAsync(flag, 0, sizeof(unsigned), s));
    k_constrained_nonzero<<<constrained_grid(m), 256, 0, s>>>(m.M, m.Nu, m.faces, src, flag);
    EVAP_CHECK_LAUNCH("constrained_nonzero");
    unsigned hv = 0;
    EVAP_CUDA(cudaMemcpyAsync(&hv, flag, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    EVAP_CUDA(cudaStreamSynchronize(s));
    *any = hv != 0;
    return EVAP_OK;
}

template <typename T>
int launch_momentum(evap_mesh* h, const T* x, T* y, T* yp, cudaStream_t s, bool init, const T* p, bool all_columns) {
    MeshArgs<double> m = h->m;
    if (all_columns) {
        // the unconstrained operator (no face read as 0), then the identity rows of the real faces
        if (sizeof(T) != 8 || !init) return EVAP_EINVAL;
        m.faces = 0u;
    }
    if (init) {
        const int64_t lines = 3 * (int64_t)m.M * m.M;
        const unsigned grid = (unsigned)std::min<int64_t>((lines + 7) / 8, 152 * 16);
        k_momentum_init<T><<<grid, 256, 0, s>>>(m.M, m.Nu, m.faces, x, y, yp, m.Np);  // y_p: pressure space
        EVAP_CHECK_LAUNCH("momentum_init");
    }
    if constexpr (sizeof(T) == 4) {  // FP32: line-oriented kernel (momentum32.cu)
        if (p) return EVAP_EINVAL;  // the pressure term is FP64 only
        return launch_momentum32(h, x, y, yp, s);
    } else {  // FP64-accurate: double-float arithmetic on the FP32 pipe (momentum_df.cu)
        int rc = launch_momentum_df(h, m, x, y, yp, p, s);
        if (rc) return rc;
        if (all_columns) return launch_constrained_copy(h, x, y, s);
        return EVAP_OK;
    }
}
template int launch_momentum<double>(evap_mesh*, const double*, double*, double*, cudaStream_t, bool, const double*,
                                     bool);
template int launch_momentum<float>(evap_mesh*, const float*, float*, float*, cudaStream_t, bool, const float*, bool);

}  // namespace evap
