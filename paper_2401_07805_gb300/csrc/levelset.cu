// Matrix-free Q1 level-set operators with the 2^3 Gauss rule (Sec. 2.5), one thread per cell:
//   EVAP_ADVECT      y_i = sum_q W [ N_i x + theta dt N_i (u_Gamma . grad x) ]            Eq. (weakFormLevelSet), CN
//   EVAP_REINIT      y_i = sum_q W [ N_i x / dtau + eps (grad N_i . n)(grad x . n) ]      Eq. (reinitialization)
//   EVAP_REINIT_RHS  y_i = sum_q W [ N_i x / dtau + (grad N_i . n) (1 - x^2) / 2 ]        explicit compressive flux
// The FP64 pipe bounds the FP64 reinitialization operators, so they run by sum factorization (q1_points.cuh).  Measured at
// 64^3 (us): operator 454 -> 208, explicit side 413 -> 180 (direct sums over nodes and points before).
// with n the frozen normal at the quadrature point: grad phi / |grad phi| of the level set (Eq. normal_vector), or,
// when a nodal normal field is set (e.g. the projected normal of Eq. normal_vector_regularized), its normalized
// interpolant (frozen_normals).  The FP64 advection runs in double-float arithmetic (the FP64 pipe bounds the FP64
// version), sum-factorized (k_levelset_advect_sf); the reinitialization operators stay in FP64.
#include <type_traits>

#include "df_lines.cuh"
#include "q1_points.cuh"

namespace evap {

template <typename T, int MODE, bool DET>
__global__ void __launch_bounds__(128) k_levelset(MeshArgs<T> m, T wm, T wd, const T* __restrict__ phi,
                                                  const T* __restrict__ nf, const T* __restrict__ ug,
                                                  const T* __restrict__ x, T* __restrict__ y, int colour) {
    int cx, cy, cz;
    if constexpr (DET) {
        if (!colour_cell(blockIdx.x * (int64_t)blockDim.x + threadIdx.x, m.n, colour, cx, cy, cz)) return;
    } else {  // written out: the shared helper's form of this test cost the atomic variant 100 registers
        const int64_t cell = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        if (cell >= m.ncell) return;
        cx = (int)(cell % m.n), cy = (int)((cell / m.n) % m.n), cz = (int)(cell / ((int64_t)m.n * m.n));
    }
    const int n = m.n;
    const int64_t m1 = n + 1;
    int64_t node[8];
    T xv[8], pv[8], uv[3][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        node[j] = (cx + (j & 1)) + m1 * ((cy + ((j >> 1) & 1)) + m1 * (cz + (j >> 2)));
        xv[j] = x[node[j]];
        if (MODE == EVAP_ADVECT) {
#pragma unroll
            for (int k = 0; k < 3; ++k) uv[k][j] = ug[k * m.Nphi + node[j]];
        } else if (nf) {
#pragma unroll
            for (int k = 0; k < 3; ++k) uv[k][j] = nf[k * m.Nphi + node[j]];
            pv[j] = T(0);
        } else {
            pv[j] = phi[node[j]];
        }
    }
    T out[8], X[8], gx[4], gy[4], gz[4];  // values and reference gradient (physical gradient = reference / h)
    const T ih = m.inv_h;
    const T W = T(0.125) * m.vol_w;  // 2-point Gauss weights 1/2 in each direction
    q1_points(xv, X, gx, gy, gz);
    if (MODE == EVAP_ADVECT) {
        T U[3][8], F[8], d0[4], d1[4], d2[4];
#pragma unroll
        for (int k = 0; k < 3; ++k) q1_points(uv[k], U[k], d0, d1, d2);
        const T c = m.theta * m.dt * ih;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int qx = q & 1, qy = (q >> 1) & 1, qz = q >> 2;
            F[q] = W * (X[q] + c * (U[0][q] * gx[qy + 2 * qz] + U[1][q] * gy[qx + 2 * qz] + U[2][q] * gz[qx + 2 * qy]));
        }
        q1_test<false>(F, F, F, F, out);
    } else {
        T nv[8][3], F[8], G0[8], G1[8], G2[8];  // G: flux tested with the reference gradients (physical flux / h)
        frozen_normals<T>(nf != nullptr, uv, pv, nv);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int qx = q & 1, qy = (q >> 1) & 1, qz = q >> 2;
            F[q] = wm * X[q];
            const T s = MODE == EVAP_REINIT
                            ? wd * (gx[qy + 2 * qz] * nv[q][0] + gy[qx + 2 * qz] * nv[q][1] + gz[qx + 2 * qy] * nv[q][2])
                            : wd * (T(1) - X[q] * X[q]);
            G0[q] = s * nv[q][0];
            G1[q] = s * nv[q][1];
            G2[q] = s * nv[q][2];
        }
        q1_test<true>(F, G0, G1, G2, out);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) acc_add(&y[node[j]], out[j], DET);
}

// EVAP_ADVECT for the FP64 applies in double-float arithmetic (dfloat.cuh) with x converted per node, u_Gamma read from its
// double-float copy and the scatter in FP64, by sum factorization: the trilinear interpolation of x and u_Gamma to the 2^3 Gauss points and
// the testing with the shape functions as three 1D sweeps of the 2 x 2 matrix N[q][j] (N_0 = 1 - t, N_1 = t at the
// Gauss points t), the reference gradient of x as differences along its own direction interpolated along the other
// two: 132 two-term double-float dot products per cell in place of the direct sums' 8 x 7 eight-term ones.
__device__ __forceinline__ dfl dot2(dfl c0, dfl v0, dfl c1, dfl v1) {
    dfl s = df_prod(c0, v0);
    df_fma(s, c1, v1);
    return df_norm(s);
}
template <bool DET>
__global__ void __launch_bounds__(128) k_levelset_advect_sf(MeshArgs<double> m, dfl W, dfl thdt_ih,
                                                            const float2* __restrict__ ug, const double* __restrict__ x,
                                                            double* __restrict__ y, int colour) {
    int cx, cy, cz;
    if constexpr (DET) {
        if (!colour_cell(blockIdx.x * (int64_t)blockDim.x + threadIdx.x, m.n, colour, cx, cy, cz)) return;
    } else {
        const int64_t cell = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        if (cell >= m.ncell) return;
        cx = (int)(cell % m.n), cy = (int)((cell / m.n) % m.n), cz = (int)(cell / ((int64_t)m.n * m.n));
    }
    constexpr double t0 = g2_point(0), t1 = g2_point(1);
    // N[q][j]: shape function j (0: 1 - t, 1: t) at Gauss point q
    const dfl N[2][2] = {{EVAP_DFK(1.0 - t0), EVAP_DFK(t0)}, {EVAP_DFK(1.0 - t1), EVAP_DFK(t1)}};
    const int n = m.n;
    const int64_t m1 = n + 1;
    int64_t node[8];  // j = ja + 2 jb + 4 jc
#pragma unroll
    for (int j = 0; j < 8; ++j) node[j] = (cx + (j & 1)) + m1 * ((cy + ((j >> 1) & 1)) + m1 * (cz + (j >> 2)));
    // values of a nodal field at the points q = qx + 2 qy + 4 qz
    auto interp = [&](const dfl* f, dfl* out) {
        dfl fx[8], fxy[8];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) fx[q + 2 * r] = dot2(N[q][0], f[2 * r], N[q][1], f[2 * r + 1]);
#pragma unroll
        for (int jc = 0; jc < 2; ++jc)
#pragma unroll
            for (int qy = 0; qy < 2; ++qy)
#pragma unroll
                for (int qx = 0; qx < 2; ++qx)
                    fxy[qx + 2 * (qy + 2 * jc)] = dot2(N[qy][0], fx[qx + 2 * (0 + 2 * jc)], N[qy][1], fx[qx + 2 * (1 + 2 * jc)]);
#pragma unroll
        for (int qz = 0; qz < 2; ++qz)
#pragma unroll
            for (int r = 0; r < 4; ++r) out[r + 4 * qz] = dot2(N[qz][0], fxy[r], N[qz][1], fxy[r + 4]);
    };
    dfl X[8], GXx[4], GXy[4], GXz[4];  // GXx[qy + 2 qz], GXy[qx + 2 qz], GXz[qx + 2 qy] (reference gradient)
    {
        dfl f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = df_from_double(x[node[j]]);
        dfl fx[8], dx[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
#pragma unroll
            for (int q = 0; q < 2; ++q) fx[q + 2 * r] = dot2(N[q][0], f[2 * r], N[q][1], f[2 * r + 1]);
            dx[r] = df_sub(f[2 * r + 1], f[2 * r]);  // r = jb + 2 jc
        }
        dfl fxy[8], dxb[4], dy[4];
#pragma unroll
        for (int jc = 0; jc < 2; ++jc) {
#pragma unroll
            for (int qy = 0; qy < 2; ++qy) {
#pragma unroll
                for (int qx = 0; qx < 2; ++qx)
                    fxy[qx + 2 * (qy + 2 * jc)] = dot2(N[qy][0], fx[qx + 2 * (0 + 2 * jc)], N[qy][1], fx[qx + 2 * (1 + 2 * jc)]);
                dxb[qy + 2 * jc] = dot2(N[qy][0], dx[0 + 2 * jc], N[qy][1], dx[1 + 2 * jc]);
            }
#pragma unroll
            for (int qx = 0; qx < 2; ++qx) dy[qx + 2 * jc] = df_sub(fx[qx + 2 * (1 + 2 * jc)], fx[qx + 2 * (0 + 2 * jc)]);
        }
#pragma unroll
        for (int qz = 0; qz < 2; ++qz) {
#pragma unroll
            for (int r = 0; r < 4; ++r) X[r + 4 * qz] = dot2(N[qz][0], fxy[r], N[qz][1], fxy[r + 4]);
#pragma unroll
            for (int qy = 0; qy < 2; ++qy) GXx[qy + 2 * qz] = dot2(N[qz][0], dxb[qy], N[qz][1], dxb[qy + 2]);
#pragma unroll
            for (int qx = 0; qx < 2; ++qx) GXy[qx + 2 * qz] = dot2(N[qz][0], dy[qx], N[qz][1], dy[qx + 2]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) GXz[r] = df_sub(fxy[r + 4], fxy[r]);
    }
    dfl Fv[8];
    {
        dfl U[3][8];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            dfl f[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) f[j] = ld_df(ug + d * m.Nphi + node[j]);
            interp(f, U[d]);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int qx = q & 1, qy = (q >> 1) & 1, qz = q >> 2;
            dfl ug_gx = df_prod(U[0][q], GXx[qy + 2 * qz]);
            df_fma(ug_gx, U[1][q], GXy[qx + 2 * qz]);
            df_fma(ug_gx, U[2][q], GXz[qx + 2 * qy]);
            dfl v = X[q];
            df_fma(v, thdt_ih, df_norm(ug_gx));
            Fv[q] = df_mul(W, df_norm(v));
        }
    }
    // test: out_j = sum_q N_j(q) Fv_q by the transposed sweeps z, y, x
    dfl T1[8], T2[8];
#pragma unroll
    for (int jc = 0; jc < 2; ++jc)
#pragma unroll
        for (int r = 0; r < 4; ++r) T1[r + 4 * jc] = dot2(N[0][jc], Fv[r], N[1][jc], Fv[r + 4]);  // r = qx + 2 qy
#pragma unroll
    for (int jc = 0; jc < 2; ++jc)
#pragma unroll
        for (int jb = 0; jb < 2; ++jb)
#pragma unroll
            for (int qx = 0; qx < 2; ++qx)
                T2[qx + 2 * (jb + 2 * jc)] = dot2(N[0][jb], T1[qx + 2 * (0 + 2 * jc)], N[1][jb], T1[qx + 2 * (1 + 2 * jc)]);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int ja = 0; ja < 2; ++ja) {
            const dfl o = dot2(N[0][ja], T2[2 * r], N[1][ja], T2[2 * r + 1]);
            acc_add(&y[node[ja + 2 * r]], df_to_double(o), DET);
        }
}

// (The sum-factorized advection took 45.2 us per apply at 64^3, 275 k DoFs, where direct 8-point sums took 57.8.)
template <typename T>
int launch_levelset(evap_mesh* h, int mode, const T* x, T* y, cudaStream_t s) {
    const MeshArgs<T> m = ls_args<T>(h);  // Q1 on the level-set mesh
    // factors of the mass and the flux term of the reinitialization operators, formed in FP64 and rounded once: a rounded
    // factor is wrong by the same amount at every point
    const MeshArgs<double> md = ls_args<double>(h);
    const double Wd = 0.125 * md.vol_w;
    const T wm = (T)(Wd / md.dtau);
    const T wd = (T)(mode == EVAP_REINIT ? Wd * md.eps * md.inv_h * md.inv_h : Wd * 0.5 * md.inv_h);
    const bool dbl = sizeof(T) == 8;
    const T* phi = dbl ? (const T*)h->phi : (const T*)h->phi32;
    const T* ug = dbl ? (const T*)h->ugamma : (const T*)h->ugamma32;
    const T* nf = dbl ? (const T*)h->ls_normal : (const T*)h->ls_normal32;
    int rc = launch_fill<T>(y, m.Nphi, T(0), s);
    if (rc) return rc;
    const int threads = 128;
    // colour passes (deterministic) or one atomic pass, each variant compiled apart
    auto go = [&](auto det) -> int {
        constexpr bool DET = decltype(det)::value;
        for (int colour = DET ? 0 : -1; colour < (DET ? 8 : 0); ++colour) {
            const int64_t cells = colour_cells(m.n, colour);
            if (cells == 0) continue;
            const unsigned grid = (unsigned)((cells + threads - 1) / threads);
            if (mode == EVAP_ADVECT) {
                if constexpr (sizeof(T) == 8) {  // FP64-accurate advection in double-float arithmetic
                    const dfl W = df_from_double(0.125 * (double)m.vol_w);  // 2-point Gauss weights 1/2 per direction
                    const dfl thdt_ih = df_from_double((double)m.theta * (double)m.dt * (double)m.inv_h);
                    k_levelset_advect_sf<DET><<<grid, threads, 0, s>>>(m, W, thdt_ih, (const float2*)h->ugammadf,
                                                                       (const double*)x, (double*)y, colour);
                } else {
                    k_levelset<T, EVAP_ADVECT, DET><<<grid, threads, 0, s>>>(m, wm, wd, phi, nullptr, ug, x, y, colour);
                }
            } else if (mode == EVAP_REINIT) {
                k_levelset<T, EVAP_REINIT, DET><<<grid, threads, 0, s>>>(m, wm, wd, phi, nf, ug, x, y, colour);
            } else {
                k_levelset<T, EVAP_REINIT_RHS, DET><<<grid, threads, 0, s>>>(m, wm, wd, phi, nf, ug, x, y, colour);
            }
            EVAP_CHECK_LAUNCH("levelset");
        }
        return EVAP_OK;
    };
    return h->deterministic ? go(std::true_type{}) : go(std::false_type{});
}
template int launch_levelset<double>(evap_mesh*, int, const double*, double*, cudaStream_t);
template int launch_levelset<float>(evap_mesh*, int, const float*, float*, cudaStream_t);

}  // namespace evap
