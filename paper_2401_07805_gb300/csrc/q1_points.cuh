// Q1 fields at the 2^3 Gauss points of a cell and their testing, by sum factorization with compile-time points: along a
// line with end values f0, f1 and d = f1 - f0 the points t, 1 - t of the 2-point rule hold f0 + t d and f0 + (1 - t) d,
// and d itself is the reference derivative.  Values, reference gradient and test of one field cost 54 and up to 120
// operations a cell, where direct sums over the 8 nodes at 8 points take 256 and 256.  On GB300 the FP64 pipe bounds the
// kernels built on this (2 FMA per cycle and SM), so operations are what counts.
// Index order everywhere: node j = ja + 2 jb + 4 jc, point q = qx + 2 qy + 4 qz, x fastest.
#pragma once

#include "physics.cuh"

namespace evap {

// values X[q] and reference gradient: d/dx at [qy + 2 qz], d/dy at [qx + 2 qz], d/dz at [qx + 2 qy] (constant along
// their own direction)
template <typename T>
__device__ __forceinline__ void q1_points(const T (&f)[8], T (&X)[8], T (&gx)[4], T (&gy)[4], T (&gz)[4]) {
    constexpr T t0 = T(g2_point(0)), t1 = T(g2_point(1));
    T vx[8], dx[4], vxy[8], dy[4], dxy[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // r = jb + 2 jc
        dx[r] = f[2 * r + 1] - f[2 * r];
        vx[2 * r] = f[2 * r] + t0 * dx[r];
        vx[2 * r + 1] = f[2 * r] + t1 * dx[r];
    }
#pragma unroll
    for (int jc = 0; jc < 2; ++jc) {
#pragma unroll
        for (int qx = 0; qx < 2; ++qx) {
            const T a = vx[qx + 4 * jc], d = vx[qx + 2 + 4 * jc] - a;
            dy[qx + 2 * jc] = d;
            vxy[qx + 4 * jc] = a + t0 * d;
            vxy[qx + 2 + 4 * jc] = a + t1 * d;
        }
        const T a = dx[2 * jc], d = dx[2 * jc + 1] - a;
        dxy[2 * jc] = a + t0 * d;
        dxy[2 * jc + 1] = a + t1 * d;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // r = qx + 2 qy
        const T a = vxy[r], d = vxy[r + 4] - a;
        gz[r] = d;
        X[r] = a + t0 * d;
        X[r + 4] = a + t1 * d;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const T ax = dxy[q], ex = dxy[q + 2] - ax, ay = dy[q], ey = dy[q + 2] - ay;
        gx[q] = ax + t0 * ex;
        gx[q + 2] = ax + t1 * ex;
        gy[q] = ay + t0 * ey;
        gy[q + 2] = ay + t1 * ey;
    }
}

template <typename T>
__device__ __forceinline__ T inv_norm(T g2) {
    return T(1) / sqrt(g2);
}
template <>
__device__ __forceinline__ double inv_norm<double>(double g2) {
    return rsqrt(g2);
}

// Frozen normals of the reinitialization operators at the 8 points (Eq. reinitialization): with a nodal field nf (its
// values at the cell's nodes) the normalized interpolant n_h / |n_h|, zero where |n_h| <= 1e-4, else the unit normal of the
// level set pv, zero where |grad phi| h <= GRAD_TINY (the reference gradient's norm).
template <typename T>
__device__ __forceinline__ void frozen_normals(bool nodal, const T (&nf)[3][8], const T (&pv)[8], T (&nv)[8][3]) {
    T X[8], gx[4], gy[4], gz[4];
    if (nodal) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            q1_points(nf[d], X, gx, gy, gz);
#pragma unroll
            for (int q = 0; q < 8; ++q) nv[q][d] = X[q];
        }
    } else {
        q1_points(pv, X, gx, gy, gz);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int qx = q & 1, qy = (q >> 1) & 1, qz = q >> 2;
            nv[q][0] = gx[qy + 2 * qz];
            nv[q][1] = gy[qx + 2 * qz];
            nv[q][2] = gz[qx + 2 * qy];
        }
    }
    constexpr T least = T(NODAL_NORMAL_TINY * NODAL_NORMAL_TINY);
    static_assert(NODAL_NORMAL_TINY == GRAD_TINY, "one threshold for both kinds of normal");
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const T g2 = nv[q][0] * nv[q][0] + nv[q][1] * nv[q][1] + nv[q][2] * nv[q][2];
        const T ig = g2 > least ? inv_norm(g2) : T(0);
#pragma unroll
        for (int d = 0; d < 3; ++d) nv[q][d] = g2 > least ? nv[q][d] * ig : T(0);
    }
}

// out_j = sum_q N_j(q) F_q (+ the reference gradients of N_j against G when GRAD): transposed sweeps z, y, x
template <bool GRAD, typename T>
__device__ __forceinline__ void q1_test(const T (&F)[8], const T (&Gx)[8], const T (&Gy)[8], const T (&Gz)[8], T (&out)[8]) {
    constexpr T t0 = T(g2_point(0)), t1 = T(g2_point(1));
    T a[8], bx[8], by[8];  // [qx + 2 qy + 4 jc]
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        T o1 = t0 * F[r] + t1 * F[r + 4];
        if (GRAD) o1 += Gz[r] + Gz[r + 4];
        a[r + 4] = o1;
        a[r] = (F[r] + F[r + 4]) - o1;
        if (GRAD) {
            bx[r + 4] = t0 * Gx[r] + t1 * Gx[r + 4];
            bx[r] = (Gx[r] + Gx[r + 4]) - bx[r + 4];
            by[r + 4] = t0 * Gy[r] + t1 * Gy[r + 4];
            by[r] = (Gy[r] + Gy[r + 4]) - by[r + 4];
        }
    }
    T c[8], cx[8];  // [qx + 2 jb + 4 jc]
#pragma unroll
    for (int jc = 0; jc < 2; ++jc)
#pragma unroll
        for (int qx = 0; qx < 2; ++qx) {
            const int p0 = qx + 4 * jc, p1 = p0 + 2;
            T o1 = t0 * a[p0] + t1 * a[p1];
            if (GRAD) o1 += by[p0] + by[p1];
            c[p1] = o1;
            c[p0] = (a[p0] + a[p1]) - o1;
            if (GRAD) {
                cx[p1] = t0 * bx[p0] + t1 * bx[p1];
                cx[p0] = (bx[p0] + bx[p1]) - cx[p1];
            }
        }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        T o1 = t0 * c[2 * r] + t1 * c[2 * r + 1];
        if (GRAD) o1 += cx[2 * r] + cx[2 * r + 1];
        out[2 * r + 1] = o1;
        out[2 * r] = (c[2 * r] + c[2 * r + 1]) - o1;
    }
}

}  // namespace evap
