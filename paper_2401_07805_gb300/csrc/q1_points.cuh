// Q1 fields at the 2^3 Gauss points of a cell and their testing, by sum factorization with compile-time points: along a
// line with end values f0, f1 and d = f1 - f0 the points t, 1 - t of the 2-point rule hold f0 + t d and f0 + (1 - t) d,
// and d itself is the reference derivative.  Values, reference gradient and test of one field cost 54 and up to 120
// operations a cell, where direct sums over the 8 nodes at 8 points take 256 and 256.  On GB300 the FP64 pipe bounds the
// kernels built on this (2 FMA per cycle and SM), so operations are what counts.
// Index order everywhere: node j = ja + 2 jb + 4 jc, point q = qx + 2 qy + 4 qz, x fastest.
#pragma once

#include "physics.cuh"

namespace evap {

// The values v0, v1 at the two points of a line with end values f0, f1 and d = f1 - f0.  FP64 takes the fewest operations; in
// FP32, where the arithmetic is no limit, two-term sums, which round less than the differences.
template <typename T>
__device__ __forceinline__ void q1_line(T f0, T f1, T d, T& v0, T& v1) {
    constexpr T t0 = T(g2_point(0)), t1 = T(g2_point(1));
    if constexpr (sizeof(T) == 4) {
        v0 = t1 * f0 + t0 * f1;
        v1 = t0 * f0 + t1 * f1;
    } else {
        v0 = f0 + t0 * d;
        v1 = f0 + t1 * d;
    }
}
// One line of a transposed sweep: (o0, o1) = sum of the shape values (1 - t, t) times F, with g added to o1 and taken from o0
// (the derivative test); in FP32 again as two sums, in FP64 o0 as the rest.  With both, and the factors of the operators rounded
// once (levelset.cu), the FP32 reinitialization operators have 0.97 times the error against 64 bits of direct sums over nodes
// and points (60 drawn level sets), 1.21 without.
template <typename T>
__device__ __forceinline__ void q1_lineT(T F0, T F1, T g, bool grad, T& o0, T& o1) {
    constexpr T t0 = T(g2_point(0)), t1 = T(g2_point(1));
    o1 = t0 * F0 + t1 * F1;
    if (grad) o1 += g;
    if constexpr (sizeof(T) == 4) {
        o0 = t1 * F0 + t0 * F1;
        if (grad) o0 -= g;
    } else {
        o0 = (F0 + F1) - o1;
    }
}

// values X[q] and reference gradient: d/dx at [qy + 2 qz], d/dy at [qx + 2 qz], d/dz at [qx + 2 qy] (constant along
// their own direction)
template <typename T>
__device__ __forceinline__ void q1_points(const T (&f)[8], T (&X)[8], T (&gx)[4], T (&gy)[4], T (&gz)[4]) {
    T vx[8], dx[4], vxy[8], dy[4], dxy[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // r = jb + 2 jc
        dx[r] = f[2 * r + 1] - f[2 * r];
        q1_line(f[2 * r], f[2 * r + 1], dx[r], vx[2 * r], vx[2 * r + 1]);
    }
#pragma unroll
    for (int jc = 0; jc < 2; ++jc) {
#pragma unroll
        for (int qx = 0; qx < 2; ++qx) {
            const T a = vx[qx + 4 * jc], b = vx[qx + 2 + 4 * jc], d = b - a;
            dy[qx + 2 * jc] = d;
            q1_line(a, b, d, vxy[qx + 4 * jc], vxy[qx + 2 + 4 * jc]);
        }
        q1_line(dx[2 * jc], dx[2 * jc + 1], dx[2 * jc + 1] - dx[2 * jc], dxy[2 * jc], dxy[2 * jc + 1]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // r = qx + 2 qy
        const T a = vxy[r], b = vxy[r + 4], d = b - a;
        gz[r] = d;
        q1_line(a, b, d, X[r], X[r + 4]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        q1_line(dxy[q], dxy[q + 2], dxy[q + 2] - dxy[q], gx[q], gx[q + 2]);
        q1_line(dy[q], dy[q + 2], dy[q + 2] - dy[q], gy[q], gy[q + 2]);
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
    const T zero = T(0);
    T a[8], bx[8], by[8];  // [qx + 2 qy + 4 jc]
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        q1_lineT(F[r], F[r + 4], GRAD ? Gz[r] + Gz[r + 4] : zero, GRAD, a[r], a[r + 4]);
        if (GRAD) {
            q1_lineT(Gx[r], Gx[r + 4], zero, false, bx[r], bx[r + 4]);
            q1_lineT(Gy[r], Gy[r + 4], zero, false, by[r], by[r + 4]);
        }
    }
    T c[8], cx[8];  // [qx + 2 jb + 4 jc]
#pragma unroll
    for (int jc = 0; jc < 2; ++jc)
#pragma unroll
        for (int qx = 0; qx < 2; ++qx) {
            const int p0 = qx + 4 * jc, p1 = p0 + 2;
            q1_lineT(a[p0], a[p1], GRAD ? by[p0] + by[p1] : zero, GRAD, c[p0], c[p1]);
            if (GRAD) q1_lineT(bx[p0], bx[p1], zero, false, cx[p0], cx[p1]);
        }
#pragma unroll
    for (int r = 0; r < 4; ++r)
        q1_lineT(c[2 * r], c[2 * r + 1], GRAD ? cx[2 * r] + cx[2 * r + 1] : zero, GRAD, out[2 * r], out[2 * r + 1]);
}

}  // namespace evap
