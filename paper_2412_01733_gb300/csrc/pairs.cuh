// pairs.cuh -- packed FP32 pair terms (two sources per instruction) and the
// compensated fold, shared by the walk and the direct sum.
#pragma once

#include <cfloat>

#include "common.cuh"

namespace treegb {

// --- packed FP32 pair terms: two sources per instruction ---------------------
// 1/r for two pairs.  Softened (SOFT): r^2 >= eps^2, and the FP32 walk takes
// this variant only when eps^2 is a normal FP32 number, so r^2 is never
// subnormal and the PTX approximate reciprocal square root with subnormal
// inputs flushed (rsqrt.approx.ftz.f32) serves; for normal inputs it gave the
// same bits as rsqrtf on sm_103a over a sweep of all normal exponents, and it
// saves rsqrtf's handling of subnormal inputs (the far-cell loop ran 6.6 %
// faster).  Unsoftened: rsqrtf, and a coincident pair (r^2 = 0) contributes
// nothing.
template <bool SOFT>
__device__ __forceinline__ float2 rsqrt_pair(float2 r2) {
    float2 ri;
    if (SOFT) {
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ri.x) : "f"(r2.x));
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ri.y) : "f"(r2.y));
    } else {
        ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
        ri.x = r2.x > 0.f ? ri.x : 0.f;
        ri.y = r2.y > 0.f ? ri.y : 0.f;
    }
    return ri;
}

// Each float2 holds one quantity of two sources (or two cells); the target is
// held negated and duplicated, nP = (-p, -p), so every difference is an add.
// PP: d = r_s - r_i, accumulates m d / r^3 and -m / r for both sources.
template <bool SOFT>
__device__ __forceinline__ void pp_pair(float2 nx, float2 ny, float2 nz, float2 X, float2 Y, float2 Z, float2 M,
                                        float2 eps2, float2 neg1, float2 (&acc)[4]) {
    const float2 dx = __fadd2_rn(X, nx), dy = __fadd2_rn(Y, ny), dz = __fadd2_rn(Z, nz);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, eps2)));
    const float2 ri = rsqrt_pair<SOFT>(r2);
    const float2 ri2 = __fmul2_rn(ri, ri);
    const float2 mr = __fmul2_rn(M, ri);
    const float2 mr3 = __fmul2_rn(mr, ri2);
    acc[0] = __ffma2_rn(mr3, dx, acc[0]);
    acc[1] = __ffma2_rn(mr3, dy, acc[1]);
    acc[2] = __ffma2_rn(mr3, dz, acc[2]);
    acc[3] = __ffma2_rn(neg1, mr, acc[3]);
}

// PC for two cells.  With u = R - r_i (= -y) and the negated quadrupole
// Qn = -Q (the FP32 cell copies store -Q), w = Qn u equals Q y, u.w = -(y.Q.y), and the terms of
// pc_term become a = [M/r^3 - 5/2 (u.w)/r^7] u + w/r^5, phi = -M/r + 1/2 (u.w)/r^5.
// R5 (quadrupole only) takes r^-5 out of the acceleration: with t = (u.w)/r^4,
// a = r^-5 (k u + w), k = r^2 (M - 5/2 t), and accumulates -phi = (M - 1/2 t) / r in acc[3]
// (neg1 must then hold -1/2): 32 packed operations for two cells instead of 34.  It forms
// r^-5 and M r^2 u, so the walk takes it only where pc_r5_fits holds.  This loop alone bounds the
// large walks (FMA pipe); staged cells only, it does 9.1e11 pairs/s (33 operations, without the
// shared t: 8.7e11).
template <bool QUAD, bool SOFT, bool R5 = false>
__device__ __forceinline__ void pc_pair(float2 nx, float2 ny, float2 nz, const float4 &A, const float4 &B,
                                        const float4 &C, const float4 &D, const float4 &E, float2 eps2,
                                        float2 neg1, float2 half, float2 m25, float2 (&acc)[4]) {
    const float2 ux = __fadd2_rn(make_float2(A.x, A.y), nx);
    const float2 uy = __fadd2_rn(make_float2(A.z, A.w), ny);
    const float2 uz = __fadd2_rn(make_float2(B.x, B.y), nz);
    const float2 M = make_float2(B.z, B.w);
    const float2 r2 = __ffma2_rn(ux, ux, __ffma2_rn(uy, uy, __ffma2_rn(uz, uz, eps2)));
    const float2 ri = rsqrt_pair<SOFT>(r2);
    const float2 ri2 = __fmul2_rn(ri, ri);
    const float2 Mr = __fmul2_rn(M, ri);
    const float2 Mr3 = __fmul2_rn(Mr, ri2);
    if (QUAD) {
        const float2 qxx = make_float2(C.x, C.y), qyy = make_float2(C.z, C.w);
        const float2 qzz = make_float2(D.x, D.y), qxy = make_float2(D.z, D.w);
        const float2 qxz = make_float2(E.x, E.y), qyz = make_float2(E.z, E.w);
        const float2 wx = __ffma2_rn(qxx, ux, __ffma2_rn(qxy, uy, __fmul2_rn(qxz, uz)));
        const float2 wy = __ffma2_rn(qxy, ux, __ffma2_rn(qyy, uy, __fmul2_rn(qyz, uz)));
        const float2 wz = __ffma2_rn(qxz, ux, __ffma2_rn(qyz, uy, __fmul2_rn(qzz, uz)));
        const float2 uw = __ffma2_rn(ux, wx, __ffma2_rn(uy, wy, __fmul2_rn(uz, wz)));
        if (R5) {
            const float2 ri4 = __fmul2_rn(ri2, ri2);
            const float2 r5 = __fmul2_rn(ri4, ri);
            const float2 t = __fmul2_rn(uw, ri4);
            const float2 k = __fmul2_rn(r2, __ffma2_rn(m25, t, M));
            acc[0] = __ffma2_rn(r5, __ffma2_rn(k, ux, wx), acc[0]);
            acc[1] = __ffma2_rn(r5, __ffma2_rn(k, uy, wy), acc[1]);
            acc[2] = __ffma2_rn(r5, __ffma2_rn(k, uz, wz), acc[2]);
            acc[3] = __ffma2_rn(ri, __ffma2_rn(neg1, t, M), acc[3]);
        } else {
            const float2 r3 = __fmul2_rn(ri, ri2);
            const float2 r5 = __fmul2_rn(r3, ri2);
            const float2 t = __fmul2_rn(uw, r5);
            const float2 c = __ffma2_rn(t, __fmul2_rn(ri2, m25), Mr3);
            acc[0] = __ffma2_rn(c, ux, __ffma2_rn(r5, wx, acc[0]));
            acc[1] = __ffma2_rn(c, uy, __ffma2_rn(r5, wy, acc[1]));
            acc[2] = __ffma2_rn(c, uz, __ffma2_rn(r5, wz, acc[2]));
            acc[3] = __ffma2_rn(neg1, Mr, __ffma2_rn(half, t, acc[3]));
        }
    } else {
        acc[0] = __ffma2_rn(Mr3, ux, acc[0]);
        acc[1] = __ffma2_rn(Mr3, uy, acc[1]);
        acc[2] = __ffma2_rn(Mr3, uz, acc[2]);
        acc[3] = __ffma2_rn(neg1, Mr, acc[3]);
    }
}

template <typename Real, bool KAHAN>
__device__ __forceinline__ void fold(Real (&sum)[4], Real (&cmp)[4], const Real (&part)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (KAHAN) {
            const Real y = part[c] - cmp[c];
            const Real t = sum[c] + y;
            cmp[c] = (t - sum[c]) - y;
            sum[c] = t;
        } else {
            sum[c] += part[c];
        }
    }
}

// The FP32 softened pair terms need eps^2 to be a normal FP32 number (see
// rsqrt_pair); a smaller eps^2 takes the unsoftened variant, which still adds
// it to r^2 and drops coincident pairs.
inline bool walk_soft_f32(double eps) { return (float)(eps * eps) >= FLT_MIN; }

}  // namespace treegb
