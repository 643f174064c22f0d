// Pair terms of the blob mobility for two targets at once, in the lanes of
// float2 registers.
#pragma once
#include "rpy_pair.cuh"

namespace am {

// ---- paired FP32 arithmetic: two targets per thread in the lanes of float2
// registers (__ffma2_rn and friends: one instruction for both targets), the
// source values in shared memory already duplicated and negated so that one
// 128-bit load gives ready register pairs.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 bc2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 rsq2(float2 a) { return make_float2(rsq(a.x), rsq(a.y)); }

// (hi, lo) += t exactly in each lane (Knuth's TwoSum of hi and t, the
// rounding error added to lo): the compensated accumulation of the tile sums
__device__ __forceinline__ void two_sum_acc2(float2& hi, float2& lo, float2 t) {
    const float2 m1 = bc2(-1.f);
    const float2 s = add2(hi, t);
    const float2 v = fma2(hi, m1, s);                          // s - hi
    const float2 e = add2(fma2(fma2(v, m1, s), m1, hi),        // hi - (s - v)
                          fma2(v, m1, t));                      // + (t - v)
    hi = s;
    lo = add2(lo, e);
}

// Free-space pair plus wall image in both lanes: pair_free_r2 and pair_wall_r2
// of rpy_pair.cuh (the same operations, rounded alike), with the free-space
// coefficients of the far branch; pairs closer than 2a in either lane take
// free_coefs per lane.  nx3 = -x3 per lane.
template <bool WALL>
__device__ __forceinline__ void pair2(float2 dx, float2 dy, float2 dz, float2 rxy2, float2 r2, float2 Rz, float2 h2,
                                      float2 nx3, float2 lx, float2 ly, float2 lz, const RpyK<float>& k,
                                      float2& ux, float2& uy, float2& uz) {
    const float2 one = bc2(1.f);
    float2 c1f, c2f;
    if (r2.x < k.four_a2 || r2.y < k.four_a2) {
        free_coefs<float>(r2.x, k, c1f.x, c2f.x);
        free_coefs<float>(r2.y, k, c1f.y, c2f.y);
    } else {
        const float2 ri = rsq2(r2);
        const float2 ri2 = mul2(ri, ri);
        c1f = mul2(ri, fma2(bc2(k.kf2), ri2, one));
        c2f = mul2(mul2(ri, ri2), fma2(bc2(-k.kf3), ri2, one));
    }
    if (!WALL) {
        const float2 sdl = mul2(c2f, fma2(dx, lx, fma2(dy, ly, mul2(dz, lz))));
        ux = fma2(c1f, lx, fma2(sdl, dx, ux));
        uy = fma2(c1f, ly, fma2(sdl, dy, uy));
        uz = fma2(c1f, lz, fma2(sdl, dz, uz));
        return;
    }
    const float2 dlxy = fma2(dx, lx, mul2(dy, ly));
    const float2 Df = fma2(dz, lz, dlxy);
    const float2 sdl = mul2(c2f, Df);
    const float2 Rz2 = mul2(Rz, Rz);
    const float2 Di = fma2(Rz, lz, dlxy);
    const float2 s = rsq2(add2(rxy2, Rz2));
    const float2 w = mul2(s, s), s3 = mul2(s, w), w2 = mul2(w, w);
    const float2 c1 = fma2(h2, nx3, bc2(k.wc1));
    const float2 c2 = fma2(Rz2, bc2(k.w2a2), bc2(k.wc2));
    const float2 c3 = mul2(Rz2, bc2(k.wc3));
    const float2 x1 = fma2(w, c3, c2);
    const float2 cI = fma2(w, fma2(w, x1, c1), bc2(-1.f));
    const float2 y = fma2(w, c3, x1);
    const float2 yz = fma2(w, c3, y);
    const float2 cRR = fma2(mul2(w2, y), bc2(-2.f), fma2(cI, bc2(-3.f), bc2(-4.f)));
    const float2 A4w2n = mul2(w2, bc2(-k.wa4));
    const float2 inner = fma2(cRR, bc2(-2.f), fma2(A4w2n, bc2(-1.f), bc2(-2.f)));
    const float2 P = mul2(s3, fma2(cRR, Di, mul2(fma2(Rz, inner, h2), lz)));
    const float2 QX = fma2(h2, Df, fma2(mul2(A4w2n, Rz), Di, mul2(mul2(w, fma2(yz, bc2(-2.f), bc2(k.wi2))), lz)));
    const float2 uq = fma2(s3, QX, uz);  // rounds as the compiler contracts uz + s3 QX in pair_wall_r2
    const float2 cc = fma2(s, cI, c1f);
    const float2 pp = add2(sdl, P);
    ux = fma2(cc, lx, fma2(pp, dx, ux));
    uy = fma2(cc, ly, fma2(pp, dy, uy));
    uz = fma2(cc, lz, fma2(sdl, dz, fma2(P, Rz, uq)));
}

}  // namespace am
