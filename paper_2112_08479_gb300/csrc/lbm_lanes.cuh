// lbm_lanes.cuh -- arithmetic of the collisions on one node (float) or on two
// nodes side by side (float2, the packed FP32 instructions of sm_100 and
// later: one issue slot for the same operation on both halves).
//
// Every operation is written out (no contraction is left to the compiler), so
// a collision gives the same bits for a node whether it is computed alone or
// as either half of a pair.
#pragma once

#include "lbm_common.cuh"

namespace lbmgpu {

struct One {
    using V = float;
    static __device__ __forceinline__ V set(float a) { return a; }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ V sub(V a, V b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ V neg(V a) { return -a; }
    static __device__ __forceinline__ V rcp0(V a) { return __fdividef(1.0f, a); }
    static __device__ __forceinline__ V rsqrt0(V a) { return rsqrtf(fmaxf(a, 1e-37f)); }
};

struct Two {
    using V = float2;
    static __device__ __forceinline__ V set(float a) { return make_float2(a, a); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
    // a - b: the product with -1 is exact, so this rounds once, as a subtraction
    static __device__ __forceinline__ V sub(V a, V b) { return __ffma2_rn(b, set(-1.0f), a); }
    // (PTX: the compiler fuses a product of __fmul2_rn into a following __fadd2_rn)
    static __device__ __forceinline__ V mul(V a, V b) {
        V d;
        asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
            "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
            : "=f"(d.x), "=f"(d.y)
            : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
        return d;
    }
    static __device__ __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
    static __device__ __forceinline__ V rcp0(V a) {
        return make_float2(One::rcp0(a.x), One::rcp0(a.y));
    }
    static __device__ __forceinline__ V rsqrt0(V a) {
        return make_float2(One::rsqrt0(a.x), One::rsqrt0(a.y));
    }
};

// 1 / a and sqrt(a): the hardware estimate (relative error about 1e-7) and one
// Newton-Raphson step, to about half a unit in the last place, in packed
// arithmetic.  sqrt takes a >= 0; the estimate is taken of at least 1e-37 so
// that sqrt(0) = 0.  (1 / a of a > 2^126 is 0, the hardware estimate's.  sqrt of
// infinity is NaN, where the BGK collision would form inf / inf from infinity.)
template <typename L>
__device__ __forceinline__ typename L::V lane_rcp(typename L::V a) {
    const typename L::V r = L::rcp0(a);
    return L::fma(r, L::fma(L::neg(a), r, L::set(1.0f)), r);
}
template <typename L>
__device__ __forceinline__ typename L::V lane_sqrt(typename L::V a) {
    const typename L::V y = L::rsqrt0(a);
    const typename L::V s = L::mul(a, y);
    return L::fma(L::fma(L::neg(s), s, a), L::mul(L::set(0.5f), y), s);
}

}  // namespace lbmgpu
