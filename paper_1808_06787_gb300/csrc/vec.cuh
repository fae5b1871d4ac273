// Arithmetic of the node functions, written out operation by operation.
//
// Every add, multiply and fused multiply-add below is explicit and rounds to
// nearest, so the result of a node does not depend on the kernel it is inlined
// into (the compiler contracts nothing), and the same function runs on one node
// (float, double) or on two at once (f2: sm_100's packed FP32 instructions, one
// issue slot for both nodes, each half rounded as the scalar instruction rounds).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbms {

// Two FP32 values of two nodes, in a 64-bit register pair.
struct f2 {
    unsigned long long v;
};

__device__ __forceinline__ f2 pack2(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo(f2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return x;
}
__device__ __forceinline__ float hi(f2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return y;
}

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }

__device__ __forceinline__ f2 vadd(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 vmul(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 vsub(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// A product that an add follows: rounded by itself in every type.  (The assembler fuses
// mul.rn.f32x2 with a following packed add, so the packed product is written as a
// fused multiply-add of +0, which differs from the product in the sign of a zero only.)
__device__ __forceinline__ float vprod(float a, float b) { return vmul(a, b); }
__device__ __forceinline__ double vprod(double a, double b) { return vmul(a, b); }
__device__ __forceinline__ f2 vprod(f2 a, f2 b) { return vfma(a, b, pack2(0.0f, 0.0f)); }

__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ f2 vneg(f2 a) { return vmul(a, pack2(-1.0f, -1.0f)); }
// -(a b): the sign is free in a scalar instruction's operand, but not in a packed one's.
__device__ __forceinline__ float vnmul(float a, float b) { return -__fmul_rn(a, b); }
__device__ __forceinline__ double vnmul(double a, double b) { return -__dmul_rn(a, b); }
__device__ __forceinline__ f2 vnmul(f2 a, f2 b) { return vmul(vmul(a, pack2(-1.0f, -1.0f)), b); }

// A constant or uniform value in every lane of V.
template <typename V>
struct Vec {
    using scalar = V;
    static __device__ __forceinline__ V all(V x) { return x; }
};
template <>
struct Vec<f2> {
    using scalar = float;
    static __device__ __forceinline__ f2 all(float x) { return pack2(x, x); }
};

// Reciprocal of the per-node solve: the fast hardware approximation in FP32
// (well inside the FP32 tolerance), the IEEE division in FP64.
__device__ __forceinline__ float recip(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ double recip(double v) { return 1.0 / v; }
__device__ __forceinline__ f2 recip(f2 v) { return pack2(recip(lo(v)), recip(hi(v))); }

}  // namespace lbms
