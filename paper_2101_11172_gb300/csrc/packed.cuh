// Packed FP32 pairs (sm_100 and later: add, sub, mul and fma.rn.f32x2).
#pragma once

#include <cuda_runtime.h>

namespace ws {

// Complex arithmetic on packed pairs (add/mul/fma.rn.f32x2): one instruction
// works on both components, and an operand's swapped or broadcast components
// cost nothing (they are operand forms of the instruction).  The transforms
// are bound by instruction issue as much as by the FP32 pipe, and a complex add
// is one instruction here instead of two, a product two to three instead of four.
__device__ __forceinline__ unsigned long long bits2(float2 a) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a.x), "f"(a.y));
    return d;
}
__device__ __forceinline__ float2 pair2(unsigned long long d) {
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(d));
    return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(bits2(a)), "l"(bits2(b)));
    return pair2(d);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(bits2(a)), "l"(bits2(b)));
    return pair2(d);
}
// componentwise product and fused multiply-add
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(bits2(a)), "l"(bits2(b)));
    return pair2(d);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(bits2(a)), "l"(bits2(b)), "l"(bits2(c)));
    return pair2(d);
}
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }
// a times b, given b's quarter turn r = (-b.y, b.x): (a.x b.x - a.y b.y, a.x b.y + a.y b.x),
// the products with a.y rounded first
__device__ __forceinline__ float2 cmul_rot(float2 a, float2 b, float2 r) {
    return fma2(dup2(a.x), b, mul2(dup2(a.y), r));
}
__device__ __forceinline__ float2 turn2(float2 b) { return mul2(swap2(b), make_float2(-1.f, 1.f)); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return cmul_rot(a, b, turn2(b)); }
// a + (-+ i) b (forward -, inverse +) and a - (-+ i) b; the products by 1 are exact
__device__ __forceinline__ float2 add_rot(float2 a, float2 b, bool inv) {
    return fma2(swap2(b), inv ? make_float2(-1.f, 1.f) : make_float2(1.f, -1.f), a);
}
__device__ __forceinline__ float2 sub_rot(float2 a, float2 b, bool inv) { return add_rot(a, b, !inv); }
// multiply by -i (forward) or +i (inverse)
__device__ __forceinline__ float2 rot_q(float2 a, bool inv) {
    return inv ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

}  // namespace ws
