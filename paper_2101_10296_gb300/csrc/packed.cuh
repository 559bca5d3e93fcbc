// Packed FP32 pairs: two independent FP32 values in one 64-bit register, on
// which the FP32x2 instructions work.  Their rounding is that of the scalar
// instructions; negating a value, exchanging the halves and using one half for
// both are operand modifiers, so lo/hi/neg/swap/splat of existing pairs cost no
// instruction.  The pair is a 64-bit integer to the compiler: kept as float2, a
// chain of packed operations was taken apart into scalars and moves (3.6
// instructions per operation in a sequence of butterflies, 1.0 in this form).
#pragma once

#include <cstdint>

namespace qaoa {

struct P2 {
    unsigned long long v;
};

__device__ __forceinline__ P2 p2(float lo, float hi) {
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 halves(P2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ float lo(P2 a) { return halves(a).x; }
__device__ __forceinline__ float hi(P2 a) { return halves(a).y; }
__device__ __forceinline__ P2 splat(float a) { return p2(a, a); }
__device__ __forceinline__ P2 neg(P2 a) {
    const float2 h = halves(a);
    return p2(-h.x, -h.y);
}
__device__ __forceinline__ P2 swap(P2 a) {
    const float2 h = halves(a);
    return p2(h.y, h.x);
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c) {
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ P2 mul2(P2 a, P2 b) {
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 add2(P2 a, P2 b) {
    P2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// Two complex numbers: real parts r, imaginary parts i.
struct C2 {
    P2 r, i;
};

// a b, a conj(b) and Im(conj(a) b); which product is rounded by itself follows
// what the compiler made of cmul, cmulc and imconj (dev_math.cuh) in the scalar
// kernels: the imaginary part of a product had a.i b.r in the FMA in the
// register kernel (cmul) and a.r b.i in the large-state kernels (cmul_ri)
__device__ __forceinline__ C2 cmul(const C2 &a, const C2 &b) {
    return C2{fma2(a.r, b.r, neg(mul2(a.i, b.i))), fma2(a.i, b.r, mul2(a.r, b.i))};
}
__device__ __forceinline__ C2 cmul_ri(const C2 &a, const C2 &b) {
    return C2{fma2(a.r, b.r, neg(mul2(a.i, b.i))), fma2(a.r, b.i, mul2(a.i, b.r))};
}
__device__ __forceinline__ C2 cmulc(const C2 &a, const C2 &b) {
    return C2{fma2(a.r, b.r, mul2(a.i, b.i)), fma2(a.i, b.r, neg(mul2(a.r, b.i)))};
}
__device__ __forceinline__ P2 imconj(const C2 &a, const C2 &b) { return fma2(a.r, b.i, neg(mul2(a.i, b.r))); }
// d += Im(conj(a) b), the two products added one after the other
__device__ __forceinline__ void acc_imconj(P2 &d, const C2 &a, const C2 &b) {
    d = fma2(a.r, b.i, d);
    d = fma2(neg(a.i), b.r, d);
}
__device__ __forceinline__ C2 neg(const C2 &a) { return C2{neg(a.r), neg(a.i)}; }
__device__ __forceinline__ C2 swap(const C2 &a) { return C2{swap(a.r), swap(a.i)}; }
// u - i tau v
__device__ __forceinline__ C2 bfly(const C2 &u, const C2 &v, float tau) {
    return C2{fma2(splat(tau), v.i, u.r), fma2(splat(-tau), v.r, u.i)};
}
// (I - i tau X) on qubit 0 (pairs (0,1), (2,3)), then on qubit 1 ((0,2), (1,3))
__device__ __forceinline__ void mix01(C2 (&x)[4], float tau) {
    C2 a = x[0], b = x[1];
    x[0] = bfly(a, b, tau);
    x[1] = bfly(b, a, tau);
    a = x[2];
    b = x[3];
    x[2] = bfly(a, b, tau);
    x[3] = bfly(b, a, tau);
    a = x[0];
    b = x[2];
    x[0] = bfly(a, b, tau);
    x[2] = bfly(b, a, tau);
    a = x[1];
    b = x[3];
    x[1] = bfly(a, b, tau);
    x[3] = bfly(b, a, tau);
}
__device__ __forceinline__ P2 shfl_xor(P2 a, int m) {
    const float2 h = halves(a);
    return p2(__shfl_xor_sync(0xffffffffu, h.x, m), __shfl_xor_sync(0xffffffffu, h.y, m));
}
__device__ __forceinline__ C2 shfl_xor(const C2 &a, int m) { return C2{shfl_xor(a.r, m), shfl_xor(a.i, m)}; }

// Four bytes at a shared-memory address.
__device__ __forceinline__ float lds1(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(addr));
    return v;
}
// Keeps what is derived from v from being carried in registers from one use to
// the next (recomputing it is one instruction).
__device__ __forceinline__ void opaque(uint32_t &v) { asm volatile("" : "+r"(v)); }

}  // namespace qaoa
