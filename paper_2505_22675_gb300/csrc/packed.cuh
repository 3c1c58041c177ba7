// Packed two-lane FP32 arithmetic (sm_100 and later).
#pragma once

namespace bg {

using u64 = unsigned long long;

// Packed two-lane FP32 arithmetic (one instruction for two IEEE single
// operations, each lane rounded as its scalar counterpart): two floats in one
// 64-bit register pair.
__device__ __forceinline__ unsigned long long pk2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(unsigned long long p, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ u64 dup2(float a) { return pk2(a, a); }
__device__ __forceinline__ float lo2(u64 p) {
    float a, b;
    upk2(p, a, b);
    return a;
}
__device__ __forceinline__ float hi2(u64 p) {
    float a, b;
    upk2(p, a, b);
    return b;
}
__device__ __forceinline__ float lane2(u64 p, int i) { return i ? hi2(p) : lo2(p); }

}  // namespace bg
