// Pairs of fp32 values handled by the packed instructions of sm_100 (add / sub / mul / fma .f32x2).
//
// A packed instruction does two fp32 operations with the rounding of the scalar ones, from one
// issue slot.  The fp32 pipe itself is no faster (measured on B200: 128 lane-operations per clock
// and SM either way), so the packed form pays where a kernel is held by instruction issue: the
// transforms of n = 64 and 128 on pairs of columns, and the FP32 contraction, which keeps its multiply-adds at half of the issue
// slots and has the other half for loads and address arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fc {

struct F2 {
    unsigned long long b;       // low half: first value
};

__device__ __forceinline__ F2 f2_pack(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.b) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.b));
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a) {
    float lo, hi;
    f2_unpack(a, lo, hi);
    return f2_pack(-lo, -hi);
}
// a * b + c, element by element
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.b) : "l"(a.b), "l"(b.b), "l"(c.b));
    return r;
}

}  // namespace fc
