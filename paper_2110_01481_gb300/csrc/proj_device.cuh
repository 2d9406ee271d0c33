// Device helpers shared by the projectors: loads of 16-bit basis elements, the
// fractional part of a fixed-point position, and floor and fraction of two
// positions in packed FP32 pairs.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ctg_internal.cuh"

namespace {

// Inputs that are Krylov basis vectors may be stored in BF16 or FP16.
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_f(__half v) { return __half2float(v); }

__device__ __forceinline__ float fx_frac(long long U) {
    // top 24 bits of the 40-bit fraction of a 24.40 value, in [0, 1)
    const unsigned f24 = (unsigned)((unsigned long long)U >> (CTG_FX_BITS - 24)) & 0xFFFFFFu;
    return (float)f24 * (1.0f / 16777216.0f);
}

// floor(u) by the round-down magic-number add, for two positions at once in
// packed FP32 pairs: t = u + M rounded down (M = 1.5 * 2^23, so the bits of t
// are those of M plus floor(u), negative ones too, for |u| < 2^22) and f = u -
// (t - M), exactly the scalar sequence per position, with half the instructions.
__device__ __forceinline__ void floor_frac2(float u0, float u1, float &t0, float &t1, float &f0,
                                            float &f1) {
    asm("{\n\t.reg .b64 u, m, t, f;\n\t"
        "mov.b64 u, {%4, %5};\n\t"
        "mov.b64 m, {%6, %6};\n\t"
        "add.rm.f32x2 t, u, m;\n\t"
        "sub.rn.f32x2 f, t, m;\n\t"
        "sub.rn.f32x2 f, u, f;\n\t"
        "mov.b64 {%0, %1}, t;\n\t"
        "mov.b64 {%2, %3}, f;\n\t}"
        : "=f"(t0), "=f"(t1), "=f"(f0), "=f"(f1)
        : "f"(u0), "f"(u1), "f"(12582912.0f));
}

}  // namespace
