// npw_bits.cuh -- integer format changes between binary32 and binary64 and the reciprocal estimate,
// shared by the mixed-precision and the double-precision arithmetic: none of them occupies the FP64
// pipe (on GB300 a float<->double conversion takes FP64-pipe slots like an FP64 add).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace npw {
namespace fast {

// reciprocal to about one ulp for a normal argument (subnormal results flushed): one instruction,
// where a quotient only needs to be an estimate
__device__ __forceinline__ float rcp_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// widen for a zero or normal x (the common case): the exponent field is rebiased in place.
__device__ __forceinline__ double widen_nz(float x) {
    const uint32_t b = __float_as_uint(x), t = b & 0x7FFFFFFFu;
    const uint32_t hi = t != 0u ? (t >> 3) + (896u << 20) : 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}
// seed_f: a binary64 value whose magnitude lies in [2^-99, 2^99) truncated to binary32
// (relative error below 2^-23), for a reciprocal seed; false outside that range (zero,
// subnormal, huge, infinite or NaN), where the caller divides in double instead.
__device__ __forceinline__ bool seed_f(double v, float* out) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const uint32_t E = (uint32_t)(b >> 52) & 0x7FFu;
    *out = __uint_as_float(((uint32_t)(b >> 29) - (896u << 23)) | ((uint32_t)(b >> 32) & 0x80000000u));
    return E - 924u < 198u;
}

}  // namespace fast
}  // namespace npw
