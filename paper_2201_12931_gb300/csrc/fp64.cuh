// FP64 helpers in few FP64 instructions.  FP64 instructions and FP64 <-> FP32
// conversions run at 2 lanes per clock and SM on this part, 1/64 of the
// integer and FP32 rates, so conversions go through integer words and the
// iterations start from an FP32 seed.
#pragma once

#include <cuda_runtime.h>

namespace topo {

// FP32 value of a non-negative double, truncated (relative error below 2^-23;
// 0 below FP32's normal range, infinity above)
__device__ __forceinline__ float trunc_f32(double v) {
    const int hi = __double2hiint(v);
    if (hi < (897 << 20)) return 0.0f;
    if (hi >= (1151 << 20)) return __int_as_float(0x7f800000);
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(v), (unsigned)hi, 3) - 0xc0000000u);
}
// a positive normal FP32 value, exactly
__device__ __forceinline__ double widen_f32(float v) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}
// The conversions (float)v and (double)v bit for bit on integer words; values
// outside FP32's normal range (other than zeros) take the instructions
__device__ __forceinline__ float narrow(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    if (((hi >> 20) & 0x7ffu) - 897u < 254u) {
        unsigned b = (__funnelshift_l(lo, hi & 0x7fffffffu, 3) - 0xc0000000u);   // truncated magnitude
        b += (lo << 3) + (b & 1u) > 0x80000000u ? 1u : 0u;                       // to nearest, ties to even
        return __uint_as_float(b | (hi & 0x80000000u));
    }
    if (((hi & 0x7fffffffu) | lo) == 0u) return __uint_as_float(hi);
    return (float)v;
}
__device__ __forceinline__ double widen(float v) {
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    if ((m >> 23) - 1u < 254u) return __hiloint2double((int)(((m >> 3) + (896u << 20)) | (b & 0x80000000u)), (int)(b << 29));
    if (m == 0u) return __hiloint2double((int)b, 0);
    return (double)v;
}
// the FP32 reciprocal y0 of b, 2^-100 <= b < 2^100: relative error below 2^-21
__device__ __forceinline__ double recip_seed(double b) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(trunc_f32(b)));
    return widen_f32(r);
}
__device__ __forceinline__ bool seed_range(double b) {
    return (unsigned)((__double2hiint(b) >> 20) - (1023 - 100)) < 200u;
}

}  // namespace topo
