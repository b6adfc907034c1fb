// Rounding of samples to the tensor cores' operand formats, shared by the quantiser
// (pnce_quant.cu) and by the transform kernel that rounds in registers (pnce_mst.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "pnce_internal.h"

namespace pnce {

template <int DT> struct Fmt;
template <> struct Fmt<PNCE_FP16> { static constexpr int target = 15; using T = uint16_t; };
template <> struct Fmt<PNCE_BF16> { static constexpr int target = 0; using T = uint16_t; };
template <> struct Fmt<PNCE_TF32> { static constexpr int target = 0; using T = uint32_t; };
template <> struct Fmt<PNCE_FP8E4M3> { static constexpr int target = 8; using T = uint8_t; };

__device__ __forceinline__ uint16_t to_f16(float x) {
    return __half_as_ushort(__float2half_rn(x));
}
__device__ __forceinline__ uint16_t to_bf16(float x) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}
__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
// two e4m3 codes (lo from a, hi from b), round to nearest even, saturate to +-448
__device__ __forceinline__ uint16_t to_e4m3x2(float a, float b) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %2, %1;" : "=h"(r) : "f"(a), "f"(b));
    return r;
}

// s of the scale 2^s for an antenna whose peak component is m: 2^s m in [2^(target-1),
// 2^target), s clamped to [-100, 100]; 0 for formats without a target (target 0), for an
// all-zero antenna and for a peak that is not finite
__device__ __forceinline__ int scale_exponent(int target, float m) {
    if (target == 0 || !(m > 0.f) || !isfinite(m)) return 0;
    int ex;
    frexpf(m, &ex);                          // m = mant * 2^ex, mant in [0.5, 1)
    const int se = target - ex;
    return se < -100 ? -100 : (se > 100 ? 100 : se);
}

// one complex sample rounded to the format and back
template <int DT>
__device__ __forceinline__ float2 round_through(float2 v) {
    if constexpr (DT == PNCE_FP16)
        return __half22float2(__floats2half2_rn(v.x, v.y));
    else if constexpr (DT == PNCE_BF16)
        return __bfloat1622float2(__floats2bfloat162_rn(v.x, v.y));
    else if constexpr (DT == PNCE_TF32)
        return make_float2(__uint_as_float(to_tf32(v.x)), __uint_as_float(to_tf32(v.y)));
    else
        return __half22float2(__half2(
            __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)to_e4m3x2(v.x, v.y), __NV_E4M3)));
}

// one complex sample from its stored codes
template <int DT>
__device__ __forceinline__ float2 decode(typename Fmt<DT>::T re, typename Fmt<DT>::T im) {
    if constexpr (DT == PNCE_FP16)
        return make_float2(__half2float(__ushort_as_half(re)), __half2float(__ushort_as_half(im)));
    else if constexpr (DT == PNCE_BF16)
        return make_float2(__uint_as_float((uint32_t)re << 16), __uint_as_float((uint32_t)im << 16));
    else if constexpr (DT == PNCE_TF32)
        return make_float2(__uint_as_float(re), __uint_as_float(im));
    else
        return __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(
            (__nv_fp8x2_storage_t)(re | (uint16_t)im << 8), __NV_E4M3)));
}

}  // namespace pnce
