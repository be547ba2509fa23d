// What the norm kernels share: reductions and roundings that have to give the same bits in every one of them.
#pragma once
#include "odb_internal.cuh"

namespace odb {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ uint2 pack4_bf16(float a, float b, float c, float d) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b);
    const __nv_bfloat162 hi = __floats2bfloat162_rn(c, d);
    uint2 pk;
    pk.x = *reinterpret_cast<const uint32_t*>(&lo);
    pk.y = *reinterpret_cast<const uint32_t*>(&hi);
    return pk;
}

// x^2 + y^2 + z^2 + w^2 with the roundings spelled out, so that every variant of an RMSNorm kernel gives the same bits
// (a last bit here flips bf16 roundings in every layer behind): SECOND_FIRST starts with y^2, as the few-row kernel does.
template <bool SECOND_FIRST>
__device__ __forceinline__ float squares4(const float4& v) {
    const float t = SECOND_FIRST ? __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y)) : __fmaf_rn(v.y, v.y, __fmul_rn(v.x, v.x));
    return __fmaf_rn(v.w, v.w, __fmaf_rn(v.z, v.z, t));
}

}  // namespace odb
