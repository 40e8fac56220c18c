// Cache codes as 16-bit operands of a tensor-core product, for the attention kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>

namespace resq {

// Eight codes as halves minus their centre: a word of nibbles (order 0 4 1 5 2 6 3 7), or eight bytes.
__device__ __forceinline__ uint32_t centred(uint32_t biased, uint16_t bias) {
    const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&biased), __half2half2(__ushort_as_half(bias)));
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint4 nibbles_centred(uint32_t w) {
    uint32_t v[4];
    const __half2 sixteenth = __half2half2(__ushort_as_half(0x2C00)), bias = __half2half2(__ushort_as_half(0xD480));  // 1/16, -(64 + 8)
#pragma unroll
    for (int m = 0; m < 4; m += 2, w >>= 8) {
        v[m] = centred((w & 0x000F000Fu) | 0x64006400u, 0x6408);  // 1024 + 8
        const uint32_t high = (w & 0x00F000F0u) | 0x64006400u;    // 1024 + 16 code: no shift, exact by one multiply-add
        const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&high), sixteenth, bias);
        v[m + 1] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(v[0], v[1], v[2], v[3]);
}
// Two bytes of nibbles, one in each half of a word, as halves minus 8: low nibbles, high nibbles.
__device__ __forceinline__ uint2 byte_pair_centred(uint32_t w) {
    const __half2 sixteenth = __half2half2(__ushort_as_half(0x2C00)), bias = __half2half2(__ushort_as_half(0xD480));  // 1/16, -(64 + 8)
    const uint32_t high = (w & 0x00F000F0u) | 0x64006400u;
    const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&high), sixteenth, bias);
    return make_uint2(centred((w & 0x000F000Fu) | 0x64006400u, 0x6408), *reinterpret_cast<const uint32_t*>(&h));
}
__device__ __forceinline__ uint4 bytes_centred(uint2 w) {
    const uint16_t b = 0x6480;  // 1024 + 128
    return make_uint4(centred(__byte_perm(w.x, 0x64646464u, 0x4140), b), centred(__byte_perm(w.x, 0x64646464u, 0x4342), b),
                      centred(__byte_perm(w.y, 0x64646464u, 0x4140), b), centred(__byte_perm(w.y, 0x64646464u, 0x4342), b));
}

// The same as bf16.  bf16 holds 128 + (0..127) exactly: the
// bytes' upper bits move the centre.
__device__ __forceinline__ uint32_t minus_bf16(uint32_t v, uint32_t centre) {
    const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&v), *reinterpret_cast<const __nv_bfloat162*>(&centre));
    return *reinterpret_cast<const uint32_t*>(&d);
}
// The nibbles in bits 0-3 of a word's halves, or their bytes.
__device__ __forceinline__ uint32_t nibble_pair_bf16(uint32_t w) {
    return minus_bf16((w & 0x000F000Fu) | 0x43004300u, 0x43084308u);  // 128 + 8
}
__device__ __forceinline__ uint32_t byte_pair_bf16(uint32_t w) {  // code < 128: (128 + code) - 256, else (128 + code - 128) - 128
    return minus_bf16((w & 0x007F007Fu) | 0x43004300u, (~w & 0x00800080u) | 0x43004300u);
}

__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

}  // namespace resq
