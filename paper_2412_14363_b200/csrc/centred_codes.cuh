// Cache codes as 16-bit operands of a tensor-core product, for the attention kernels.
#pragma once
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
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = centred(((w >> (4 * m)) & 0x000F000Fu) | 0x64006400u, 0x6408);  // 1024 + 8
    return make_uint4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ uint4 bytes_centred(uint2 w) {
    const uint16_t b = 0x6480;  // 1024 + 128
    return make_uint4(centred(__byte_perm(w.x, 0x64646464u, 0x4140), b), centred(__byte_perm(w.x, 0x64646464u, 0x4342), b),
                      centred(__byte_perm(w.y, 0x64646464u, 0x4140), b), centred(__byte_perm(w.y, 0x64646464u, 0x4342), b));
}

__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

}  // namespace resq
