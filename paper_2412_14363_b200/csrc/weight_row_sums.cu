// Row sums of the weight codes: what asymmetric activations (Eq. 1, second form; Section 5.1) add to the epilogue.
// (The asymmetric quantizer is a form of the row quantizer in quantize.cu.)
#include "internal.h"

namespace resq {
namespace {

// Row sums of the weight codes of one output channel: one warp per channel.
__global__ void __launch_bounds__(256)
weight_row_sums_kernel(const int8_t* __restrict__ w8, const uint8_t* __restrict__ w4, int N, int r, int row4,
                       int32_t* __restrict__ wsum8, int32_t* __restrict__ wsum4) {
    const int n = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (n >= N) return;
    int a8 = 0, a4 = 0;
    const uint32_t* p8 = reinterpret_cast<const uint32_t*>(w8 + static_cast<size_t>(n) * r);
    for (int i = lane; i < (r >> 2); i += 32) a8 = __dp4a(static_cast<int>(p8[i]), 0x01010101, a8);
    const uint32_t* p4 = reinterpret_cast<const uint32_t*>(w4 + static_cast<size_t>(n) * row4);
    for (int i = lane; i < (row4 >> 2); i += 32) {
        const uint32_t w = p4[i];
        // both nibble sets as int8 lanes times 16; the sum is divided by 16 at the end (exact)
        a4 = __dp4a(static_cast<int>((w << 4) & 0xF0F0F0F0u), 0x01010101, a4);
        a4 = __dp4a(static_cast<int>(w & 0xF0F0F0F0u), 0x01010101, a4);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a8 += __shfl_xor_sync(0xffffffffu, a8, o);
        a4 += __shfl_xor_sync(0xffffffffu, a4, o);
    }
    if (lane == 0) {
        wsum8[n] = a8;
        wsum4[n] = a4 >> 4;
    }
}

}  // namespace

cudaError_t launch_weight_row_sums(const int8_t* w8, const uint8_t* w4, int N, int K, int r, int32_t* wsum8,
                                   int32_t* wsum4, cudaStream_t st) {
    count_launch();
    weight_row_sums_kernel<<<(N + 7) / 8, 256, 0, st>>>(w8, w4, N, r, (K - r) / 2, wsum8, wsum4);
    return cudaGetLastError();
}

}  // namespace resq
