// Per-row split quantization (Eq. 1 applied per segment, Eq. 2 / Eq. 3): HBM-bound.
//
// One CTA per row.  Each thread owns 8-element chunks (one 128-bit bf16 load, or two for fp32),
// keeps up to kMaxChunks of them in registers so the row is read from memory once, reduces the two
// per-segment absmax values with warp shuffles + one shared-memory step, then emits int8 codes
// (8-byte stores) and packed int4 codes (4-byte stores).
#include <algorithm>
#include <cmath>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "internal.h"
#include "packed_fp32.cuh"
#include "ptx.cuh"
#include "row_codes.cuh"

namespace resq {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxChunks = 8;  // register-cached chunks per thread: rows up to 8*8*256 = 16384 wide

// code = clamp(round-half-even(x / s)); IEEE division, no reciprocal.
__device__ __forceinline__ int quant1(float x, float s, float lo, float hi) {
    float q = rintf(__fdiv_rn(x, s));
    q = fminf(fmaxf(q, lo), hi);
    return static_cast<int>(q);
}

template <bool F32>
__device__ __forceinline__ void store_chunk(const Chunk<F32>& ch, int col, int r, float s8, float s4, int8_t* q8row,
                                            uint8_t* q4row, int8_t* q4e_row) {
    if (col < r) {
        uint32_t w0 = 0, w1 = 0;
        if (s8 > 0.f) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                w0 |= (static_cast<uint32_t>(quant1(ch.get(i), s8, -128.f, 127.f)) & 0xFFu) << (8 * i);
                w1 |= (static_cast<uint32_t>(quant1(ch.get(4 + i), s8, -128.f, 127.f)) & 0xFFu) << (8 * i);
            }
        }
        *reinterpret_cast<uint2*>(q8row + col) = make_uint2(w0, w1);
    } else {
        const int j = col - r;
        uint32_t packed = 0, w0 = 0, w1 = 0;
        if (s4 > 0.f) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                uint32_t q = static_cast<uint32_t>(quant1(ch.get(i), s4, -8.f, 7.f));
                packed |= (q & 0xFu) << (4 * i);
                if (i < 4) w0 |= (q & 0xFFu) << (8 * i);
                else w1 |= (q & 0xFFu) << (8 * (i - 4));
            }
        }
        if (q4row) *reinterpret_cast<uint32_t*>(q4row + (j >> 1)) = packed;
        if (q4e_row) *reinterpret_cast<uint2*>(q4e_row + j) = make_uint2(w0, w1);
    }
}

template <bool F32>
__global__ void __launch_bounds__(kThreads)
split_quantize_kernel(const void* __restrict__ in, size_t in_row_bytes, size_t rows, int K, int r,
                      int8_t* __restrict__ q8, uint8_t* __restrict__ q4, void* __restrict__ s8_out,
                      void* __restrict__ s4_out, int scale_fp16, int8_t* __restrict__ q4e) {
    __shared__ float red[2][kThreads / 32];
    const int nchunks = K >> 3;
    const int K4 = K - r;
    for (size_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const char* rp = reinterpret_cast<const char*>(in) + row * in_row_bytes;
        Chunk<F32> cache[kMaxChunks];
        float a8 = 0.f, a4 = 0.f;
#pragma unroll
        for (int i = 0; i < kMaxChunks; ++i) {
            const int c = threadIdx.x + i * kThreads;
            if (c < nchunks) {
                cache[i] = load_chunk<F32>(rp, c);
                const float m = chunk_absmax(cache[i]);
                if (c * 8 < r) a8 = fmaxf(a8, m);
                else a4 = fmaxf(a4, m);
            }
        }
        for (int c = threadIdx.x + kMaxChunks * kThreads; c < nchunks; c += kThreads) {  // rows wider than the cache
            const float m = chunk_absmax(load_chunk<F32>(rp, c));
            if (c * 8 < r) a8 = fmaxf(a8, m);
            else a4 = fmaxf(a4, m);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a8 = fmaxf(a8, __shfl_xor_sync(0xffffffffu, a8, o));
            a4 = fmaxf(a4, __shfl_xor_sync(0xffffffffu, a4, o));
        }
        __syncthreads();  // previous row's readers of `red` are done
        if ((threadIdx.x & 31) == 0) {
            red[0][threadIdx.x >> 5] = a8;
            red[1][threadIdx.x >> 5] = a4;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            a8 = fmaxf(a8, red[0][w]);
            a4 = fmaxf(a4, red[1][w]);
        }
        float s8 = __fdiv_rn(a8, 127.f), s4 = __fdiv_rn(a4, 7.f);
        if (scale_fp16) {
            s8 = __half2float(__float2half_rn(s8));
            s4 = __half2float(__float2half_rn(s4));
        }
        if (threadIdx.x == 0) {
            if (scale_fp16) {
                reinterpret_cast<__half*>(s8_out)[row] = __float2half_rn(s8);
                reinterpret_cast<__half*>(s4_out)[row] = __float2half_rn(s4);
            } else {
                reinterpret_cast<float*>(s8_out)[row] = s8;
                reinterpret_cast<float*>(s4_out)[row] = s4;
            }
        }
        int8_t* q8row = q8 + row * static_cast<size_t>(r);
        uint8_t* q4row = q4 ? q4 + row * static_cast<size_t>(K4 >> 1) : nullptr;
        int8_t* q4e_row = q4e ? q4e + row * static_cast<size_t>(K4) : nullptr;
#pragma unroll
        for (int i = 0; i < kMaxChunks; ++i) {
            const int c = threadIdx.x + i * kThreads;
            if (c < nchunks) store_chunk(cache[i], c * 8, r, s8, s4, q8row, q4row, q4e_row);
        }
        for (int c = threadIdx.x + kMaxChunks * kThreads; c < nchunks; c += kThreads)
            store_chunk(load_chunk<F32>(rp, c), c * 8, r, s8, s4, q8row, q4row, q4e_row);
    }
}

// ---------------------------------------------------------------------------------------------
// Fast path (fp32 scales).  Same codes as the kernel above, bit for bit, at a fraction of its
// instructions and with the row staged in shared memory instead of registers.
//
// Staging.  A CTA takes a group of 1, 2, 4 or 8 consecutive rows (about 32 KB); one thread issues a
// bulk copy (cp.async.bulk, completion counted on an mbarrier) per row, so the whole group is in
// flight at once and several CTAs per SM keep HBM busy while others compute.  Each row is then read
// twice from shared memory: once for the two absmax values, once for the codes.
//
// Rounding: row_codes.cuh.
constexpr int kFastGroupBytes = 32 * 1024;
constexpr int kFastMaxRowBytes = 200 * 1024;

template <bool F32>
__device__ __forceinline__ Chunk<F32> lds_chunk(const uint8_t* row, int c) {
    Chunk<F32> o;
    if constexpr (F32) {
        const uint4* p = reinterpret_cast<const uint4*>(row) + 2 * c;
        const uint4 a = p[0], b = p[1];
        o.w[0] = a.x; o.w[1] = a.y; o.w[2] = a.z; o.w[3] = a.w;
        o.w[4] = b.x; o.w[5] = b.y; o.w[6] = b.z; o.w[7] = b.w;
    } else {
        const uint4 u = reinterpret_cast<const uint4*>(row)[c];
        o.w[0] = u.x; o.w[1] = u.y; o.w[2] = u.z; o.w[3] = u.w;
    }
    return o;
}

// ASYM: asymmetric codes (unsigned), with the zero-points z8_out / z4_out; else symmetric ones.
template <bool F32, bool ASYM>
__global__ void __launch_bounds__(kThreads)
split_quantize_fast_kernel(const void* in, size_t in_row_bytes, size_t rows, int K, int r,
                           int rows_per_cta, int nstages, int8_t* __restrict__ q8, uint8_t* __restrict__ q4,
                           float* __restrict__ s8_out, float* __restrict__ s4_out, float* __restrict__ z8_out,
                           float* __restrict__ z4_out, int8_t* __restrict__ q4e, int* __restrict__ status) {
    extern __shared__ __align__(128) uint8_t stage[];
    __shared__ uint64_t bar[2];
    __shared__ int abort_flag;
    __shared__ float red[ASYM ? 4 : 2][kThreads / 32];
    // Enqueued with programmatic stream serialization, this grid may have been scheduled before its input was complete:
    // wait for the preceding grid.  Only then may the kernel enqueued behind this one start its own prologue, so that a
    // dependent that is running finds everything enqueued before this grid complete (the product that follows in
    // resq_linear streams its weights at once; it still waits for this grid before it reads the codes).
    griddep_wait();
    griddep_launch_dependents();
    const uint32_t row_bytes = static_cast<uint32_t>(K) * (F32 ? 4u : 2u);
    const size_t group_bytes = static_cast<size_t>(row_bytes) * rows_per_cta;
    const size_t groups = (rows + rows_per_cta - 1) / rows_per_cta;
    auto rows_of = [&](size_t g) {
        const size_t row0 = g * rows_per_cta;
        return static_cast<int>(rows - row0 < static_cast<size_t>(rows_per_cta) ? rows - row0 : rows_per_cta);
    };
    auto issue = [&](size_t g, int buf) {  // one thread: the rows of group g, one bulk copy each
        const int n = rows_of(g);
        mbar_arrive_expect_tx(&bar[buf], row_bytes * static_cast<uint32_t>(n));
        for (int i = 0; i < n; ++i)
            bulk_load(stage + buf * group_bytes + static_cast<size_t>(i) * row_bytes,
                      reinterpret_cast<const char*>(in) + (g * rows_per_cta + i) * in_row_bytes, row_bytes, &bar[buf]);
    };
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
        if (blockIdx.x < groups) issue(blockIdx.x, 0);
    }
    __syncthreads();

    const int tpr = kThreads / rows_per_cta;  // threads per row, a multiple of 32
    const int grp = threadIdx.x / tpr, j = threadIdx.x - grp * tpr;
    const int nchunks = K >> 3, rchunks = r >> 3;
    const int K4 = K - r;

    // The CTA walks its groups (grid-stride); with two stages the rows of the next group are in flight while this
    // one is quantized, so the copy engine never waits for the arithmetic of the same CTA.
    int it = 0;
    for (size_t g = blockIdx.x; g < groups; g += gridDim.x, ++it) {
        const int buf = nstages == 2 ? (it & 1) : 0;
        const uint32_t parity = nstages == 2 ? (it >> 1) & 1 : it & 1;
        const bool more = g + gridDim.x < groups;
        if (nstages == 2 && more && threadIdx.x == 0) issue(g + gridDim.x, buf ^ 1);
        const bool landed = mbar_wait(&bar[buf], parity, &abort_flag, status);
        if (__syncthreads_or(!landed)) {
            // The copy did not land in time: report it and leave the outputs of the remaining groups unwritten.
            if (threadIdx.x == 0) {
                atomicOr(status, kStatusBitTimeout);
                if (nstages == 2 && more) {  // the copies of the next group are still this CTA's to wait for
                    int keep_waiting = 0;
                    (void)mbar_wait(&bar[buf ^ 1], ((it + 1) >> 1) & 1, &keep_waiting, status);
                }
            }
            return;
        }
        const int nrows = rows_of(g);
        const size_t row0 = g * rows_per_cta;
        const bool live = grp < nrows;
        const uint8_t* srow = stage + buf * group_bytes + static_cast<size_t>(live ? grp : 0) * row_bytes;

        // ---- pass 1: the largest magnitude of the two segments (a8, a4), or their ranges ([lo8, a8], [lo4, a4])
        constexpr float kBig = 3.402823466e38f;
        float a8 = ASYM ? -kBig : 0.f, a4 = a8, lo8 = kBig, lo4 = kBig;
        if constexpr (ASYM) {
            if (live) {
                if constexpr (F32) {
                    auto acc = [](const Chunk<F32>& ch, float& lo, float& hi) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) { lo = fminf(lo, ch.get(i)); hi = fmaxf(hi, ch.get(i)); }
                    };
                    for (int c = j; c < rchunks; c += tpr) acc(lds_chunk<F32>(srow, c), lo8, a8);
                    for (int c = rchunks + j; c < nchunks; c += tpr) acc(lds_chunk<F32>(srow, c), lo4, a4);
                } else {
                    // bf16 rows: extrema kept as packed pairs until the end (two operations per pair)
                    const uint4* v = reinterpret_cast<const uint4*>(srow);
                    auto acc = [](const uint4 u, __nv_bfloat162& lo, __nv_bfloat162& hi) {
                        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
                            lo = __hmin2(lo, x);
                            hi = __hmax2(hi, x);
                        }
                    };
                    const uint32_t big = 0x7F7F7F7Fu, small = 0xFF7FFF7Fu;  // the largest finite bf16, and its negative
                    __nv_bfloat162 l8 = *reinterpret_cast<const __nv_bfloat162*>(&big), h8 = *reinterpret_cast<const __nv_bfloat162*>(&small);
                    __nv_bfloat162 l4 = l8, h4 = h8;
                    for (int c = j; c < rchunks; c += tpr) acc(v[c], l8, h8);
#pragma unroll 2
                    for (int c = rchunks + j; c < nchunks; c += tpr) acc(v[c], l4, h4);
                    lo8 = fminf(__low2float(l8), __high2float(l8)); a8 = fmaxf(__low2float(h8), __high2float(h8));
                    lo4 = fminf(__low2float(l4), __high2float(l4)); a4 = fmaxf(__low2float(h4), __high2float(h4));
                }
            }
        } else {
            if (live) {
                if constexpr (F32) {
                    for (int c = j; c < rchunks; c += tpr) a8 = fmaxf(a8, chunk_absmax(lds_chunk<F32>(srow, c)));
                    float m0 = 0.f, m1 = 0.f;  // two chains: the INT4 segment is 7/8 of the row
                    int c = rchunks + j;
                    for (; c + tpr < nchunks; c += 2 * tpr) {
                        m0 = fmaxf(m0, chunk_absmax(lds_chunk<F32>(srow, c)));
                        m1 = fmaxf(m1, chunk_absmax(lds_chunk<F32>(srow, c + tpr)));
                    }
                    if (c < nchunks) m0 = fmaxf(m0, chunk_absmax(lds_chunk<F32>(srow, c)));
                    a4 = fmaxf(m0, m1);
                } else {
                    // bf16 rows: sign bits cleared, maxima kept as packed pairs until the end (two operations per pair)
                    const uint4* v = reinterpret_cast<const uint4*>(srow);
                    uint32_t m8 = 0, m4a = 0, m4b = 0;
                    auto acc = [](uint32_t& m, const uint4 u) {
                        const uint32_t w[4] = {u.x & 0x7FFF7FFFu, u.y & 0x7FFF7FFFu, u.z & 0x7FFF7FFFu, u.w & 0x7FFF7FFFu};
                        __nv_bfloat162 mm = *reinterpret_cast<const __nv_bfloat162*>(&m);
#pragma unroll
                        for (int i = 0; i < 4; ++i) mm = __hmax2(mm, *reinterpret_cast<const __nv_bfloat162*>(&w[i]));
                        m = *reinterpret_cast<const uint32_t*>(&mm);
                    };
                    for (int c = j; c < rchunks; c += tpr) acc(m8, v[c]);
                    int c = rchunks + j;
#pragma unroll 2
                    for (; c + tpr < nchunks; c += 2 * tpr) {
                        acc(m4a, v[c]);
                        acc(m4b, v[c + tpr]);
                    }
                    if (c < nchunks) acc(m4a, v[c]);
                    auto unpack = [](uint32_t m) { return fmaxf(__uint_as_float(m << 16), __uint_as_float(m & 0xFFFF0000u)); };
                    a8 = unpack(m8);
                    a4 = fmaxf(unpack(m4a), unpack(m4b));
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a8 = fmaxf(a8, __shfl_xor_sync(0xffffffffu, a8, o));
            a4 = fmaxf(a4, __shfl_xor_sync(0xffffffffu, a4, o));
            if constexpr (ASYM) {
                lo8 = fminf(lo8, __shfl_xor_sync(0xffffffffu, lo8, o));
                lo4 = fminf(lo4, __shfl_xor_sync(0xffffffffu, lo4, o));
            }
        }
        if (tpr > 32) {
            const int warp = threadIdx.x >> 5, wpr = tpr >> 5;
            if ((threadIdx.x & 31) == 0) {
                red[0][warp] = a8;
                red[1][warp] = a4;
                if constexpr (ASYM) {
                    red[2][warp] = lo8;
                    red[3][warp] = lo4;
                }
            }
            __syncthreads();
            for (int w = 0; w < wpr; ++w) {
                a8 = fmaxf(a8, red[0][grp * wpr + w]);
                a4 = fmaxf(a4, red[1][grp * wpr + w]);
                if constexpr (ASYM) {
                    lo8 = fminf(lo8, red[2][grp * wpr + w]);
                    lo4 = fminf(lo4, red[3][grp * wpr + w]);
                }
            }
        }
        if (live) {
            const size_t row = row0 + grp;
            if (ASYM && rchunks == 0) lo8 = a8 = 0.f;  // uniform 4-bit layer: the empty INT8 segment has s = 0, z = 0
            const float s8 = ASYM ? __fdiv_rn(__fsub_rn(a8, lo8), 255.f) : __fdiv_rn(a8, 127.f);
            const float s4 = ASYM ? __fdiv_rn(__fsub_rn(a4, lo4), 15.f) : __fdiv_rn(a4, 7.f);
            const ScaleInv i8(s8), i4(s4);
            const float inv8 = i8.inv, inv4 = i4.inv;
            const bool exact8 = i8.exact, exact4 = i4.exact;
            if (j == 0) {
                s8_out[row] = s8;
                s4_out[row] = s4;
                if constexpr (ASYM) {
                    z8_out[row] = lo8;
                    z4_out[row] = lo4;
                }
            }
            auto codes = [&](const Chunk<F32>& ch, float z, float s, float inv, bool exact, float qmax, uint32_t (&t)[8]) {
                if constexpr (ASYM) fast_codes_asym(ch, z, s, inv, exact, qmax, t);
                else fast_codes(ch, s, inv, exact, t);
            };
            int8_t* q8row = q8 + row * static_cast<size_t>(r);
            uint8_t* q4row = q4 ? q4 + row * static_cast<size_t>(K4 >> 1) : nullptr;
            int8_t* q4e_row = q4e ? q4e + row * static_cast<size_t>(K4) : nullptr;

            for (int c = j; c < rchunks; c += tpr) {
                uint32_t t[8];
                if (s8 > 0.f) codes(lds_chunk<F32>(srow, c), lo8, s8, inv8, exact8, 255.f, t);
                else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) t[k] = 0;
                }
                *reinterpret_cast<uint2*>(q8row + c * 8) =
                    make_uint2(pack_low_bytes(t[0], t[1], t[2], t[3]), pack_low_bytes(t[4], t[5], t[6], t[7]));
            }
#pragma unroll 2
            for (int c = rchunks + j; c < nchunks; c += tpr) {
                uint32_t t[8];
                if (s4 > 0.f) codes(lds_chunk<F32>(srow, c), lo4, s4, inv4, exact4, 15.f, t);
                else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) t[k] = 0;
                }
                const int jj = (c - rchunks) * 8;
                const uint32_t lo = pack_low_bytes(t[0], t[1], t[2], t[3]), hi = pack_low_bytes(t[4], t[5], t[6], t[7]);
                if (q4e_row) *reinterpret_cast<uint2*>(q4e_row + jj) = make_uint2(lo, hi);
                if (q4row) {
                    // two's-complement nibbles of the eight bytes: byte pairs (b0 | b1 << 4) sit in bytes 0 and 2 of
                    // x | x >> 4 once the high nibbles are cleared
                    const uint32_t xl = lo & 0x0F0F0F0Fu, xh = hi & 0x0F0F0F0Fu;
                    *reinterpret_cast<uint32_t*>(q4row + (jj >> 1)) = __byte_perm(xl | (xl >> 4), xh | (xh >> 4), 0x6420);
                }
            }
        }
        __syncthreads();  // every thread is done with this stage (and with `red`) before it is refilled
        if (nstages == 1 && more && threadIdx.x == 0) issue(g + gridDim.x, 0);
    }
}

template <bool UNSIGNED>
__global__ void unpack_int4_kernel(const uint8_t* __restrict__ packed, int8_t* __restrict__ out, size_t nwords) {
    // one 32-bit packed word (8 codes) per thread -> 8 bytes
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < nwords;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const uint32_t w = reinterpret_cast<const uint32_t*>(packed)[i];
        uint32_t o[2] = {0, 0};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            int v = static_cast<int>((w >> (4 * k)) & 0xFu);
            if (!UNSIGNED) v = (v ^ 8) - 8;  // sign-extend the nibble
            o[k >> 2] |= (static_cast<uint32_t>(v) & 0xFFu) << (8 * (k & 3));
        }
        reinterpret_cast<uint2*>(out)[i] = make_uint2(o[0], o[1]);
    }
}

// ---------------------------------------------------------------------------------------------
// Hadamard basis for the down_proj input (Section 4.3: U_D is a Hadamard matrix so that the projection
// that cannot be folded costs a fast transform instead of a dense product), fused with the per-token
// quantizer: C = X * H_K / sqrt(K), H_K = Sylvester(2^k) (x) H_m with coefficient index a * m + b, m = 1, or
// m = 12 / 28 with Paley's second construction (q = 5 / 13).  One CTA per row: the row is widened to fp32
// in shared memory, multiplied group-wise by the small factor (a compile-time table), run through the
// Sylvester butterflies up to five index bits per pass (32 values in registers),
// scaled, and then quantized exactly as in the fast path above (absmax per segment, reciprocal-product
// rounding with the exact fallback).  r = 0 gives the paper's uniform INT4 down_proj input.
// What bounds it: instructions.  So the factor's p and m halves, neighbouring coefficients of a butterfly and of the code
// rounding go two to an instruction, and through shared memory 8 bytes at a time: 1537 rows of 14336 45.2 -> 37.6 us, 4096
// 114 -> 96 (the row quantizers above, which share the rounding: 4096 x 4096 24.5 -> 23.7).
// Paley's second construction for a prime q = 1 (mod 4): H = S (x) [[1,1],[1,-1]] + I (x) [[1,-1],[-1,-1]] of order
// 2 (q + 1), with S = [[0, 1^T], [1, chi(i - j)]] and chi the quadratic character of GF(q).  S is evaluated at compile
// time, so the product with H is additions and subtractions only: with p_i = x_2i + x_2i+1 and m_i = x_2i - x_2i+1,
//   y_2j = m_j + sum_i S_ij p_i,   y_2j+1 = -p_j + sum_i S_ij m_i,
// and the circulant block of S needs only its quadratic-residue half (see the kernel): about 290 operations for
// M = 28, not M * M = 784.
constexpr int quad_char(int q, int a) {
    a = ((a % q) + q) % q;
    if (a == 0) return 0;
    for (int x = 1; x < q; ++x)
        if ((x * x) % q == a) return 1;
    return -1;
}
template <int M>
struct Conference {
    int s[M / 2][M / 2];
    constexpr Conference() : s() {
        constexpr int q = M / 2 - 1;
        for (int i = 0; i < M / 2; ++i)
            for (int j = 0; j < M / 2; ++j)
                s[i][j] = i == 0 ? (j == 0 ? 0 : 1) : (j == 0 ? 1 : quad_char(q, (i - 1) - (j - 1)));
    }
};

constexpr int kWideThreads = 1024;  // threads per row when there are at most kWideMaxRows rows (one CTA per SM)
constexpr int kWideMaxRows = 148;
// Place of group a of M coefficients in the row buffer: one group is left free behind every 2^run, a run being what a thread of the first
// pass walks through.  The threads of a warp take neighbouring runs there, which all begin at the same bank otherwise (2^run * M words, 2 ways).
__device__ __forceinline__ int slot_of(int a, int run) { return a + (a >> run); }
__device__ __forceinline__ int slot_stride(int s, int run) { return (1 << s) + (s >= run ? 1 << (s - run) : 0); }  // of index bit s
// One pass of the Sylvester butterflies: index bits [s, s + NB) of a, 2^NB values per thread in registers.  The last
// pass also scales by 1 / sqrt(K) and collects the two absmax values (elements below r belong to the INT8 segment).
template <int M, int NT, int NB>
__device__ __forceinline__ void butterfly_pass(float* hrow, int K, int s, int tid, bool last, float inv_sqrt_k, int r,
                                               float& a8, float& a4) {
    constexpr int N = 1 << NB;
    const int count = K >> NB;
    const int stride = M << s;
    for (int i = tid; i < count; i += NT) {
        const int arest = i / M, b = i - arest * M;
        const int a0 = ((arest >> s) << (s + NB)) | (arest & ((1 << s) - 1));
        float* base = hrow + a0 * M + b;
        float v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = base[j * stride];
#pragma unroll
        for (int bit = 0; bit < NB; ++bit) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (!(j & (1 << bit))) {
                    const float lo = v[j], hi = v[j | (1 << bit)];
                    v[j] = lo + hi;
                    v[j | (1 << bit)] = lo - hi;
                }
            }
        }
        if (last) {
            const int e0 = a0 * M + b;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                v[j] *= inv_sqrt_k;
                if (e0 + j * stride < r) a8 = fmaxf(a8, fabsf(v[j]));
                else a4 = fmaxf(a4, fabsf(v[j]));
            }
        }
#pragma unroll
        for (int j = 0; j < N; ++j) base[j * stride] = v[j];
    }
}

// The same for M even, a thread taking coefficients b and b + 1 of its 2^NB groups as pairs: half the instructions.
template <int M, int NT, int NB>
__device__ __forceinline__ void butterfly_pairs(float* hrow, int K, int s, int run, int tid, bool last, float inv_sqrt_k, int r, float& a8,
                                                float& a4) {
    constexpr int N = 1 << NB;
    const int count = K >> (NB + 1);
    const int estride = M << s, stride = slot_stride(s, run) * M;  // of the coefficients, of their places
    for (int i = tid; i < count; i += NT) {
        const int arest = i / (M / 2), b = 2 * (i - arest * (M / 2));
        const int a0 = ((arest >> s) << (s + NB)) | (arest & ((1 << s) - 1));
        f2* base = reinterpret_cast<f2*>(hrow + slot_of(a0, run) * M + b);
        f2 v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = base[j * (stride / 2)];
#pragma unroll
        for (int bit = 0; bit < NB; ++bit) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (!(j & (1 << bit))) {
                    const f2 lo = v[j], hi = v[j | (1 << bit)];
                    v[j] = add2(lo, hi);
                    v[j | (1 << bit)] = sub2(lo, hi);
                }
            }
        }
        if (last) {
            const f2 scale = pack2(inv_sqrt_k, inv_sqrt_k);
            const int e0 = a0 * M + b;  // r is a multiple of 8: a pair is in one segment
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = mul2(v[j], scale);
            if (e0 >= r) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const float2 x = unpack2(v[j]);
                    a4 = fmaxf(a4, fmaxf(fabsf(x.x), fabsf(x.y)));
                }
            } else {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const float2 x = unpack2(v[j]);
                    float& m = e0 + j * estride < r ? a8 : a4;
                    m = fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y)));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < N; ++j) base[j * (stride / 2)] = v[j];
    }
}

// Rows of 2^k with PAIRS: the first four index bits are the "small factor", groups of M = 16 coefficients.  Group a's 16-byte quarters sit
// in the order q ^ (a >> 1 & 3), so that eight groups' quarters, which eight threads write together, cover all banks (in order: 4 ways).
__device__ __forceinline__ int quarter_at(int a, int q, int run) { return 16 * slot_of(a, run) + 4 * (q ^ ((a >> 1) & 3)); }

// butterfly_pairs over these groups.  FIRST: s = 0, and the threads' groups are whole runs of 2^NB, NB >= 3, so the order of quarters
// follows from j; later passes have s >= 3, and it is the same for all j.
template <int NT, int NB, bool FIRST>
__device__ __forceinline__ void butterfly_sixteens(float* hrow, int K, int s, int run, int tid, bool last, float inv_sqrt_k, int r, float& a8, float& a4) {
    constexpr int N = 1 << NB;
    const int count = K >> (NB + 1);
    for (int i = tid; i < count; i += NT) {
        const int arest = i >> 3, b = 2 * (i & 7);
        const int a0 = FIRST ? arest << NB : ((arest >> s) << (s + NB)) | (arest & ((1 << s) - 1));
        const int estride = FIRST ? 16 : 16 << s, stride = FIRST ? 16 : 16 * slot_stride(s, run);
        float* at[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) at[c] = hrow + quarter_at(a0, (b >> 2) ^ (FIRST ? c : 0), run) + (b & 2);
        auto place = [&](int j) { return reinterpret_cast<f2*>(at[FIRST ? (j >> 1) & 3 : 0] + j * stride); };
        f2 v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = *place(j);
#pragma unroll
        for (int bit = 0; bit < NB; ++bit) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (!(j & (1 << bit))) {
                    const f2 lo = v[j], hi = v[j | (1 << bit)];
                    v[j] = add2(lo, hi);
                    v[j | (1 << bit)] = sub2(lo, hi);
                }
            }
        }
        if (last) {
            const f2 scale = pack2(inv_sqrt_k, inv_sqrt_k);
            const int e0 = a0 * 16 + b;  // r is a multiple of 8: a pair is in one segment
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = mul2(v[j], scale);
            if (e0 >= r) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const float2 x = unpack2(v[j]);
                    a4 = fmaxf(a4, fmaxf(fabsf(x.x), fabsf(x.y)));
                }
            } else {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const float2 x = unpack2(v[j]);
                    float& m = e0 + j * estride < r ? a8 : a4;
                    m = fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y)));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < N; ++j) *place(j) = v[j];
    }
}

// NT threads per row: 256 when rows outnumber the SMs (throughput: several CTAs per SM), 1024 for the few rows of a
// generation step, where one row's chain of passes is all there is to wait for.
// PAIRS: butterflies of two neighbours to a thread, for rows of kPairWidth and more.  Narrower ones have fewer pairs than threads: with
// M = 12 and 28 and pairs, rows of 384 to 896 took 2 to 6 % longer than now (1537 rows of 384 9.7 us, 9.0 now; 1000 rows of 1536
// 8.2, 8.1; of 1792 8.5, singly 9.1).
constexpr int kPairWidth = 1792;
// Rows of 2^k: groups of sixteen from here on, for any number of rows, 256 threads a row.  us, three index bits a pass (of 1024 threads a row up to
// 148 rows) / groups: 1537 rows of 1024 11.6 / 10.0, 2048 16.9 / 11.1, 8192 56.5 / 23.9, 32768 285 / 168; one row of 1024 4.2 / 2.9, 8192
// 8.5 / 4.6; but 1537 rows of 512 8.6 / 9.8.  One row of 512, 1024 / 256 threads: 3.8 / 2.8.
constexpr int kSixteensWidth = 1024;
template <int M, int NT, bool PAIRS = (M > 1 && NT == kThreads)>
__global__ void __launch_bounds__(NT, NT == kThreads ? (M > 1 ? 3 : 5) : 1)
hadamard_quantize_kernel(const __nv_bfloat16* X, size_t rows, int K, int kbits, int run, int r, float inv_sqrt_k,
                         int8_t* __restrict__ q8, uint8_t* __restrict__ q4, float* __restrict__ s8_out,
                         float* __restrict__ s4_out, int8_t* __restrict__ q4e) {
    extern __shared__ __align__(16) float hrow[];  // [K], and the places left free behind runs (slot_of)
    __shared__ float red[2][NT / 32];
    const int tid = threadIdx.x;
    const int nchunks = K >> 3, rchunks = r >> 3;
    const int K4 = K - r;
    const uint8_t* srow = reinterpret_cast<const uint8_t*>(hrow);
    griddep_wait();  // launched with programmatic stream serialization
    griddep_launch_dependents();
    for (size_t row = blockIdx.x; row < rows; row += gridDim.x) {
        // 1. widen the bf16 row (M = 1; otherwise the small factor below reads its groups straight from global memory)
        const uint4* xp = reinterpret_cast<const uint4*>(X + row * static_cast<size_t>(K));
        for (int c = tid; M == 1 && c < nchunks; c += NT) {
            const uint4 u = xp[c];
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
            float4 a, b;
            a.x = __uint_as_float(w[0] << 16); a.y = __uint_as_float(w[0] & 0xFFFF0000u);
            a.z = __uint_as_float(w[1] << 16); a.w = __uint_as_float(w[1] & 0xFFFF0000u);
            b.x = __uint_as_float(w[2] << 16); b.y = __uint_as_float(w[2] & 0xFFFF0000u);
            b.z = __uint_as_float(w[3] << 16); b.w = __uint_as_float(w[3] & 0xFFFF0000u);
            reinterpret_cast<float4*>(hrow)[2 * c] = a;
            reinterpret_cast<float4*>(hrow)[2 * c + 1] = b;
        }
        if constexpr (M == 1) __syncthreads();
        // 2. the small factor, one group of M consecutive coefficients per thread: bf16 from global memory (M * 2 bytes
        //    per group, a multiple of 8), fp32 result to the row buffer
        if constexpr (M == 16) {  // bits 0 to 3 of a row of 2^k
            for (int a = tid; a < (K >> 4); a += NT) {
                const uint4* xg = xp + 2 * a;
                const uint4 u0 = xg[0], u1 = xg[1];
                const uint32_t w[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
                f2 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xFFFF0000u);
                    v[i] = add2(pack2(lo, lo), pack2(hi, -hi));
                }
#pragma unroll
                for (int bit = 1; bit < 8; bit *= 2)
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (!(i & bit)) {
                            const f2 lo = v[i], hi = v[i | bit];
                            v[i] = add2(lo, hi);
                            v[i | bit] = sub2(lo, hi);
                        }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 lo = unpack2(v[2 * q]), hi = unpack2(v[2 * q + 1]);
                    *reinterpret_cast<float4*>(hrow + quarter_at(a, q, run)) = make_float4(lo.x, lo.y, hi.x, hi.y);
                }
            }
            __syncthreads();
        } else if constexpr (M > 1) {
            constexpr Conference<M> conf{};
            constexpr int H2 = M / 2;
            for (int a = tid; a < (K / M); a += NT) {
                // M * 4 bytes is a multiple of 16: the group moves as float4s (conflict-free at this stride)
                float4* gp = reinterpret_cast<float4*>(hrow + (PAIRS ? slot_of(a, run) : a) * M);
                const uint2* xg = reinterpret_cast<const uint2*>(X + row * static_cast<size_t>(K) + static_cast<size_t>(a) * M);
                float y[M];
                f2 pm[H2];  // (x_2i + x_2i+1, x_2i - x_2i+1)
#pragma unroll
                for (int i = 0; i < M / 4; ++i) {
                    const uint2 u = xg[i];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t w = h ? u.y : u.x;
                        const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xFFFF0000u);
                        pm[2 * i + h] = add2(pack2(lo, lo), pack2(hi, -hi));
                    }
                }
                // S = [[0, 1^T], [1, Q]] with Q_ij = chi(i - j) circulant of order q = M / 2 - 1.  With t = sum of the
                // q inner entries and R_j = sum over the quadratic residues k of entry (j + k) mod q, the non-residues
                // sum to t - entry_j - R_j, so (Q v)_j = 2 R_j - t + v_j: (q - 1) / 2 + 2 operations instead of q - 1, on the
                // p and m halves in one instruction.
                constexpr int Q = H2 - 1;
                const f2 two = pack2(2.f, 2.f);
                f2 t = pm[1];
#pragma unroll
                for (int i = 2; i < H2; ++i) t = add2(t, pm[i]);
                const float2 first = unpack2(pm[0]), tt = unpack2(t);
                y[0] = first.y + tt.x;
                y[1] = tt.y - first.x;
#pragma unroll
                for (int jp = 0; jp < Q; ++jp) {
                    f2 res = 0ull;
                    bool any = false;
#pragma unroll
                    for (int k = 1; k < Q; ++k) {
                        if (conf.s[1 + k][1] > 0) {  // chi(k) = +1
                            res = any ? add2(res, pm[1 + (jp + k) % Q]) : pm[1 + (jp + k) % Q];
                            any = true;
                        }
                    }
                    const float2 own = unpack2(pm[jp + 1]);
                    const f2 q = fma2(two, res, sub2(pm[jp + 1], t));
                    const float2 o = unpack2(add2(add2(pack2(own.y, -own.x), pack2(first.x, first.y)), q));
                    y[2 * (jp + 1)] = o.x;
                    y[2 * (jp + 1) + 1] = o.y;
                }
#pragma unroll
                for (int i = 0; i < M / 4; ++i) gp[i] = make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
            }
            __syncthreads();
        }
        // 3. Sylvester butterflies over the index bits of a, up to five bits (32 values in registers) per pass.  With
        //    M = 1 a thread's values of the first pass are 2^nb consecutive words, i.e. the lanes of a warp sit 2^nb
        //    banks apart: three bits per pass there (an 8-way conflict on one pass instead of a 32-way one).
        constexpr int kMaxBits = M == 1 ? 3 : 5;
        float a8 = 0.f, a4 = 0.f;
        for (int s = 0; s < kbits;) {
            const int left = kbits - s;
            const int nb = left <= kMaxBits ? left : (left <= 2 * kMaxBits ? (left + 1) / 2 : kMaxBits);
            const bool last = s + nb >= kbits;
            if constexpr (M == 16) {
                auto pass = [&](auto bits, auto first) {
                    butterfly_sixteens<NT, decltype(bits)::value, decltype(first)::value>(hrow, K, s, run, tid, last, inv_sqrt_k, r, a8, a4);
                };
                using std::integral_constant;
                if (s == 0) {
                    if (nb == 3) pass(integral_constant<int, 3>(), std::true_type());
                    else if (nb == 4) pass(integral_constant<int, 4>(), std::true_type());
                    else pass(integral_constant<int, 5>(), std::true_type());
                } else if (nb == 3) pass(integral_constant<int, 3>(), std::false_type());
                else if (nb == 4) pass(integral_constant<int, 4>(), std::false_type());
                else pass(integral_constant<int, 5>(), std::false_type());
            } else if constexpr (PAIRS) {  // 1024 threads have no registers for 32 pairs; M = 1 has odd neighbours in the first pass
                if (nb == 1) butterfly_pairs<M, NT, 1>(hrow, K, s, run, tid, last, inv_sqrt_k, r, a8, a4);
                else if (nb == 2) butterfly_pairs<M, NT, 2>(hrow, K, s, run, tid, last, inv_sqrt_k, r, a8, a4);
                else if (nb == 3) butterfly_pairs<M, NT, 3>(hrow, K, s, run, tid, last, inv_sqrt_k, r, a8, a4);
                else if (nb == 4) butterfly_pairs<M, NT, 4>(hrow, K, s, run, tid, last, inv_sqrt_k, r, a8, a4);
                else butterfly_pairs<M, NT, 5>(hrow, K, s, run, tid, last, inv_sqrt_k, r, a8, a4);
            } else if (nb == 1) butterfly_pass<M, NT, 1>(hrow, K, s, tid, last, inv_sqrt_k, r, a8, a4);
            else if (nb == 2) butterfly_pass<M, NT, 2>(hrow, K, s, tid, last, inv_sqrt_k, r, a8, a4);
            else if (nb == 3) butterfly_pass<M, NT, 3>(hrow, K, s, tid, last, inv_sqrt_k, r, a8, a4);
            else if constexpr (kMaxBits > 3) {
                if (nb == 4) butterfly_pass<M, NT, 4>(hrow, K, s, tid, last, inv_sqrt_k, r, a8, a4);
                else butterfly_pass<M, NT, 5>(hrow, K, s, tid, last, inv_sqrt_k, r, a8, a4);
            }
            s += nb;
            __syncthreads();
        }
        // 4. (no butterfly pass: K = M) scale and absmax in a pass of their own
        for (int c = tid; kbits == 0 && c < nchunks; c += NT) {
            float4* p = reinterpret_cast<float4*>(hrow) + 2 * c;
            float4 a = p[0], b = p[1];
            a.x *= inv_sqrt_k; a.y *= inv_sqrt_k; a.z *= inv_sqrt_k; a.w *= inv_sqrt_k;
            b.x *= inv_sqrt_k; b.y *= inv_sqrt_k; b.z *= inv_sqrt_k; b.w *= inv_sqrt_k;
            p[0] = a; p[1] = b;
            const float m = fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                                  fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
            if (c < rchunks) a8 = fmaxf(a8, m);
            else a4 = fmaxf(a4, m);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a8 = fmaxf(a8, __shfl_xor_sync(0xffffffffu, a8, o));
            a4 = fmaxf(a4, __shfl_xor_sync(0xffffffffu, a4, o));
        }
        if ((tid & 31) == 0) {
            red[0][tid >> 5] = a8;
            red[1][tid >> 5] = a4;
        }
        __syncthreads();  // also: every thread's scaled values are in place
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) {
            a8 = fmaxf(a8, red[0][w]);
            a4 = fmaxf(a4, red[1][w]);
        }
        // 5. codes
        const float s8 = __fdiv_rn(a8, 127.f), s4 = __fdiv_rn(a4, 7.f);
        const float inv8 = s8 > 0.f ? __frcp_rn(s8) : 0.f, inv4 = s4 > 0.f ? __frcp_rn(s4) : 0.f;
        const bool exact8 = s8 > 0.f && !(inv8 >= 1.1754944e-38f && inv8 <= 3.0e38f);
        const bool exact4 = s4 > 0.f && !(inv4 >= 1.1754944e-38f && inv4 <= 3.0e38f);
        if (tid == 0) {
            s8_out[row] = s8;
            s4_out[row] = s4;
        }
        int8_t* q8row = q8 + row * static_cast<size_t>(r);
        uint8_t* q4row = q4 ? q4 + row * static_cast<size_t>(K4 >> 1) : nullptr;
        int8_t* q4e_row = q4e ? q4e + row * static_cast<size_t>(K4) : nullptr;
        for (int c = tid; c < nchunks; c += NT) {
            uint32_t t[8];
            const bool seg8 = c < rchunks;
            const float s = seg8 ? s8 : s4;
            Chunk<true> ch;
            if constexpr (M == 16) {
                const int a = c >> 1, q = 2 * (c & 1);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4 u = *reinterpret_cast<const uint4*>(hrow + quarter_at(a, q + h, run));
                    ch.w[4 * h] = u.x; ch.w[4 * h + 1] = u.y; ch.w[4 * h + 2] = u.z; ch.w[4 * h + 3] = u.w;
                }
            } else {  // no run ends within a chunk
                const uint4* p = reinterpret_cast<const uint4*>(srow) + 2 * c + (PAIRS ? M / 4 * ((8 * c / M) >> run) : 0);
                const uint4 u = p[0], v = p[1];
                ch.w[0] = u.x; ch.w[1] = u.y; ch.w[2] = u.z; ch.w[3] = u.w;
                ch.w[4] = v.x; ch.w[5] = v.y; ch.w[6] = v.z; ch.w[7] = v.w;
            }
            if (s > 0.f) fast_codes(ch, s, seg8 ? inv8 : inv4, seg8 ? exact8 : exact4, t);
            else {
#pragma unroll
                for (int k = 0; k < 8; ++k) t[k] = 0;
            }
            const uint32_t w0 = pack_low_bytes(t[0], t[1], t[2], t[3]), w1 = pack_low_bytes(t[4], t[5], t[6], t[7]);
            if (seg8) {
                *reinterpret_cast<uint2*>(q8row + c * 8) = make_uint2(w0, w1);
            } else {
                const int jj = (c - rchunks) * 8;
                if (q4e_row) *reinterpret_cast<uint2*>(q4e_row + jj) = make_uint2(w0, w1);
                if (q4row) {
                    const uint32_t x = w0 & 0x0F0F0F0Fu, y = w1 & 0x0F0F0F0Fu;
                    *reinterpret_cast<uint32_t*>(q4row + (jj >> 1)) = __byte_perm(x | (x >> 4), y | (y >> 4), 0x6420);
                }
            }
        }
        __syncthreads();  // the row buffer is reused by the next row
    }
}

}  // namespace

namespace {

// The fast kernel on `rows` rows that fit its staging (launch_split_quantize, launch_split_quantize_asym).
template <bool F32, bool ASYM>
cudaError_t launch_fast(const void* in, size_t rows, int K, int r, int8_t* q8, uint8_t* q4, float* s8, float* s4, float* z8,
                        float* z4, int8_t* q4_i8, size_t in_row_stride_bytes, cudaStream_t st) {
    const size_t row_bytes = static_cast<size_t>(K) * (F32 ? 4 : 2);
    int rpc = 1;  // rows per CTA and step: 1, 2, 4 or 8, about half of kFastGroupBytes of staging
    while (rpc < 8 && row_bytes * rpc * 2 <= static_cast<size_t>(kFastGroupBytes)) rpc *= 2;
    while (rpc > 1 && rows / rpc < 148) rpc /= 2;  // few rows (a generation step): all threads of a CTA on one row
    const size_t groups = (rows + rpc - 1) / rpc;
    const size_t group_bytes = row_bytes * rpc;
    auto kern = split_quantize_fast_kernel<F32, ASYM>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kFastMaxRowBytes);
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set[dev] = true;
    }
    auto ctas_per_sm = [](size_t smem) {  // shared memory and the 2048-thread limit; registers allow 8 CTAs of 256
        const size_t by_smem = (227u * 1024u) / (smem + 1024u);
        return by_smem < 1 ? size_t(1) : (by_smem > 8 ? size_t(8) : by_smem);
    };
    // Two stages when they are cheap (several CTAs per SM still fit) and a CTA has more than one group to do.  Asymmetric rows
    // take more arithmetic per byte and gain from more warps per SM instead: a CTA per group, one stage (8192 rows of 2048 /
    // 4096 / 14336: 19.0 / 34.6 / 100.4 us against 21.7 / 37.0 / 105.5 with two stages).
    // With one stage a CTA per group, too, for wide symmetric rows: the next CTA's copy starts as soon as one has left (fp32 rows, us, a walk of as many
    // CTAs as fit / this: 4096 of 14336 59.8 / 57.0, of 16384 64.5 / 61.1, 2048 of 28672 61.1 / 59.7, 1024 of 14336
    // 17.5 / 16.5; bf16 rows 4096 of 20480 77 / 61.6, of 28672 91.2 / 87, 1000 of 28672 29.2 / 27).
    int nstages = 1;
    size_t grid = groups;
    if (!ASYM && groups > 148 * ctas_per_sm(group_bytes) && 2 * group_bytes <= 64u * 1024u) {
        nstages = 2;
        grid = 148 * ctas_per_sm(2 * group_bytes);
    }
    if (grid > groups) grid = groups;
    // The kernel waits for the preceding grid itself (griddepcontrol.wait on entry), so it may always be scheduled
    // while that grid drains; for the few rows of a generation step this hides most of its launch.
    count_launch();
    return launch_programmatic(kern, grid, kThreads, group_bytes * nstages, st, in, in_row_stride_bytes, rows, K, r, rpc, nstages, q8,
                               q4, s8, s4, z8, z4, q4_i8, device_status_ptr());
}

}  // namespace

cudaError_t launch_split_quantize_asym(const void* in, bool in_is_f32, size_t rows, int K, int r, uint8_t* u8,
                                       uint8_t* u4, float* s8, float* s4, float* z8, float* z4, uint8_t* u4_u8,
                                       size_t in_row_stride_bytes, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    const size_t row_bytes = static_cast<size_t>(K) * (in_is_f32 ? 4 : 2);
    if (row_bytes > static_cast<size_t>(kFastMaxRowBytes) || in_row_stride_bytes % 16 != 0) return cudaErrorNotSupported;
    auto launch = in_is_f32 ? launch_fast<true, true> : launch_fast<false, true>;
    return launch(in, rows, K, r, reinterpret_cast<int8_t*>(u8), u4, s8, s4, z8, z4, reinterpret_cast<int8_t*>(u4_u8),
                  in_row_stride_bytes, st);
}

cudaError_t launch_split_quantize(const void* in, bool in_is_f32, size_t rows, int K, int r, int8_t* q8,
                                  uint8_t* q4, void* s8, void* s4, bool scale_fp16, int8_t* q4_i8,
                                  size_t in_row_stride_bytes, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    const size_t row_bytes = static_cast<size_t>(K) * (in_is_f32 ? 4 : 2);
    if (!scale_fp16 && row_bytes <= static_cast<size_t>(kFastMaxRowBytes) && in_row_stride_bytes % 16 == 0) {
        auto launch = in_is_f32 ? launch_fast<true, false> : launch_fast<false, false>;
        return launch(in, rows, K, r, q8, q4, static_cast<float*>(s8), static_cast<float*>(s4), nullptr, nullptr, q4_i8,
                      in_row_stride_bytes, st);
    }
    const unsigned grid = static_cast<unsigned>(rows < 148u * 64u ? rows : 148u * 64u);
    count_launch();
    if (in_is_f32)
        split_quantize_kernel<true><<<grid, kThreads, 0, st>>>(in, in_row_stride_bytes, rows, K, r, q8, q4, s8, s4,
                                                               scale_fp16 ? 1 : 0, q4_i8);
    else
        split_quantize_kernel<false><<<grid, kThreads, 0, st>>>(in, in_row_stride_bytes, rows, K, r, q8, q4, s8, s4,
                                                                scale_fp16 ? 1 : 0, q4_i8);
    return cudaGetLastError();
}

cudaError_t launch_unpack_int4(const uint8_t* packed, int8_t* out, size_t rows, size_t cols, cudaStream_t st,
                               bool codes_unsigned) {
    const size_t nwords = rows * cols / 8;
    if (nwords == 0) return cudaSuccess;
    size_t blocks = (nwords + 255) / 256;
    if (blocks > 148 * 32) blocks = 148 * 32;
    count_launch();
    if (codes_unsigned) unpack_int4_kernel<true><<<static_cast<unsigned>(blocks), 256, 0, st>>>(packed, out, nwords);
    else unpack_int4_kernel<false><<<static_cast<unsigned>(blocks), 256, 0, st>>>(packed, out, nwords);
    return cudaGetLastError();
}


// K = 2^k * m with m in {28, 12, 1} (largest first); false if K has no such form.
bool hadamard_factor(int K, int* kbits, int* m) {
    for (int mm : {28, 12, 1}) {
        if (K % mm) continue;
        const int a = K / mm;
        if (a & (a - 1)) continue;
        int kb = 0;
        while ((1 << kb) < a) ++kb;
        *kbits = kb;
        *m = mm;
        return true;
    }
    return false;
}

cudaError_t launch_hadamard_quantize(const void* X, size_t rows, int K, int r, int8_t* q8, uint8_t* q4, float* s8,
                                     float* s4, int8_t* q4_i8, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    int kbits = 0, m = 0;
    if (!hadamard_factor(K, &kbits, &m)) return cudaErrorNotSupported;
    constexpr size_t kMaxSmem = 200 * 1024;
    size_t smem = static_cast<size_t>(K) * 4;
    if (smem > kMaxSmem) return cudaErrorNotSupported;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    static bool ready[64] = {};
    if (dev < 64 && !ready[dev]) {
        // Once per device: the shared-memory limit of the kernels.
        for (auto k : {hadamard_quantize_kernel<1, kThreads>, hadamard_quantize_kernel<12, kThreads>,
                       hadamard_quantize_kernel<28, kThreads>, hadamard_quantize_kernel<12, kThreads, false>,
                       hadamard_quantize_kernel<28, kThreads, false>, hadamard_quantize_kernel<16, kThreads>,
                       hadamard_quantize_kernel<12, kWideThreads>, hadamard_quantize_kernel<28, kWideThreads>})
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem)) != cudaSuccess)
                return e;
        ready[dev] = true;
    }
    // 1024 threads per row only when rows do not outnumber the SMs: at 28672-wide rows (two 256-thread CTAs per SM)
    // the wide form measured slower for many rows (0.89 against 0.72 ms at 8192 rows).
    const bool wide = rows <= kWideMaxRows && m != 1;
    if (m == 1 && K >= kSixteensWidth) { m = 16; kbits -= 4; }  // the group's own bits
    const bool pairs = !wide && m > 1 && (m == 16 || K >= kPairWidth);
    // A place left free behind every run of the first pass (slot_of), unless fewer CTAs then fit an SM (rows of 28672: two).  1537 rows, us, without
    // / with: 6144 22.4 / 19.4, 8192 23.9 / 22.1, 14336 39.2 / 37.1, 24576 103 / 87; in the other forms it cost 3 to 8 % (28672, 1024 threads a row).
    int run = 31;
    if (pairs && kbits > 5) {
        const int first = kbits > 10 ? 5 : (kbits + 1) / 2;
        const size_t spaced = smem + static_cast<size_t>((K / m) >> first) * m * 4;
        auto ctas = [](size_t bytes) { return std::min<size_t>(3, 228 * 1024 / (bytes + 1280)); };
        if (spaced <= kMaxSmem && ctas(spaced) == ctas(smem)) {
            run = first;
            smem = spaced;
        }
    }
    const float inv_sqrt_k = static_cast<float>(1.0 / sqrt(static_cast<double>(K)));
    const unsigned grid = static_cast<unsigned>(rows < 148u * 16u ? rows : 148u * 16u);
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(X);
    auto kern = wide ? (m == 12 ? hadamard_quantize_kernel<12, kWideThreads> : hadamard_quantize_kernel<28, kWideThreads>)
                : m == 1  ? hadamard_quantize_kernel<1, kThreads>
                : m == 16 ? hadamard_quantize_kernel<16, kThreads>
                : !pairs  ? (m == 12 ? hadamard_quantize_kernel<12, kThreads, false> : hadamard_quantize_kernel<28, kThreads, false>)
                          : (m == 12 ? hadamard_quantize_kernel<12, kThreads> : hadamard_quantize_kernel<28, kThreads>);
    count_launch();
    return launch_programmatic(kern, grid, wide ? kWideThreads : kThreads, smem, st, x, rows, K, kbits, run, r, inv_sqrt_k, q8, q4,
                               s8, s4, q4_i8);
}

}  // namespace resq
