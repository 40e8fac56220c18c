// Eight neighbouring values of a row and their codes (Eq. 1, both forms), for the row quantizers and the product that quantizes its own
// rows.
//
// Rounding.  The definition is code = round-half-even(fl(x / s)) with an IEEE division.  Here
// t = fma(x, v, M) with M = 1.5 * 2^23 rounds the exact product x * v to the nearest integer (ties to
// even) in one instruction, and the low byte of t's bit pattern is the two's-complement code.  It is
// evaluated for two factors that bracket 1 / s, v_lo = RN(inv (1 - 2^-20)) and v_hi = RN(inv (1 + 2^-20))
// with inv = RN(1 / s): fl(x / s) lies between x * v_lo and x * v_hi (the division and the reciprocal
// are each off by at most 2^-24 relative, the bracket is 2^-21 wide at least on either side), rounding to
// nearest is monotone, so when both products round to the same integer, that integer is the defined code;
// when they differ (the quotient is within |x / s| * 2^-19 of a half-integer, ties included) the chunk is
// redone with the true division.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>

#include "packed_fp32.cuh"

namespace resq {

constexpr float kRowMagic = 12582912.f;              // 1.5 * 2^23
constexpr float kRowBracket = 9.5367431640625e-07f;  // 2^-20

// A chunk is kept in registers in its storage format: 4 words of bf16 pairs, or 8 fp32 words.
template <bool F32>
struct Chunk {
    uint32_t w[F32 ? 8 : 4];
    __device__ __forceinline__ float get(int i) const {
        if constexpr (F32) return __uint_as_float(w[i]);
        else return (i & 1) ? __uint_as_float(w[i >> 1] & 0xFFFF0000u) : __uint_as_float(w[i >> 1] << 16);
    }
};

template <bool F32>
__device__ __forceinline__ Chunk<F32> load_chunk(const void* row, int c) {
    Chunk<F32> o;
    if constexpr (F32) {
        const uint4* p = reinterpret_cast<const uint4*>(row) + 2 * c;
        uint4 a = p[0], b = p[1];
        o.w[0] = a.x; o.w[1] = a.y; o.w[2] = a.z; o.w[3] = a.w;
        o.w[4] = b.x; o.w[5] = b.y; o.w[6] = b.z; o.w[7] = b.w;
    } else {
        uint4 u = reinterpret_cast<const uint4*>(row)[c];
        o.w[0] = u.x; o.w[1] = u.y; o.w[2] = u.z; o.w[3] = u.w;
    }
    return o;
}

template <bool F32>
__device__ __forceinline__ float chunk_absmax(const Chunk<F32>& c) {
    if constexpr (F32) {
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(c.get(i)));
        return m;
    } else {
        // bf16 pairs: clear the signs, then compare as packed bf16 (exact: max selects one of its inputs)
        __nv_bfloat162 m = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t a = c.w[i] & 0x7FFF7FFFu;
            m = __hmax2(m, *reinterpret_cast<const __nv_bfloat162*>(&a));
        }
        return fmaxf(__low2float(m), __high2float(m));
    }
}

template <bool F32>
__device__ __forceinline__ void fast_codes(const Chunk<F32>& ch, float s, float inv, bool exact_only, uint32_t (&t)[8]) {
    const float v_lo = fmaf(inv, -kRowBracket, inv), v_hi = fmaf(inv, kRowBracket, inv);
    const f2 vl = pack2(v_lo, v_lo), vh = pack2(v_hi, v_hi), magic = pack2(kRowMagic, kRowMagic);
    uint32_t differ = 0;
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        const f2 x = pack2(ch.get(i), ch.get(i + 1));
        const float2 a = unpack2(fma2(x, vl, magic)), b = unpack2(fma2(x, vh, magic));
        t[i] = __float_as_uint(a.x);
        t[i + 1] = __float_as_uint(a.y);
        differ |= t[i] ^ __float_as_uint(b.x);
        differ |= t[i + 1] ^ __float_as_uint(b.y);
    }
    if (exact_only || differ != 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = __float_as_uint(rintf(__fdiv_rn(ch.get(i), s)) + kRowMagic);
    }
}

// The asymmetric form (Eq. 1, second form): code = round-half-even(fl(fl(x - z) / s)) clamped to [0, qmax].  The same
// bracket around 1 / s on d = fl(x - z): quotients reach 255, where a bracketed product still rounds to an integer in one
// fma and the argument above is about relative errors only.
template <bool F32>
__device__ __forceinline__ void fast_codes_asym(const Chunk<F32>& ch, float z, float s, float inv, bool exact_only, float qmax,
                                                uint32_t (&t)[8]) {
    const float v_lo = fmaf(inv, -kRowBracket, inv), v_hi = fmaf(inv, kRowBracket, inv);
    const f2 vl = pack2(v_lo, v_lo), vh = pack2(v_hi, v_hi), magic = pack2(kRowMagic, kRowMagic), mz = pack2(-z, -z);
    uint32_t differ = 0;
    float d[8];
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        const f2 x = add2(pack2(ch.get(i), ch.get(i + 1)), mz);
        const float2 u = unpack2(x), a = unpack2(fma2(x, vl, magic)), b = unpack2(fma2(x, vh, magic));
        d[i] = u.x;
        d[i + 1] = u.y;
        t[i] = __float_as_uint(a.x);
        t[i + 1] = __float_as_uint(a.y);
        differ |= t[i] ^ __float_as_uint(b.x);
        differ |= t[i + 1] ^ __float_as_uint(b.y);
    }
    if (exact_only || differ != 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = __float_as_uint(fminf(fmaxf(rintf(__fdiv_rn(d[i], s)), 0.f), qmax) + kRowMagic);
    }
}

// Low bytes of four words -> one word.
__device__ __forceinline__ uint32_t pack_low_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// Reciprocal of a scale; whether the product form may use it (finite, normal): otherwise every chunk takes the division.
struct ScaleInv {
    float inv;
    bool exact;
    __device__ __forceinline__ explicit ScaleInv(float s) {
        inv = s > 0.f ? __frcp_rn(s) : 0.f;
        exact = s > 0.f && !(inv >= 1.1754944e-38f && inv <= 3.0e38f);
    }
};

}  // namespace resq
