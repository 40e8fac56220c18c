// Attention-block path, cache side (Section 4.3, Eq. 8; Section 5.1), d_head = 128 and 64: the 8-bit online U_C
// projection of query and key head vectors, and the per-head asymmetric 8/4-bit quantizer that writes key and value
// into the blocked cache.  A few MB per call at most.  Two forms, chosen by the number of head vectors (launch_project):
//
// kv_project_kernel (many): one warp owns 16 head vectors (rows) at a time and contracts them on mma.sync s8
// fragments taken straight from the global loads.  Lane (g, c) = (lane / 4, lane % 4) loads, for rows g and g + 8, the
// elements [32 b + 8c, +8), 16 bytes at a time: the bytes of its A fragments of mma.m16n8k32, in an order of the reduction that
// U_C's staged rows share.  The product's columns are dealt out in the same way (a permutation of U_C's rows, free with
// ldmatrix), so outputs leave 16 bytes at a time too, and key and value share the cache quantizer.
// What bounds it: instructions, their fetch first (120 KB of straight code at d = 128, 70 at 64); 2048 tokens of 32 + 16 vectors take
// 27.2 us at d = 128 (before 32.0; the 100 MB would take 15) and 13.6 at 64 (before 18.1).  128 registers at d = 128 spill 76 bytes.  Rows of a key or value tile are 16 tokens of one head: their records are
// neighbours in the cache.  The next tile's rows are on their way during the products.  Roundings are checked for a whole lane
// at once (two bracketing products, packed pairs) instead of one by one with a branch each.
// head_vector_kernel (few, a generation step): one warp per head vector, lane l owning coefficients l + 32 i, dp4a
// against U_C's codes in shared memory.  A step is latency: one vector's chain is shorter than a 16-vector tile's and so is
// the code, which counts in a step, where every kernel runs once between others.  16 tokens (512 query, 256 key and value
// vectors) at d = 128: 15.0 -> 8.6 us by themselves, 37 -> 10.6 us right after an attention call on a 140 MB cache.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "internal.h"
#include "packed_fp32.cuh"
#include "plans.h"
#include "ptx.cuh"
#include "../../include/resq_kv.h"

namespace resq {
namespace {

constexpr int kWarps = 4;
template <int D>
struct Head {  // geometry of a head vector and of its cache block (resq_kv.h)
    static constexpr int kR8 = D / 8;                          // coefficients in 8 bits
    static constexpr int kB4 = (D - kR8) / 2;                  // bytes of 4-bit codes
    static constexpr int kC8 = RESQ_KV_BLOCK * kR8, kC4 = RESQ_KV_BLOCK * kB4;
    static constexpr int kHalf = kC8 + kC4 + RESQ_KV_BLOCK * 16, kBlock = 2 * kHalf;
    static constexpr int kWStride = D + 16;  // bytes per W_C row as head_vector_kernel stages it: the lanes' rows hit all banks
};
static_assert(Head<128>::kBlock == RESQ_KV_BLOCK_BYTES, "block layout");
// Head vectors of a call up to which one warp takes one of them.  Event times in us, one per warp / 16 per warp, 32 + 16 vectors per
// token: d = 128, 100 tokens 7.9 / 9.0, 128 10.7 / 9.2, 256 15.0 / 10.1, but with cold caches, as in a step of a model, 128 tokens
// 14.3 / 16.4, 192 16.4 / 16.4, 256 18.4 / 16.4: 9216 vectors.  d = 64: 80 tokens 5.2 / 5.4, 100
// 5.7 / 5.4, 256 9.7 / 6.1; cold, 64 tokens 10.2 / 10.2, 128 12.3 / 10.2.
template <int D>
constexpr long long kFewVectors = D == 128 ? 9216 : 4096;
constexpr float kMagic = 12582912.f;  // 1.5 * 2^23
constexpr float kBracket = 9.5367431640625e-7f;  // 2^-20
constexpr int kTileWarps = 8;            // of a kv_project_kernel CTA, two per SM

// round-half-even(x / s) with the IEEE quotient's rounding: the product with inv = RN(1/s) lies within 2^-15
// (|q| <= 127) / 2^-14 (|q| <= 255) of the quotient, so the two can only round apart when the product is that
// close to a half-integer; there the true division decides.
__device__ __forceinline__ float code_rn(float x, float s, float inv, bool exact_only, float guard) {
    const float tf = fmaf(x, inv, kMagic);
    const float q = tf - kMagic;
    const float res = fabsf(fmaf(x, inv, -q));
    if (exact_only || !(res < guard)) return rintf(__fdiv_rn(x, s));
    return q;
}
__device__ __forceinline__ bool needs_division(float inv) { return !(inv >= 1.1754944e-38f && inv <= 3.0e38f); }

__device__ __forceinline__ void mma_s8(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float quad_max(float v) {
    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_min(float v) {
    v = fminf(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return fminf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}

// Asymmetric parameters of one segment from its (min, max): s, 1/s, whether the division must be used.
struct Asym {
    float z, s, inv;
    bool exact;
    __device__ __forceinline__ Asym(float lo, float hi, float qmax) {
        z = lo;
        s = __fdiv_rn(__fsub_rn(hi, lo), qmax);
        inv = s > 0.f ? __frcp_rn(s) : 0.f;
        exact = s > 0.f && needs_division(inv);
    }
    __device__ __forceinline__ uint32_t code(float x, float qmax) const {
        if (!(s > 0.f)) return 0u;
        const float q = code_rn(__fsub_rn(x, z), s, inv, exact, 0.5f - 0.00006103515625f);
        return static_cast<uint32_t>(fminf(fmaxf(q, 0.f), qmax));
    }
};

// Byte offset in the cache of the block that holds head h of token t, plus the token's slot in it (below 32; blocks are multiples
// of 32 bytes), or -1.
template <int D>
__device__ __forceinline__ long long cache_slot(int t, int h, int n_kv_heads, int n_seqs, int capacity, const int32_t* seq_ids,
                                                const int32_t* positions, int* status) {
    const int b = seq_ids[t], pos = positions[t];
    if (b < 0 || b >= n_seqs || pos < 0 || pos >= capacity) {
        atomicOr(status, kStatusBitIndex);
        return -1;
    }
    const long long blk = (static_cast<long long>(b) * n_kv_heads + h) * (capacity / RESQ_KV_BLOCK) + pos / RESQ_KV_BLOCK;
    return blk * Head<D>::kBlock + (pos % RESQ_KV_BLOCK);
}

struct ProjectParams {
    const __nv_bfloat16* q;  // [q_rows][128] or null
    const __nv_bfloat16* k;  // [kv_rows][128] or null
    const __nv_bfloat16* v;
    long long q_rows, kv_rows;
    const int8_t* wq;
    const float* s_u;
    __half* q_out;
    uint8_t* cache;
    int n_seqs, n_kv_heads, capacity;
    const int32_t* seq_ids;
    const int32_t* positions;
    int* status;
    bool together;  // append_tiles_together
};

// W_C's codes and scales into shared memory.
template <int D>
__device__ __forceinline__ void stage_uc(const int8_t* wq, const float* s_u, uint8_t* w_s, float* su_s) {
    for (int i = threadIdx.x; i < D * (D / 16); i += blockDim.x) {  // 16-byte pieces
        const int n = i / (D / 16), pc = i % (D / 16);
        *reinterpret_cast<uint4*>(w_s + n * Head<D>::kWStride + pc * 16) = reinterpret_cast<const uint4*>(wq + n * D)[pc];
    }
    for (int i = threadIdx.x; i < D; i += blockDim.x) su_s[i] = s_u[i];
}

// Rounds N values x / s (after x - z) to codes 0 .. qmax or of either sign, t[i] = code + kMagic as bits: x v for the two factors
// v = RN(inv (1 -+ 2^-20)) that bracket 1 / s, inv = RN(1 / s).  Where both products round to the same integer it is the rounded
// IEEE quotient; else, or where one is NaN, the true divisions decide for all of the lane's values.
template <int N>
__device__ __forceinline__ void round_codes(const f2* d, float s, float inv, bool exact, float lo, float hi, uint32_t (&t)[N]) {
    const float v_lo = fmaf(inv, -kBracket, inv), v_hi = fmaf(inv, kBracket, inv);
    const f2 vl = pack2(v_lo, v_lo), vh = pack2(v_hi, v_hi), magic = pack2(kMagic, kMagic);
    uint32_t differ = 0, seen = 0;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float2 a = unpack2(fma2(d[i], vl, magic)), b = unpack2(fma2(d[i], vh, magic));
        t[2 * i] = __float_as_uint(a.x);
        t[2 * i + 1] = __float_as_uint(a.y);
        differ |= t[2 * i] ^ __float_as_uint(b.x);
        differ |= t[2 * i + 1] ^ __float_as_uint(b.y);
        seen |= t[2 * i] | t[2 * i + 1];
    }
    if (exact || differ != 0 || (seen & 0x34000000u) != 0) {  // kMagic plus a code has none of these bits, NaN has
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const float2 x = unpack2(d[i]);
            const float qa = rintf(__fdiv_rn(x.x, s)), qb = rintf(__fdiv_rn(x.y, s));
            t[2 * i] = __float_as_uint((qa == qa ? fminf(fmaxf(qa, lo), hi) : 0.f) + kMagic);  // NaN: 0
            t[2 * i + 1] = __float_as_uint((qb == qb ? fminf(fmaxf(qb, lo), hi) : 0.f) + kMagic);
        }
    }
}
__device__ __forceinline__ uint32_t low_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// Staging of a warp's 16 records.
template <int D>
struct Records {
    alignas(16) uint8_t c8[16][Head<D>::kR8];
    alignas(16) uint8_t c4[16][Head<D>::kB4];
    float4 meta[16];
    long long slot[16];
};

// The asymmetric 8/4-bit record of a row held by a quad, v[4 b + i]: columns 32 b + 8c + 2i and the next.  Values that are
// all NaN (a key with an infinity has them) leave z = inf and s = -inf, as in head_vector_kernel.
template <int D>
__device__ __forceinline__ void quantize_record(const f2 (&v)[D / 8], int c, Records<D>& rec, int row) {
    const bool in8 = 8 * c < Head<D>::kR8;  // the lane's first eight values; the others are in the 4-bit segment for every lane
    float hmin = INFINITY, hmax = -INFINITY, lo4 = INFINITY, hi4 = -INFINITY;
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
        const float2 x = unpack2(v[i]);
        float& lo = i < 4 ? hmin : lo4;
        float& hi = i < 4 ? hmax : hi4;
        lo = fminf(lo, fminf(x.x, x.y));
        hi = fmaxf(hi, fmaxf(x.x, x.y));
    }
    const Asym q8(quad_min(in8 ? hmin : INFINITY), quad_max(in8 ? hmax : -INFINITY), 255.f);
    const Asym q4(quad_min(in8 ? lo4 : fminf(lo4, hmin)), quad_max(in8 ? hi4 : fmaxf(hi4, hmax)), 15.f);
#pragma unroll
    for (int b = 0; b < D / 32; ++b) {
        const bool wide = b == 0 && in8;
        const Asym& q = wide ? q8 : q4;
        const f2 mz = pack2(-q.z, -q.z);
        f2 d[4];
        uint32_t t[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = add2(v[4 * b + i], mz);
        round_codes<8>(d, q.s, q.inv, q.exact, 0.f, wide ? 255.f : 15.f, t);
        const uint32_t lo = q.s > 0.f ? low_bytes(t[0], t[1], t[2], t[3]) : 0u, hi = q.s > 0.f ? low_bytes(t[4], t[5], t[6], t[7]) : 0u;
        if (wide) {
            *reinterpret_cast<uint2*>(rec.c8[row] + 8 * c) = make_uint2(lo, hi);
        } else {  // eight nibbles
            const uint32_t x = lo & 0x0F0F0F0Fu, y = hi & 0x0F0F0F0Fu;
            *reinterpret_cast<uint32_t*>(rec.c4[row] + 16 * b + 4 * c - Head<D>::kR8 / 2) = __byte_perm(x | (x >> 4), y | (y >> 4), 0x6420);
        }
    }
    if (c == 0) rec.meta[row] = make_float4(q8.s, q8.z, q4.s, q4.z);
}

// Copies the 16 staged records into the cache (half 0: key, 1: value).
template <int D>
__device__ __forceinline__ void flush_records(const Records<D>& rec, uint8_t* cache, int half, int lane) {
    using H = Head<D>;
    using Byte8 = typename std::conditional<D == 128, uint4, uint2>::type;   // a record's 8-bit codes
    using Unit = typename std::conditional<D == 128, uint2, uint32_t>::type;  // a seventh of its 4-bit codes
    const int row = lane & 15;
    const long long mine = rec.slot[row];
    if (mine >= 0) {
        uint8_t* blk = cache + (mine & ~31ll) + half * H::kHalf;
        const int p = static_cast<int>(mine & 31);
        if (lane < 16) *reinterpret_cast<Byte8*>(blk + p * H::kR8) = *reinterpret_cast<const Byte8*>(rec.c8[row]);
        else *reinterpret_cast<float4*>(blk + H::kC8 + H::kC4 + p * 16) = rec.meta[row];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int u = i * 32 + lane, r = u / 7, part = u - 7 * r;
        if (u >= 112) break;
        const long long sl = rec.slot[r];
        if (sl < 0) continue;
        uint8_t* dst = cache + (sl & ~31ll) + half * H::kHalf + H::kC8 + static_cast<int>(sl & 31) * H::kB4;
        reinterpret_cast<Unit*>(dst)[part] = reinterpret_cast<const Unit*>(rec.c4[r])[part];
    }
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// Tiles of 16 head vectors: the keys' (16 tokens of one head: projected, quantized, appended), the values' (quantized, appended), the
// query's (16 rows: projected, written as half).  All warps go through them in this order: longest first, and at any time an SM's
// warps run one kind's code (2048 tokens of 32 + 16 vectors of 128: 27.8 us; queries before values 36.6).  Neighbours are in
// different CTAs, or (append_tiles_together) in the warps of one, which start each round together; a last round that is
// not full is spread over the CTAs either way.
template <int D>
__global__ void __launch_bounds__(kTileWarps * 32, 2) kv_project_kernel(const ProjectParams p) {
    constexpr int KS = D / 32;  // k steps, blocks of 32 columns
    __shared__ __align__(128) uint8_t w_s[D * D];  // chunk j of row n at chunk j ^ swizzle(n)
    __shared__ __align__(16) float su_s[D];
    __shared__ __align__(16) Records<D> rec_s[kTileWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    Records<D>& rec = rec_s[warp];
    const int T = p.n_kv_heads ? static_cast<int>(p.kv_rows / p.n_kv_heads) : 0;
    const int kv_tiles = (T + 15) / 16 * p.n_kv_heads, q_tiles = static_cast<int>((p.q_rows + 15) / 16);
    const int tiles = q_tiles + 2 * kv_tiles, stride = static_cast<int>(gridDim.x) * kTileWarps;  // 2^31 tiles would be terabytes
    // an ldmatrix reads rows 0 1 8 9 16 17 24 25 of 32 at once, or those plus 2, 4, 6
    auto swizzle = [](int n) { return D == 128 ? (n & 1) | ((n >> 2) & 6) : (n >> 3) & 3; };

    int kind = 0, t0 = 0, head = 0;  // 0 query, 1 key, 2 value; first token; head
    const __nv_bfloat16* rows[2];
    bool live[2];
    uint4 raw[2][KS];
    auto load = [&](int tile) {
        kind = tile < kv_tiles ? 1 : tile < 2 * kv_tiles ? 2 : 0;
        if (kind == 0) {
            const long long r0 = static_cast<long long>(tile - 2 * kv_tiles) * 16 + g;
            t0 = tile - 2 * kv_tiles;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                live[i] = r0 + 8 * i < p.q_rows;
                rows[i] = p.q + (r0 + 8 * i) * D;
            }
        } else {
            const unsigned kt = static_cast<unsigned>(kind == 1 ? tile : tile - kv_tiles);
            t0 = static_cast<int>(kt / static_cast<unsigned>(p.n_kv_heads));
            head = static_cast<int>(kt - static_cast<unsigned>(t0) * p.n_kv_heads);
            t0 *= 16;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int t = t0 + g + 8 * i;
                live[i] = t < T;
                rows[i] = (kind == 1 ? p.k : p.v) + (static_cast<long long>(t) * p.n_kv_heads + head) * D;
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int b = 0; b < KS; ++b)
                raw[i][b] = live[i] ? *reinterpret_cast<const uint4*>(rows[i] + 32 * b + 8 * c) : make_uint4(0u, 0u, 0u, 0u);
    };
    griddep_wait();  // launched with programmatic stream serialization
    griddep_launch_dependents();
    const int apart = warp * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);
    const int full = p.together ? tiles / stride * stride : 0;  // the rounds in which every warp has a tile
    int tile = p.together ? static_cast<int>(blockIdx.x) * kTileWarps + warp : apart;
    if (tile < tiles) load(tile);  // on its way while U_C is staged
    for (int i = threadIdx.x; i < D * (D / 16); i += kTileWarps * 32) {
        // the reduction's order: of 32 bytes first the even words, then the odd ones
        const int n = i / (D / 16), j = i % (D / 16);
        const uint4* src = reinterpret_cast<const uint4*>(p.wq + n * D) + (j & ~1);
        const uint4 x = src[0], y = src[1];
        *reinterpret_cast<uint4*>(w_s + n * D + ((j ^ swizzle(n)) << 4)) = j & 1 ? make_uint4(x.y, x.w, y.y, y.w) : make_uint4(x.x, x.z, y.x, y.z);
    }
    for (int i = threadIdx.x; i < D; i += kTileWarps * 32) su_s[i] = p.s_u[i];
    __syncthreads();
    const int w_row = 8 * ((lane & 7) >> 1) + (lane & 1) + 2 * (lane >> 4);  // of a block: the lane's ldmatrix row
    uint32_t w_addr[2][KS];  // of block 0: products 0 and 1, or 2 and 3
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
            w_addr[h][ks] = smem_u32(w_s) + (w_row + 4 * h) * D + (((2 * ks + ((lane >> 3) & 1)) ^ swizzle(w_row + 4 * h)) << 4);

    while (tile < tiles) {
        if (tile < full) __syncthreads();  // together: all of the CTA's warps are in the round
        const int now = kind, tok = t0, h = head;
        const bool ok0 = live[0], ok1 = live[1];
        if (now != 0) {
            if (lane < 16)
                rec.slot[lane] = tok + lane < T ? cache_slot<D>(tok + lane, h, p.n_kv_heads, p.n_seqs, p.capacity, p.seq_ids, p.positions, p.status)
                                                : -1;
        }
        auto pairs_of = [](uint4 u, f2* x) {
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
        };
        tile = tile < full && tile + stride >= full ? full + apart : tile + stride;
        if (now == 2) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                f2 x[D / 8];
#pragma unroll
                for (int b = 0; b < KS; ++b) pairs_of(raw[i][b], x + 4 * b);
                quantize_record<D>(x, c, rec, g + 8 * i);
            }
            if (tile < tiles) load(tile);
            __syncwarp();
            flush_records<D>(rec, p.cache, 1, lane);
            __syncwarp();
            continue;
        }
        // ---- symmetric INT8 codes, packed as the A fragments: a[ks][0] row g, [1] row g + 8: the first four elements of eight;
        // [2], [3]: the others
        uint32_t a[KS][4];
        float sx[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            f2 x[D / 8];
            float m = 0.f;
#pragma unroll
            for (int b = 0; b < KS; ++b) pairs_of(raw[i][b], x + 4 * b);
#pragma unroll
            for (int j = 0; j < D / 8; ++j) {
                const float2 u = unpack2(x[j]);
                m = fmaxf(m, fmaxf(fabsf(u.x), fabsf(u.y)));
            }
            m = quad_max(m);
            const float s = __fdiv_rn(m, 127.f), inv = s > 0.f ? __frcp_rn(s) : 0.f;
            sx[i] = s;
            const bool exact = s > 0.f && needs_division(inv);
#pragma unroll
            for (int b = 0; b < KS; b += 2) {
                uint32_t t[16];
                round_codes<16>(x + 4 * b, s, inv, exact, -128.f, 127.f, t);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    a[b + (j >> 1)][2 * (j & 1) + i] = s > 0.f ? low_bytes(t[4 * j], t[4 * j + 1], t[4 * j + 2], t[4 * j + 3]) : 0u;
            }
        }
        // ---- y = x W_C^T, a block of 32 columns at a time: the lane gets columns 32 b + 8c .. + 7 of rows g and g + 8
        auto product = [&](int b, f2 (&y0)[4], f2 (&y1)[4]) {
            const float4 u0 = *reinterpret_cast<const float4*>(su_s + 32 * b + 8 * c), u1 = *reinterpret_cast<const float4*>(su_s + 32 * b + 8 * c + 4);
            const f2 u[4] = {pack2(u0.x, u0.y), pack2(u0.z, u0.w), pack2(u1.x, u1.y), pack2(u1.z, u1.w)};
            const f2 s0 = pack2(sx[0], sx[0]), s1 = pack2(sx[1], sx[1]);
            int acc[4][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t w[4];
                    ldsm4(w, w_addr[h][ks] + b * 32 * D);
                    mma_s8(acc[2 * h], a[ks], w[0], w[1]);
                    mma_s8(acc[2 * h + 1], a[ks], w[2], w[3]);
                }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                y0[j] = mul2(pack2(static_cast<float>(acc[j][0]), static_cast<float>(acc[j][1])), mul2(s0, u[j]));
                y1[j] = mul2(pack2(static_cast<float>(acc[j][2]), static_cast<float>(acc[j][3])), mul2(s1, u[j]));
            }
        };
        if (now == 0) {
            if (tile < tiles) load(tile);
            __half* dst = p.q_out + (static_cast<long long>(tok) * 16 + g) * D + 8 * c;
#pragma unroll 1  // the code of a kind stays small
            for (int b = 0; b < KS; ++b) {
                f2 y[2][4];
                product(b, y[0], y[1]);
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (i == 0 ? ok0 : ok1)
                        *reinterpret_cast<uint4*>(dst + 8 * i * D + 32 * b) =
                            make_uint4(half_pair(y[i][0]), half_pair(y[i][1]), half_pair(y[i][2]), half_pair(y[i][3]));
            }
            continue;
        }
        f2 y[2][D / 8];
#pragma unroll
        for (int b = 0; b < KS; ++b) {
            f2 y0[4], y1[4];
            product(b, y0, y1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                y[0][4 * b + j] = y0[j];
                y[1][4 * b + j] = y1[j];
            }
        }
        quantize_record<D>(y[0], c, rec, g);
        quantize_record<D>(y[1], c, rec, g + 8);
        if (tile < tiles) load(tile);
        __syncwarp();
        flush_records<D>(rec, p.cache, 0, lane);
        __syncwarp();
    }
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// One warp per head vector, lane l owning coefficients l + 32 i; items: queries, keys, values.
template <int D>
__global__ void __launch_bounds__(kWarps * 32) head_vector_kernel(const ProjectParams p) {
    using H = Head<D>;
    constexpr int N = D / 32;
    __shared__ __align__(16) uint8_t w_s[D * H::kWStride];
    __shared__ float su_s[D];
    __shared__ __align__(16) int8_t xs_s[kWarps][D];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long total = p.q_rows + 2 * p.kv_rows, step = static_cast<long long>(gridDim.x) * kWarps;
    long long item = static_cast<long long>(blockIdx.x) * kWarps + warp;
    auto locate = [&](long long it, int& kind, long long& row) {
        kind = it < p.q_rows ? 0 : it < p.q_rows + p.kv_rows ? 1 : 2;  // query, key, value
        row = kind == 0 ? it : kind == 1 ? it - p.q_rows : it - p.q_rows - p.kv_rows;
    };
    griddep_wait();  // launched with programmatic stream serialization
    griddep_launch_dependents();
    int kind = 0;
    long long row = 0;
    float x[N];
    auto load = [&] {
        const __nv_bfloat16* src = (kind == 0 ? p.q : kind == 1 ? p.k : p.v) + row * D + lane;
#pragma unroll
        for (int i = 0; i < N; ++i) x[i] = __bfloat162float(src[32 * i]);
    };
    if (item < total) {
        locate(item, kind, row);
        load();  // on its way while U_C is staged
    }
    stage_uc<D>(p.wq, p.s_u, w_s, su_s);
    __syncthreads();
    for (; item < total; item += step) {
        long long slot = -1;
        if (kind != 0) {
            if (lane == 0) {
                const unsigned t = static_cast<unsigned>(row) / static_cast<unsigned>(p.n_kv_heads);
                slot = cache_slot<D>(static_cast<int>(t), static_cast<int>(row - static_cast<long long>(t) * p.n_kv_heads), p.n_kv_heads, p.n_seqs,
                                     p.capacity, p.seq_ids, p.positions, p.status);
            }
            slot = __shfl_sync(0xffffffffu, slot, 0);
        }
        float y[N];
#pragma unroll
        for (int i = 0; i < N; ++i) y[i] = x[i];
        if (kind != 2) {  // y = x U_C through the 8-bit product
            float m = 0.f;
#pragma unroll
            for (int i = 0; i < N; ++i) m = fmaxf(m, fabsf(x[i]));
            const float s = __fdiv_rn(warp_max(m), 127.f);
            const float inv = s > 0.f ? __frcp_rn(s) : 0.f;
            const bool exact = needs_division(inv);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < N; ++i)
                xs_s[warp][lane + 32 * i] =
                    s > 0.f ? static_cast<int8_t>(static_cast<int>(code_rn(x[i], s, inv, exact, 0.5f - 0.000030517578125f))) : 0;
            __syncwarp();
            int acc[N];
#pragma unroll
            for (int i = 0; i < N; ++i) acc[i] = 0;
#pragma unroll 2
            for (int k = 0; k < D / 16; ++k) {
                const int4 xc = *reinterpret_cast<const int4*>(xs_s[warp] + 16 * k);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int4 w = *reinterpret_cast<const int4*>(w_s + (lane + 32 * i) * H::kWStride + 16 * k);
                    acc[i] = __dp4a(xc.x, w.x, __dp4a(xc.y, w.y, __dp4a(xc.z, w.z, __dp4a(xc.w, w.w, acc[i]))));
                }
            }
#pragma unroll
            for (int i = 0; i < N; ++i) y[i] = __fmul_rn(static_cast<float>(acc[i]), __fmul_rn(s, su_s[lane + 32 * i]));
        }
        if (kind == 0) {
#pragma unroll
            for (int i = 0; i < N; ++i) p.q_out[row * D + lane + 32 * i] = __float2half_rn(y[i]);
        } else if (slot >= 0) {  // the whole warp
            const bool in8 = lane < H::kR8;  // of coefficient `lane`; the others are all in the 4-bit segment
            float lo4 = in8 ? INFINITY : y[0], hi4 = in8 ? -INFINITY : y[0];
#pragma unroll
            for (int i = 1; i < N; ++i) { lo4 = fminf(lo4, y[i]); hi4 = fmaxf(hi4, y[i]); }
            const Asym q8(warp_min(in8 ? y[0] : INFINITY), warp_max(in8 ? y[0] : -INFINITY), 255.f);
            const Asym q4(warp_min(lo4), warp_max(hi4), 15.f);
            uint8_t* half = p.cache + (slot & ~31ll) + (kind == 2 ? H::kHalf : 0);
            const int ps = static_cast<int>(slot & 31);
            uint8_t* c4 = half + H::kC8 + ps * H::kB4;
#pragma unroll
            for (int i = 0; i < N; ++i) {  // a 4-bit coefficient j is nibble j - kR8; kR8 is even, so pairs start at even lanes
                const uint32_t code = i == 0 && in8 ? q8.code(y[i], 255.f) : q4.code(y[i], 15.f);
                const uint32_t next = __shfl_down_sync(0xffffffffu, code, 1);
                if (i == 0 && in8) half[ps * H::kR8 + lane] = static_cast<uint8_t>(code);
                else if ((lane & 1) == 0) c4[(lane + 32 * i - H::kR8) >> 1] = static_cast<uint8_t>(code | (next << 4));
            }
            if (lane == 0) *reinterpret_cast<float4*>(half + H::kC8 + H::kC4 + ps * 16) = make_float4(q8.s, q8.z, q4.s, q4.z);
        }
        if (item + step < total) {
            locate(item + step, kind, row);
            load();
        }
    }
}

// W_C = U_C^T [D][D] fp32 -> symmetric per-row INT8 (one warp per row; offline, true divisions).
template <int D>
__global__ void __launch_bounds__(32) uc_quantize_kernel(const float* __restrict__ W, int8_t* __restrict__ wq,
                                                         float* __restrict__ s_u) {
    const int row = blockIdx.x, lane = threadIdx.x;
    float x[D / 32], m = 0.f;
#pragma unroll
    for (int i = 0; i < D / 32; ++i) {
        x[i] = W[row * D + lane + 32 * i];
        m = fmaxf(m, fabsf(x[i]));
    }
    const float s = __fdiv_rn(warp_max(m), 127.f);
#pragma unroll
    for (int i = 0; i < D / 32; ++i)
        wq[row * D + lane + 32 * i] =
            s > 0.f ? static_cast<int8_t>(static_cast<int>(fminf(fmaxf(rintf(__fdiv_rn(x[i], s)), -127.f), 127.f))) : 0;
    if (lane == 0) s_u[row] = s;
}

template <int D>
cudaError_t launch_project(const ProjectParams& p, cudaStream_t st) {
    const long long vectors = p.q_rows + 2 * p.kv_rows;
    if (vectors == 0) return cudaSuccess;
    count_launch();
    if (vectors <= kFewVectors<D>) {
        const long long ctas = (vectors + kWarps - 1) / kWarps;
        return launch_programmatic(head_vector_kernel<D>, ctas < 148 * 8 ? ctas : 148 * 8, kWarps * 32, 0, st, p);
    }
    const long long T = p.n_kv_heads ? p.kv_rows / p.n_kv_heads : 0;
    const long long kv_tiles = 2 * ((T + 15) / 16) * p.n_kv_heads, tiles = (p.q_rows + 15) / 16 + kv_tiles;
    const long long ctas = (tiles + kTileWarps - 1) / kTileWarps;
    ProjectParams tp = p;
    tp.together = append_tiles_together(D, kv_tiles, tiles);
    static_assert(kTileWarps * 148 * 2 == kAppendWarps, "a round");
    return launch_programmatic(kv_project_kernel<D>, ctas < 148 * 2 ? ctas : 148 * 2, kTileWarps * 32, 0, st, tp);
}

}  // namespace

cudaError_t launch_uc_quantize(const float* W_C, int d_head, int8_t* wq, float* s_u, cudaStream_t st) {
    count_launch();
    if (d_head == 64) uc_quantize_kernel<64><<<64, 32, 0, st>>>(W_C, wq, s_u);
    else uc_quantize_kernel<128><<<128, 32, 0, st>>>(W_C, wq, s_u);
    return cudaGetLastError();
}

// q (q_rows head vectors) and / or k, v (T tokens) in one launch; either part may be absent (null / 0).
cudaError_t launch_qkv_project_append(const resq_kv_cache_t* cache, int d_head, const void* q, long long q_rows, void* q_out,
                                      const void* k, const void* v, long long T, const int32_t* seq_ids,
                                      const int32_t* positions, const int8_t* wq, const float* s_u, cudaStream_t st) {
    ProjectParams p{};
    p.q = static_cast<const __nv_bfloat16*>(q);
    p.q_rows = q ? q_rows : 0;
    p.q_out = static_cast<__half*>(q_out);
    p.wq = wq;
    p.s_u = s_u;
    p.status = device_status_ptr();
    if (cache && k) {
        p.k = static_cast<const __nv_bfloat16*>(k);
        p.v = static_cast<const __nv_bfloat16*>(v);
        p.kv_rows = T * cache->n_kv_heads;
        p.cache = static_cast<uint8_t*>(cache->data);
        p.n_seqs = cache->n_seqs;
        p.n_kv_heads = cache->n_kv_heads;
        p.capacity = cache->capacity;
        p.seq_ids = seq_ids;
        p.positions = positions;
    }
    return d_head == 64 ? launch_project<64>(p, st) : launch_project<128>(p, st);
}

}  // namespace resq
