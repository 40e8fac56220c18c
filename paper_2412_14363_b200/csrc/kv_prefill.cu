// Causal attention of a run of new tokens over the quantized KV cache (Section 4.3, Eq. 8; cache format of
// Section 5.1) on the tcgen05 tensor cores: the prefill form, where every cache block is read once per CTA instead of
// once per query.  d_head = 128 and 64.
//
// Rows are (token, query head) pairs that share a KV head, tokens ascending; a tile is 128 of them.  A CTA walks the cache of its
// sequence in steps of 64 positions (two cache blocks).  Roles:
//   expand   3 warps: raw blocks (bulk copies, two steps ahead) -> operand tiles [position][coefficient], keys K-major, values
//            N-major (so neither is transposed), and the step's per-position constants; three stages.  The codes become exact
//            halves, centred (code - 128, code - 8); values at d = 64 become s (code - centre) as three bf16 parts.
//   mma      one warp: S8 and S4, the products of the two segments, into TMEM; later the output product with the weights taken
//            from TMEM.
//   softmax  2 or 4 threads per row, each with a share of the step's positions: score = s8 S8 + s4 S4 + (z8 + 128 s8) sum(q8) +
//            (z4 + 8 s4) sum(q4) in fp32 minus the row's reference (the part without S while S is on its way), p = 2^score,
//            and the operands of the output product over the scores in TMEM.
// d = 128: P8 = half(p s8_v 2^-E), P4 = half(p s4_v 2^-E) times the exact codes, sums of p and of p (z + c0 s) in fp32.  2^E is the
// largest finite value scale of the positions the CTA visits (read ahead of the walk), so the products stay in half's normal
// range.  The outputs are accumulated in TMEM.
// d = 64, whose outputs keep fp32's precision (relative error against 64 bits 0.8e-7 to 2.6e-7; the mma.sync tiles before 0.9e-7 to 3.3e-7):
// p as three bf16 parts of all its 24 bits (bf16 has fp32's range: a value scale 2^28 above the others' beside next to no weight
// costs nothing) times the parts of the values without their zero-points, six products, those left out below 2^-26.  The tensor core
// truncates its fp32 sums, so a step's product is added to the thread's registers, with rounding, and the zero-points, in which a
// common mean of the values lies, are summed in fp32.  The row's reference comes off a score last, when it is small.
// The reference of a row is the maximum of its first step and is raised only when a score exceeds it by 2^8; in that rare step the
// row's outputs are rescaled.  So there is one pass over the cache, and weights are no smaller against the row's maximum than
// 2^-8 of those with an exact one (d = 64: values are taken times 2^-8, so that no sum is larger than with weights up to 1).
// Two things are in flight, so that the products of one run under the softmax of the other: two steps of one tile, or (PAIR, d = 128,
// where there are tiles enough) two tiles.  A CTA may take a long and a short tile in turn; the roles run on from one to the other.
// With few CTAs a cluster splits the steps, and every rank merges the sums of a share of the rows through distributed shared memory.
//
// The coefficients of a 32-bit word of nibbles are kept in the order 0 4 1 5 2 6 3 7 (one shift and mask per pair of
// tile elements); the query tile is written in the same order and the output un-permuted on the way out.
// Positions beyond a row's own are masked by selection in the scores; the constants of positions past the tile's last are
// zeroed by selection, and so are a value's constants that are not finite (they would turn a hidden position's weight of 0 into
// NaN); the first such position is noted for the rows that do see it.  So unwritten cache positions of a loaded block, and later
// tokens, may hold anything.  All waits are bounded; after a failed wait every role leaves its loop, copies and products in
// flight are waited for, and TMEM is freed.
//
// What bounds it: the instructions of softmax and expansion (60 % of the issue slots, 63 at d = 64) and the latency of their chains.
// us per step: d = 128, two tiles together 2.03, one tile 1.33; d = 64, one tile 1.87 (1.62 with the zero-points inside the values'
// parts).  The expansion sets the pace where its words are read, converted and written one by one; so all words are on their way
// first, with addresses of a register and a constant.  Divisions by the group size took 5 us of a call, outputs stored row by row 2 us.
// us, 32 query / 8 KV heads: d = 128, 2048 tokens behind 4096 400 -> 349 (1310 with one 128-row tile per CTA in two passes), 1000
// tokens 49 -> 37; d = 64, 1000 tokens 60 -> 43 (mma.sync tiles of 64 rows), 2048 behind 4096 828 -> 580.  A run of one step (32
// tokens of 8 / 8 heads at position 0: 7.2 -> 8.0) and, at d = 64, of a few tokens there (5.6 -> 6.9) is slower than before: more of it
// is set-up.
#include "centred_codes.cuh"
#include "internal.h"
#include "packed_fp32.cuh"
#include "plans.h"
#include "ptx.cuh"

#include <cuda_fp16.h>

#include <cfloat>
#include <climits>

namespace resq {
namespace {

constexpr int kRows = 128;          // rows of a tile = TMEM lanes
constexpr int kStep = 64;           // cache positions per step
constexpr int kStages = 3;          // expanded steps
constexpr int kExpandWarps = 3;
constexpr uint32_t kTmemCols = 512, kColS4 = 64;  // the 4-bit segment's scores behind the 8-bit one's
constexpr float kSlack = 8.f;       // log2 of how far a score may rise above a row's first maximum before its reference is raised

// What depends on the head width.  Operand tiles have rows of 128 bytes (64 coefficients of 16 bits).
template <int D>
struct Head {
    static constexpr int kR8 = D / 8, kB4 = (D - kR8) / 2;                  // coefficients in 8 bits, bytes of the 4-bit ones
    static constexpr int kOffK4 = 32 * kR8, kOffKm = kOffK4 + 32 * kB4, kOffV8 = kOffKm + 512;  // parts of a cache block
    static constexpr int kOffV4 = kOffV8 + kOffK4, kOffVm = kOffV8 + kOffKm, kBlockBytes = 2 * kOffV8;
    static constexpr int kRawBytes = 2 * kBlockBytes;
    static constexpr int kTile = kStep * 128;                               // an operand tile of 64 positions
    static constexpr int kQBytes = D / 64 * kRows * 128;
    // A stage.  D = 128: keys in two halves of 64 coefficients, 4-bit values in two halves (64 and 48), 8-bit values.
    // D = 64: 4-bit keys in chunks (of 8 coefficients) 1-7, 8-bit keys in chunk 0 of a tile of their own, the chunks beside them 0;
    // three tiles that add up to the values (chunks 0-6 the 4-bit segment, chunk 7 the other).
    static constexpr int kStageBytes = 5 * kTile, kOffStageV4 = 2 * kTile, kOffStageV8 = 4 * kTile;
    static constexpr int kWeights = D == 128 ? 2 : 3;                       // 16-bit operands of a weight
    static constexpr int kRecPitch = D + 4;                                 // floats per row of a record: sums, reference, sum of weights
};
static_assert(Head<128>::kBlockBytes == RESQ_KV_BLOCK_BYTES && Head<128>::kOffVm == 5120, "block layout");

struct Shared {
    // per stage and pair of positions: keys (s8 s8 s4 s4) (z8 z8 z4 z4) times log2(e) / sqrt(d), the zero-points with the
    // centre; values, D = 128: (s8 s8 s4 s4) times 2^-E, (z8 z8 z4 z4) with the centre
    float4 col_k[kStages][kStep], col_v[kStages][kStep];
    float2 row_sum[2][kRows];   // of the query, by tile: 8-bit, 4-bit segment
    // what the threads of a row tell each other (PAIR: [tile][thread], else [thread]): sums of weights and zero-points, maxima (w)
    float4 row_part[4][kRows];
    float warp_max[20];           // one per warp
    int bad8, bad4;  // the first position visited whose value constants of the 8-bit / 4-bit segment are infinite or NaN
    uint64_t raw_full[2], kv_full[kStages], kv_empty[kStages], s_full[2], s_read[2], p_full[2], pv_done[2], drain;
    uint32_t tmem_base;
    int abort_flag;
};

// WAYS: threads of a row, each with that share of a step's positions and of the output.  PAIR: two tiles in flight with one score
// buffer each; otherwise two steps of one.
template <int D, int WAYS, bool PAIR>
struct Geometry {
    static constexpr int kGroupWarps = 4 * WAYS;  // of a tile
    static constexpr int kSoftmaxWarps = kGroupWarps * (PAIR ? 2 : 1), kMmaWarp = kSoftmaxWarps + kExpandWarps, kThreads = 32 * (kMmaWarp + 1);
    static constexpr int kPart = kStep / WAYS, kPairs = kPart / 2, kOutCols = D / WAYS;
    static constexpr size_t kTiles = 2 * static_cast<size_t>(Head<D>::kQBytes) + kStages * Head<D>::kStageBytes;
    // a warp's outputs on their way from rows to contiguous stores: over the tile's query where that is large enough
    static constexpr int kOutBlock = kOutCols < 32 ? kOutCols : 32, kOutBytes = 32 * kOutBlock * 4;
    static constexpr size_t kOutStage = D == 128 ? 0 : kSoftmaxWarps * kOutBytes;
    static_assert(D == 64 || kGroupWarps * kOutBytes <= Head<D>::kQBytes, "outputs fit");
    static constexpr size_t kSmem = 1024 + kTiles + kOutStage + 2 * Head<D>::kRawBytes + sizeof(Shared);
    static_assert(kSmem <= 227 * 1024 && kMmaWarp < 20 && (!PAIR || (D == 128 && WAYS == 2)), "one CTA per SM");
    static_assert(kTiles >= static_cast<size_t>(kRows) * Head<D>::kRecPitch * 4, "records fit");
    // TMEM: score buffers (8-bit and 4-bit segment, the weights over them; PAIR: one per tile, else one per stage), then the outputs:
    // PAIR: one per tile; D = 128: one, which the tensor core adds up; D = 64: two, by turns
    static constexpr uint32_t kBufCols = 128, kColOut = (PAIR ? 2 : kStages) * kBufCols, kOutPitch = PAIR ? 128 : D == 128 ? 0 : 64;
    static_assert(kColOut + kOutPitch + D <= kTmemCols, "TMEM");
};

struct PrefillParams {
    const uint8_t* blocks;  // first cache block of the sequence (KV head 0)
    size_t head_stride;     // bytes between the KV heads of the sequence
    const __half* q;        // [T][Hq][D]
    float* out;             // [T][Hq][D]
    int T, Hq, Hkv, g, pos0, splits, tiles;  // splits: CTAs of a cluster; tiles: per CTA, in turn, 1 or 2
    unsigned g_inv;  // 2^32 / g rounded up
    int* status;
};

__host__ __device__ constexpr uint32_t make_idesc_f16(int M, int N) {  // f16 x f16 -> f32, K-major A and B
    return (1u << 4) | (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
constexpr uint32_t kBNMajor = 1u << 16;

// Two pairs from shared memory, where the program has it (hoisted reads would not fit the registers).
struct f2x2 {
    f2 x, y;
};
__device__ __forceinline__ f2x2 lds_pairs(uint32_t addr) {
    f2x2 d;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(d.x), "=l"(d.y) : "r"(addr));
    return d;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t d;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(d) : "r"(addr));
    return d;
}
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 d;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(d.x), "=r"(d.y) : "r"(addr));
    return d;
}
__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
    float4 d;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(d.x), "=f"(d.y), "=f"(d.z), "=f"(d.w) : "r"(addr));
    return d;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts_f(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }
// Two floats as three pairs of bf16 that add up to all of their 24 bits: each part is what the ones before leave, rounded.
__device__ __forceinline__ uint32_t bf16_pair(f2 v) {
    const float2 f = unpack2(v);
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(f.y), "f"(f.x));
    return d;
}
__device__ __forceinline__ f2 minus_pair(f2 v, uint32_t pair) {
    return fma2(pack2(__uint_as_float(pair << 16), __uint_as_float(pair & 0xFFFF0000u)), pack2(-1.f, -1.f), v);
}
__device__ __forceinline__ void split_bf16(f2 v, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    p0 = bf16_pair(v);
    v = minus_pair(v, p0);
    p1 = bf16_pair(v);
    p2 = bf16_pair(minus_pair(v, p1));
}

// One step of the expanding warps, lane = position of a block.  Warps 0 and 1 take a block each: the words of nibbles of the keys and
// the first of the values'; warp 2 the rest of both blocks.  Every address is a register and a constant, and a warp's words are
// all on their way before the first is written: few warps expand, so the length of their chain counts.  The constants of
// positions from n_valid on, and a value's that are not finite, become 0; bad8 / bad4 note the latter (j0: the first position).
template <int D>
__device__ __forceinline__ void expand_step(uint32_t raw, uint32_t stage, uint32_t col_k, uint32_t col_v, int warp, int lane,
                                            int n_valid, float p_scale, int j0, int* bad8, int* bad4) {
    using H = Head<D>;
    constexpr int kWords = H::kB4 / 4, kFirst = D == 128 ? 8 : 5, kByteChunks = H::kR8 / 8;
    const float kScore = 1.4426950408889634f * (D == 128 ? 0.08838834764831845f : 0.125f);  // log2(e) / sqrt(D)
    // a position's row of an operand tile, chunk c at row ^ (c << 4) (128-byte swizzle; rows are 128-byte aligned)
    auto row_of = [&](int blk) { return stage + blk * (32 * 128) + lane * 128 + ((lane & 7) << 4); };
    auto key_chunk = [&](uint32_t row, int w) {
        constexpr int kAt = D == 128 ? 2 : 1;
        return (row ^ (((w + kAt) & 7) << 4)) + ((w + kAt) >> 3) * H::kTile;
    };
    auto constants = [&](float4 c, int blk, bool is_v, float fs, float fz) {
        const int j = 32 * blk + lane;
        if (j >= n_valid) c = make_float4(0.f, 0.f, 0.f, 0.f);
        const float up = D == 64 && is_v ? 0.5f : 0.f;  // value_parts
        c.y = fmaf(128.f - up, c.x, c.y);
        c.w = fmaf(8.f - up, c.z, c.w);
        if (is_v && !(fabsf(c.x) <= FLT_MAX && fabsf(c.y) <= FLT_MAX)) {
            c.x = c.y = 0.f;
            atomicMin(bad8, j0 + j);
        }
        if (is_v && !(fabsf(c.z) <= FLT_MAX && fabsf(c.w) <= FLT_MAX)) {
            c.z = c.w = 0.f;
            atomicMin(bad4, j0 + j);
        }
        return make_float4(c.x * fs, c.y * fz, c.z * fs, c.w * fz);
    };
    auto store_constants = [&](uint32_t col, int blk, float4 c) {  // pair j / 2, element j % 2 of each pair
        const uint32_t dst = col + (32 * blk + lane >> 1) * 32 + (lane & 1) * 4;
        sts_f(dst, c.x);
        sts_f(dst + 8, c.z);
        sts_f(dst + 16, c.y);
        sts_f(dst + 24, c.w);
    };
    // D = 64: eight values without their zero-point, s (code - centre), as three chunks of bf16.  The centre is half a code lower, in the
    // middle of the codes: sums that the tensor core truncates shall not lean to one side.
    auto value_parts = [&](uint32_t at, const f2 (&code)[4], float scale) {
        uint32_t p[3][4];
        const f2 half = pack2(0.5f * scale, 0.5f * scale);
#pragma unroll
        for (int m = 0; m < 4; ++m) split_bf16(fma2(code[m], pack2(scale, scale), half), p[0][m], p[1][m], p[2][m]);
#pragma unroll
        for (int k = 0; k < 3; ++k) sts128(at + k * H::kTile, make_uint4(p[k][0], p[k][1], p[k][2], p[k][3]));
    };
    auto centred_floats = [&](uint4 h, f2 (&code)[4]) {
        const uint32_t v[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v[m]));
            code[m] = pack2(f.x, f.y);
        }
    };
    auto value_word = [&](uint32_t row, int w, uint32_t word, float4 c) {
        if constexpr (D == 128) {
            sts128((row ^ ((w & 7) << 4)) + H::kOffStageV4 + (w >> 3) * H::kTile, nibbles_centred(word));
        } else {
            f2 code[4];
            centred_floats(nibbles_centred(word), code);
            value_parts((row ^ (w << 4)) + H::kOffStageV4, code, c.z);
        }
    };
    if (warp < 2) {
        const uint32_t src = raw + warp * H::kBlockBytes, row = row_of(warp);
        uint32_t k[kWords], v[kFirst];
        float4 mk, mv;
        uint2 k8;
#pragma unroll
        for (int w = 0; w < kWords; ++w) k[w] = lds32(src + lane * H::kB4 + H::kOffK4 + 4 * w);
#pragma unroll
        for (int w = 0; w < kFirst; ++w) v[w] = lds32(src + lane * H::kB4 + H::kOffV4 + 4 * w);
        if (D == 64) {
            mk = lds_f4(src + H::kOffKm + lane * 16);
            mv = lds_f4(src + H::kOffVm + lane * 16);
            k8 = lds64(src + lane * H::kR8);
        }
#pragma unroll
        for (int w = 0; w < kWords; ++w) sts128(key_chunk(row, w), nibbles_centred(k[w]));
        if (D == 64) {
            sts128(row + H::kTile, bytes_centred(k8));
            store_constants(col_k, warp, constants(mk, warp, false, kScore, kScore));
            mv = constants(mv, warp, true, p_scale, p_scale);
        }
#pragma unroll
        for (int w = 0; w < kFirst; ++w) value_word(row, w, v[w], mv);
        return;
    }
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        const uint32_t src = raw + blk * H::kBlockBytes, row = row_of(blk);
        uint32_t v[kWords - kFirst];
        uint2 k8[kByteChunks], v8[kByteChunks];
        float4 mk, mv = lds_f4(src + H::kOffVm + lane * 16);
        if (D == 128) mk = lds_f4(src + H::kOffKm + lane * 16);
#pragma unroll
        for (int w = kFirst; w < kWords; ++w) v[w - kFirst] = lds32(src + lane * H::kB4 + H::kOffV4 + 4 * w);
#pragma unroll
        for (int c = 0; c < kByteChunks; ++c) {
            if (D == 128) k8[c] = lds64(src + lane * H::kR8 + 8 * c);
            v8[c] = lds64(src + lane * H::kR8 + H::kOffV8 + 8 * c);
        }
        mv = constants(mv, blk, true, p_scale, D == 128 ? 1.f : p_scale);
        if (D == 128) store_constants(col_k, blk, constants(mk, blk, false, kScore, kScore));
        store_constants(col_v, blk, mv);
#pragma unroll
        for (int w = kFirst; w < kWords; ++w) value_word(row, w, v[w - kFirst], mv);
        if constexpr (D == 128) {
#pragma unroll
            for (int c = 0; c < kByteChunks; ++c) {
                sts128(row ^ (c << 4), bytes_centred(k8[c]));
                sts128((row ^ (c << 4)) + H::kOffStageV8, bytes_centred(v8[c]));
            }
        } else {
            f2 code[4];
            centred_floats(bytes_centred(v8[0]), code);
            value_parts((row ^ (7 << 4)) + H::kOffStageV4, code, mv.x);
        }
    }
}

// Running state of a row over the positions of one of its threads, by the parity of the position.
struct RowState {
    float m;       // reference, log2 units; -inf: no position seen yet.  The same in all
    f2 l, z8, z4;  // sums of p and of p times the zero-points (with the centre)
};

// Constants of a pair of positions (Shared::col_k, col_v).
__device__ __forceinline__ f2x2 pair_scales(uint32_t col, int pair) { return lds_pairs(col + 32 * pair); }
__device__ __forceinline__ f2x2 pair_zeros(uint32_t col, int pair) { return lds_pairs(col + 32 * pair + 16); }

// What the zero-points give to the scores of the thread's positions (D = 128: minus the row's reference), as pairs: known before the
// products.
template <int D, int PAIRS>
__device__ __forceinline__ void step_offsets(f2 (&sc)[PAIRS], uint32_t col_k, f2 q8, f2 q4, float neg_m) {
    const f2 nm = pack2(neg_m, neg_m);
#pragma unroll
    for (int pr = 0; pr < PAIRS; ++pr) {
        const f2x2 z = pair_zeros(col_k, pr);
        sc[pr] = fma2(z.x, q8, D == 128 ? fma2(z.y, q4, nm) : mul2(z.y, q4));
    }
}

// The scores on top of that, against the row's reference; returns their maximum.  D = 64 takes the reference off last: what is left of
// the scores that count is small and so is its rounding.  tmem_s, col_k: at the first of the positions; those beyond `last` are
// hidden from the row.
template <int D, bool MASKED, int PAIRS>
__device__ __forceinline__ float step_scores(f2 (&sc)[PAIRS], uint32_t tmem_s, uint32_t col_k, float neg_m, int last) {
    const f2 nm = pack2(neg_m, neg_m);
    float mx = -INFINITY;
#pragma unroll
    for (int part = 0; part < PAIRS / 4; ++part) {  // eight positions
        uint32_t a8[8], a4[8];
        f2x2 s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = pair_scales(col_k, 4 * part + i);
        tmem_ld8x2(tmem_s + 8 * part, tmem_s + kColS4 + 8 * part, a8, a4);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            sc[4 * part + i] = fma2(s[i].y, pack2(__uint_as_float(a4[2 * i]), __uint_as_float(a4[2 * i + 1])), sc[4 * part + i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int pr = 4 * part + i;
            sc[pr] = fma2(s[i].x, pack2(__uint_as_float(a8[2 * i]), __uint_as_float(a8[2 * i + 1])), sc[pr]);
            if (D == 64) sc[pr] = add2(sc[pr], nm);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int pr = 4 * part + i;
            float2 f = unpack2(sc[pr]);
            if (MASKED) {
                if (2 * pr > last) f.x = -INFINITY;
                if (2 * pr + 1 > last) f.y = -INFINITY;
                sc[pr] = pack2(f.x, f.y);
            }
            mx = fmaxf(mx, fmaxf(f.x, f.y));
        }
    }
    return mx;
}

// Weights of those positions: their sums into the row's state, the operands of the output product over the scores in TMEM.
// tmem_p, col_v: at the first of the positions.  The exponentials first, in place: one behind the other they would each wait for
// the special function unit.
template <int D, int PAIRS>
__device__ __forceinline__ void step_weights(RowState& st, f2 (&sc)[PAIRS], uint32_t tmem_p, uint32_t col_v) {
    constexpr int kStore = 4;  // pairs per store
    f2x2 s[2], z[2];
    RowState sum{0.f, 0ull, 0ull, 0ull};  // D = 64: of the step, so that most of the additions round small sums
    RowState& to = D == 128 ? st : sum;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (D == 128) s[i] = pair_scales(col_v, i);
        z[i] = pair_zeros(col_v, i);
    }
#pragma unroll
    for (int pr = 0; pr < PAIRS; ++pr) {
        const float2 f = unpack2(sc[pr]);
        sc[pr] = pack2(exp2_approx(f.x), exp2_approx(f.y));
    }
#pragma unroll
    for (int g = 0; g < PAIRS / kStore; ++g) {
        uint32_t w[Head<D>::kWeights][kStore];
#pragma unroll
        for (int i = 0; i < kStore; ++i) {
            const int pr = kStore * g + i, b = pr & 1;
            to.l = add2(to.l, sc[pr]);
            to.z8 = fma2(sc[pr], z[b].x, to.z8);
            to.z4 = fma2(sc[pr], z[b].y, to.z4);
            if constexpr (D == 128) {
                w[0][i] = half_pair(mul2(sc[pr], s[b].x));
                w[1][i] = half_pair(mul2(sc[pr], s[b].y));
                if (pr + 2 < PAIRS) s[b] = pair_scales(col_v, pr + 2);
            } else {
                split_bf16(sc[pr], w[0][i], w[1][i], w[2][i]);
            }
            if (pr + 2 < PAIRS) z[b] = pair_zeros(col_v, pr + 2);
        }
#pragma unroll
        for (int k = 0; k < Head<D>::kWeights; ++k) tmem_st4(tmem_p + 32 * k + kStore * g, w[k]);
    }
    if (D == 64) {
        st.l = add2(st.l, sum.l);
        st.z8 = add2(st.z8, sum.z8);
        st.z4 = add2(st.z4, sum.z4);
    }
}

// Barrier of the THREADS / 32 warps that share 32 rows; whether the predicate holds in any of their threads.
template <int THREADS>
__device__ __forceinline__ bool group_any(int id, bool pred) {
    int any;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\t"
                 "selp.b32 %0, 1, 0, q;\n\t}" : "=r"(any) : "r"(pred ? 1 : 0), "r"(id), "n"(THREADS) : "memory");
    return any != 0;
}

template <int D, int WAYS, bool PAIR>
__global__ void __launch_bounds__(Geometry<D, WAYS, PAIR>::kThreads, 1) attention_prefill_kernel(const PrefillParams p) {
    using H = Head<D>;
    using G = Geometry<D, WAYS, PAIR>;
    constexpr float kUnit = D == 128 ? 1.f : 256.f;  // of the outputs before their division
    constexpr int kThreads = G::kThreads, kSoftmaxWarps = G::kSoftmaxWarps, kMmaWarp = G::kMmaWarp;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + (-smem_u32(smem_raw) & 1023u);  // (through an integer the compiler would lose that it is shared memory)
    uint8_t* Qs = base;
    uint8_t* stages = Qs + 2 * H::kQBytes;
    uint8_t* out_stage_d64 = stages + kStages * H::kStageBytes;
    uint8_t* raw = out_stage_d64 + G::kOutStage;
    Shared* sh = reinterpret_cast<Shared*>(raw + 2 * H::kRawBytes);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int splits = PAIR ? 1 : p.splits;
    const int rank = PAIR ? 0 : static_cast<int>(blockIdx.x % splits), item = static_cast<int>(blockIdx.x / splits);
    const int kvh = item % p.Hkv, n_tiles = (p.T * p.g + kRows - 1) / kRows;
    const uint8_t* blocks = p.blocks + static_cast<size_t>(kvh) * p.head_stride;
    // token of row R, and the row's place among the head vectors [token][head] (a division by g by its reciprocal: rows are below 2^32 / g)
    auto token_of = [&](int R) { return p.g == 1 ? R : static_cast<int>(__umulhi(static_cast<unsigned>(R), p.g_inv)); };
    auto head_vector = [&](int R) {
        const int t = token_of(R);
        return static_cast<size_t>(t) * p.Hq + kvh * p.g + (R - t * p.g);
    };
    auto positions_seen = [&](int tile) { return p.pos0 + min(p.T - 1, token_of(tile * kRows + kRows - 1)) + 1; };
    auto first_step = [&](int limit, int r) {  // of rank r's steps
        return static_cast<int>(static_cast<long long>((limit + kStep - 1) / kStep) * r / splits);
    };
    // long tiles of all heads first; a second one from the other end (an odd number of tiles: the middle one is alone)
    // (PAIR: two neighbours instead, which walk together)
    const int long_tile = PAIR ? (n_tiles - 1 | 1) - 2 * (item / p.Hkv) : n_tiles - 1 - item / p.Hkv;
    const int short_tile = PAIR ? long_tile - 1 : item / p.Hkv;
    const int tiles = !PAIR && p.tiles == 2 && short_tile < long_tile ? 2 : 1;
    struct Tile {
        int limit, first, n_steps;  // positions any row sees; this rank's steps
    };
    auto tile_of = [&](int ti) {
        Tile t;
        t.limit = positions_seen(ti == 0 ? long_tile : short_tile);
        t.first = first_step(t.limit, rank);
        t.n_steps = first_step(t.limit, rank + 1) - t.first;
        return t;
    };
    const Tile tile0 = tile_of(0);
    const int total_steps = tile0.n_steps + (tiles == 2 ? tile_of(1).n_steps : 0);
    // copies of the CTA's step N, counted over its tiles
    auto issue_load = [&](int N) {
        const bool second = N >= tile0.n_steps;
        const int b0 = 2 * (second ? N - tile0.n_steps : tile0.first + N);  // (two tiles: not split)
        const int n_blocks = ((second ? positions_seen(short_tile) : tile0.limit) + RESQ_KV_BLOCK - 1) / RESQ_KV_BLOCK;
        const uint32_t bytes = static_cast<uint32_t>(min(2, n_blocks - b0)) * H::kBlockBytes;
        mbar_arrive_expect_tx(&sh->raw_full[N & 1], bytes);
        bulk_load(raw + (N & 1) * H::kRawBytes, blocks + static_cast<size_t>(b0) * H::kBlockBytes, bytes, &sh->raw_full[N & 1]);
    };
    const bool loader = tid == 32 * kSoftmaxWarps;  // sets the barriers up and issues the copies

    if (loader) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh->raw_full[i], 1);
            mbar_init(&sh->s_full[i], 1);
            mbar_init(&sh->s_read[i], G::kGroupWarps);
            mbar_init(&sh->p_full[i], G::kGroupWarps);
            mbar_init(&sh->pv_done[i], 1);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&sh->kv_full[i], kExpandWarps);
            mbar_init(&sh->kv_empty[i], 1);
        }
        mbar_init(&sh->drain, 1);
        sh->abort_flag = 0;
        sh->bad8 = sh->bad4 = INT_MAX;
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        __syncwarp();
        tmem_alloc(&sh->tmem_base, kTmemCols);
        tmem_relinquish();
    }
    if (D == 64) {  // the chunks that stay 0 in every stage (Head)
        for (int i = tid; i < kStages * 2 * kStep; i += kThreads) {
            const int j = i & (kStep - 1), t = (i / kStep) & 1;  // chunk 0 of the 4-bit keys, chunk 1 of the 8-bit ones
            *reinterpret_cast<uint4*>(stages + (i / (2 * kStep)) * H::kStageBytes + t * H::kTile + j * 128 + ((t ^ (j & 7)) << 4)) =
                make_uint4(0, 0, 0, 0);
        }
    }

    griddep_wait();  // the set-up above ran under the tail of the preceding grid
    griddep_launch_dependents();
    if (loader)
        for (int N = 0; N < min(2, total_steps); ++N) issue_load(N);
    // ---- D = 128: the largest value scale of the positions visited
    float p_scale = D == 128 ? 1.f : 0.00390625f, out_scale = 1.f;
    if (D == 128) {
        float vmax = 0.f;
        const int limit = positions_seen(long_tile), end = min(limit, first_step(limit, rank + 1) * kStep);
        for (int j = first_step(limit, rank) * kStep + tid; j < end; j += kThreads) {
            const float4 m = reinterpret_cast<const float4*>(blocks + static_cast<size_t>(j >> 5) * H::kBlockBytes + H::kOffVm)[j & 31];
            // a scale that is not finite makes the rows that see it infinite or NaN whatever E is
            vmax = fmaxf(vmax, fmaxf(m.x <= FLT_MAX ? m.x : 0.f, m.z <= FLT_MAX ? m.z : 0.f));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if (lane == 0) sh->warp_max[warp] = vmax;
    }

    const bool softmax = warp < kSoftmaxWarps;
    const int part = (warp >> 2) % WAYS;  // of a softmax warp: WAYS threads per row share the positions; its TMEM lanes follow from warp % 4
    const int buf0 = PAIR ? warp >> 3 & 1 : 0;  // PAIR: its tile and score buffer; 0: the short one
    const int row = tid & (kRows - 1);
    const int group = 3 + 4 * buf0 + (warp & 3);  // barrier of the warps of these rows
    float4(*const row_part)[kRows] = sh->row_part + WAYS * buf0;
    // ---- query tiles: chunks of eight coefficients, neighbouring lanes neighbouring chunks
    if (softmax) {
        constexpr int kChunks = D / 8, kRounds = kRows * kChunks / (32 * G::kGroupWarps);
        const int first_chunk = (PAIR ? warp & 7 : warp) * 32 + lane;
        for (int ti = 0; ti < tiles; ++ti) {
            const int q_tile = PAIR ? buf0 : ti, tile_row = (PAIR ? short_tile + buf0 : ti == 0 ? long_tile : short_tile) * kRows;
            uint4 qv[kRounds];  // all on their way before anything is stored
#pragma unroll
            for (int i = 0; i < kRounds; ++i) {
                const int chunk = first_chunk + i * 32 * G::kGroupWarps, R = tile_row + chunk / kChunks, c = chunk % kChunks;
                qv[i] = make_uint4(0, 0, 0, 0);
                if (R < p.T * p.g)
                    qv[i] = reinterpret_cast<const uint4*>(p.q + head_vector(R) * D)[c];
            }
#pragma unroll
            for (int i = 0; i < kRounds; ++i) {
                const int chunk = first_chunk + i * 32 * G::kGroupWarps, r = chunk / kChunks, c = chunk % kChunks;
                uint4 v = qv[i];
                const __half2* h = reinterpret_cast<const __half2*>(&v);
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 f = __half22float2(h[k]);
                    s += f.x + f.y;
                }
                const bool seg8 = c < H::kR8 / 8;  // chunk 0, at D = 128 chunks 0 and 1
                float s8 = s, s4 = seg8 ? 0.f : s;
                if (tile_row + chunk / 32 * 32 / kChunks < p.T * p.g) {  // any row of the warp's chunks
                    if (D == 128) s8 += __shfl_xor_sync(0xffffffffu, s8, 1);
#pragma unroll
                    for (int o = 1; o < kChunks; o <<= 1) s4 += __shfl_xor_sync(0xffffffffu, s4, o);
                }
                if (c == 0) sh->row_sum[q_tile][r] = make_float2(s8, s4);
                if (!seg8)
                    v = make_uint4(__byte_perm(v.x, v.z, 0x5410), __byte_perm(v.x, v.z, 0x7632), __byte_perm(v.y, v.w, 0x5410),
                                   __byte_perm(v.y, v.w, 0x7632));
                *reinterpret_cast<uint4*>(Qs + q_tile * H::kQBytes + r * 128 + (c >> 3) * (kRows * 128) + (((c & 7) ^ (r & 7)) << 4)) = v;
            }
        }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    if (D == 128) {
        float vmax = 0.f;
#pragma unroll
        for (int i = 0; i <= kMmaWarp; ++i) vmax = fmaxf(vmax, sh->warp_max[i]);
        int e = 0;
        if (vmax > 0.f) e = min(max(ilogbf(vmax), -100), 100);
        p_scale = ldexpf(1.f, -e);
        out_scale = ldexpf(1.f, e);
    }

    bool ok = true;
    int stage = 0, stage_parity = 0;  // of the role's next step
    if (softmax) {
        const uint32_t tmem_row = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        auto buffer = [&](int N) { return PAIR ? buf0 : N & 1; };  // whose barriers (and output) step N uses, and their parity
        auto parity = [&](int N) { return PAIR ? N & 1 : N >> 1 & 1; };
        auto out_columns = [&](int N) { return tmem_row + G::kColOut + part * G::kOutCols + buffer(N) * G::kOutPitch; };
        const uint32_t cols_k = smem_u32(sh->col_k) + part * (G::kPart * 16), cols_v = smem_u32(sh->col_v) + part * (G::kPart * 16);
        for (int ti = 0, done = 0; ti < tiles && ok; ++ti) {  // done: steps of the tiles before
            const Tile tile = tile_of(ti);
            const int R0 = (PAIR ? short_tile + buf0 : ti == 0 ? long_tile : short_tile) * kRows, n_steps = tile.n_steps;
            const int pos_first = p.pos0 + token_of(R0);  // position of the first row: the smallest
            const int pos_i = R0 + row < p.T * p.g ? p.pos0 + token_of(R0 + row) : -1;
            RowState st{-INFINITY, 0ull, 0ull, 0ull};
            f2 O[D == 64 ? G::kOutCols / 2 : 1];  // D = 64: they are summed here, with rounding (the tensor core truncates its sums)
            if constexpr (D == 64) {
#pragma unroll
                for (int i = 0; i < G::kOutCols / 2; ++i) O[i] = 0ull;
            }
            // Waits for the output product of the CTA's step N, counted over its tiles: of a buffer's every one in turn (PAIR: the last
            // alone; the next scores are behind the others).
            auto output_ready = [&](int N) {
                ok = mbar_wait(&sh->pv_done[buffer(N)], parity(N), &sh->abort_flag, p.status);
                ok = !__any_sync(0xffffffffu, !ok);
                tc_fence_after();
                return ok;
            };
            auto add_output = [&](int N) {  // D = 64: that step's product
                if constexpr (D == 64) {
#pragma unroll
                    for (int c = 0; c < G::kOutCols / 16; ++c) {
                        uint32_t o[16];
                        __syncwarp();
                        tmem_ld16(out_columns(N) + 16 * c, o);
#pragma unroll
                        for (int i = 0; i < 8; ++i) O[8 * c + i] = add2(O[8 * c + i], pack2(__uint_as_float(o[2 * i]), __uint_as_float(o[2 * i + 1])));
                    }
                }
            };
            bool added = false;  // the previous step's output is in O already
            for (int n = 0; n < n_steps; ++n) {
                const int N = done + n;
                const int j0 = (tile.first + n) * kStep + part * G::kPart;
                const uint32_t col_k = cols_k + stage * (kStep * 16), col_v = cols_v + stage * (kStep * 16);
                const uint32_t tmem_s = tmem_row + (PAIR ? buf0 : stage) * G::kBufCols;
                f2 sc[G::kPairs];
                const float m_use = st.m == -INFINITY ? 0.f : st.m;
                float mx = -INFINITY;
                ok = mbar_wait(&sh->kv_full[stage], stage_parity, &sh->abort_flag, p.status);
                ok = !__any_sync(0xffffffffu, !ok);
                const float2 q = sh->row_sum[PAIR ? buf0 : ti][row];  // read again each step: cheaper than its registers
                step_offsets<D>(sc, col_k, pack2(q.x, q.x), pack2(q.y, q.y), -m_use);  // under the wait for the products
                if (++stage == kStages) {
                    stage = 0;
                    stage_parity ^= 1;
                }
                if (!PAIR && n >= 2 && ok && output_ready(N - 2) && !added) add_output(N - 2);
                added = false;
                ok = ok && mbar_wait(&sh->s_full[buffer(N)], parity(N), &sh->abort_flag, p.status);
                ok = !__any_sync(0xffffffffu, !ok);
                tc_fence_after();
                if (ok) {
                    const bool masked = j0 + G::kPart - 1 > pos_first;
                    const int last = pos_i - j0;  // the last of these positions that this row sees
                    if (masked) mx = step_scores<D, true>(sc, tmem_s + part * G::kPart, col_k, -m_use, last);
                    else mx = step_scores<D, false>(sc, tmem_s + part * G::kPart, col_k, -m_use, last);
                }
                if constexpr (PAIR) {  // the 4-bit segment's next scores may come: the weights go over the other's only
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh->s_read[buf0]);
                }
                // ---- raise the reference where a score leaves it too far behind (and set it at the first position seen).  Behind
                // the barrier all warps of the rows have read the scores that the weights go over, and all leave if a wait of one failed
                tc_fence_before();
                const bool rare = group_any<32 * WAYS>(group, !ok || mx > (st.m == -INFINITY ? -INFINITY : kSlack));
                tc_fence_after();
                if (rare) {
                    row_part[part][row].w = mx;
                    if (!PAIR && n > 0 && ok && output_ready(N - 1) && D == 64) {  // its weights are behind the old reference
                        add_output(N - 1);
                        added = true;
                    }
                    if (group_any<32 * WAYS>(group, !ok)) {
                        ok = false;
                        break;
                    }
#pragma unroll
                    for (int i = 0; i < WAYS; ++i) mx = fmaxf(mx, row_part[i][row].w);
                    const bool raise = mx > (st.m == -INFINITY ? -INFINITY : kSlack);
                    const float d = raise ? mx : 0.f;
                    const float f = raise ? (st.m == -INFINITY ? 0.f : exp2_approx(-d)) : 1.f;
                    const f2 d2 = pack2(-d, -d), ff = pack2(f, f);
#pragma unroll
                    for (int i = 0; i < G::kPairs; ++i) sc[i] = add2(sc[i], d2);
                    st.l = mul2(st.l, ff);
                    st.z8 = mul2(st.z8, ff);
                    st.z4 = mul2(st.z4, ff);
                    if (raise) st.m = m_use + d;
                    if constexpr (D == 64) {
#pragma unroll
                        for (int i = 0; i < G::kOutCols / 2; ++i) O[i] = mul2(O[i], ff);
                    } else if (n > 0) {
#pragma unroll
                        for (int c = 0; c < G::kOutCols / 16; ++c) {
                            uint32_t o[16];
                            __syncwarp();
                            tmem_ld16(out_columns(N) + 16 * c, o);
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                            tmem_st16(out_columns(N) + 16 * c, o);
                        }
                    }
                }
                // ---- weights, their sums, the operands of the output product
                step_weights<D>(st, sc, tmem_s + part * (G::kPart / 2), col_v);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh->p_full[buffer(N)]);
            }
            for (int n = max(n_steps - (PAIR ? 1 : 2), 0); n < n_steps && ok; ++n)
                if (output_ready(done + n) && !(added && n == n_steps - 2)) add_output(done + n);
            // a row that sees a value whose constants are not finite gets NaN in that segment
            if (pos_i >= sh->bad8) st.z8 = pack2(NAN, NAN);
            if (pos_i >= sh->bad4) st.z4 = pack2(NAN, NAN);
            done += n_steps;

            // ---- out = (O 2^E + zero-point sums) / sum of p; the row's outputs leave in the coefficients' own order
            const float2 l2 = unpack2(st.l), z8p = unpack2(st.z8), z4p = unpack2(st.z4);
            row_part[part][row] = make_float4(l2.x + l2.y, z8p.x + z8p.y, z4p.x + z4p.y, 0.f);
            if (group_any<32 * WAYS>(group, !ok)) ok = false;  // the warps of these rows leave together: they would meet at the next tile's barrier
            float l = 0.f, z8 = 0.f, z4 = 0.f;
#pragma unroll
            for (int i = 0; i < WAYS; ++i) {
                const float4 v = row_part[i][row];
                l += v.x;
                z8 += v.y;
                z4 += v.z;
            }
            // A block of the warp's columns goes through shared memory (to a split walk's record, or a patch of the warp's own): stored
            // from rows, every 16 bytes would be a line of their own (2 us per tile).
            float* record = reinterpret_cast<float*>(base) + row * H::kRecPitch;  // over the tiles: every product of the CTA is done
            const float inv = splits > 1 ? 1.f : l > 0.f ? kUnit / l : 0.f;
            if (splits > 1 && part == 0 && ok) {
                record[D] = st.m;
                record[D + 1] = l;
            }
            constexpr int kCols = G::kOutBlock, kQuads = kCols / 4;
            auto coefficient = [&](int n0) { return n0 >= D - H::kR8 ? n0 - (D - H::kR8) : H::kR8 + n0; };  // of the first of eight columns
            uint8_t* patch = D == 128 ? Qs + (PAIR ? buf0 : ti) * H::kQBytes + (warp & 7) * G::kOutBytes : out_stage_d64 + warp * G::kOutBytes;
#pragma unroll
            for (int c = 0; c < G::kOutCols / kCols; ++c) {
                if (R0 + (warp & 3) * 32 >= p.T * p.g && splits == 1) break;  // none of the warp's rows exists
                float o[kCols];
                if constexpr (D == 64) {
#pragma unroll
                    for (int i = 0; i < kCols / 2; ++i) {
                        const float2 f = unpack2(O[c * kCols / 2 + i]);
                        o[2 * i] = f.x;
                        o[2 * i + 1] = f.y;
                    }
                } else {
                    uint32_t u[2][16];
                    __syncwarp();
                    tmem_ld16(out_columns(0) + 32 * c, u[0]);
                    tmem_ld16(out_columns(0) + 32 * c + 16, u[1]);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __uint_as_float(u[i >> 4][i & 15]);
                }
                const int block = part * G::kOutCols + kCols * c;
                __syncwarp();  // the patch has been read
#pragma unroll
                for (int grp = 0; grp < kCols / 8; ++grp) {  // eight columns = eight coefficients
                    const int n0 = block + 8 * grp;
                    const bool seg8 = n0 >= D - H::kR8;
                    const float z = seg8 ? z8 : z4;
                    float f[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) f[i] = (n_steps > 0 ? fmaf(o[8 * grp + i], out_scale, z) : 0.f) * inv;
                    const float4 lo = seg8 ? make_float4(f[0], f[1], f[2], f[3]) : make_float4(f[0], f[2], f[4], f[6]);
                    const float4 hi = seg8 ? make_float4(f[4], f[5], f[6], f[7]) : make_float4(f[1], f[3], f[5], f[7]);
                    if (splits > 1) {
                        if (ok) {
                            *reinterpret_cast<float4*>(record + coefficient(n0)) = lo;
                            *reinterpret_cast<float4*>(record + coefficient(n0) + 4) = hi;
                        }
                    } else {  // quad q of the row's block at q ^ (lane % kQuads)
                        float4* r = reinterpret_cast<float4*>(patch) + lane * kQuads;
                        r[(2 * grp) ^ (lane & (kQuads - 1))] = lo;
                        r[(2 * grp + 1) ^ (lane & (kQuads - 1))] = hi;
                    }
                }
                if (splits == 1) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < kQuads; ++i) {
                        const int r = i * (32 / kQuads) + lane / kQuads, q = lane % kQuads, R = R0 + (warp & 3) * 32 + r;
                        const float4 v = reinterpret_cast<const float4*>(patch)[r * kQuads + (q ^ (r & (kQuads - 1)))];
                        if (ok && R < p.T * p.g)
                            *reinterpret_cast<float4*>(p.out + head_vector(R) * D +
                                                       coefficient(block + 8 * (q >> 1)) + 4 * (q & 1)) = v;
                    }
                }
            }
            tc_fence_before();  // the next tile's products go over the output
        }
    } else if (warp < kMmaWarp) {
        int N = 0;
        for (; N < total_steps; ++N) {
            ok = mbar_wait(&sh->raw_full[N & 1], (N >> 1) & 1, &sh->abort_flag, p.status);
            if (ok && N >= kStages) ok = mbar_wait(&sh->kv_empty[stage], stage_parity ^ 1, &sh->abort_flag, p.status);
            int all_ok;  // the warps leave together (they meet at a barrier below)
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 2, %2, p;\n\t"
                         "selp.b32 %0, 1, 0, q;\n\t}" : "=r"(all_ok) : "r"(ok ? 1 : 0), "n"(32 * kExpandWarps) : "memory");
            if (!all_ok) { ok = false; break; }
            const bool second = N >= tile0.n_steps;
            const int j0 = (second ? N - tile0.n_steps : tile0.first + N) * kStep;
            expand_step<D>(smem_u32(raw) + (N & 1) * H::kRawBytes, smem_u32(stages) + stage * H::kStageBytes, smem_u32(sh->col_k[stage]),
                           smem_u32(sh->col_v[stage]), warp - kSoftmaxWarps, lane, (second ? positions_seen(short_tile) : tile0.limit) - j0,
                           p_scale, j0, &sh->bad8, &sh->bad4);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->kv_full[stage]);
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kExpandWarps) : "memory");  // everybody has read the raw buffer
            if (loader && N + 2 < total_steps) issue_load(N + 2);
            if (++stage == kStages) {
                stage = 0;
                stage_parity ^= 1;
            }
        }
        if (loader && !ok) {  // copies still in flight are waited for (bounded; the shared flag is set by now)
            int keep_waiting = 0;
            for (int i = N; i < min(N + 2, total_steps); ++i) (void)mbar_wait(&sh->raw_full[i & 1], (i >> 1) & 1, &keep_waiting, p.status);
        }
    } else {  // the whole warp, converged; one lane issues
        const bool leader = elect_one();
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            if (ok) ok = !__any_sync(0xffffffffu, !mbar_wait(bar, parity, &sh->abort_flag, p.status));
            tc_fence_after();
            return ok;
        };
        const uint32_t idS = make_idesc_f16(kRows, kStep);
        // the 4-bit segment's scores at d = 128, beside the weights
        auto segment4_scores = [&](int q_tile, int buf, int st) {
            const uint32_t q = smem_u32(Qs) + q_tile * H::kQBytes, k = smem_u32(stages) + st * H::kStageBytes;
            const uint64_t q0 = make_smem_desc_k128(q), k0 = make_smem_desc_k128(k), k1 = make_smem_desc_k128(k + H::kTile);
            const uint64_t q1 = make_smem_desc_k128(q + kRows * 128);
            const uint32_t d = tmem + buf * G::kBufCols + kColS4;
#pragma unroll
            for (int i = 1; i < 4; ++i) mma_f16_ss_if(leader, d, q0 + 2 * i, k0 + 2 * i, idS, i > 1);
#pragma unroll
            for (int i = 0; i < 4; ++i) mma_f16_ss_if(leader, d, q1 + 2 * i, k1 + 2 * i, idS, 1);
        };
        // the scores that the weights lie over (PAIR: the 8-bit segment's alone, behind the others), then all of them are announced
        auto score_product = [&](int q_tile, int buf, int st, int bar) {
            const uint32_t q = smem_u32(Qs) + q_tile * H::kQBytes, k = smem_u32(stages) + st * H::kStageBytes;
            const uint64_t q0 = make_smem_desc_k128(q), k0 = make_smem_desc_k128(k), k1 = make_smem_desc_k128(k + H::kTile);
            const uint32_t d = tmem + buf * G::kBufCols;
            if constexpr (D == 128) {
                mma_f16_ss_if(leader, d, q0, k0, idS, 0);
                if constexpr (!PAIR) segment4_scores(q_tile, buf, st);
            } else {  // each segment's keys are 0 where the other's coefficients are
                mma_f16_ss_if(leader, d, q0, k1, idS, 0);
#pragma unroll
                for (int i = 0; i < 4; ++i) mma_f16_ss_if(leader, d + kColS4, q0 + 2 * i, k0 + 2 * i, idS, i > 0);
            }
            tc_commit_if(leader, &sh->s_full[bar]);
        };
        auto output_product = [&](int buf, int out, bool fresh, int st) {
            const uint32_t v = smem_u32(stages) + st * H::kStageBytes + H::kOffStageV4;
            const uint64_t v4 = make_smem_desc_mn128(v, H::kTile);
            const uint32_t w = tmem + buf * G::kBufCols;  // the weights
            const uint32_t d = tmem + G::kColOut + out * G::kOutPitch;
            if constexpr (D == 128) {
                const uint64_t v8 = make_smem_desc_mn128(v + H::kOffStageV8 - H::kOffStageV4, H::kTile);
                const uint32_t id8 = make_idesc_f16(kRows, 16) | kBNMajor, id4 = make_idesc_f16(kRows, 112) | kBNMajor;
#pragma unroll
                for (int i = 0; i < kStep / 16; ++i) {  // 16 positions: 8 columns of weights, 16 rows of 128 bytes
                    const uint32_t acc = (!fresh || i > 0) ? 1u : 0u;
                    mma_f16_ts_if(leader, d + 112, w + 8 * i, v8 + (2048 >> 4) * i, id8, acc);
                    mma_f16_ts_if(leader, d, w + 32 + 8 * i, v4 + (2048 >> 4) * i, id4, acc);
                }
            } else {  // parts of the weights times parts of the values, the small products first; those left out are below 2^-26
                const uint32_t id = make_idesc_bf16(kRows, 64) | kBNMajor;
#pragma unroll
                for (int order = 2; order >= 0; --order)
#pragma unroll
                    for (int k = order; k >= 0; --k)
#pragma unroll
                        for (int i = 0; i < kStep / 16; ++i)
                            mma_f16_ts_if(leader, d, w + 32 * k + 8 * i, v4 + (((order - k) * H::kTile + 2048 * i) >> 4), id,
                                          order < 2 || k < 2 || i > 0);
            }
        };
        // the stage of the next scores, once its keys are in place
        auto keys_ready = [&] { return wait(&sh->kv_full[stage], stage_parity); };
        auto next_stage = [&] {
            if (++stage == kStages) {
                stage = 0;
                stage_parity ^= 1;
            }
        };
        // Scores go over the weights of an earlier output product, which has to be complete: two products are ordered by their issue only
        // if they share accumulator and shape.  PAIR: the weights lie over the 8-bit segment's scores, so only that product, one
        // instruction, waits for the output product; the 4-bit segment's follow as soon as the softmax has read the ones before, under
        // its weights (2048 tokens behind 4096: 338.6 us; both products behind it 346.6).  Otherwise a stage has its score buffer, and its keys
        // are in place only after the output product of the step that had the stage before has freed it.
        int out_stage = 0;
        if constexpr (PAIR) {
            if (total_steps > 0 && keys_ready()) {
                for (int t = 0; t < 2; ++t) {
                    segment4_scores(t, t, stage);
                    score_product(t, t, stage, t);
                }
                next_stage();
            }
            for (int n = 0; n < total_steps && ok; ++n) {
                const bool more = n + 1 < total_steps;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (more) {
                        if (t == 0 && !keys_ready()) break;
                        if (!wait(&sh->s_read[t], n & 1)) break;
                        segment4_scores(t, t, stage);
                    }
                    if (!wait(&sh->p_full[t], n & 1)) break;
                    output_product(t, t, n == 0, out_stage);
                    tc_commit_if(leader, &sh->pv_done[t]);
                    if (t == 1) tc_commit_if(leader, &sh->kv_empty[out_stage]);
                    if (more) {
                        if (!wait(&sh->pv_done[t], n & 1)) break;
                        score_product(t, t, stage, t);
                    }
                }
                if (++out_stage == kStages) out_stage = 0;
                if (more) next_stage();
            }
        } else {
            auto scores = [&](int N) {
                if (!keys_ready()) return;
                score_product(N >= tile0.n_steps, stage, stage, N & 1);
                next_stage();
            };
            for (int N = 0; N < min(2, total_steps) && ok; ++N) scores(N);
            for (int N = 0; N < total_steps && ok; ++N) {
                if (!wait(&sh->p_full[N & 1], (N >> 1) & 1)) break;
                output_product(out_stage, N & 1, N == 0 || N == tile0.n_steps, out_stage);
                tc_commit_if(leader, &sh->pv_done[N & 1]);
                tc_commit_if(leader, &sh->kv_empty[out_stage]);
                if (++out_stage == kStages) out_stage = 0;
                if (N + 2 < total_steps) scores(N + 2);
            }
        }
        if (!ok) {  // products in flight finish before TMEM and shared memory are given back (bounded)
            int keep_waiting = 0;
            tc_commit_if(leader, &sh->drain);
            (void)mbar_wait(&sh->drain, 0, &keep_waiting, p.status);
        }
    }
    if (splits > 1) {
        float* rec = reinterpret_cast<float*>(base);
        const int R0 = long_tile * kRows;
        __syncwarp();
        cluster_sync_all();
        // every rank merges a share of the rows, all ranks' records of an item on their way at once
        const int share = (kRows + splits - 1) / splits, end = min(share * (rank + 1), kRows) * (D / 4);
        for (int i = share * rank * (D / 4) + tid; i < end; i += kThreads) {
            const int rr = i / (D / 4), c4 = i % (D / 4), Ro = R0 + rr;
            if (Ro >= p.T * p.g) continue;
            const uint32_t local = smem_u32(rec + rr * H::kRecPitch);
            float2 ml[8];
            float4 o[8];
#pragma unroll
            for (int rk = 0; rk < 8; ++rk) {
                ml[rk] = make_float2(-INFINITY, 0.f);
                o[rk] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (rk < splits) {
                    const uint32_t a = cluster_map_addr(local, rk);
                    ml[rk] = ld_cluster_f2(a + D * 4);
                    o[rk] = ld_cluster_f4(a + c4 * 16);
                }
            }
            float M = -INFINITY, L = 0.f;
#pragma unroll
            for (int rk = 0; rk < 8; ++rk) M = fmaxf(M, ml[rk].x);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int rk = 0; rk < 8; ++rk) {
                const float f = rk < splits ? exp2_approx(ml[rk].x - M) : 0.f;
                L = fmaf(ml[rk].y, f, L);
                acc = make_float4(fmaf(o[rk].x, f, acc.x), fmaf(o[rk].y, f, acc.y), fmaf(o[rk].z, f, acc.z), fmaf(o[rk].w, f, acc.w));
            }
            const float inv = L > 0.f ? kUnit / L : 0.f;
            *reinterpret_cast<float4*>(p.out + head_vector(Ro) * D + 4 * c4) =
                make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
        __syncwarp();
        cluster_sync_all();  // the records stay until all have read them
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && sh->abort_flag) atomicOr(p.status, kStatusBitTimeout);
    if (warp == kMmaWarp) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(sh->tmem_base, kTmemCols);
    }
}

template <int D, int WAYS, bool PAIR>
cudaError_t launch_prefill(const PrefillParams& p, long long ctas, cudaStream_t st) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(attention_prefill_kernel<D, WAYS, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(Geometry<D, WAYS, PAIR>::kSmem));
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(ctas));
    cfg.blockDim = dim3(Geometry<D, WAYS, PAIR>::kThreads);
    cfg.dynamicSmemBytes = Geometry<D, WAYS, PAIR>::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(p.splits);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // More CTAs than SMs start in order of length only behind a drained grid.
    cfg.numAttrs = ctas <= 148 ? 2 : 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, attention_prefill_kernel<D, WAYS, PAIR>, p);
}

}  // namespace

cudaError_t launch_attention_prefill(const resq_kv_cache_t& cache, const void* q16, int n_q_heads, int seq, int pos0,
                                     int T, float* out, cudaStream_t st, int d_head) {
    PrefillParams p;
    const size_t nblk = static_cast<size_t>(cache.capacity / RESQ_KV_BLOCK);
    p.head_stride = nblk * (d_head == 64 ? Head<64>::kBlockBytes : Head<128>::kBlockBytes);
    p.blocks = static_cast<const uint8_t*>(cache.data) + static_cast<size_t>(seq) * cache.n_kv_heads * p.head_stride;
    p.q = static_cast<const __half*>(q16);
    p.out = out;
    p.T = T;
    p.Hq = n_q_heads;
    p.Hkv = cache.n_kv_heads;
    p.g = n_q_heads / cache.n_kv_heads;
    p.g_inv = static_cast<unsigned>(((1ull << 32) + p.g - 1) / p.g);
    p.pos0 = pos0;
    p.status = device_status_ptr();
    const PrefillPlan pl = prefill_plan(pos0, T, p.g, p.Hkv, d_head);
    p.splits = pl.splits;
    p.tiles = pl.tiles_per_cta;
    const long long ctas = pl.row_groups * p.Hkv * pl.splits;
    if (d_head == 64) return launch_prefill<64, 4, false>(p, ctas, st);
    return pl.pair ? launch_prefill<128, 2, true>(p, ctas, st) : launch_prefill<128, 2, false>(p, ctas, st);
}

}  // namespace resq
