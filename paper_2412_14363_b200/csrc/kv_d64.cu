// Attention over the quantized cache for d_head = 64 (Section 4.3, Eq. 8; Section 5.1), all three forms: the cache format
// of d_head = 128 with the first d/8 = 8 coefficients in 8 bits and the other 56 in 4, on mma.sync tiles with
// fp32-accurate weights.  (Projection and cache update: kv_cache.cu.)
//
// Block layout for d_head = 64 (the d = 128 layout with every code array halved): per half (key, then value)
//   c8 [32][8] | c4 [32][28] | meta [32][4] fp32      = 256 + 896 + 512 = 1664 bytes, 3328 per block.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cfloat>
#include <climits>

#include "centred_codes.cuh"
#include "internal.h"
#include "plans.h"
#include "ptx.cuh"

namespace resq {
namespace {

constexpr int D = 64, R8 = D / 8, N4 = D - R8;
constexpr int kC8 = 32 * R8, kC4 = 32 * (N4 / 2), kHalf = kC8 + kC4 + 512, kBlock = 2 * kHalf;

// ---- attention -------------------------------------------------------------------------------------------------
// Rows (a query row's head vectors that share a KV head) meet STEP cache positions at a time on mma.sync m16n8k16 /
// m16n8k8, 16 rows per warp, fp32 accumulators.  Two forms of one kernel:
//   TEAM = 4  four warps share a tile of 64 rows -- 64 / g consecutive tokens of one sequence times the g heads -- and
//             walk the sequence together (a causal run of new tokens);
//   TEAM = 1  the g <= 8 rows of one (query row, KV head) -- an item -- are alone: the warps of the CTA take every NW-th
//             step each, with a tile of their own, and their sums are merged at the end (single-query and many-query forms).
//             NW = 12, one CTA per SM, for few items.  From 888 of them (two rounds of 3 x 148 CTAs) NW = 4, three CTAs
//             per SM, which overlap each other's start and merge.  With more items than SMs, NW neighbouring ones whose
//             lengths are short (the lengths are on the device) are taken by one CTA, a warp each; with NW = 4 all are
//             once they fill four rounds that way.  us for rows of 32 positions, 8 KV heads, one / four heads per group,
//             a CTA of twelve warps per item -> now: 110 rows 21 / 22 -> 11 / 12, 1000 rows 177 / 187 -> 21 / 24, 4096 rows
//             713 / 754 -> 74 / 82 (one warp per query head: 13 / 15, 31 / 89, 92 / 333).
// With few CTAs a cluster splits the steps further and rank 0 merges the sums through distributed shared memory, so
// no global scratch is needed.
//
// A step: the raw blocks arrive by cp.async two steps ahead; the codes are expanded, centred (code - 128, code - 8), in two
// tiles [position][64 coefficients], keys as exact halves, values as exact bf16; K fragments come from ldmatrix, V
// fragments from ldmatrix.trans, P straight from the score accumulators.  Scales and zero-points act in fp32 on the
// accumulators:
//   score = s8 S8 + s4 S4 + (z8 + 128 s8) sum(q8) + (z4 + 8 s4) sum(q4)         (q half, codes exact: products exact)
//   out   = sum_j p_j s_j (c_j - c0) + sum_j p_j (z_j + c0 s_j)
// The weights p_j s_j enter the second product as they are in fp32: as three bf16 values of 8 bits each, which add up to
// all 24, three products per fragment (TEAM = 1: two, its rows fill half a fragment).  (Two halves under a common power of
// two hold 22 bits of the largest weight only: a value scale 2^20 above the others, on a position with next to no
// weight, left 2e-5 of the rest.)
// The eight coefficients of a 32-bit word of nibbles are stored in the order 0 4 1 5 2 6 3 7 (one shift and mask per
// pair); the query fragments are gathered in that order and the outputs put back.
//
// What bounds it: the softmax arithmetic and the operand conversions on the CUDA cores (about 20 instructions per score
// of which two thirds per pair) and, for few rows, the latency of a step; not HBM, not the tensor pipe (26 % busy).
// 32 query / 8 KV heads, project-and-append included: 1000 new tokens 1355 -> 71 us (two halves per weight: 68), a step of
// 16 sequences of 1024-2048 positions 507 -> 21.7 us (20.6), against one warp per (row, query head) that dequantized each
// position per head.
struct Attn64Params {
    const uint8_t* cache;
    const __half* q;   // [rows][Hq][64]
    float* out;
    int rows, Hq, Hkv, g, n_seqs, capacity, splits;  // splits: CTAs of a cluster
    int pack, short_steps;      // TEAM = 1: whether a CTA takes NW neighbouring items, a warp each (Pack); up to how many steps
    const int32_t* seq_of_row;  // null: seq_const if >= 0, else the row index
    const int32_t* len_of_row;  // null: len0 + row + 1
    int seq_const, len0;
    int* status;
};

constexpr int kPitch = 144;        // bytes per position of an expanded tile: 64 halves + 16 (ldmatrix without conflicts)
constexpr int kRecPitch = 68;      // floats per row of a record: 64 sums, maximum, sum of weights

template <int TEAM, int NW>  // NW: warps of a CTA
struct A64 {
    static constexpr int kStep = TEAM == 1 ? 32 : 64;
    static constexpr int kNWarps = NW;
    static constexpr int kRaw = kStep / 32 * kBlock;
    static constexpr int kTeamBytes = 2 * kRaw + 2 * kStep * kPitch + 2 * kStep * 16 + 16;
    static constexpr int kSmem = kTeamBytes * (kNWarps / TEAM);
    static constexpr int kRows = TEAM == 1 ? 8 : 16;  // rows of a warp in use
};
static_assert(A64<1, 4>::kTeamBytes >= 8 * kRecPitch * 4 && A64<4, 4>::kSmem >= 4 * 16 * kRecPitch * 4, "records fit");

__device__ __forceinline__ void mma16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma16_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t h2_bits(__half2 v) { return *reinterpret_cast<const uint32_t*>(&v); }
// The bits of a float that bf16 keeps.
__device__ __forceinline__ float bf16_part(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFF0000u); }
// a, b as three pairs of bf16 that add up to them exactly: 8 bits each, cut off, of what the ones before leave.
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t (&part)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        part[i] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
        a -= bf16_part(a);
        b -= bf16_part(b);
    }
}
// Eight codes as bf16 minus their centre (centred_codes.cuh has them as halves).  bf16 holds 128 + (0..127) exactly: the
// bytes' upper bits move the centre.
__device__ __forceinline__ uint32_t minus_bf16(uint32_t v, uint32_t centre) {
    const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&v), *reinterpret_cast<const __nv_bfloat162*>(&centre));
    return *reinterpret_cast<const uint32_t*>(&d);
}
__device__ __forceinline__ uint4 nibbles_centred_bf16(uint32_t word) {
    uint32_t v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = minus_bf16(((word >> (4 * m)) & 0x000F000Fu) | 0x43004300u, 0x43084308u);  // 128 + 8
    return make_uint4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ uint4 bytes_centred_bf16(uint2 w) {
    uint32_t v[4] = {__byte_perm(w.x, 0u, 0x4140), __byte_perm(w.x, 0u, 0x4342), __byte_perm(w.y, 0u, 0x4140), __byte_perm(w.y, 0u, 0x4342)};
#pragma unroll
    for (int m = 0; m < 4; ++m)  // code < 128: (128 + code) - 256, else (128 + code - 128) - 128
        v[m] = minus_bf16((v[m] & 0x007F007Fu) | 0x43004300u, (~v[m] & 0x00800080u) | 0x43004300u);
    return make_uint4(v[0], v[1], v[2], v[3]);
}
// Coefficient at element e (0..7) of chunk j (0: the 8-bit segment, 1..7: words of nibbles).
__device__ __forceinline__ int coef64(int j, int e) { return j == 0 ? e : 8 * j + (e >> 1) + ((e & 1) << 2); }

// Sequence and attended positions of query row `row` (TEAM = 1); out-of-range entries are clamped and, if asked, reported.
__device__ __forceinline__ int row_length(const Attn64Params& p, int row, bool report, int& b) {
    b = p.seq_of_row ? p.seq_of_row[row] : (p.seq_const >= 0 ? p.seq_const : row);
    int len = p.len_of_row ? p.len_of_row[row] : p.len0 + row + 1;
    if (b < 0 || b >= p.n_seqs) {
        if (report) atomicOr(p.status, kStatusBitIndex);
        b = 0;
        len = 0;
    }
    if (len < 0 || len > p.capacity) {
        if (report) atomicOr(p.status, kStatusBitIndex);
        len = len < 0 ? 0 : p.capacity;
    }
    return len;
}

template <int TEAM, int NW>
__global__ void __launch_bounds__(NW * 32, NW == 4 ? 3 : 1) attention64_kernel(const Attn64Params p) {
    using C = A64<TEAM, NW>;
    constexpr int STEP = C::kStep, NT = STEP / 8;
    constexpr bool TWO = TEAM != 1;  // rows lane / 4 + 8 are in use
    constexpr int RH = TWO ? 2 : 1;
    constexpr int PARTS = TWO ? 3 : 2;  // products per fragment for a weight's three parts
    extern __shared__ __align__(128) uint8_t smem64[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gr = lane >> 2, c = lane & 3;
    const int team = warp / TEAM, tt = threadIdx.x - team * TEAM * 32;  // thread of the team
    uint8_t* raw = smem64 + static_cast<size_t>(team) * C::kTeamBytes;
    uint8_t* Kt = raw + 2 * C::kRaw;
    uint8_t* Vt = Kt + STEP * kPitch;
    float4* colK = reinterpret_cast<float4*>(Vt + STEP * kPitch);
    float4* colV = colK + STEP;
    int* bad = reinterpret_cast<int*>(colV + STEP);  // the first position whose value's 8-bit / 4-bit constants are not finite
    const int rank = static_cast<int>(blockIdx.x % p.splits);
    int item = static_cast<int>(blockIdx.x / p.splits);
    int part = 0, parts = 1;  // TEAM = 1: this warp's place among the warps that share an item
    griddep_wait();  // launched with programmatic stream serialization
    griddep_launch_dependents();
    if (TEAM == 1) {
        part = warp;
        parts = NW;
        if (p.pack) {
            const int n_items = p.rows * p.Hkv, base = p.pack == kPackAlways ? item * NW : item / NW * NW;
            bool together = p.pack == kPackAlways;
            if (!together) {
                const int last = min(base + NW, n_items) - 1, row = min(base / p.Hkv + lane, last / p.Hkv);  // at most NW rows
                int seq;
                together = __reduce_max_sync(0xffffffffu, row_length(p, row, false, seq)) <= p.short_steps * C::kStep;
                if (together && item != base) return;  // the block's first CTA takes them all
            }
            if (together) {
                item = base + warp;
                part = 0;
                parts = 1;
            }
            if (item >= n_items) return;
        }
    }
    const int kvh = item % p.Hkv, n_tiles = static_cast<int>(gridDim.x) / p.splits / p.Hkv;
    const int tile = TEAM == 1 ? item / p.Hkv : n_tiles - 1 - item / p.Hkv;  // long tiles of all heads first
    auto team_sync = [&] {
        if (TEAM == 1) __syncwarp();
        else __syncthreads();
    };

    // ---- rows of this lane, positions they see, the sequence
    int tok[RH], head[RH], pos_i[RH];
    int b, limit, pos_min;  // positions any row of the tile sees; the smallest of the rows' own positions
    if (TEAM == 1) {
        const int row = tile;
        const int len = row_length(p, row, kvh == 0 && rank == 0 && part == 0 && lane == 0, b);
        limit = len;
        pos_min = len - 1;
        tok[0] = gr < p.g ? row : -1;
        head[0] = kvh * p.g + gr;
        pos_i[0] = len - 1;
    } else {
        b = p.seq_const;
        const int R0 = tile * 64, n_rows = p.rows * p.g;
        pos_min = p.len0 + R0 / p.g;
        limit = p.len0 + min(p.rows - 1, (R0 + 63) / p.g) + 1;
#pragma unroll
        for (int h = 0; h < RH; ++h) {
            const int R = R0 + warp * 16 + gr + 8 * h;
            tok[h] = R < n_rows ? R / p.g : -1;
            head[h] = kvh * p.g + R % p.g;
            pos_i[h] = tok[h] >= 0 ? p.len0 + tok[h] : -1;
        }
    }
    const uint8_t* blocks = p.cache + (static_cast<size_t>(b) * p.Hkv + kvh) * (p.capacity / RESQ_KV_BLOCK) * kBlock;
    const int n_blocks = (limit + 31) >> 5, n_steps = (limit + STEP - 1) / STEP;
    // this team's steps: first, first + stride, .. < end
    const int first = TEAM == 1 ? rank * parts + part : static_cast<int>(static_cast<long long>(n_steps) * rank / p.splits);
    const int end = TEAM == 1 ? n_steps : static_cast<int>(static_cast<long long>(n_steps) * (rank + 1) / p.splits);
    const int stride = TEAM == 1 ? parts * p.splits : 1;

    auto issue = [&](int s, int buf) {  // copies of step s (if it exists) into a raw buffer; always one group
        if (s < end) {
            const int nb = min(STEP / 32, n_blocks - s * (STEP / 32));
            const uint8_t* src = blocks + static_cast<size_t>(s) * C::kRaw;
            for (int i = tt; i < nb * (kBlock / 16); i += TEAM * 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(raw + buf * C::kRaw + i * 16)), "l"(src + i * 16)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (TWO && tt == 0) bad[0] = bad[1] = INT_MAX;
    issue(first, 0);
    issue(first + stride, 1);

    // ---- query fragments: chunk 0 (m16n8k8), chunks 1-6 as three k16 pairs, chunk 7 (m16n8k8); sums per segment
    uint32_t qa[8][2];
    float qs8[2] = {0.f, 0.f}, qs4[2] = {0.f, 0.f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const bool ok = h < RH && tok[h < RH ? h : 0] >= 0;
        const __half* qrow = p.q + (static_cast<size_t>(ok ? tok[h < RH ? h : 0] : 0) * p.Hq + (ok ? head[h < RH ? h : 0] : 0)) * D;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            __half2 v = __floats2half2_rn(0.f, 0.f);
            if (ok) v = __halves2half2(qrow[coef64(j, 2 * c)], qrow[coef64(j, 2 * c + 1)]);
            qa[j][h] = h2_bits(v);
            const float2 f = __half22float2(v);
            if (j == 0) qs8[h] += f.x + f.y;
            else qs4[h] += f.x + f.y;
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            qs8[h] += __shfl_xor_sync(0xffffffffu, qs8[h], o);
            qs4[h] += __shfl_xor_sync(0xffffffffu, qs4[h], o);
        }
    }

    float O[8][4], m_run[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, zs8[2] = {0.f, 0.f}, zs4[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 8; ++j) O[j][0] = O[j][1] = O[j][2] = O[j][3] = 0.f;
    const float kScore = 1.4426950408889634f * 0.125f;  // log2(e) / sqrt(64)
    const uint32_t k_addr = smem_u32(Kt) + (lane & 7) * kPitch + (lane >> 3) * 16;
    const uint32_t v_addr = smem_u32(Vt) + ((lane & 7) + ((lane >> 3) & 1) * 8) * kPitch + (lane >> 4) * 16;

    int buf = 0;
    for (int s = first; s < end; s += stride, buf ^= 1) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        team_sync();  // the step's bytes are in place and nobody reads the previous tiles
        const uint8_t* rb = raw + buf * C::kRaw;
        const int j0 = s * STEP;
        // ---- expand: items of eight coefficients, chunks 0-7 of the keys then of the values
#pragma unroll
        for (int i = 0; i < STEP * 16 / (TEAM * 32); ++i) {
            const int item = i * TEAM * 32 + tt, pos = item % STEP, ch = item / STEP;  // ch is uniform over a warp
            const uint8_t* half_base = rb + (pos >> 5) * kBlock + (ch >= 8 ? kHalf : 0);
            const int j = ch & 7, pp = pos & 31;
            uint4 v;
            if (j == 0) {
                const uint2 w = *reinterpret_cast<const uint2*>(half_base + pp * R8);
                v = ch >= 8 ? bytes_centred_bf16(w) : bytes_centred(w);
            } else {
                const uint32_t w = *reinterpret_cast<const uint32_t*>(half_base + kC8 + pp * (N4 / 2) + 4 * (j - 1));
                v = ch >= 8 ? nibbles_centred_bf16(w) : nibbles_centred(w);
            }
            *reinterpret_cast<uint4*>((ch >= 8 ? Vt : Kt) + pos * kPitch + j * 16) = v;
        }
        // ---- per-position constants; positions past the tile's limit hold anything and are zeroed by selection
#pragma unroll
        for (int i = 0; i < (2 * STEP) / (TEAM * 32); ++i) {
            const int item = i * TEAM * 32 + tt, pos = item % STEP;
            const bool is_v = item >= STEP;
            float4 m = *reinterpret_cast<const float4*>(rb + (pos >> 5) * kBlock + (is_v ? kHalf : 0) + kC8 + kC4 + (pos & 31) * 16);
            if (j0 + pos >= limit) m = make_float4(0.f, 0.f, 0.f, 0.f);
            m.y = fmaf(128.f, m.x, m.y);
            m.w = fmaf(8.f, m.z, m.w);
            if (is_v) {
                // A causal run: a value's constants that are not finite become 0 (they would turn a hidden position's weight of 0
                // into NaN); the first such position is noted for the rows that see it.  Rows that are alone see every position.
                if (TWO && !(fabsf(m.x) <= FLT_MAX && fabsf(m.y) <= FLT_MAX)) {
                    m.x = m.y = 0.f;
                    atomicMin(bad, j0 + pos);
                }
                if (TWO && !(fabsf(m.z) <= FLT_MAX && fabsf(m.w) <= FLT_MAX)) {
                    m.z = m.w = 0.f;
                    atomicMin(bad + 1, j0 + pos);
                }
                colV[pos] = m;
            } else colK[pos] = make_float4(m.x * kScore, m.y * kScore, m.z * kScore, m.w * kScore);
        }
        team_sync();
        issue(s + 2 * stride, buf);  // everybody is done with this raw buffer

        // ---- scores
        float sc[NT][2 * RH];
        float mx[2] = {-INFINITY, -INFINITY};
        const bool masked = j0 + STEP - 1 > pos_min;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            uint32_t k0[4], k1[4];
            ldsm4(k0, k_addr + nt * 8 * kPitch);
            ldsm4(k1, k_addr + nt * 8 * kPitch + 64);
            float s8[4] = {0.f, 0.f, 0.f, 0.f}, s4[4] = {0.f, 0.f, 0.f, 0.f};
            mma8(s8, qa[0][0], qa[0][1], k0[0]);
            mma16(s4, qa[1][0], qa[1][1], qa[2][0], qa[2][1], k0[1], k0[2]);
            mma16(s4, qa[3][0], qa[3][1], qa[4][0], qa[4][1], k0[3], k1[0]);
            mma16(s4, qa[5][0], qa[5][1], qa[6][0], qa[6][1], k1[1], k1[2]);
            mma8(s4, qa[7][0], qa[7][1], k1[3]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int pos = 8 * nt + 2 * c + e;
                const float4 k = colK[pos];
#pragma unroll
                for (int h = 0; h < RH; ++h) {
                    float x = fmaf(k.x, s8[2 * h + e], fmaf(k.z, s4[2 * h + e], fmaf(k.y, qs8[h], k.w * qs4[h])));
                    if (masked && j0 + pos > pos_i[h]) x = -INFINITY;
                    sc[nt][2 * h + e] = x;
                    mx[h] = fmaxf(mx[h], x);
                }
            }
        }
        // ---- running maximum
        float m_use[RH], corr[RH];
        bool moved = false;
#pragma unroll
        for (int h = 0; h < RH; ++h) {
            mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
            mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
            const float m_new = fmaxf(m_run[h], mx[h]);
            m_use[h] = m_new == -INFINITY ? 0.f : m_new;
            corr[h] = exp2_approx(m_run[h] - m_use[h]);
            moved |= m_new != m_run[h];
            m_run[h] = m_new;
        }
        if (__any_sync(0xffffffffu, moved)) {
#pragma unroll
            for (int h = 0; h < RH; ++h) {
                l[h] *= corr[h];
                zs8[h] *= corr[h];
                zs4[h] *= corr[h];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    O[j][2 * h] *= corr[h];
                    O[j][2 * h + 1] *= corr[h];
                }
            }
        }
        // ---- weights and the second product, 32 positions at a time: the tensor core's fp32 sums are truncated, so a
        // chain of products runs over 32 positions only and is then added to the running sums with rounding
#pragma unroll
        for (int kp = 0; kp < STEP / 32; ++kp) {
            uint32_t p8[2][PARTS][4], p4[2][PARTS][4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int nt = 4 * kp + t, pos = 8 * nt + 2 * c;
                const float4 va = colV[pos], vb = colV[pos + 1];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = 2 * (t & 1) + h;
                    uint32_t w8[3], w4[3];
                    if (h < RH) {
                        const float pa = exp2_approx(sc[nt][2 * (h % RH)] - m_use[h % RH]);
                        const float pb = exp2_approx(sc[nt][2 * (h % RH) + 1] - m_use[h % RH]);
                        l[h] += pa + pb;
                        zs8[h] = fmaf(pa, va.y, fmaf(pb, vb.y, zs8[h]));
                        zs4[h] = fmaf(pa, va.w, fmaf(pb, vb.w, zs4[h]));
                        split_bf16(pa * va.x, pb * vb.x, w8);
                        split_bf16(pa * va.z, pb * vb.z, w4);
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (TWO) {
                            p8[t >> 1][k][i] = w8[k];
                            p4[t >> 1][k][i] = w4[k];
                        } else if (h == 0) {  // the middle part takes the unused rows of the first one's product
                            p8[t >> 1][k == 2][i + (k == 1)] = w8[k];
                            p4[t >> 1][k == 2][i + (k == 1)] = w4[k];
                        } else if (k == 0) {
                            p8[t >> 1][1][i] = p4[t >> 1][1][i] = 0u;
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
                uint32_t v[2][4];
                ldsm4t(v[0], v_addr + 2 * kp * 16 * kPitch + j * 16);
                ldsm4t(v[1], v_addr + (2 * kp + 1) * 16 * kPitch + j * 16);
#pragma unroll
                for (int k = PARTS - 1; k >= 0; --k)  // the small parts first
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {
                        mma16_bf16(d0, j == 0 ? p8[ks][k] : p4[ks][k], v[ks][0], v[ks][1]);
                        mma16_bf16(d1, p4[ks][k], v[ks][2], v[ks][3]);
                    }
#pragma unroll
                for (int e = 0; e < 2 * RH; ++e) {
                    O[j][e] += TWO ? d0[e] : d0[e] + d0[2 + e];
                    O[j + 1][e] += TWO ? d1[e] : d1[e] + d1[2 + e];
                }
            }
        }
    }

    // ---- records of the warps (unnormalised sums with the zero-points, maximum, sum of weights), then the merge
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    team_sync();
    const int bad8 = TWO ? bad[0] : INT_MAX, bad4 = TWO ? bad[1] : INT_MAX;
    // over the warp's own tiles, or (TEAM = 4) over the CTA's: [row][kRecPitch]
    float* rec = reinterpret_cast<float*>(TEAM == 1 ? raw : smem64 + warp * C::kRows * kRecPitch * 4);
#pragma unroll
    for (int h = 0; h < RH; ++h) {
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            l[h] += __shfl_xor_sync(0xffffffffu, l[h], o);
            zs8[h] += __shfl_xor_sync(0xffffffffu, zs8[h], o);
            zs4[h] += __shfl_xor_sync(0xffffffffu, zs4[h], o);
        }
        float* r = rec + (gr + 8 * h) * kRecPitch;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float z = TWO && pos_i[h] >= (j == 0 ? bad8 : bad4) ? NAN : j == 0 ? zs8[h] : zs4[h];
            r[coef64(j, 2 * c)] = O[j][2 * h] + z;
            r[coef64(j, 2 * c + 1)] = O[j][2 * h + 1] + z;
        }
        if (c == 0) {
            r[D] = m_run[h];
            r[D + 1] = l[h];
        }
    }
    __syncwarp();
    if (p.splits > 1) cluster_sync_all();
    else if (TEAM != 1 || parts > 1) __syncthreads();
    if (rank == 0) {
        const int n_rows = TEAM == 1 ? p.g : 64;
        const int sharers = TEAM == 1 ? parts * 32 : NW * 32, me = TEAM == 1 ? part * 32 + lane : static_cast<int>(threadIdx.x);
        uint8_t* rec0 = TEAM == 1 ? raw - part * C::kTeamBytes : smem64;  // the item's first record
        for (int i = me; i < n_rows * (D / 4); i += sharers) {
            const int row = i / (D / 4), c4 = i % (D / 4);
            const int R = tile * 64 + row;
            if (TEAM != 1 && R >= p.rows * p.g) continue;
            const uint32_t local = smem_u32(rec0) + row * kRecPitch * 4;  // TEAM = 4: warps' rows follow one another
            float M = -INFINITY, L = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int rk = 0; rk < p.splits; ++rk) {
                const uint32_t base = cluster_map_addr(local, rk);
#pragma unroll 4
                for (int w = 0; w < parts; ++w) {
                    const uint32_t a = base + w * C::kTeamBytes;
                    const float2 ml = ld_cluster_f2(a + D * 4);
                    const float4 o = ld_cluster_f4(a + c4 * 16);
                    const float m_new = fmaxf(M, ml.x);
                    const float ref = m_new == -INFINITY ? 0.f : m_new;
                    const float f0 = exp2_approx(M - ref), f1 = exp2_approx(ml.x - ref);
                    L = L * f0 + ml.y * f1;
                    acc = make_float4(acc.x * f0 + o.x * f1, acc.y * f0 + o.y * f1, acc.z * f0 + o.z * f1, acc.w * f0 + o.w * f1);
                    M = m_new;
                }
            }
            const float inv = L > 0.f ? 1.f / L : 0.f;
            const int t = TEAM == 1 ? tile : R / p.g, hq = kvh * p.g + (TEAM == 1 ? row : R % p.g);
            *reinterpret_cast<float4*>(p.out + (static_cast<size_t>(t) * p.Hq + hq) * D + 4 * c4) =
                make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
    }
    __syncwarp();
    if (p.splits > 1) cluster_sync_all();  // the records stay until rank 0 has read them
}

template <int TEAM, int NW>
cudaError_t launch_attention64_form(const Attn64Params& p, long long ctas, cudaStream_t st) {
    using C = A64<TEAM, NW>;
    const auto kern = attention64_kernel<TEAM, NW>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem);
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(ctas));
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = C::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(p.splits);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // The causal form's CTAs (three per SM, long tiles first) would crowd the SMs that drain first: 58 -> 68 us.
    cfg.numAttrs = TEAM == 1 || cfg.gridDim.x <= 148 ? 2 : 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace

size_t kv64_block_bytes() { return kBlock; }

cudaError_t launch_attention64(const resq_kv_cache_t& cache, const void* q16, int n_q_heads, int rows,
                               const int32_t* seq_of_row, const int32_t* len_of_row, int seq_const, int len0, float* out,
                               cudaStream_t st) {
    Attn64Params p{};
    p.cache = static_cast<const uint8_t*>(cache.data);
    p.q = static_cast<const __half*>(q16);
    p.out = out;
    p.rows = rows;
    p.Hq = n_q_heads;
    p.Hkv = cache.n_kv_heads;
    p.g = n_q_heads / cache.n_kv_heads;
    p.n_seqs = cache.n_seqs;
    p.capacity = cache.capacity;
    p.seq_of_row = seq_of_row;
    p.len_of_row = len_of_row;
    p.seq_const = seq_const;
    p.len0 = len0;
    p.status = device_status_ptr();
    const bool run = seq_const >= 0 && !seq_of_row && !len_of_row;  // a causal run of one sequence
    const Attn64Plan pl = run ? attention64_run_plan(len0, rows, p.g, p.Hkv) : attention64_rows_plan(rows, p.Hkv, cache.capacity);
    p.splits = pl.splits;
    p.pack = pl.pack;
    p.short_steps = pl.short_steps;
    if (run) return launch_attention64_form<4, 4>(p, pl.ctas, st);
    return pl.warps == 4 ? launch_attention64_form<1, 4>(p, pl.ctas, st) : launch_attention64_form<1, 12>(p, pl.ctas, st);
}

}  // namespace resq
