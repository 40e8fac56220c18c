// Attention over the quantized cache for d_head = 64 (Section 4.3, Eq. 8; Section 5.1), rows that are alone: the cache format
// of d_head = 128 with the first d/8 = 8 coefficients in 8 bits and the other 56 in 4, on mma.sync tiles with
// fp32-accurate weights.  (A causal run: kv_prefill.cu.  Projection and cache update: kv_cache.cu.)
//
// Block layout for d_head = 64 (the d = 128 layout with every code array halved): per half (key, then value)
//   c8 [32][8] | c4 [32][28] | meta [32][4] fp32      = 256 + 896 + 512 = 1664 bytes, 3328 per block.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "centred_codes.cuh"
#include "internal.h"
#include "plans.h"
#include "ptx.cuh"

namespace resq {
namespace {

constexpr int D = 64, R8 = D / 8, N4 = D - R8;
constexpr int kC8 = 32 * R8, kC4 = 32 * (N4 / 2), kHalf = kC8 + kC4 + 512, kBlock = 2 * kHalf;

// ---- attention -------------------------------------------------------------------------------------------------
// Rows (a query row's head vectors that share a KV head) meet 32 cache positions at a time on mma.sync m16n8k16 /
// m16n8k8, fp32 accumulators.  The g <= 8 rows of one (query row, KV head) are an item: the warps of the CTA take every NW-th
// step each, with a tile of their own, and their sums are merged at the end (single-query and many-query forms).
// NW = 12, one CTA per SM, for few items.  From 888 of them (two rounds of 3 x 148 CTAs) NW = 4, three CTAs
// per SM, which overlap each other's start and merge.  With more items than SMs, NW neighbouring ones whose
// lengths are short (the lengths are on the device) are taken by one CTA, a warp each; with NW = 4 all are
// once they fill four rounds that way.  us for rows of 32 positions, 8 KV heads, one / four heads per group,
// a CTA of twelve warps per item -> now: 110 rows 21 / 22 -> 11 / 12, 1000 rows 177 / 187 -> 21 / 24, 4096 rows
// 713 / 754 -> 74 / 82 (one warp per query head: 13 / 15, 31 / 89, 92 / 333).
// With few CTAs a cluster splits the steps further and rank 0 merges the sums through distributed shared memory, so
// no global scratch is needed.
//
// A step: a block arrives by cp.async three steps ahead.  Positions are the rows of the score product and heads its columns, coefficients the
// rows of the second product; both take their codes straight from the block's bytes, a lane reading the pieces of the positions
// and coefficients that are its own in the fragments, centred (code - 128, code - 8), keys as exact halves, values as exact bf16:
// expanded into shared memory and read back with ldmatrix, a step moved 236 shared-memory wavefronts, three quarters of what twelve
// warps had of them, and now some 140.  The weights become the second product's columns by 8 x 8 transposes.  Scales and
// zero-points act in fp32 on the accumulators:
//   score = s8 S8 + s4 S4 + (z8 + 128 s8) sum(q8) + (z4 + 8 s4) sum(q4)         (q half, codes exact: products exact)
//   out   = sum_j p_j s_j (c_j - c0) + sum_j p_j (z_j + c0 s_j)
// The weights p_j s_j enter the second product as they are in fp32: as three bf16 values of 8 bits each, which add up to
// all 24.  (Two halves under a common power of
// two hold 22 bits of the largest weight only: a value scale 2^20 above the others, on a position with next to no
// weight, left 2e-5 of the rest.)  A head's reference is raised when a score exceeds it by 2^2; against 64 bits the outputs are as far off as with
// an exact maximum (1.2 to 4.2e-7 over seven distributions, the form before 1.2 to 4.2e-7; with 2^8 and one chain for all parts up to 11 % more).
//
// What bounds it: shared memory and issue slots about equally; not HBM, not the tensor pipe.
// 32 query / 8 KV heads, project-and-append included: a step of 16 sequences of 1024-2048 positions 507 us (one warp per (row, query head) that
// dequantized each position per head) -> 19.7 -> 18.0; the attention alone 15.2 -> 13.4; 64 sequences of 1000 positions 35.1 -> 30.6, with eight heads in a
// group 36.9 -> 31.0.
struct Attn64Params {
    const uint8_t* cache;
    const __half* q;   // [rows][Hq][64]
    float* out;
    int rows, Hq, Hkv, g, n_seqs, capacity, splits;  // splits: CTAs of a cluster
    int pack, short_steps;      // whether a CTA takes NW neighbouring items, a warp each (Pack); up to how many steps
    const int32_t* seq_of_row;  // null: the row index
    const int32_t* len_of_row;
    int* status;
};

constexpr int kRecPitch = 68;      // floats per row of a record: 64 sums, maximum, sum of weights

constexpr int kStep = 32;          // positions of a step: a cache block
constexpr int kStages = 3;         // blocks of a warp's ring
constexpr int kWarpBytes = kStages * kBlock;  // of a warp's shared memory
static_assert(kWarpBytes >= 8 * kRecPitch * 4 && kWarpBytes % 16 == 0, "records fit");
constexpr float kSlack = 2.f;      // log2 of the largest weight before the reference is raised

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
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(x));
    return d;
}
__device__ __forceinline__ uint32_t lds32(const uint8_t* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ uint32_t lds16(const uint8_t* p) { return *reinterpret_cast<const uint16_t*>(p); }
__device__ __forceinline__ float4 lds_f4(const uint8_t* p) { return *reinterpret_cast<const float4*>(p); }
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
// Sequence and attended positions of query row `row`; out-of-range entries are clamped and, if asked, reported.
__device__ __forceinline__ int row_length(const Attn64Params& p, int row, bool report, int& b) {
    b = p.seq_of_row ? p.seq_of_row[row] : row;
    int len = p.len_of_row[row];
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

template <int NW>  // warps of a CTA
__global__ void __launch_bounds__(NW * 32, NW == 4 ? 3 : 1) attention64_kernel(const Attn64Params p) {
    extern __shared__ __align__(128) uint8_t smem64[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gr = lane >> 2, c = lane & 3;
    uint8_t* raw = smem64 + static_cast<size_t>(warp) * kWarpBytes;
    const int rank = static_cast<int>(blockIdx.x % p.splits);
    int item = static_cast<int>(blockIdx.x / p.splits);
    griddep_wait();  // launched with programmatic stream serialization
    griddep_launch_dependents();
    int part = warp, parts = NW;  // this warp's place among the warps that share an item
    if (p.pack) {
        const int n_items = p.rows * p.Hkv, base = p.pack == kPackAlways ? item * NW : item / NW * NW;
        bool together = p.pack == kPackAlways;
        if (!together) {
            const int last = min(base + NW, n_items) - 1, row = min(base / p.Hkv + lane, last / p.Hkv);  // at most NW rows
            int seq;
            together = __reduce_max_sync(0xffffffffu, row_length(p, row, false, seq)) <= p.short_steps * kStep;
            if (together && item != base) return;  // the block's first CTA takes them all
        }
        if (together) {
            item = base + warp;
            part = 0;
            parts = 1;
        }
        if (item >= n_items) return;
    }
    // ---- the item's row: its head vectors are the lanes' rows, lane / 4
    const int kvh = item % p.Hkv, row = item / p.Hkv;
    int b;
    const int limit = row_length(p, row, kvh == 0 && rank == 0 && part == 0 && lane == 0, b);  // positions it sees
    const uint8_t* blocks = p.cache + (static_cast<size_t>(b) * p.Hkv + kvh) * (p.capacity / RESQ_KV_BLOCK) * kBlock;
    const int n_steps = (limit + kStep - 1) / kStep;
    const int first = rank * parts + part, stride = parts * p.splits;  // this warp's steps

    auto issue = [&](int s, int buf) {  // copies of step s (if it exists) into a raw buffer; always one group
        if (s < n_steps) {
            const uint8_t* src = blocks + static_cast<size_t>(s) * kBlock;
            for (int i = lane; i < kBlock / 16; i += 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(raw + buf * kBlock + i * 16)), "l"(src + i * 16)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kStages; ++i) issue(first + i * stride, i);

    // ---- the query as the products' column operand: column gr is head gr; coefficients in the order in which the keys' pieces come (below)
    uint32_t qa[8];
    float qs8 = 0.f, qs4 = 0.f;
    {
        const __half* qrow = p.q + (static_cast<size_t>(row) * p.Hq + kvh * p.g + (gr < p.g ? gr : 0)) * D;
        uint32_t q0 = 0u, q3 = 0u;
        uint4 q1 = make_uint4(0u, 0u, 0u, 0u);
        uint2 q2 = make_uint2(0u, 0u);
        if (gr < p.g) {
            q0 = *reinterpret_cast<const uint32_t*>(qrow + 2 * c);
            q1 = *reinterpret_cast<const uint4*>(qrow + R8 + 8 * c);
            q2 = *reinterpret_cast<const uint2*>(qrow + R8 + 32 + 4 * c);
            q3 = *reinterpret_cast<const uint32_t*>(qrow + R8 + 48 + 2 * c);
        }
        qa[0] = q0;
        qa[1] = __byte_perm(q1.x, q1.z, 0x5410);  // 0 4 | 1 5, then 2 6 | 3 7 of a word of nibbles
        qa[2] = __byte_perm(q1.x, q1.z, 0x7632);
        qa[3] = __byte_perm(q1.y, q1.w, 0x5410);
        qa[4] = __byte_perm(q1.y, q1.w, 0x7632);
        qa[5] = __byte_perm(q2.x, q2.y, 0x5410);  // 0 2 | 1 3 of two bytes
        qa[6] = __byte_perm(q2.x, q2.y, 0x7632);
        qa[7] = q3;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&qa[j]));
            if (j == 0) qs8 += f.x + f.y;
            else qs4 += f.x + f.y;
        }
    }
    const float kScore = 1.4426950408889634f * 0.125f;  // log2(e) / sqrt(64)
    float kq8[2], kq4[2];  // of heads 2 c, 2 c + 1, the columns of a lane's scores
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        qs8 += __shfl_xor_sync(0xffffffffu, qs8, o);
        qs4 += __shfl_xor_sync(0xffffffffu, qs4, o);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        kq8[e] = kScore * __shfl_sync(0xffffffffu, qs8, 4 * (2 * c + e));
        kq4[e] = kScore * __shfl_sync(0xffffffffu, qs4, 4 * (2 * c + e));
    }

    // Outputs: rows are coefficients (gr, gr + 8), columns heads 2 c, 2 c + 1.  O[0]: the 8-bit segment in rows 0-7; O[1 + 2 i + t]: byte t of
    // half-word gr + 8 i of the 4-bit codes (i = 1: rows 6 and 7 are nobody's), the low nibble in row gr, the high one in row gr + 8.
    float O[5][4], m_run[2], l[2], zs8[2], zs4[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        m_run[e] = -INFINITY;
        l[e] = zs8[e] = zs4[e] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 5; ++j) O[j][0] = O[j][1] = O[j][2] = O[j][3] = 0.f;

    int buf = 0;
    for (int s = first; s < n_steps; s += stride) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
        __syncwarp();  // the step's bytes are in place
        const uint8_t* kb = raw + buf * kBlock;
        const uint8_t* vb = kb + kHalf;
        const int j0 = s * kStep;
        const bool masked = j0 + kStep > limit;

        // ---- scores of two tiles of 16 positions: row gr is position 2 gr of the tile, row gr + 8 the one behind it
        float sc[2][2][2];  // [tile][position][head]
        float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int tok = 16 * m + 2 * gr;
            const uint8_t* k4 = kb + kC8 + tok * (N4 / 2);
            uint32_t w[2], h[2], x[2], y[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                w[i] = lds32(k4 + i * (N4 / 2) + 4 * c);
                h[i] = lds16(k4 + i * (N4 / 2) + 16 + 2 * c);
                y[i] = k4[i * (N4 / 2) + 24 + c];
                x[i] = lds16(kb + (tok + i) * R8 + 2 * c);
            }
            const uint4 va = nibbles_centred(w[0]), vn = nibbles_centred(w[1]);
            float s8[4] = {0.f, 0.f, 0.f, 0.f}, s4[4] = {0.f, 0.f, 0.f, 0.f};
            mma8(s8, centred(__byte_perm(x[0], 0x64646464u, 0x4140), 0x6480), centred(__byte_perm(x[1], 0x64646464u, 0x4140), 0x6480), qa[0]);
            mma16(s4, va.x, vn.x, va.y, vn.y, qa[1], qa[2]);
            mma16(s4, va.z, vn.z, va.w, vn.w, qa[3], qa[4]);
            const uint2 ha = byte_pair_centred(__byte_perm(h[0], 0u, 0x4140)), hn = byte_pair_centred(__byte_perm(h[1], 0u, 0x4140));
            mma16(s4, ha.x, hn.x, ha.y, hn.y, qa[5], qa[6]);
            mma8(s4, centred(((y[0] * 0x1001u) & 0x000F000Fu) | 0x64006400u, 0x6408), centred(((y[1] * 0x1001u) & 0x000F000Fu) | 0x64006400u, 0x6408), qa[7]);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float4 k = lds_f4(kb + kC8 + kC4 + (tok + i) * 16);
                const bool hidden = masked && j0 + tok + i >= limit;
                if (hidden) k = make_float4(0.f, 0.f, 0.f, 0.f);
                k.y = fmaf(128.f, k.x, k.y);
                k.w = fmaf(8.f, k.z, k.w);
                k.x *= kScore;
                k.z *= kScore;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float v = fmaf(k.x, s8[2 * i + e], fmaf(k.z, s4[2 * i + e], fmaf(k.y, kq8[e], k.w * kq4[e])));
                    sc[m][i][e] = hidden ? -INFINITY : v;
                    mx[e] = fmaxf(mx[e], sc[m][i][e]);
                }
            }
        }
        // ---- reference of a head, the same in the lanes that share it: raised only when a score exceeds it by kSlack (and at first)
        if (__any_sync(0xffffffffu, mx[0] > m_run[0] + kSlack || mx[1] > m_run[1] + kSlack)) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float v = mx[e];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
                const float m_new = fmaxf(m_run[e], v);
                const float f = exp2_approx(m_run[e] - (m_new == -INFINITY ? 0.f : m_new));
                m_run[e] = m_new;
                l[e] *= f;
                zs8[e] *= f;
                zs4[e] *= f;
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    O[j][e] *= f;
                    O[j][2 + e] *= f;
                }
            }
        }
        // ---- weights times the value scales as three bf16 parts, transposed into the second product's column operand
        uint32_t w8[2][3][2], w4[2][3][2];  // [tile][part][positions 0 2 | 1 3 of the lane's four]
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int tok = 16 * m + 2 * gr + i;
                float4 v = lds_f4(vb + kC8 + kC4 + tok * 16);
                if (masked && j0 + tok >= limit) v = make_float4(0.f, 0.f, 0.f, 0.f);
                v.y = fmaf(128.f, v.x, v.y);
                v.w = fmaf(8.f, v.z, v.w);
                float pw[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    pw[e] = exp2_approx(sc[m][i][e] - (m_run[e] == -INFINITY ? 0.f : m_run[e]));
                    l[e] += pw[e];
                    zs8[e] = fmaf(pw[e], v.y, zs8[e]);
                    zs4[e] = fmaf(pw[e], v.w, zs4[e]);
                }
                uint32_t part[3];
                split_bf16(pw[0] * v.x, pw[1] * v.x, part);
#pragma unroll
                for (int k = 0; k < 3; ++k) w8[m][k][i] = movmatrix_trans(part[k]);
                split_bf16(pw[0] * v.z, pw[1] * v.z, part);
#pragma unroll
                for (int k = 0; k < 3; ++k) w4[m][k][i] = movmatrix_trans(part[k]);
            }
        // ---- the second product: the tensor core's fp32 sums are truncated, so a chain of products runs over
        // 32 positions only and is then added to the running sums with rounding; the first parts in a chain of their own.
        auto add_product = [&](float (&o)[4], const uint32_t (&a)[2][4], const uint32_t (&b)[2][3][2]) {
            float d[4] = {0.f, 0.f, 0.f, 0.f}, rest[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int m = 0; m < 2; ++m) mma16_bf16(rest, a[m], b[m][2][0], b[m][2][1]);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                mma16_bf16(rest, a[m], b[m][1][0], b[m][1][1]);
                mma16_bf16(d, a[m], b[m][0][0], b[m][0][1]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] += d[i] + rest[i];
        };
        {
            uint32_t a[2][4];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const uint8_t* v8 = vb + (16 * m + 4 * c) * R8 + gr;
                a[m][0] = byte_pair_bf16(__byte_perm(v8[0], v8[2 * R8], 0x5410));
                a[m][2] = byte_pair_bf16(__byte_perm(v8[R8], v8[3 * R8], 0x5410));
                a[m][1] = a[m][3] = 0u;
            }
            add_product(O[0], a, w8);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t w02[2], w13[2];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const uint8_t* v4 = vb + kC8 + (16 * m + 4 * c) * (N4 / 2) + 2 * (i == 0 ? gr : 8 + min(gr, 5));
                w02[m] = __byte_perm(lds16(v4), lds16(v4 + N4), 0x5410);
                w13[m] = __byte_perm(lds16(v4 + N4 / 2), lds16(v4 + 3 * (N4 / 2)), 0x5410);
            }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                uint32_t a[2][4];
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    a[m][0] = nibble_pair_bf16(w02[m] >> (8 * t));
                    a[m][1] = nibble_pair_bf16(w02[m] >> (8 * t + 4));
                    a[m][2] = nibble_pair_bf16(w13[m] >> (8 * t));
                    a[m][3] = nibble_pair_bf16(w13[m] >> (8 * t + 4));
                }
                add_product(O[1 + 2 * i + t], a, w4);
            }
        }
        __syncwarp();  // everybody is done with this block
        issue(s + kStages * stride, buf);
        if (++buf == kStages) buf = 0;
    }

    // ---- records of the warps (unnormalised sums with the zero-points, reference, sum of weights) over their rings, then the merge
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            l[e] += __shfl_xor_sync(0xffffffffu, l[e], o);
            zs8[e] += __shfl_xor_sync(0xffffffffu, zs8[e], o);
            zs4[e] += __shfl_xor_sync(0xffffffffu, zs4[e], o);
        }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        float* r = reinterpret_cast<float*>(raw) + (2 * c + e) * kRecPitch;
        r[gr] = O[0][e] + zs8[e];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (i == 1 && gr >= 6) continue;
            float* q = r + R8 + 4 * (gr + 8 * i);
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                q[2 * t] = O[1 + 2 * i + t][e] + zs4[e];
                q[2 * t + 1] = O[1 + 2 * i + t][2 + e] + zs4[e];
            }
        }
        if (gr == 0) {
            r[D] = m_run[e];
            r[D + 1] = l[e];
        }
    }
    __syncwarp();
    if (p.splits > 1) cluster_sync_all();
    else if (parts > 1) __syncthreads();
    if (rank == 0) {
        const uint8_t* rec0 = raw - part * kWarpBytes;  // the item's first record
        for (int i = part * 32 + lane; i < p.g * (D / 4); i += parts * 32) {
            const int hr = i / (D / 4), c4 = i % (D / 4);
            const uint32_t local = smem_u32(rec0) + hr * kRecPitch * 4;
            float M = -INFINITY, L = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int rk = 0; rk < p.splits; ++rk) {
                const uint32_t base = cluster_map_addr(local, rk);
#pragma unroll 4
                for (int w = 0; w < parts; ++w) {
                    const uint32_t a = base + w * kWarpBytes;
                    const float2 ml = ld_cluster_f2(a + D * 4);
                    const float4 o = ld_cluster_f4(a + c4 * 16);
                    const float m_all = fmaxf(M, ml.x);
                    const float ref = m_all == -INFINITY ? 0.f : m_all;
                    const float f0 = exp2_approx(M - ref), f1 = exp2_approx(ml.x - ref);
                    L = L * f0 + ml.y * f1;
                    acc = make_float4(acc.x * f0 + o.x * f1, acc.y * f0 + o.y * f1, acc.z * f0 + o.z * f1, acc.w * f0 + o.w * f1);
                    M = m_all;
                }
            }
            const float inv = L > 0.f ? 1.f / L : 0.f;
            *reinterpret_cast<float4*>(p.out + (static_cast<size_t>(row) * p.Hq + kvh * p.g + hr) * D + 4 * c4) =
                make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
    }
    __syncwarp();
    if (p.splits > 1) cluster_sync_all();  // the records stay until rank 0 has read them
}

template <int NW>
cudaError_t launch_attention64_form(const Attn64Params& p, long long ctas, cudaStream_t st) {
    const auto kern = attention64_kernel<NW>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, NW * kWarpBytes);
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(ctas));
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = NW * kWarpBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(p.splits);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace

size_t kv64_block_bytes() { return kBlock; }

cudaError_t launch_attention64(const resq_kv_cache_t& cache, const void* q16, int n_q_heads, int rows,
                               const int32_t* seq_of_row, const int32_t* len_of_row, float* out, cudaStream_t st) {
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
    p.status = device_status_ptr();
    const Attn64Plan pl = attention64_rows_plan(rows, p.Hkv, cache.capacity);
    p.splits = pl.splits;
    p.pack = pl.pack;
    p.short_steps = pl.short_steps;
    return pl.warps == 4 ? launch_attention64_form<4>(p, pl.ctas, st) : launch_attention64_form<12>(p, pl.ctas, st);
}

}  // namespace resq
