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
// A step: the raw blocks arrive by cp.async two steps ahead; the codes are expanded, centred (code - 128, code - 8), in two
// tiles [position][64 coefficients], keys as exact halves, values as exact bf16; K fragments come from ldmatrix, V
// fragments from ldmatrix.trans, P straight from the score accumulators.  Scales and zero-points act in fp32 on the
// accumulators:
//   score = s8 S8 + s4 S4 + (z8 + 128 s8) sum(q8) + (z4 + 8 s4) sum(q4)         (q half, codes exact: products exact)
//   out   = sum_j p_j s_j (c_j - c0) + sum_j p_j (z_j + c0 s_j)
// The weights p_j s_j enter the second product as they are in fp32: as three bf16 values of 8 bits each, which add up to
// all 24, in two products per fragment, since the rows fill half of one.  (Two halves under a common power of
// two hold 22 bits of the largest weight only: a value scale 2^20 above the others, on a position with next to no
// weight, left 2e-5 of the rest.)
// The eight coefficients of a 32-bit word of nibbles are stored in the order 0 4 1 5 2 6 3 7 (one shift and mask per
// pair); the query fragments are gathered in that order and the outputs put back.
//
// What bounds it: the latency of a step and the operand conversions on the CUDA cores; not HBM, not the tensor pipe.
// 32 query / 8 KV heads, project-and-append included: a step of 16 sequences of 1024-2048 positions 507 -> 19.7 us (21.7 while the words
// of a step were read and expanded one by one), against one warp per (row, query head) that dequantized each position per head.
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

constexpr int kPitch = 144;        // bytes per position of an expanded tile: 64 halves + 16 (ldmatrix without conflicts)
constexpr int kRecPitch = 68;      // floats per row of a record: 64 sums, maximum, sum of weights

constexpr int kStep = 32, kNT = kStep / 8;  // positions of a step, score fragments
constexpr int kWarpBytes = 2 * kBlock + 2 * kStep * kPitch + 2 * kStep * 16;  // of a warp's shared memory
static_assert(kWarpBytes >= 8 * kRecPitch * 4 && kWarpBytes % 16 == 0, "records fit");

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
// Coefficient at element e (0..7) of chunk j (0: the 8-bit segment, 1..7: words of nibbles).
__device__ __forceinline__ int coef64(int j, int e) { return j == 0 ? e : 8 * j + (e >> 1) + ((e & 1) << 2); }

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
    uint8_t* Kt = raw + 2 * kBlock;
    uint8_t* Vt = Kt + kStep * kPitch;
    float4* colK = reinterpret_cast<float4*>(Vt + kStep * kPitch);
    float4* colV = colK + kStep;
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
    issue(first, 0);
    issue(first + stride, 1);

    // ---- query fragments: chunk 0 (m16n8k8), chunks 1-6 as three k16 pairs, chunk 7 (m16n8k8); sums per segment
    uint32_t qa[8];
    float qs8 = 0.f, qs4 = 0.f;
    const __half* qrow = p.q + (static_cast<size_t>(row) * p.Hq + kvh * p.g + (gr < p.g ? gr : 0)) * D;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        __half2 v = __floats2half2_rn(0.f, 0.f);
        if (gr < p.g) v = __halves2half2(qrow[coef64(j, 2 * c)], qrow[coef64(j, 2 * c + 1)]);
        qa[j] = h2_bits(v);
        const float2 f = __half22float2(v);
        if (j == 0) qs8 += f.x + f.y;
        else qs4 += f.x + f.y;
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        qs8 += __shfl_xor_sync(0xffffffffu, qs8, o);
        qs4 += __shfl_xor_sync(0xffffffffu, qs4, o);
    }
    const uint32_t none = 0u;  // rows 8-15 of a fragment

    float O[8][2], m_run = -INFINITY, l = 0.f, zs8 = 0.f, zs4 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) O[j][0] = O[j][1] = 0.f;
    const float kScore = 1.4426950408889634f * 0.125f;  // log2(e) / sqrt(64)
    const uint32_t k_addr = smem_u32(Kt) + (lane & 7) * kPitch + (lane >> 3) * 16;
    const uint32_t v_addr = smem_u32(Vt) + ((lane & 7) + ((lane >> 3) & 1) * 8) * kPitch + (lane >> 4) * 16;

    int buf = 0;
    for (int s = first; s < n_steps; s += stride, buf ^= 1) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();  // the step's bytes are in place and nobody reads the previous tiles
        const uint8_t* rb = raw + buf * kBlock;
        const int j0 = s * kStep;
        // ---- expand: chunks of eight coefficients, lane = position.  Every word is read before the first chunk is written: one by one
        // they would each wait for shared memory (16 rows of 2048 positions, 8 KV heads, with the append: 21.7 -> 19.7 us).
        {
            uint32_t w4[2][7];
            uint2 w8[2];
            float4 m[2];
#pragma unroll
            for (int is_v = 0; is_v < 2; ++is_v) {
                const uint8_t* half_base = rb + is_v * kHalf;
                w8[is_v] = *reinterpret_cast<const uint2*>(half_base + lane * R8);
#pragma unroll
                for (int j = 0; j < 7; ++j) w4[is_v][j] = *reinterpret_cast<const uint32_t*>(half_base + kC8 + lane * (N4 / 2) + 4 * j);
                m[is_v] = *reinterpret_cast<const float4*>(half_base + kC8 + kC4 + lane * 16);
            }
            uint4* krow = reinterpret_cast<uint4*>(Kt + lane * kPitch);
            uint4* vrow = reinterpret_cast<uint4*>(Vt + lane * kPitch);
            krow[0] = bytes_centred(w8[0]);
            vrow[0] = bytes_centred_bf16(w8[1]);
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                krow[1 + j] = nibbles_centred(w4[0][j]);
                vrow[1 + j] = nibbles_centred_bf16(w4[1][j]);
            }
            // per-position constants; positions past the row's last hold anything and are zeroed by selection
#pragma unroll
            for (int is_v = 0; is_v < 2; ++is_v) {
                if (j0 + lane >= limit) m[is_v] = make_float4(0.f, 0.f, 0.f, 0.f);
                m[is_v].y = fmaf(128.f, m[is_v].x, m[is_v].y);
                m[is_v].w = fmaf(8.f, m[is_v].z, m[is_v].w);
            }
            colK[lane] = make_float4(m[0].x * kScore, m[0].y * kScore, m[0].z * kScore, m[0].w * kScore);
            colV[lane] = m[1];
        }
        __syncwarp();
        issue(s + 2 * stride, buf);  // everybody is done with this raw buffer

        // ---- scores
        float sc[kNT][2];
        float mx = -INFINITY;
        const bool masked = j0 + kStep > limit;
#pragma unroll
        for (int nt = 0; nt < kNT; ++nt) {
            uint32_t k0[4], k1[4];
            ldsm4(k0, k_addr + nt * 8 * kPitch);
            ldsm4(k1, k_addr + nt * 8 * kPitch + 64);
            float s8[4] = {0.f, 0.f, 0.f, 0.f}, s4[4] = {0.f, 0.f, 0.f, 0.f};
            mma8(s8, qa[0], none, k0[0]);
            mma16(s4, qa[1], none, qa[2], none, k0[1], k0[2]);
            mma16(s4, qa[3], none, qa[4], none, k0[3], k1[0]);
            mma16(s4, qa[5], none, qa[6], none, k1[1], k1[2]);
            mma8(s4, qa[7], none, k1[3]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int pos = 8 * nt + 2 * c + e;
                const float4 k = colK[pos];
                float x = fmaf(k.x, s8[e], fmaf(k.z, s4[e], fmaf(k.y, qs8, k.w * qs4)));
                if (masked && j0 + pos >= limit) x = -INFINITY;
                sc[nt][e] = x;
                mx = fmaxf(mx, x);
            }
        }
        // ---- running maximum
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx), m_use = m_new == -INFINITY ? 0.f : m_new;
        const float corr = exp2_approx(m_run - m_use);
        const bool moved = m_new != m_run;
        m_run = m_new;
        if (__any_sync(0xffffffffu, moved)) {
            l *= corr;
            zs8 *= corr;
            zs4 *= corr;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                O[j][0] *= corr;
                O[j][1] *= corr;
            }
        }
        // ---- weights and the second product: the tensor core's fp32 sums are truncated, so a chain of products runs over
        // 32 positions only and is then added to the running sums with rounding.  The middle part of a weight takes the unused rows
        // of the first one's product.
        uint32_t p8[2][2][4], p4[2][2][4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int pos = 8 * t + 2 * c, i = 2 * (t & 1);
            const float4 va = colV[pos], vb = colV[pos + 1];
            uint32_t w8[3], w4[3];
            const float pa = exp2_approx(sc[t][0] - m_use), pb = exp2_approx(sc[t][1] - m_use);
            l += pa + pb;
            zs8 = fmaf(pa, va.y, fmaf(pb, vb.y, zs8));
            zs4 = fmaf(pa, va.w, fmaf(pb, vb.w, zs4));
            split_bf16(pa * va.x, pb * vb.x, w8);
            split_bf16(pa * va.z, pb * vb.z, w4);
            p8[t >> 1][0][i] = w8[0];
            p8[t >> 1][0][i + 1] = w8[1];
            p8[t >> 1][1][i] = w8[2];
            p4[t >> 1][0][i] = w4[0];
            p4[t >> 1][0][i + 1] = w4[1];
            p4[t >> 1][1][i] = w4[2];
            p8[t >> 1][1][i + 1] = p4[t >> 1][1][i + 1] = none;
        }
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
            uint32_t v[2][4];
            ldsm4t(v[0], v_addr + j * 16);
            ldsm4t(v[1], v_addr + 16 * kPitch + j * 16);
#pragma unroll
            for (int k = 1; k >= 0; --k)  // the small parts first
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    mma16_bf16(d0, j == 0 ? p8[ks][k] : p4[ks][k], v[ks][0], v[ks][1]);
                    mma16_bf16(d1, p4[ks][k], v[ks][2], v[ks][3]);
                }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                O[j][e] += d0[e] + d0[2 + e];
                O[j + 1][e] += d1[e] + d1[2 + e];
            }
        }
    }

    // ---- records of the warps (unnormalised sums with the zero-points, maximum, sum of weights) over their tiles, then the merge
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        l += __shfl_xor_sync(0xffffffffu, l, o);
        zs8 += __shfl_xor_sync(0xffffffffu, zs8, o);
        zs4 += __shfl_xor_sync(0xffffffffu, zs4, o);
    }
    float* r = reinterpret_cast<float*>(raw) + gr * kRecPitch;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float z = j == 0 ? zs8 : zs4;
        r[coef64(j, 2 * c)] = O[j][0] + z;
        r[coef64(j, 2 * c + 1)] = O[j][1] + z;
    }
    if (c == 0) {
        r[D] = m_run;
        r[D + 1] = l;
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
