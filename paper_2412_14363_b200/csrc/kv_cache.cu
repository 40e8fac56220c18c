// Attention-block path, cache side (Section 4.3, Eq. 8; Section 5.1), d_head = 128 and 64: the 8-bit online U_C
// projection of query and key head vectors, and the per-head asymmetric 8/4-bit quantizer that writes key and value
// into the blocked cache.  A few MB per call at most.  Two forms, chosen by the number of head vectors (launch_project):
//
// kv_project_kernel (many): one warp owns 16 consecutive head vectors (rows) and contracts them on mma.sync s8
// fragments taken straight from the global loads.  Lane (g, c) = (lane / 4, lane % 4) loads, for rows g and g + 8, the
// elements [32 ks + 4c, +4) and [32 ks + 16 + 4c, +4): exactly the bytes of its A fragments of mma.m16n8k32, and 32
// contiguous bytes per quad, so every sector fetched is used.
//
// head_vector_kernel (few, a generation step): one warp per head vector, lane l owning coefficients l + 32 i, dp4a
// against U_C's codes in shared memory.  A step is latency: one vector's chain is shorter than a 16-vector tile's and so is
// the code, which counts in a step, where every kernel runs once between others.  16 tokens (512 query, 256 key and value
// vectors) at d = 128: 15.0 -> 8.6 us by themselves, 37 -> 10.6 us right after an attention call on a 140 MB cache.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "internal.h"
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
    static constexpr int kWStride = D + 16;  // bytes per staged W_C row: the 8 rows of a B fragment hit 8 bank groups
    static constexpr int kRec = kR8 + kB4 + 16;                // staged record: code bytes, 4 floats
};
static_assert(Head<128>::kBlock == RESQ_KV_BLOCK_BYTES, "block layout");
// Head vectors of a call up to which one warp takes one of them.  Event times in us, one per warp / 16 per warp, 32 + 16
// vectors per token: d = 128, 128 tokens 12.9 / 15.0, 256 tokens 16.8 / 16.8, 512 tokens 25.0 / 17.0; d = 64, 256 tokens
// 10.9 / 12.7, 512 tokens 15.2 / 12.7.
constexpr long long kFewVectors = 12288;
constexpr float kMagic = 12582912.f;  // 1.5 * 2^23

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

// The lane's D / 4 elements of one row as fp32: v[8 ks + i] = x[32 ks + 4c + i], v[8 ks + 4 + i] = x[32 ks + 16 + 4c + i].
template <int D>
__device__ __forceinline__ void load_row(const __nv_bfloat16* row, int c, bool live, float (&v)[D / 4]) {
#pragma unroll
    for (int ks = 0; ks < D / 32; ++ks)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            uint2 u = make_uint2(0u, 0u);
            if (live) u = *reinterpret_cast<const uint2*>(row + 32 * ks + 16 * hf + 4 * c);
            float* o = v + 8 * ks + 4 * hf;
            o[0] = __uint_as_float(u.x << 16); o[1] = __uint_as_float(u.x & 0xFFFF0000u);
            o[2] = __uint_as_float(u.y << 16); o[3] = __uint_as_float(u.y & 0xFFFF0000u);
        }
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
        exact = needs_division(inv);
    }
    __device__ __forceinline__ uint32_t code(float x, float qmax) const {
        if (!(s > 0.f)) return 0u;
        const float q = code_rn(__fsub_rn(x, z), s, inv, exact, 0.5f - 0.00006103515625f);
        return static_cast<uint32_t>(fminf(fmaxf(q, 0.f), qmax));
    }
};

// Where the record of head vector `row` goes: (block index) * 32 + slot in the block, or -1.
__device__ __forceinline__ long long cache_slot(long long row, int n_kv_heads, int n_seqs, int capacity,
                                                const int32_t* seq_ids, const int32_t* positions, int* status) {
    const long long t = row / n_kv_heads;
    const int h = static_cast<int>(row - t * n_kv_heads);
    const int b = seq_ids[t], pos = positions[t];
    if (b < 0 || b >= n_seqs || pos < 0 || pos >= capacity) {
        atomicOr(status, kStatusBitIndex);
        return -1;
    }
    const long long blk = (static_cast<long long>(b) * n_kv_heads + h) * (capacity / RESQ_KV_BLOCK) + pos / RESQ_KV_BLOCK;
    return blk * RESQ_KV_BLOCK + (pos % RESQ_KV_BLOCK);
}

// Copies the 16 staged records of a warp tile into the cache blocks (key: half 0, value: half 1).
template <int D>
__device__ __forceinline__ void flush_records(const uint8_t* rec, const long long* slot, uint8_t* cache, int half,
                                              int lane) {
    using H = Head<D>;
    using Unit = typename std::conditional<D == 128, uint2, uint32_t>::type;  // what divides every part of a record
    constexpr int kU = sizeof(Unit), kN8 = H::kR8 / kU, kN4 = H::kB4 / kU, kN = H::kRec / kU;
    for (int u = lane; u < 16 * kN; u += 32) {
        const int row = u / kN, part = u - row * kN;
        const long long sl = slot[row];
        if (sl < 0) continue;
        uint8_t* blk = cache + (sl / RESQ_KV_BLOCK) * H::kBlock + half * H::kHalf;
        const int p = static_cast<int>(sl % RESQ_KV_BLOCK);
        uint8_t* dst = part < kN8         ? blk + p * H::kR8 + part * kU
                       : part < kN8 + kN4 ? blk + H::kC8 + p * H::kB4 + (part - kN8) * kU
                                          : blk + H::kC8 + H::kC4 + p * 16 + (part - kN8 - kN4) * kU;
        *reinterpret_cast<Unit*>(dst) = *reinterpret_cast<const Unit*>(rec + row * H::kRec + part * kU);
    }
}

// Symmetric INT8 codes of the lane's part of two rows, packed as the A fragments a[ks][0..3]; returns the scales.
template <int D>
__device__ __forceinline__ void sym8_fragments(const float (&xv)[2][D / 4], uint32_t (&a)[D / 32][4], float (&sx)[2]) {
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < D / 4; ++i) m = fmaxf(m, fabsf(xv[rr][i]));
        m = quad_max(m);
        const float s = __fdiv_rn(m, 127.f);
        const float inv = s > 0.f ? __frcp_rn(s) : 0.f;
        const bool exact = needs_division(inv);
        sx[rr] = s;
#pragma unroll
        for (int ks = 0; ks < D / 32; ++ks)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t w = 0;
                if (s > 0.f) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float q = code_rn(xv[rr][8 * ks + 4 * hf + i], s, inv, exact, 0.5f - 0.000030517578125f);
                        w |= (static_cast<uint32_t>(static_cast<int>(q)) & 0xFFu) << (8 * i);
                    }
                }
                a[ks][2 * hf + rr] = w;  // a0: row g, k 4c..; a1: row g+8; a2: row g, k 16+4c..; a3: row g+8
            }
    }
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
};

// Ranges of the two segments of a row held by a quad: the lane's values 0 .. N8 - 1 are in the 8-bit segment where in8,
// else in the 4-bit one with the rest.
template <int N8, int N>
__device__ __forceinline__ void quad_ranges(const float* v, bool in8, float (&lohi)[4]) {
    float lo8 = 3.402823466e38f, hi8 = -3.402823466e38f, lo4 = lo8, hi4 = hi8;
#pragma unroll
    for (int i = N8; i < N; ++i) { lo4 = fminf(lo4, v[i]); hi4 = fmaxf(hi4, v[i]); }
#pragma unroll
    for (int i = 0; i < N8; ++i) {
        if (in8) { lo8 = fminf(lo8, v[i]); hi8 = fmaxf(hi8, v[i]); }
        else { lo4 = fminf(lo4, v[i]); hi4 = fmaxf(hi4, v[i]); }
    }
    lohi[0] = quad_min(lo8); lohi[1] = quad_max(hi8); lohi[2] = quad_min(lo4); lohi[3] = quad_max(hi4);
}

// W_C's codes and scales into shared memory.
template <int D>
__device__ __forceinline__ void stage_uc(const int8_t* wq, const float* s_u, uint8_t* w_s, float* su_s) {
    for (int i = threadIdx.x; i < D * (D / 16); i += blockDim.x) {  // 16-byte pieces
        const int n = i / (D / 16), pc = i % (D / 16);
        *reinterpret_cast<uint4*>(w_s + n * Head<D>::kWStride + pc * 16) = reinterpret_cast<const uint4*>(wq + n * D)[pc];
    }
    for (int i = threadIdx.x; i < D; i += blockDim.x) su_s[i] = s_u[i];
}

// One warp per tile of 16 head vectors; the tiles of a call are the query tiles (projected, written as half),
// then the key tiles (projected, quantized, appended), then the value tiles (quantized, appended).
template <int D>
__global__ void __launch_bounds__(kWarps * 32) kv_project_kernel(const ProjectParams p) {
    using H = Head<D>;
    constexpr int KS = D / 32, NT = D / 8;
    __shared__ __align__(16) uint8_t w_s[D * H::kWStride];
    __shared__ float su_s[D];
    __shared__ __align__(16) uint8_t rec_s[kWarps][16 * H::kRec];
    __shared__ long long slot_s[kWarps][16];
    griddep_wait();  // launched with programmatic stream serialization
    griddep_launch_dependents();
    stage_uc<D>(p.wq, p.s_u, w_s, su_s);
    __syncthreads();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    const long long q_tiles = (p.q_rows + 15) / 16, kv_tiles = (p.kv_rows + 15) / 16, tiles = q_tiles + 2 * kv_tiles;
    uint8_t* rec = rec_s[warp];
    for (long long tile = static_cast<long long>(blockIdx.x) * kWarps + warp; tile < tiles;
         tile += static_cast<long long>(gridDim.x) * kWarps) {
        const int kind = tile < q_tiles ? 0 : (tile < q_tiles + kv_tiles ? 1 : 2);  // query, key, value
        const long long t0 = kind == 0 ? tile : (kind == 1 ? tile - q_tiles : tile - q_tiles - kv_tiles);
        const long long rows = kind == 0 ? p.q_rows : p.kv_rows;
        const __nv_bfloat16* x = kind == 0 ? p.q : (kind == 1 ? p.k : p.v);
        const long long r0 = t0 * 16 + g, r1 = r0 + 8;
        const bool live0 = r0 < rows, live1 = r1 < rows;
        float xv[2][D / 4];
        load_row<D>(x + r0 * D, c, live0, xv[0]);
        load_row<D>(x + r1 * D, c, live1, xv[1]);
        if (kind != 0 && lane < 16) {
            const long long r = t0 * 16 + lane;
            slot_s[warp][lane] = r < rows ? cache_slot(r, p.n_kv_heads, p.n_seqs, p.capacity, p.seq_ids, p.positions, p.status) : -1;
        }
        if (kind == 2) {
            // ---- value: the bf16 head vectors quantized directly; elements 0-3 of the lane are columns
            // [4c, 4c + 4): the 8-bit segment, of which D = 64 has only the quad's first two lanes
            const bool in8 = 4 * c < H::kR8;
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                float lohi[4];
                quad_ranges<4, D / 4>(xv[rr], in8, lohi);
                const Asym q8(lohi[0], lohi[1], 255.f), q4(lohi[2], lohi[3], 15.f);
                uint8_t* rrow = rec + (g + 8 * rr) * H::kRec;
                if (in8) {
                    uint32_t w8 = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) w8 |= q8.code(xv[rr][i], 255.f) << (8 * i);
                    *reinterpret_cast<uint32_t*>(rrow + 4 * c) = w8;
                }
#pragma unroll
                for (int ks = 0; ks < KS; ++ks)
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        if (ks == 0 && hf == 0 && in8) continue;
                        const float* e = xv[rr] + 8 * ks + 4 * hf;
                        const int col = 32 * ks + 16 * hf + 4 * c;  // >= kR8
                        *reinterpret_cast<uint16_t*>(rrow + H::kR8 + (col - H::kR8) / 2) = static_cast<uint16_t>(
                            q4.code(e[0], 15.f) | (q4.code(e[1], 15.f) << 4) | (q4.code(e[2], 15.f) << 8) | (q4.code(e[3], 15.f) << 12));
                    }
                if (c == 0) {
                    float* m = reinterpret_cast<float*>(rrow + H::kR8 + H::kB4);
                    m[0] = q8.s; m[1] = q8.z; m[2] = q4.s; m[3] = q4.z;
                }
            }
            __syncwarp();
            flush_records<D>(rec, slot_s[warp], p.cache, 1, lane);
            __syncwarp();
            continue;
        }
        float sx[2];
        uint32_t a[KS][4];
        sym8_fragments<D>(xv, a, sx);
        // ---- y = x W_C^T: column tiles of 8, exact int32
        int acc[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0;
            const uint8_t* wrow = w_s + (8 * nt + g) * H::kWStride + 4 * c;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
                mma_s8(acc[nt], a[ks], *reinterpret_cast<const uint32_t*>(wrow + 32 * ks),
                       *reinterpret_cast<const uint32_t*>(wrow + 32 * ks + 16));
        }
        // y[row g][8 nt + 2c + e] = acc[nt][e], y[row g + 8][...] = acc[nt][2 + e]
        if (kind == 0) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const float u0 = su_s[8 * nt + 2 * c], u1 = su_s[8 * nt + 2 * c + 1];
                if (live0)
                    *reinterpret_cast<__half2*>(p.q_out + r0 * D + 8 * nt + 2 * c) = __floats2half2_rn(
                        __fmul_rn(static_cast<float>(acc[nt][0]), __fmul_rn(sx[0], u0)),
                        __fmul_rn(static_cast<float>(acc[nt][1]), __fmul_rn(sx[0], u1)));
                if (live1)
                    *reinterpret_cast<__half2*>(p.q_out + r1 * D + 8 * nt + 2 * c) = __floats2half2_rn(
                        __fmul_rn(static_cast<float>(acc[nt][2]), __fmul_rn(sx[1], u0)),
                        __fmul_rn(static_cast<float>(acc[nt][3]), __fmul_rn(sx[1], u1)));
            }
            continue;
        }
        // ---- key: asymmetric 8/4-bit codes of the fp32 coefficients (the first D / 64 column tiles are the 8-bit segment)
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            float y[D / 4];  // y[2 nt + e]
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    y[2 * nt + e] = __fmul_rn(static_cast<float>(acc[nt][2 * rr + e]), __fmul_rn(sx[rr], su_s[8 * nt + 2 * c + e]));
            float lohi[4];
            quad_ranges<2 * (D / 64), D / 4>(y, true, lohi);
            const Asym q8(lohi[0], lohi[1], 255.f), q4(lohi[2], lohi[3], 15.f);
            uint8_t* rrow = rec + (g + 8 * rr) * H::kRec;
#pragma unroll
            for (int nt = 0; nt < D / 64; ++nt)
                *reinterpret_cast<uint16_t*>(rrow + 8 * nt + 2 * c) =
                    static_cast<uint16_t>(q8.code(y[2 * nt], 255.f) | (q8.code(y[2 * nt + 1], 255.f) << 8));
#pragma unroll
            for (int nt = D / 64; nt < NT; ++nt)
                rrow[H::kR8 + 4 * (nt - D / 64) + c] = static_cast<uint8_t>(q4.code(y[2 * nt], 15.f) | (q4.code(y[2 * nt + 1], 15.f) << 4));
            if (c == 0) {
                float* m = reinterpret_cast<float*>(rrow + H::kR8 + H::kB4);
                m[0] = q8.s; m[1] = q8.z; m[2] = q4.s; m[3] = q4.z;
            }
        }
        __syncwarp();
        flush_records<D>(rec, slot_s[warp], p.cache, 0, lane);
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

// One warp per head vector, lane l owning coefficients l + 32 i; items in the order of kv_project_kernel.
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
            if (lane == 0) slot = cache_slot(row, p.n_kv_heads, p.n_seqs, p.capacity, p.seq_ids, p.positions, p.status);
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
            uint8_t* half = p.cache + (slot / RESQ_KV_BLOCK) * H::kBlock + (kind == 2 ? H::kHalf : 0);
            const int ps = static_cast<int>(slot % RESQ_KV_BLOCK);
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
    const auto grid = [](long long warps) {
        const long long ctas = (warps + kWarps - 1) / kWarps;
        return static_cast<unsigned>(ctas < 148 * 8 ? ctas : 148 * 8);
    };
    if (vectors <= kFewVectors)
        return launch_programmatic(head_vector_kernel<D>, grid(vectors), kWarps * 32, 0, st, p);
    return launch_programmatic(kv_project_kernel<D>, grid((p.q_rows + 15) / 16 + 2 * ((p.kv_rows + 15) / 16)), kWarps * 32, 0, st, p);
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
