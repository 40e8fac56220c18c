// Causal attention of a run of new tokens over the quantized KV cache (Section 4.3, Eq. 8; cache format of
// Section 5.1) on the tcgen05 tensor cores: the prefill form, where every cache block is read once per CTA instead of
// once per query.
//
// A CTA owns NT = 2 (or 1) tiles of 128 rows that share a KV head -- rows are (token, query head) pairs, tokens ascending
// -- and walks the cache of its sequence in steps of 64 positions (two cache blocks).  Roles (13 or 9 warps):
//   expand   4 warps: raw blocks (bulk copies, two steps ahead) -> the codes as exact fp16 integers, centred (code - 128,
//            code - 8), in operand tiles [position][coefficient]: keys K-major, values N-major (so neither is
//            transposed), and the step's per-position constants.  Two stages.
//   mma      one warp: S8 = Q[:, :16] C8^T and S4 = Q[:, 16:] C4^T into TMEM; later O8 += P8 C8v, O4 += P4 C4v with the
//            weights taken from TMEM.
//   softmax  4 warps per tile, one row per thread: score = s8 S8 + s4 S4 + (z8 + 128 s8) sum(q8) + (z4 + 8 s4) sum(q4) in
//            fp32 minus the row's reference, p = 2^score, sums of p and of p (z + c0 s) in fp32, and the operands
//            P8 = half(p s8_v 2^-E), P4 = half(p s4_v 2^-E) written over the S8 columns it has just read.
// 2^E is the largest finite value scale of the positions the CTA visits (read ahead of the walk), so the products stay in
// half's normal range.  The reference of a row is the maximum of its first step and is raised only when a score exceeds
// it by 2^8; that rare step rescales the row's output accumulator in TMEM.  So there is one pass over the cache, weights
// are at most 2^8 (half holds 2^16) and no smaller against the row's maximum than with an exact one.
// While one tile's softmax runs, the other tile's products do; the stages let the expansion run a step ahead.  With few
// CTAs a cluster splits the steps and rank 0 merges the sums through distributed shared memory.
//
// The coefficients of a 32-bit word of nibbles are kept in the order 0 4 1 5 2 6 3 7 (one shift and mask per pair of
// tile elements); the query tile is written in the same order and the output un-permuted on the way out.
// Positions beyond a row's own are masked by selection in the scores; the constants of positions past the tile's last are
// zeroed by selection, and so are a value's constants that are not finite (they would turn a hidden position's weight of 0 into
// NaN); the first such position is noted for the rows that do see it.  So unwritten cache positions of a loaded block, and later
// tokens, may hold anything.  All waits are bounded; after a failed wait every role leaves its loop, copies and products in
// flight are waited for, and TMEM is freed.
//
// What bounds it: shared-memory traffic (the softmax constants come as broadcasts, two wavefronts per 16 bytes, beside the
// tensor core's reads of Q, K and V) and the latency of a row's chain S -> weights -> O -> next S, about 4300 cycles per
// step of 256 rows; not HBM, not the tensor pipe (42 %).  32 query / 8 KV heads, 2048 tokens behind 4096: 1310 us with
// one 128-row tile per CTA whose phases follow one another in two passes, 404 us as it stands (431 with the products
// issued by a thread alone in a branch).
#include "centred_codes.cuh"
#include "internal.h"
#include "plans.h"
#include "ptx.cuh"

#include <cuda_fp16.h>

#include <cfloat>
#include <climits>

namespace resq {
namespace {

constexpr int kRows = 128;          // rows of a tile = TMEM lanes
constexpr int kStep = 64;           // cache positions per step
constexpr int kBlockBytes = RESQ_KV_BLOCK_BYTES;
constexpr int kOffK4 = 512, kOffKm = 2304, kOffV8 = 2816, kOffV4 = 3328, kOffVm = 5120;
constexpr int kQBytes = 2 * kRows * 128;       // two 64-coefficient halves of [128 rows][128 B]
constexpr int kKBytes = 2 * kStep * 128;       // keys: two 64-coefficient halves of [64 positions][128 B]
constexpr int kV4Bytes = 2 * kStep * 128;      // 4-bit values: coefficients 0-63 and 64-111 of [64 positions][128 B]
constexpr int kV8Bytes = kStep * 128;          // 8-bit values: 16 coefficients of [64 positions][128 B]
constexpr int kStageBytes = kKBytes + kV4Bytes + kV8Bytes;
constexpr int kRawBytes = 2 * kBlockBytes;
constexpr uint32_t kColS8 = 0, kColS4 = 64, kColO4 = 128, kColO8 = 240, kTileCols = 256;  // TMEM columns of a tile
constexpr uint32_t kColP8 = 0, kColP4 = 32;    // the weights, two halves per column, over S8
constexpr int kExpandWarps = 4;
constexpr int kRecPitch = 132;      // floats per row of a record: 128 sums, reference, sum of weights
constexpr float kSlack = 8.f;       // log2 of the largest weight before a row's reference is raised

struct Shared {
    // per stage and pair of positions: keys (s8 s8 s4 s4) (z8 z8 z4 z4) times log2(e) / sqrt(d), the zero-points with the
    // centre; values (s8 s8 s4 s4) times 2^-E, (z8 z8 z4 z4) with the centre
    float4 col_k[2][kStep], col_v[2][kStep];
    float warp_max[16];
    int bad8, bad4;  // the first position visited whose value constants of the 8-bit / 4-bit segment are infinite or NaN
    uint64_t raw_full[2], kv_full[2], kv_empty[2], s_full[2], p_full[2], pv_done[2], drain;
    uint32_t tmem_base;
    int abort_flag;
};

template <int NT>
struct Geometry {
    static constexpr int kSoftmaxWarps = 4 * NT;
    static constexpr int kMmaWarp = kSoftmaxWarps + kExpandWarps;
    static constexpr int kThreads = 32 * (kMmaWarp + 1);
    static constexpr size_t kTiles = static_cast<size_t>(NT) * kQBytes + 2 * kStageBytes;
    static constexpr size_t kSmem = 1024 + kTiles + 2 * kRawBytes + sizeof(Shared);
};
static_assert(Geometry<2>::kSmem <= 227 * 1024, "one CTA per SM");
static_assert(Geometry<2>::kTiles >= 2 * kRows * kRecPitch * 4 && Geometry<1>::kTiles >= kRows * kRecPitch * 4, "records fit");

struct PrefillParams {
    const uint8_t* blocks;  // first cache block of the sequence (KV head 0)
    size_t head_stride;     // bytes between the KV heads of the sequence
    const __half* q;        // [T][Hq][128]
    float* out;             // [T][Hq][128]
    int T, Hq, Hkv, g, pos0, splits;
    int* status;
};

__host__ __device__ constexpr uint32_t make_idesc_f16(int M, int N) {  // f16 x f16 -> f32, K-major A and B
    return (1u << 4) | (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
constexpr uint32_t kBNMajor = 1u << 16;

// Packed fp32 pairs.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// Two pairs from shared memory, where the program has it (hoisted reads would not fit the registers).
struct f2x2 {
    f2 x, y;
};
__device__ __forceinline__ f2x2 lds_pairs(const float4* src) {
    f2x2 d;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(d.x), "=l"(d.y) : "r"(smem_u32(src)));
    return d;
}
// Values of TMEM loads that a wait has completed: nothing that reads them moves above this point.
__device__ __forceinline__ void arrived(uint32_t (&v)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) asm volatile("" : "+r"(v[i]));
}
__device__ __forceinline__ uint32_t half_pair(f2 v) {
    const float2 f = unpack2(v);
    const __half2 h = __floats2half2_rn(f.x, f.y);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// One step of the expanding warps: thread = (position tid % 64, chunk parity tid / 64).  The constants of
// positions from n_valid on, and a value's that are not finite, become 0; bad8 / bad4 note the latter (j0: the first position).
__device__ __forceinline__ void expand_step(const uint8_t* raw, uint8_t* stage, float4* col_k, float4* col_v, int tid,
                                            int n_valid, float p_scale, int j0, int* bad8, int* bad4) {
    const int j = tid & 63, jp = j & 31, par = tid >> 6, sw = j & 7;
    const uint8_t* blk = raw + (j >> 5) * kBlockBytes;
    uint8_t* krow = stage + j * 128;
    uint8_t* vrow = stage + kKBytes + j * 128;
    uint8_t* v8row = stage + kKBytes + kV4Bytes + j * 128;
    const uint32_t* k4 = reinterpret_cast<const uint32_t*>(blk + kOffK4 + jp * 56);
    const uint32_t* v4 = reinterpret_cast<const uint32_t*>(blk + kOffV4 + jp * 56);
    // chunk 0-1 of a key row: the 8-bit segment; chunks 2-15: words 0-13 of nibbles (chunk / 8: the tile's half)
    *reinterpret_cast<uint4*>(krow + ((par ^ sw) << 4)) = bytes_centred(*reinterpret_cast<const uint2*>(blk + jp * 16 + 8 * par));
    *reinterpret_cast<uint4*>(v8row + ((par ^ sw) << 4)) = bytes_centred(*reinterpret_cast<const uint2*>(blk + kOffV8 + jp * 16 + 8 * par));
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const int w = 2 * i + par, ch = w + 2;
        *reinterpret_cast<uint4*>(krow + (ch >> 3) * (kStep * 128) + (((ch & 7) ^ sw) << 4)) = nibbles_centred(k4[w]);
        *reinterpret_cast<uint4*>(vrow + (w >> 3) * (kStep * 128) + (((w & 7) ^ sw) << 4)) = nibbles_centred(v4[w]);
    }
    // constants: threads 0-63 the keys', 64-127 the values'; pair j / 2, element j % 2 of each pair
    const bool is_v = par != 0;
    float4 m = *reinterpret_cast<const float4*>(blk + (is_v ? kOffVm : kOffKm) + jp * 16);
    if (j >= n_valid) m = make_float4(0.f, 0.f, 0.f, 0.f);
    m.y = fmaf(128.f, m.x, m.y);
    m.w = fmaf(8.f, m.z, m.w);
    if (is_v && !(fabsf(m.x) <= FLT_MAX && fabsf(m.y) <= FLT_MAX)) {
        m.x = m.y = 0.f;
        atomicMin(bad8, j0 + j);
    }
    if (is_v && !(fabsf(m.z) <= FLT_MAX && fabsf(m.w) <= FLT_MAX)) {
        m.z = m.w = 0.f;
        atomicMin(bad4, j0 + j);
    }
    const float kScore = 1.4426950408889634f * 0.08838834764831845f;  // log2(e) / sqrt(128)
    const float fs = is_v ? p_scale : kScore, fz = is_v ? 1.f : kScore;
    float* dst = reinterpret_cast<float*>(is_v ? col_v : col_k) + (j >> 1) * 8 + (j & 1);
    dst[0] = m.x * fs;
    dst[2] = m.z * fs;
    dst[4] = m.y * fz;
    dst[6] = m.w * fz;
}

// Running state of a row, by the parity of the position.
struct RowState {
    float m;       // reference, log2 units; -inf: no position seen yet
    f2 l, z8, z4;  // sums of p and of p times the zero-points (with the centre)
};

// Scores of one step minus the row's reference, as 32 pairs; returns their maximum.  Positions of the step beyond `last` are
// hidden from the row.
template <bool MASKED>
__device__ __forceinline__ float step_scores(f2 (&sc)[32], uint32_t tmem_s, const float4* col_k, int last, f2 q8, f2 q4, float neg_m) {
    const f2 nm = pack2(neg_m, neg_m);
    float mx = -INFINITY;
    uint32_t a8[2][8], a4[2][8];
    tmem_ld8(tmem_s + kColS8, a8[0]);
    tmem_ld8(tmem_s + kColS4, a4[0]);
#pragma unroll
    for (int part = 0; part < 8; ++part) {  // eight positions; the next eight are on their way
        tmem_ld_wait();
        arrived(a8[part & 1]);
        arrived(a4[part & 1]);
        if (part < 7) {
            tmem_ld8(tmem_s + kColS8 + 8 * (part + 1), a8[(part + 1) & 1]);
            tmem_ld8(tmem_s + kColS4 + 8 * (part + 1), a4[(part + 1) & 1]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int pr = 4 * part + i;
            const f2x2 s = lds_pairs(col_k + 2 * pr);
            const f2x2 z = lds_pairs(col_k + 2 * pr + 1);
            const f2 v8 = pack2(__uint_as_float(a8[part & 1][2 * i]), __uint_as_float(a8[part & 1][2 * i + 1]));
            const f2 v4 = pack2(__uint_as_float(a4[part & 1][2 * i]), __uint_as_float(a4[part & 1][2 * i + 1]));
            sc[pr] = fma2(s.x, v8, fma2(s.y, v4, fma2(z.x, q8, fma2(z.y, q4, nm))));
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

// Weights of one step: their sums into the row's state, the operands of the output product over the scores in TMEM.
__device__ __forceinline__ void step_weights(RowState& st, const f2 (&sc)[32], uint32_t tmem_row, const float4* col_v) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t w8[8], w4[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int pr = 8 * c + i;
            const f2x2 s = lds_pairs(col_v + 2 * pr);
            const f2x2 z = lds_pairs(col_v + 2 * pr + 1);
            const float2 f = unpack2(sc[pr]);
            const f2 e = pack2(exp2_approx(f.x), exp2_approx(f.y));
            st.l = add2(st.l, e);
            st.z8 = fma2(e, z.x, st.z8);
            st.z4 = fma2(e, z.y, st.z4);
            w8[i] = half_pair(mul2(e, s.x));
            w4[i] = half_pair(mul2(e, s.y));
        }
        tmem_st8(tmem_row + kColP8 + 8 * c, w8);
        tmem_st8(tmem_row + kColP4 + 8 * c, w4);
    }
}

template <int NT>
__global__ void __launch_bounds__(Geometry<NT>::kThreads, 1) attention_prefill_kernel(const PrefillParams p) {
    using G = Geometry<NT>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* Qs = base;
    uint8_t* stages = Qs + NT * kQBytes;
    uint8_t* raw = stages + 2 * kStageBytes;
    Shared* sh = reinterpret_cast<Shared*>(raw + 2 * kRawBytes);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = static_cast<int>(blockIdx.x % p.splits), item = static_cast<int>(blockIdx.x / p.splits);
    const int kvh = item % p.Hkv, n_tiles = static_cast<int>(gridDim.x) / p.splits / p.Hkv;
    const int R0 = (n_tiles - 1 - item / p.Hkv) * NT * kRows;  // long tiles of all heads first
    const int pos_first = p.pos0 + R0 / p.g;                    // position of the first row: the smallest
    const int limit = p.pos0 + min(p.T - 1, (R0 + NT * kRows - 1) / p.g) + 1;  // positions any row sees
    const int all_steps = (limit + kStep - 1) / kStep;
    const int first = static_cast<int>(static_cast<long long>(all_steps) * rank / p.splits);
    const int n_steps = static_cast<int>(static_cast<long long>(all_steps) * (rank + 1) / p.splits) - first;
    const int n_blocks = (limit + RESQ_KV_BLOCK - 1) / RESQ_KV_BLOCK;
    const uint8_t* blocks = p.blocks + static_cast<size_t>(kvh) * p.head_stride;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh->raw_full[i], 1);
            mbar_init(&sh->kv_full[i], 32 * kExpandWarps);
            mbar_init(&sh->kv_empty[i], 1);
            mbar_init(&sh->s_full[i], 1);
            mbar_init(&sh->p_full[i], kRows);
            mbar_init(&sh->pv_done[i], 1);
        }
        mbar_init(&sh->drain, 1);
        sh->abort_flag = 0;
        sh->bad8 = sh->bad4 = INT_MAX;
        fence_mbar_init();
    }
    if (warp == G::kMmaWarp) {
        __syncwarp();
        tmem_alloc(&sh->tmem_base, NT * kTileCols);
        tmem_relinquish();
    }

    griddep_wait();  // the set-up above ran under the tail of the preceding grid
    griddep_launch_dependents();
    // ---- the largest value scale of the positions visited
    {
        float vmax = 0.f;
        const int end = min(limit, (first + n_steps) * kStep);
        for (int j = first * kStep + tid; j < end; j += G::kThreads) {
            const float4 m = reinterpret_cast<const float4*>(blocks + static_cast<size_t>(j >> 5) * kBlockBytes + kOffVm)[j & 31];
            // a scale that is not finite makes the rows that see it infinite or NaN whatever E is
            vmax = fmaxf(vmax, fmaxf(m.x <= FLT_MAX ? m.x : 0.f, m.z <= FLT_MAX ? m.z : 0.f));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if (lane == 0) sh->warp_max[warp] = vmax;
    }
    // ---- query tiles: thread = row; the sums of the two segments stay with the row's softmax thread
    const int tile = warp >> 2;  // of a softmax warp
    const bool softmax = warp < G::kSoftmaxWarps;
    const int row = tid & (kRows - 1);
    const int R = R0 + tile * kRows + row;
    const bool row_ok = softmax && R < p.T * p.g;
    const int tq = row_ok ? R / p.g : 0, hq = kvh * p.g + (row_ok ? R % p.g : 0);
    float qsum8 = 0.f, qsum4 = 0.f;
    if (softmax) {
        const uint4* src = reinterpret_cast<const uint4*>(p.q + (static_cast<size_t>(tq) * p.Hq + hq) * 128);
        uint8_t* dst = Qs + tile * kQBytes + row * 128;
        const int sw = row & 7;
        uint4 qv[16];  // the whole row on its way before anything is stored
#pragma unroll
        for (int c = 0; c < 16; ++c) qv[c] = row_ok ? src[c] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            uint4 v = qv[c];
            const __half2* h = reinterpret_cast<const __half2*>(&v);
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(h[i]);
                s += f.x + f.y;
            }
            if (c < 2) {
                qsum8 += s;
            } else {
                qsum4 += s;
                v = make_uint4(__byte_perm(v.x, v.z, 0x5410), __byte_perm(v.x, v.z, 0x7632), __byte_perm(v.y, v.w, 0x5410),
                               __byte_perm(v.y, v.w, 0x7632));
            }
            *reinterpret_cast<uint4*>(dst + (c >> 3) * (kRows * 128) + (((c & 7) ^ sw) << 4)) = v;
        }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    float p_scale, out_scale;
    {
        float vmax = 0.f;
#pragma unroll
        for (int i = 0; i <= G::kMmaWarp; ++i) vmax = fmaxf(vmax, sh->warp_max[i]);
        int e = 0;
        if (vmax > 0.f) e = min(max(ilogbf(vmax), -100), 100);
        p_scale = ldexpf(1.f, -e);
        out_scale = ldexpf(1.f, e);
    }

    RowState st{-INFINITY, 0ull, 0ull, 0ull};
    bool ok = true;
    const uint32_t tmem_row = tmem + tile * kTileCols + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    if (softmax) {
        const int pos_i = row_ok ? p.pos0 + tq : -1;
        const f2 q8 = pack2(qsum8, qsum8), q4 = pack2(qsum4, qsum4);
        for (int n = 0; n < n_steps; ++n) {
            const int j0 = (first + n) * kStep;
            ok = mbar_wait(&sh->kv_full[n & 1], (n >> 1) & 1, &sh->abort_flag, p.status) &&
                 mbar_wait(&sh->s_full[tile], n & 1, &sh->abort_flag, p.status);
            if (__any_sync(0xffffffffu, !ok)) break;
            tc_fence_after();
            const float4 *col_k = sh->col_k[n & 1], *col_v = sh->col_v[n & 1];
            f2 sc[32];
            float m_use = st.m == -INFINITY ? 0.f : st.m, mx;
            const bool masked = j0 + kStep - 1 > pos_first;
            const int last = pos_i - j0;  // the step's last position that this row sees
            if (masked) mx = step_scores<true>(sc, tmem_row, col_k, last, q8, q4, -m_use);
            else mx = step_scores<false>(sc, tmem_row, col_k, last, q8, q4, -m_use);
            // ---- raise the reference where a score leaves it too far behind (and set it at the first position seen)
            const bool raise = mx > (st.m == -INFINITY ? -INFINITY : kSlack);
            if (__any_sync(0xffffffffu, raise)) {
                const float d = raise ? mx : 0.f;
                const float f = raise ? (st.m == -INFINITY ? 0.f : exp2_approx(-d)) : 1.f;
                const f2 d2 = pack2(-d, -d), ff = pack2(f, f);
#pragma unroll
                for (int i = 0; i < 32; ++i) sc[i] = add2(sc[i], d2);
                st.l = mul2(st.l, ff);
                st.z8 = mul2(st.z8, ff);
                st.z4 = mul2(st.z4, ff);
                if (raise) st.m = m_use + d;
                if (n > 0) {  // S(n) was issued after the previous output product had completed
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        uint32_t o[16];
                        tmem_ld16(tmem_row + kColO4 + 16 * c, o);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                        tmem_st16(tmem_row + kColO4 + 16 * c, o);
                    }
                }
            }
            // ---- weights, their sums, the operands of the output product
            step_weights(st, sc, tmem_row, col_v);
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(&sh->p_full[tile]);
        }
        if (!__any_sync(0xffffffffu, !ok) && n_steps > 0)
            ok = mbar_wait(&sh->pv_done[tile], (n_steps - 1) & 1, &sh->abort_flag, p.status);
        tc_fence_after();
        // a row that sees a value whose constants are not finite gets NaN in that segment
        if (pos_i >= sh->bad8) st.z8 = pack2(NAN, NAN);
        if (pos_i >= sh->bad4) st.z4 = pack2(NAN, NAN);
    } else if (warp < G::kMmaWarp) {
        const int et = tid - 32 * G::kSoftmaxWarps;
        int issued = 0;
        auto issue_load = [&](int n) {
            const int b0 = 2 * (first + n);
            const uint32_t bytes = static_cast<uint32_t>(min(2, n_blocks - b0)) * kBlockBytes;
            mbar_arrive_expect_tx(&sh->raw_full[n & 1], bytes);
            bulk_load(raw + (n & 1) * kRawBytes, blocks + static_cast<size_t>(b0) * kBlockBytes, bytes, &sh->raw_full[n & 1]);
        };
        if (et == 0)
            for (; issued < min(2, n_steps); ++issued) issue_load(issued);
        int n = 0;
        for (; n < n_steps; ++n) {
            ok = mbar_wait(&sh->raw_full[n & 1], (n >> 1) & 1, &sh->abort_flag, p.status);
            if (ok && n >= 2) ok = mbar_wait(&sh->kv_empty[n & 1], ((n >> 1) - 1) & 1, &sh->abort_flag, p.status);
            int all_ok;  // the four warps leave together (they meet at a barrier below)
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 2, 128, p;\n\t"
                         "selp.b32 %0, 1, 0, q;\n\t}" : "=r"(all_ok) : "r"(ok ? 1 : 0) : "memory");
            if (!all_ok) { ok = false; break; }
            expand_step(raw + (n & 1) * kRawBytes, stages + (n & 1) * kStageBytes, sh->col_k[n & 1], sh->col_v[n & 1], et,
                        limit - (first + n) * kStep, p_scale, (first + n) * kStep, &sh->bad8, &sh->bad4);
            fence_proxy_async_smem();
            mbar_arrive(&sh->kv_full[n & 1]);
            asm volatile("bar.sync 1, 128;" ::: "memory");  // everybody has read the raw buffer
            if (et == 0 && n + 2 < n_steps) {
                issue_load(n + 2);
                ++issued;
            }
        }
        if (et == 0 && !ok) {  // copies still in flight are waited for (bounded; the shared flag is set by now)
            int keep_waiting = 0;
            for (int i = max(n, 0); i < issued; ++i) (void)mbar_wait(&sh->raw_full[i & 1], (i >> 1) & 1, &keep_waiting, p.status);
        }
    } else if (n_steps > 0) {  // the whole warp, converged; one lane issues
        const bool leader = elect_one();
        const uint32_t idS = make_idesc_f16(kRows, kStep);
        const uint32_t idO8 = make_idesc_f16(kRows, 16) | kBNMajor, idO4 = make_idesc_f16(kRows, 112) | kBNMajor;
        auto score_product = [&](int t, int n) {
            const uint32_t q = smem_u32(Qs + t * kQBytes), k = smem_u32(stages + (n & 1) * kStageBytes);
            const uint64_t q0 = make_smem_desc_k128(q), q1 = make_smem_desc_k128(q + kRows * 128);
            const uint64_t k0 = make_smem_desc_k128(k), k1 = make_smem_desc_k128(k + kStep * 128);
            const uint32_t d = tmem + t * kTileCols;
            mma_f16_ss_if(leader, d + kColS8, q0, k0, idS, 0);
#pragma unroll
            for (int i = 1; i < 4; ++i) mma_f16_ss_if(leader, d + kColS4, q0 + 2 * i, k0 + 2 * i, idS, i > 1);
#pragma unroll
            for (int i = 0; i < 4; ++i) mma_f16_ss_if(leader, d + kColS4, q1 + 2 * i, k1 + 2 * i, idS, 1);
            tc_commit_if(leader, &sh->s_full[t]);
        };
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            if (ok) ok = !__any_sync(0xffffffffu, !mbar_wait(bar, parity, &sh->abort_flag, p.status));
            tc_fence_after();
            return ok;
        };
        if (wait(&sh->kv_full[0], 0))
            for (int t = 0; t < NT; ++t) score_product(t, 0);
        for (int n = 0; n < n_steps && ok; ++n) {
            const uint32_t v = smem_u32(stages + (n & 1) * kStageBytes + kKBytes);
            const uint64_t v4 = make_smem_desc_mn128(v, kStep * 128), v8 = make_smem_desc_mn128(v + kV4Bytes, kStep * 128);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                if (!wait(&sh->p_full[t], n & 1)) break;
                const uint32_t d = tmem + t * kTileCols;
#pragma unroll
                for (int i = 0; i < kStep / 16; ++i) {  // 16 positions: 8 columns of weights, 16 rows of 128 bytes
                    const uint32_t acc = (n > 0 || i > 0) ? 1u : 0u;
                    mma_f16_ts_if(leader, d + kColO8, d + kColP8 + 8 * i, v8 + (2048 >> 4) * i, idO8, acc);
                    mma_f16_ts_if(leader, d + kColO4, d + kColP4 + 8 * i, v4 + (2048 >> 4) * i, idO4, acc);
                }
                tc_commit_if(leader, &sh->pv_done[t]);
                if (t == NT - 1) tc_commit_if(leader, &sh->kv_empty[n & 1]);
                if (n + 1 < n_steps) {
                    // the next scores go over the weights just read: their product has to be complete
                    if (t == 0 && !wait(&sh->kv_full[(n + 1) & 1], ((n + 1) >> 1) & 1)) break;
                    if (!wait(&sh->pv_done[t], n & 1)) break;
                    score_product(t, n + 1);
                }
            }
        }
        if (!ok) {  // products in flight finish before TMEM and shared memory are given back (bounded)
            int keep_waiting = 0;
            tc_commit_if(leader, &sh->drain);
            (void)mbar_wait(&sh->drain, 0, &keep_waiting, p.status);
        }
    }
    __syncwarp();

    // ---- out = (O 2^E + zero-point sums) / sum of p; the row's outputs leave in the coefficients' own order
    const float2 l2 = unpack2(st.l), z8p = unpack2(st.z8), z4p = unpack2(st.z4);
    const float l = l2.x + l2.y, z8 = z8p.x + z8p.y, z4 = z4p.x + z4p.y;
    auto row_outputs = [&](float* dst, float inv) {  // whole, converged warps; the stores are predicated by dst
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            __syncwarp();
            tmem_ld32(tmem_row + kColO4 + 32 * c, o);
            tmem_ld_wait();
#pragma unroll
            for (int grp = 0; grp < 4; ++grp) {  // eight columns = eight coefficients
                const int n0 = 32 * c + 8 * grp;
                const bool seg8 = n0 >= 112;
                const float z = seg8 ? z8 : z4;
                float f[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    f[i] = (n_steps > 0 ? fmaf(__uint_as_float(o[8 * grp + i]), out_scale, z) : 0.f) * inv;
                if (!dst) continue;
                float* d = dst + (seg8 ? n0 - 112 : 16 + n0);
                *reinterpret_cast<float4*>(d) = seg8 ? make_float4(f[0], f[1], f[2], f[3]) : make_float4(f[0], f[2], f[4], f[6]);
                *reinterpret_cast<float4*>(d + 4) = seg8 ? make_float4(f[4], f[5], f[6], f[7]) : make_float4(f[1], f[3], f[5], f[7]);
            }
        }
    };
    const bool warp_ok = !__any_sync(0xffffffffu, !ok);
    if (p.splits == 1) {
        if (softmax && warp_ok)
            row_outputs(row_ok ? p.out + (static_cast<size_t>(tq) * p.Hq + hq) * 128 : nullptr, l > 0.f ? 1.f / l : 0.f);
    } else {
        __syncthreads();  // every product of the CTA is done: the records go over the tiles
        float* rec = reinterpret_cast<float*>(base);
        if (softmax && warp_ok) {
            float* r = rec + (tile * kRows + row) * kRecPitch;
            row_outputs(r, 1.f);
            r[128] = st.m;
            r[129] = l;
        }
        __syncwarp();
        cluster_sync_all();
        if (rank == 0) {
            for (int i = tid; i < NT * kRows * 32; i += G::kThreads) {
                const int rr = i >> 5, c4 = i & 31, Ro = R0 + rr;
                if (Ro >= p.T * p.g) continue;
                const uint32_t local = smem_u32(rec + rr * kRecPitch);
                float M = -INFINITY;
                for (int rk = 0; rk < p.splits; ++rk) M = fmaxf(M, ld_cluster_f2(cluster_map_addr(local, rk) + 128 * 4).x);
                float L = 0.f;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int rk = 0; rk < p.splits; ++rk) {
                    const uint32_t a = cluster_map_addr(local, rk);
                    const float2 ml = ld_cluster_f2(a + 128 * 4);
                    const float4 o = ld_cluster_f4(a + c4 * 16);
                    const float f = exp2_approx(ml.x - M);
                    L = fmaf(ml.y, f, L);
                    acc = make_float4(fmaf(o.x, f, acc.x), fmaf(o.y, f, acc.y), fmaf(o.z, f, acc.z), fmaf(o.w, f, acc.w));
                }
                const float inv = L > 0.f ? 1.f / L : 0.f;
                *reinterpret_cast<float4*>(p.out + (static_cast<size_t>(Ro / p.g) * p.Hq + kvh * p.g + Ro % p.g) * 128 + 4 * c4) =
                    make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
            }
        }
        __syncwarp();
        cluster_sync_all();  // the records stay until rank 0 has read them
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && sh->abort_flag) atomicOr(p.status, kStatusBitTimeout);
    if (warp == G::kMmaWarp) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, NT * kTileCols);
    }
}

template <int NT>
cudaError_t launch_prefill(const PrefillParams& p, long long tiles, cudaStream_t st) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(attention_prefill_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(Geometry<NT>::kSmem));
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(tiles * p.Hkv * p.splits));
    cfg.blockDim = dim3(Geometry<NT>::kThreads);
    cfg.dynamicSmemBytes = Geometry<NT>::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(p.splits);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // More CTAs than SMs start in order of length only behind a drained grid.
    cfg.numAttrs = tiles * p.Hkv * p.splits <= 148 ? 2 : 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, attention_prefill_kernel<NT>, p);
}

}  // namespace

cudaError_t launch_attention_prefill(const resq_kv_cache_t& cache, const void* q16, int n_q_heads, int seq, int pos0,
                                     int T, float* out, cudaStream_t st) {
    PrefillParams p;
    const size_t nblk = static_cast<size_t>(cache.capacity / RESQ_KV_BLOCK);
    p.head_stride = nblk * kBlockBytes;
    p.blocks = static_cast<const uint8_t*>(cache.data) + static_cast<size_t>(seq) * cache.n_kv_heads * p.head_stride;
    p.q = static_cast<const __half*>(q16);
    p.out = out;
    p.T = T;
    p.Hq = n_q_heads;
    p.Hkv = cache.n_kv_heads;
    p.g = n_q_heads / cache.n_kv_heads;
    p.pos0 = pos0;
    p.status = device_status_ptr();
    const PrefillPlan pl = prefill_plan(pos0, T, p.g, p.Hkv);
    p.splits = pl.splits;
    return pl.tiles_per_cta == 1 ? launch_prefill<1>(p, pl.row_groups, st) : launch_prefill<2>(p, pl.row_groups, st);
}

}  // namespace resq
