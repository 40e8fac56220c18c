// Mixed-precision GEMM (Eq. 4 + dequantizing epilogue) for token counts between the weight-streaming kernel and the
// large-tile kernel: ragged batches, chunked prefill beside generation, a few hundred tokens at most.
//
// The large-tile kernel (mixed_gemm.cu) gives a CTA pair 256 tokens x 256 channels.  With few tokens that leaves most SMs
// idle (a 4096-channel layer is 16 tiles), computes rows of padding, and walks the whole reduction serially.  Here
//   * the operands change places: 256 channels are the M rows of the pair's product (cta_group::2), the tokens are its N
//     columns, N a multiple of 32 up to 256, so the padding is at most 31 tokens per tile;
//   * the reduction is cut over the S = 1, 2 or 3 pairs of a cluster: each pair streams its share of the k-blocks (INT4
//     blocks first, then INT8 ones) and accumulates exact int32 sums in its own TMEM; the pairs then exchange partial sums
//     through distributed shared memory (over the drained ring), each finishing the 16-token groups g with g % S = its
//     index.  Integer sums: the result does not depend on S, and no global scratch is needed.
//   * a lane is a channel, so the stores of one token are contiguous across the warp.
// Roles per CTA as in mixed_gemm.cu: TMA producer, MMA issuer (even CTA of a pair), 8 epilogue warps; one tile per cluster,
// no persistence.  The rule that picks this kernel, N and S is mid_plan (plans.h).  All waits are bounded.
//
// What bounds it: the latency of the TMA ring up to N = 128 (0.21 us per k-block of 24 KB, 8 stages), operand delivery beyond,
// and about 6 us of launch, first copies, epilogue and drain.  us, tile kernel -> this one: 4096 x 6144 at 17 / 128 / 300 /
// 700 tokens 17.5 -> 8.7, 24 -> 12.3, 24.7 -> 14.3, 24.9 -> 19.6; 14336 x 4096 at 17 / 300 / 1537 tokens 41 -> 15.3, 47 -> 23,
// 89 -> 68.5.  Products issued by a thread alone in a branch: 0.27 us per k-block whatever N.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "byte_map.h"
#include "internal.h"
#include "plans.h"
#include "ptx.cuh"

namespace resq {
namespace {

constexpr int BM = 128, BK = 128;  // channel rows per CTA; bytes (= codes) per k-block
constexpr int kMaxStages = 10;
constexpr int A_BYTES = BM * BK;
constexpr int kRingBytes = 6 * (A_BYTES + 128 * BK);  // a stage holds 128 channel rows and ntok / 2 token rows (at most 128)
constexpr int kThreads = 320;
constexpr uint32_t kTmemCols = 512, kColAcc4 = 256;
constexpr int kTok = 8;  // tokens that an epilogue thread finishes at a time
constexpr int kGroupBytes = 16 * BM * 4;  // partial sums of 16 tokens x 128 channels

struct Params {
    int T, N, kb4, kb8;
    int ntok, tok_tiles, splits, stages;
    const float* s_x8;
    const float* s_x4;
    const void* s_w8;
    const void* s_w4;
    int w_fp16;
    const float* z_x8;  // asymmetric activations only
    const float* z_x4;
    const int32_t* wsum8;
    const int32_t* wsum4;
    void* Y;
    int y_dtype;
    int32_t* dbg8;
    int32_t* dbg4;
    int* status;
};

struct __align__(16) Shared {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t acc_full;
    uint32_t tmem_base;
    int abort_flag;
    alignas(16) float sx8[256];  // of the tile's tokens, 0 behind the last
    alignas(16) float sx4[256];
    alignas(16) float zx8[256];
    alignas(16) float zx4[256];
};

constexpr size_t kSmemBytes = 1024 + kRingBytes + sizeof(Shared);

__device__ __forceinline__ float load_scale(const void* p, int i, int fp16) {
    return fp16 ? __half2float(reinterpret_cast<const __half*>(p)[i]) : reinterpret_cast<const float*>(p)[i];
}

template <int S>
struct Count {
    static constexpr int value = S;
};

__device__ __forceinline__ void put_value(float* dst, float y) { *dst = y; }
__device__ __forceinline__ void put_value(__nv_bfloat16* dst, float y) { *dst = __float2bfloat16_rn(y); }

// Slot of 16-token group g among the groups that pair `owner` of `splits` does not finish itself.
__device__ __forceinline__ int slot_of(int g, int owner, int splits) { return g - (g + splits - 1 - owner) / splits; }

template <bool ASYM>
__global__ void __launch_bounds__(kThreads, 1)
mixed_gemm_mid_kernel(const __grid_constant__ CUtensorMap tmW8, const __grid_constant__ CUtensorMap tmW4,
                      const __grid_constant__ CUtensorMap tmX8, const __grid_constant__ CUtensorMap tmX4, const Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Shared* sh = reinterpret_cast<Shared*>(smem + kRingBytes);
    const uint32_t stage_bytes = A_BYTES + static_cast<uint32_t>(p.ntok / 2) * BK;
    volatile int* abort_flag = &sh->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = static_cast<int>(cluster_ctarank()), pair = rank >> 1, h = rank & 1;
    const int tile = static_cast<int>(blockIdx.x) / (2 * p.splits);
    const int t0 = (tile % p.tok_tiles) * p.ntok;                    // the tile's first token
    const int n0 = (tile / p.tok_tiles) * (2 * BM) + h * BM;         // this CTA's first channel
    const int kbt = p.kb4 + p.kb8;
    const int kb0 = kbt * pair / p.splits, kb1 = kbt * (pair + 1) / p.splits;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->empty[s], 1);
        }
        mbar_init(&sh->acc_full, 1);
        sh->abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmW8);
        tma_prefetch_desc(&tmW4);
        tma_prefetch_desc(&tmX8);
        tma_prefetch_desc(&tmX4);
    }
    if (warp == 1) {
        tmem_alloc_pair(&sh->tmem_base, kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // the other CTAs' barriers exist before anything is signalled across
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    griddep_wait();  // the set-up above ran under the tail of the preceding grid
    griddep_launch_dependents();

    const int quad = warp & 3, part = (warp - 2) >> 2;  // epilogue warps: TMEM lane quadrant, which half of the groups
    const int groups = p.ntok / 16;
    const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
    const int row = quad * 32 + lane;
    // Slice i of the reduction holds INT4 blocks / INT8 blocks.
    auto has4 = [&](int i) { return kbt * i / p.splits < p.kb4; };
    auto has8 = [&](int i) { return kbt * (i + 1) / p.splits > p.kb4; };
    const uint32_t part8 = static_cast<uint32_t>(groups - groups / p.splits) * kGroupBytes;  // INT8 sums behind the INT4 ones
    bool ok = true;
    // An epilogue thread's channel, and its scales: asked for before the products are awaited.
    const int n = n0 + row;
    const bool n_in = warp >= 2 && n < p.N;
    float sw8 = 0.f, sw4 = 0.f, zc8 = 0.f, zc4 = 0.f;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!mbar_wait(&sh->empty[stage], phase ^ 1, abort_flag, p.status)) { ok = false; break; }
                // The even CTA arms its barrier for the bytes of both CTAs; the odd one only sends its bytes there (if
                // they land first, the pending arrival keeps the phase open).
                const uint32_t full_addr = cluster_map(&sh->full[stage], rank & ~1);
                if (h == 0) mbar_arrive_expect_tx(&sh->full[stage], 2 * stage_bytes);
                const bool seg4 = kb < p.kb4;
                const int x = (seg4 ? kb : kb - p.kb4) * BK;
                tma_load_2d_pair(smem + stage * stage_bytes, seg4 ? &tmW4 : &tmW8, full_addr, x, n0);
                tma_load_2d_pair(smem + stage * stage_bytes + A_BYTES, seg4 ? &tmX4 : &tmX8, full_addr, x, t0 + h * (p.ntok / 2));
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
            if (!ok) {  // give the copies already in flight time to land before the CTA gives up its shared memory
                const uint64_t since = global_timer_ns();
                while (global_timer_ns() - since < 1000000ull) {}
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (even CTA of the pair): the whole warp,
        // converged, one lane issues (by a thread alone in a branch: 0.27 us per k-block whatever N)
        if (h == 0) {
            const bool leader = elect_one();
            // signed weights times signed or unsigned activations
            const uint32_t idesc = (2u << 4) | (1u << 7) | (ASYM ? 0u : 1u << 10) | (static_cast<uint32_t>(p.ntok >> 3) << 17) |
                                   (static_cast<uint32_t>(2 * BM >> 4) << 24);
            const uint16_t both = static_cast<uint16_t>(3u << (rank & ~1));
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                ok = !__any_sync(0xffffffffu, !mbar_wait(&sh->full[stage], phase, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
                const uint32_t base = smem_u32(smem) + stage * stage_bytes;
                const uint64_t a_desc = make_smem_desc_k128(base);
                const uint64_t b_desc = make_smem_desc_k128(base + A_BYTES);
                const uint32_t d = tmem_base + (kb < p.kb4 ? kColAcc4 : 0u);
                const bool first = kb == kb0 || kb == p.kb4;
#pragma unroll
                for (int k = 0; k < BK / 32; ++k)
                    mma_i8_ss_pair_if(leader, d, a_desc + 2 * k, b_desc + 2 * k, idesc, (first && k == 0) ? 0u : 1u);
                tc_commit_pair_if(leader, &sh->empty[stage], both);
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
            if (ok) tc_commit_pair_if(leader, &sh->acc_full, both);
        }
    } else {
        // ------------------------------------------------------------ epilogue, first half: token scales, partial sums out
        const int et = threadIdx.x - 64;
        const int t = t0 + et;
        const bool live = et < p.ntok && t < p.T;
        const float sx8 = live ? p.s_x8[t] : 0.f, sx4 = live ? p.s_x4[t] : 0.f;
        const float zx8 = ASYM && live ? p.z_x8[t] : 0.f, zx4 = ASYM && live ? p.z_x4[t] : 0.f;
        sh->sx8[et] = sx8;
        sh->sx4[et] = sx4;
        if (ASYM) {
            sh->zx8[et] = zx8;
            sh->zx4[et] = zx4;
        }
        if (n_in) {
            sw8 = load_scale(p.s_w8, n, p.w_fp16);
            sw4 = load_scale(p.s_w4, n, p.w_fp16);
            if (ASYM) {
                zc8 = static_cast<float>(p.wsum8[n]) * sw8;
                zc4 = static_cast<float>(p.wsum4[n]) * sw4;
            }
        }
        ok = mbar_wait(&sh->acc_full, 0, abort_flag, p.status);
        ok = !__any_sync(0xffffffffu, !ok);
        tc_fence_after();
        if (p.splits > 1 && ok) {
            const bool w4 = has4(pair), w8 = has8(pair);
            for (int g = part; g < groups; g += 2) {
                if (g % p.splits == pair) continue;
                uint8_t* dst = smem + slot_of(g, pair, p.splits) * kGroupBytes + row * 16;
                uint32_t a[16];
                if (w4) {
                    tmem_ld16(lane_addr + kColAcc4 + 16 * g, a);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<uint4*>(dst + q * (BM * 16)) = make_uint4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]);
                }
                if (w8) {
                    tmem_ld16(lane_addr + 16 * g, a);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<uint4*>(dst + part8 + q * (BM * 16)) =
                            make_uint4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]);
                }
            }
        }
    }
    __syncwarp();
    if (p.splits > 1) cluster_sync_all();
    else __syncthreads();  // the token scales

    if (warp >= 2) {
        // ------------------------------------------------------------ epilogue, second half: sums, scales, stores
        const int tokens = n_in && ok ? min(p.ntok, p.T - t0) : 0;
        // What bounds it is the fetch of instructions: two warps a scheduler cannot hide a jump, and each skipped body (a split's sums, the sums to
        // write out, the other output type) cost 30 to 100 cycles a pass.  So one loop a split count and output type, its body straight: 8 tokens
        // take 550 cycles (two warps a scheduler, fp32 results with zero-points), 16 in one pass with those branches took 1750; the steps from
        // the last product to the last store: 128 tokens 4.2 -> 3.0 us, 192 tokens 5.1 -> 3.6.  The time of the layer, us: 4096 x 6144 at 17 / 300 /
        // 512 tokens 12.1 -> 11.4, 21.2 -> 19.8, 23.7 -> 20.7; 14336 x 4096 at 300 / 1537 tokens 32.6 -> 29.8, 94.9 -> 90.8.  The next sums asked for
        // before the stores: 0.98 of that; two passes unrolled: the same; fewer registers (112, 96): 0.99.
        auto finish = [&](auto splits, auto* Y) {
            constexpr int S = decltype(splits)::value;
            const bool w4 = has4(pair), w8 = has8(pair);
            uint32_t src[S];  // another pair's sums of this pair's first group; the next group is S - 1 slots further
            bool r4[S], r8[S];
#pragma unroll
            for (int o = 0; o < S - 1; ++o) {
                const int i = o + (o >= pair ? 1 : 0);
                src[o] = cluster_map(smem + slot_of(pair, i, S) * kGroupBytes + part * (kTok / 4 * BM * 16) + row * 16, 2 * i + h);
                r4[o] = has4(i);
                r8[o] = has8(i);
            }
            if (S == 1) {  // a segment without channels has no sums: its columns hold anything
                if (!w4) sw4 = 0.f;
                if (!w8) sw8 = 0.f;
            }
            // kTok tokens' sums over the pairs, from column t on.
            auto sums = [&](int t, uint32_t (&a4)[kTok], uint32_t (&a8)[kTok]) {
                __syncwarp();  // TMEM loads are for the whole, converged warp; lanes beyond the channels only skip their stores
                tmem_ld8x2(lane_addr + kColAcc4 + t, lane_addr + t, a4, a8);
                if (S > 1)
#pragma unroll
                    for (int j = 0; j < kTok; ++j) {
                        a4[j] = w4 ? a4[j] : 0;
                        a8[j] = w8 ? a8[j] : 0;
                    }
                const uint32_t at = static_cast<uint32_t>(t / (16 * S) * (S - 1)) * kGroupBytes;
#pragma unroll
                for (int o = 0; o < S - 1; ++o)
#pragma unroll
                    for (int q = 0; q < kTok / 4; ++q) {
                        const uint4 v4 = ld_cluster_u4_if(r4[o], src[o] + at + q * (BM * 16));
                        const uint4 v8 = ld_cluster_u4_if(r8[o], src[o] + at + part8 + q * (BM * 16));
                        a4[4 * q] += v4.x; a4[4 * q + 1] += v4.y; a4[4 * q + 2] += v4.z; a4[4 * q + 3] += v4.w;
                        a8[4 * q] += v8.x; a8[4 * q + 1] += v8.y; a8[4 * q + 2] += v8.z; a8[4 * q + 3] += v8.w;
                    }
            };
            const size_t step = static_cast<size_t>(p.N);
            const int first = 16 * pair + kTok * part;
            Y += static_cast<size_t>(t0) * step + n;
#pragma unroll 1
            for (int t = first; t < p.ntok; t += 16 * S) {
                uint32_t a4[kTok], a8[kTok];
                sums(t, a4, a8);
                float y[kTok];
#pragma unroll
                for (int q = 0; q < kTok / 4; ++q) {
                    const float4 s8 = reinterpret_cast<const float4*>(sh->sx8 + t)[q], s4 = reinterpret_cast<const float4*>(sh->sx4 + t)[q];
                    const float f8[4] = {s8.x, s8.y, s8.z, s8.w}, f4[4] = {s4.x, s4.y, s4.z, s4.w};
                    float4 z8 = {0.f, 0.f, 0.f, 0.f}, z4 = z8;
                    if (ASYM) z8 = reinterpret_cast<const float4*>(sh->zx8 + t)[q], z4 = reinterpret_cast<const float4*>(sh->zx4 + t)[q];
                    const float g8[4] = {z8.x, z8.y, z8.z, z8.w}, g4[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int j = 4 * q + i;
                        const float t8 = static_cast<float>(static_cast<int>(a8[j])) * (f8[i] * sw8);
                        const float t4 = static_cast<float>(static_cast<int>(a4[j])) * (f4[i] * sw4);
                        y[j] = t8 + t4;
                        if (ASYM) y[j] += g8[i] * zc8 + g4[i] * zc4;
                    }
                }
                auto* dst = Y + static_cast<size_t>(t) * step;
#pragma unroll
                for (int j = 0; j < kTok; ++j, dst += step)
                    if (t + j < tokens) put_value(dst, y[j]);
            }
            if (p.dbg8)
#pragma unroll 1
                for (int t = first; t < p.ntok; t += 16 * S) {
                    uint32_t a4[kTok], a8[kTok];
                    sums(t, a4, a8);
#pragma unroll
                    for (int j = 0; j < kTok; ++j)
                        if (t + j < tokens) {
                            const size_t off = static_cast<size_t>(t0 + t + j) * step + n;
                            p.dbg8[off] = w8 || S > 1 ? static_cast<int>(a8[j]) : 0;
                            p.dbg4[off] = w4 || S > 1 ? static_cast<int>(a4[j]) : 0;
                        }
                }
        };
        auto finish_as = [&](auto splits) {
            if (p.y_dtype == RESQ_Y_BF16) finish(splits, reinterpret_cast<__nv_bfloat16*>(p.Y));
            else finish(splits, reinterpret_cast<float*>(p.Y));
        };
        if (p.splits == 1) finish_as(Count<1>());
        else if (p.splits == 2) finish_as(Count<2>());
        else finish_as(Count<3>());
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // no CTA leaves while another may still read its shared memory or signal it
    if (threadIdx.x == 0 && sh->abort_flag) atomicOr(p.status, kStatusBitTimeout);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace

cudaError_t launch_mixed_gemm_mid(int T, int N, int K, int r, const int8_t* x8, const int8_t* x4e, const float* s_x8,
                                  const float* s_x4, const int8_t* w8, const int8_t* w4e, const void* s_w8,
                                  const void* s_w4, bool w_scale_fp16, void* Y, int y_dtype, int32_t* dbg8, int32_t* dbg4,
                                  cudaStream_t st, const float* z_x8, const float* z_x4, const int32_t* wsum8,
                                  const int32_t* wsum4) {
    const int K4 = K - r, kb8 = (r + BK - 1) / BK, kb4 = (K4 + BK - 1) / BK;
    const MidPlan pl = mid_plan(T, N, kb4 + kb8);
    if (!pl.use) return cudaErrorNotSupported;
    const bool asym = z_x8 != nullptr;  // then x8 / x4e hold unsigned codes
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        for (auto k : {mixed_gemm_mid_kernel<false>, mixed_gemm_mid_kernel<true>})
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemBytes))) != cudaSuccess)
                return e;
        if (dev < 64) attr_set[dev] = true;
    }
    CUtensorMap tW8, tW4, tX8, tX4;
    if (!make_map_u8(&tW4, w4e, N, K4, BM) || !make_map_u8(&tX4, x4e, T, K4, pl.ntok / 2)) return cudaErrorInvalidValue;
    if (r > 0) {
        if (!make_map_u8(&tW8, w8, N, r, BM) || !make_map_u8(&tX8, x8, T, r, pl.ntok / 2)) return cudaErrorInvalidValue;
    } else {  // uniform INT4: no INT8 blocks, these maps are never used
        tW8 = tW4;
        tX8 = tX4;
    }
    Params p;
    p.T = T; p.N = N; p.kb4 = kb4; p.kb8 = kb8;
    p.ntok = pl.ntok; p.tok_tiles = pl.tok_tiles; p.splits = pl.splits;
    p.stages = kRingBytes / (A_BYTES + pl.ntok / 2 * BK);
    if (p.stages > kMaxStages) p.stages = kMaxStages;
    p.s_x8 = s_x8; p.s_x4 = s_x4; p.s_w8 = s_w8; p.s_w4 = s_w4;
    p.w_fp16 = w_scale_fp16 ? 1 : 0;
    p.z_x8 = z_x8; p.z_x4 = z_x4; p.wsum8 = wsum8; p.wsum4 = wsum4;
    p.Y = Y; p.y_dtype = y_dtype; p.dbg8 = dbg8; p.dbg4 = dbg8 ? dbg4 : nullptr;
    p.status = device_status_ptr();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((N + 2 * BM - 1) / (2 * BM) * pl.tok_tiles * 2 * pl.splits));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(2 * pl.splits);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    count_launch();
    return cudaLaunchKernelEx(&cfg, asym ? mixed_gemm_mid_kernel<true> : mixed_gemm_mid_kernel<false>, tW8, tW4, tX8, tX4, p);
}

}  // namespace resq
