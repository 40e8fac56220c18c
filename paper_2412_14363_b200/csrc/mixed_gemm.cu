// Many-token mixed-precision GEMM (Eq. 4 + dequantizing epilogue) on tcgen05 kind::i8, CTA pairs.
//
// Persistent, warp-specialised kernel.  Two CTAs on neighbouring SMs (a cluster of 2) share one
// 256 x 256 output tile (tcgen05 cta_group::2): each stages its own 128 token rows and only its own
// 128 of the tile's 256 weight rows, 32 KB per K block, so six stages fit and the shared-memory read
// rate per MMA is a third lower than with one CTA per 128 x 256 tile.
//   warp 0     TMA producer (both CTAs): streams 128-byte-wide K blocks of the activation and weight
//              codes into the ring (128-byte swizzle), first the INT4 segment (codes one per byte, so
//              both segments run on the i8 tensor path exactly), then the INT8 one.  Completion bytes
//              of both CTAs are counted on the even CTA's barrier.
//   warp 1     TMEM allocation (both CTAs; 512 columns); MMA issue (even CTA only): the INT8 segment
//              accumulates into columns [0,256), the INT4 segment into [256,512) -- two int32
//              accumulators per output because the two segments carry different (token, channel)
//              scales.  Each CTA's TMEM receives the rows of its own 128 tokens.
//   warps 2-9  epilogue (both CTAs), two threads per tile row (128 columns each).
// Two full-width accumulators fill TMEM, so there is no second buffer; the epilogue instead frees the tensor pipe early.  As soon as
// the INT4 segment has its sums, while the INT8 segment runs in the other columns, it copies them into registers (raw int32, 128 per
// thread) and releases those columns, so the next tile's INT4 segment -- 7/8 of its work -- starts right behind the INT8 one.  Then it
// reads the INT8 accumulator, forms y = acc8*(sx8*sw8) + acc4*(sx4*sw4) in fp32, converts and stores; the INT8 columns are released
// long before the next tile's short INT8 segment needs them.  (The copy behind both segments left the tensor pipe idle for about 0.7 us
// a tile: us at 4096 tokens, 4096 x 28672, bf16 364 -> 351; 3000 tokens 2048 x 16384 114.8 -> 109, 8192 x 8192 158 -> 151.8.)
// Barriers signalled across the pair: `full` (odd CTA's copies -> even CTA), `empty`, `acc4_full` and
// `acc_full` (tcgen05.commit, multicast to both), `acc4_empty` / `acc8_empty` (epilogue threads of both CTAs ->
// even CTA).  No TMA multicast.  Out-of-range rows/columns/K are zero-filled by TMA and masked at
// the store.  All waits are bounded.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "byte_map.h"
#include "internal.h"
#include "ptx.cuh"

namespace resq {
namespace {

constexpr int BM = 128, BN = 256, BK = 128;  // BK in bytes == int8 elements
constexpr int STAGES = 6;
constexpr int BN_HALF = BN / 2;  // weight rows staged by each CTA of the pair
constexpr int A_BYTES = BM * BK, B_BYTES = BN_HALF * BK;
constexpr int kEpiThreads = 256;
constexpr int kThreads = 64 + kEpiThreads;
constexpr int kCols = BN * BM / kEpiThreads;  // of a tile row that an epilogue thread finishes
constexpr uint32_t kTmemCols = 512;

struct Params {
    int T, N, r, K4;
    int m_tiles, n_tiles, kb8, kb4;
    int bn;  // output columns per tile: a multiple of 16, <= BN (the B loads and TMEM offsets stay BN wide)
    const float* s_x8;
    const float* s_x4;
    const void* s_w8;
    const void* s_w4;
    int w_fp16;
    // asymmetric activations only: per-token zero-points and per-channel row sums of the weight codes
    const float* z_x8;
    const float* z_x4;
    const int32_t* wsum8;
    const int32_t* wsum4;
    void* Y;
    int wide;  // rows of Y start on 32 bytes
    int32_t* dbg8;
    int32_t* dbg4;
    int* status;
};

struct __align__(16) Shared {
    uint64_t full[STAGES];
    uint64_t empty[STAGES];
    uint64_t acc4_full;
    uint64_t acc_full;
    uint64_t acc4_empty;
    uint64_t acc8_empty;
    uint32_t tmem_base;
    int abort_flag;
    int epi_stop;
    alignas(16) float sw8[BN];
    alignas(16) float sw4[BN];
    alignas(16) float zc8[BN];  // asymmetric activations: (float)wsum8[n] * sw8[n], the column factor of the zero-point term
    alignas(16) float zc4[BN];
};

constexpr size_t kSmemBytes = 1024 + STAGES * (A_BYTES + B_BYTES) + sizeof(Shared);

__device__ __forceinline__ float load_scale(const void* p, int i, int fp16) {
    return fp16 ? __half2float(reinterpret_cast<const __half*>(p)[i]) : reinterpret_cast<const float*>(p)[i];
}

__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

// ASYM: the activation codes are unsigned (u8 x s8 products) and every output gets the rank-one
// zero-point terms z_x8[t] * s_w8[n] * wsum8[n] + z_x4[t] * s_w4[n] * wsum4[n] (Eq. 1, second form).
template <bool ASYM, bool BF16>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
mixed_gemm_kernel(const __grid_constant__ CUtensorMap tmA8, const __grid_constant__ CUtensorMap tmA4,
                  const __grid_constant__ CUtensorMap tmB8, const __grid_constant__ CUtensorMap tmB4,
                  const Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;
    uint8_t* sB = smem + STAGES * A_BYTES;
    Shared* sh = reinterpret_cast<Shared*>(smem + STAGES * (A_BYTES + B_BYTES));
    volatile int* abort_flag = &sh->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = static_cast<int>(cluster_ctarank());  // 0: even CTA (issues the MMAs), 1: its peer
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int num_tiles = p.m_tiles * p.n_tiles;  // m_tiles counts 256-row pair tiles
    const int kb_total = p.kb8 + p.kb4;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->empty[s], 1);
        }
        mbar_init(&sh->acc4_full, 1);
        mbar_init(&sh->acc_full, 1);
        mbar_init(&sh->acc4_empty, 2 * kEpiThreads);  // used in the even CTA: epilogue threads of both CTAs
        mbar_init(&sh->acc8_empty, 2 * kEpiThreads);
        sh->abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmA8);
        tma_prefetch_desc(&tmA4);
        tma_prefetch_desc(&tmB8);
        tma_prefetch_desc(&tmB4);
    }
    if (warp == 1) {
        tmem_alloc_pair(&sh->tmem_base, kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // the peer's barriers exist before anything is signalled across
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    // Launched with programmatic stream serialization: the set-up above ran under the tail of the preceding grid.
    griddep_wait();
    griddep_launch_dependents();

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
                const int m0 = (tile % p.m_tiles) * 2 * BM + rank * BM;        // this CTA's token rows
                const int n0 = (tile / p.m_tiles) * p.bn + rank * BN_HALF;     // this CTA's weight rows
                for (int kb = 0; kb < kb_total; ++kb) {
                    if (!mbar_wait(&sh->empty[stage], phase ^ 1, abort_flag, p.status)) { ok = false; break; }
                    // The even CTA arms its barrier for the bytes of both CTAs; the peer only sends its
                    // bytes there (if they land first, the pending arrival keeps the phase open).
                    const uint32_t full_addr = cluster_map(&sh->full[stage], 0);
                    if (rank == 0) mbar_arrive_expect_tx(&sh->full[stage], 2 * (A_BYTES + B_BYTES));
                    if (kb < p.kb4) {
                        tma_load_2d_pair(sA + stage * A_BYTES, &tmA4, full_addr, kb * BK, m0);
                        tma_load_2d_pair(sB + stage * B_BYTES, &tmB4, full_addr, kb * BK, n0);
                    } else {
                        tma_load_2d_pair(sA + stage * A_BYTES, &tmA8, full_addr, (kb - p.kb4) * BK, m0);
                        tma_load_2d_pair(sB + stage * B_BYTES, &tmB8, full_addr, (kb - p.kb4) * BK, n0);
                    }
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                }
            }
            if (!ok) {
                // Give the copies already in flight time to land before the CTA gives up its shared memory.
                const uint64_t t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 1000000ull) {}
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (even CTA only): the whole warp, converged,
        // one lane issues (4096 tokens, gate|up: 355 us; issued by a thread alone in a branch 388 us)
        if (rank == 0) {
            const bool leader = elect_one();
            const uint32_t idesc = ASYM ? make_idesc_u8s8(2 * BM, p.bn) : make_idesc_i8(2 * BM, p.bn);
            int stage = 0;
            uint32_t phase = 0, acc_phase = 0;
            auto wait = [&](uint64_t* bar, uint32_t parity) {
                const bool ok = !__any_sync(0xffffffffu, !mbar_wait(bar, parity, abort_flag, p.status));
                tc_fence_after();
                return ok;
            };
            bool ok = true;
            for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
                // INT4 columns are free once the previous tile's epilogue has copied them out.
                if (!(ok = wait(&sh->acc4_empty, acc_phase ^ 1))) break;
                for (int kb = 0; kb < kb_total; ++kb) {
                    const bool seg4 = kb < p.kb4;
                    // ... the INT8 columns once it has finished with the tile.
                    if (kb == p.kb4 && !(ok = wait(&sh->acc8_empty, acc_phase ^ 1))) break;
                    if (!(ok = wait(&sh->full[stage], phase))) break;
                    const uint64_t a_desc = make_smem_desc_k128(smem_u32(sA + stage * A_BYTES));
                    const uint64_t b_desc = make_smem_desc_k128(smem_u32(sB + stage * B_BYTES));
                    const uint32_t d = tmem_base + (seg4 ? static_cast<uint32_t>(BN) : 0u);
                    const bool first = kb == 0 || kb == p.kb4;
#pragma unroll
                    for (int k = 0; k < BK / 32; ++k)
                        mma_i8_ss_pair_if(leader, d, a_desc + 2 * k, b_desc + 2 * k, idesc, (first && k == 0) ? 0u : 1u);
                    tc_commit_pair_if(leader, &sh->empty[stage], 3);  // frees the ring slot in both CTAs once these MMAs have read it
                    if (kb == p.kb4 - 1) tc_commit_pair_if(leader, &sh->acc4_full, 3);
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                }
                if (!ok) break;
                if (p.kb4 == 0) tc_commit_pair_if(leader, &sh->acc4_full, 3);
                tc_commit_pair_if(leader, &sh->acc_full, 3);
                acc_phase ^= 1;
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int quad = warp & 3;            // TMEM lane quadrant this warp may access
        const int ch = (warp - 2) >> 2;       // column half of the tile this warp handles
        const int et = threadIdx.x - 64;
        uint32_t acc_phase = 0;
        // The epilogue threads meet at named barriers, so they must leave the loop together:
        // one thread samples the abort flag and the others take its reading.
        for (int tile = pair; tile < num_tiles; tile += npairs) {
            const int m0 = (tile % p.m_tiles) * 2 * BM + rank * BM, n0 = (tile / p.m_tiles) * p.bn;
            epi_barrier();  // previous tile's readers of sw8/sw4/epi_stop are done
            if (et == 0) sh->epi_stop = *abort_flag;
            const int n_end = min(p.N, n0 + p.bn);  // first column past this tile
            {
                const int n = n0 + et;
                const float w8s = n < n_end ? load_scale(p.s_w8, n, p.w_fp16) : 0.f;
                const float w4s = n < n_end ? load_scale(p.s_w4, n, p.w_fp16) : 0.f;
                sh->sw8[et] = w8s;
                sh->sw4[et] = w4s;
                if (ASYM) {
                    sh->zc8[et] = n < n_end ? static_cast<float>(p.wsum8[n]) * w8s : 0.f;
                    sh->zc4[et] = n < n_end ? static_cast<float>(p.wsum4[n]) * w4s : 0.f;
                }
            }
            epi_barrier();
            if (sh->epi_stop) break;
            const int row = m0 + quad * 32 + lane;
            const bool row_ok = row < p.T;
            const float sx8 = row_ok && p.kb8 ? p.s_x8[row] : 0.f;  // uniform INT4: the INT8 accumulator was never written
            const float sx4 = row_ok ? p.s_x4[row] : 0.f;
            const float zx8 = ASYM && row_ok ? p.z_x8[row] : 0.f;
            const float zx4 = ASYM && row_ok ? p.z_x4[row] : 0.f;
            // Phase 1: the INT4 accumulator values of this thread's 128 columns, raw, into registers, while the INT8 segment runs.
            // Whole warps go on together; if a wait ran out, the flag is set: leave at the next sample.
            if (__any_sync(0xffffffffu, !mbar_wait(&sh->acc4_full, acc_phase, abort_flag, p.status))) continue;
            tc_fence_after();
            const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + ch * kCols;
            uint32_t a4[kCols];
            __syncwarp();
            tmem_ld128(lane_addr + BN, a4);
            tc_fence_before();
            mbar_arrive_cluster(cluster_map(&sh->acc4_empty, 0));
            if (__any_sync(0xffffffffu, !mbar_wait(&sh->acc_full, acc_phase, abort_flag, p.status))) continue;
            acc_phase ^= 1;
            tc_fence_after();
            // Phase 2: the INT8 accumulator, the scales, the store -- 32 bytes of a row at a time, a whole sector, where rows start on 32 bytes.
            // With two warps a scheduler it is the fetch of instructions and spilled registers that bound it, and for short reductions or fp32
            // results it bounds the kernel: 16 columns loaded, scaled and stored 16 bytes at a time, with the branches on the output type and on
            // the sums to write out in each pass, took longer than the next tile's INT4 segment.  Now the kernel has the type, a load 8 columns.
            // us, before / now: 3000 tokens 2048 x 16384 bf16 108 / 90, fp32 with zero-points 154 / 124; 4096 x 28672 241 / 235 and 314 / 255;
            // 14336 x 4096 150 / 148 and 153 / 148; with stores of 16 bytes 112 and 153, with 16 warps of 64 columns (96 registers) 95 and 127.
            const int cols = row_ok ? n_end - n0 - ch * kCols : 0;  // that this thread stores
            const size_t off = static_cast<size_t>(row) * p.N + n0 + ch * kCols;
            if (p.dbg8) {
#pragma unroll
                for (int c = 0; c < kCols / 16; ++c) {
                    uint32_t a8[16];
                    __syncwarp();
                    tmem_ld16(lane_addr + c * 16, a8);
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (c * 16 + g * 4 < cols) {
                            reinterpret_cast<uint4*>(p.dbg8 + off)[4 * c + g] =
                                p.kb8 ? make_uint4(a8[4 * g], a8[4 * g + 1], a8[4 * g + 2], a8[4 * g + 3]) : make_uint4(0, 0, 0, 0);
                            reinterpret_cast<uint4*>(p.dbg4 + off)[4 * c + g] =
                                make_uint4(a4[16 * c + 4 * g], a4[16 * c + 4 * g + 1], a4[16 * c + 4 * g + 2], a4[16 * c + 4 * g + 3]);
                        }
                }
            }
            auto finish = [&](auto wide) {
#pragma unroll
                for (int c = 0; c < kCols / 16; ++c) {
                    uint32_t w[8];  // 32 bytes of the row: the chunk in bf16, half of it in fp32
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        uint32_t a8[8];
                        __syncwarp();
                        tmem_ld8(lane_addr + c * 16 + e * 8, a8);
                        const int cb = ch * kCols + c * 16 + e * 8;  // the first of these columns inside the tile
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const float4 v8 = reinterpret_cast<const float4*>(sh->sw8 + cb)[q], v4 = reinterpret_cast<const float4*>(sh->sw4 + cb)[q];
                            const float w8[4] = {v8.x, v8.y, v8.z, v8.w}, w4[4] = {v4.x, v4.y, v4.z, v4.w};
                            float4 u8 = {0.f, 0.f, 0.f, 0.f}, u4 = u8;
                            if (ASYM) u8 = reinterpret_cast<const float4*>(sh->zc8 + cb)[q], u4 = reinterpret_cast<const float4*>(sh->zc4 + cb)[q];
                            const float c8[4] = {u8.x, u8.y, u8.z, u8.w}, c4[4] = {u4.x, u4.y, u4.z, u4.w};
                            float y[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float t8 = static_cast<float>(static_cast<int>(a8[4 * q + i])) * (sx8 * w8[i]);
                                const float t4 = static_cast<float>(static_cast<int>(a4[16 * c + 8 * e + 4 * q + i])) * (sx4 * w4[i]);
                                y[i] = t8 + t4;
                                if (ASYM) y[i] += zx8 * c8[i] + zx4 * c4[i];
                            }
                            if (BF16) {
#pragma unroll
                                for (int i = 0; i < 2; ++i) {
                                    const __nv_bfloat162 h = __floats2bfloat162_rn(y[2 * i], y[2 * i + 1]);
                                    w[4 * e + 2 * q + i] = *reinterpret_cast<const uint32_t*>(&h);
                                }
                            } else {
#pragma unroll
                                for (int i = 0; i < 4; ++i) w[4 * q + i] = __float_as_uint(y[i]);
                            }
                        }
                        if (BF16 && e == 0) continue;
                        const int col = c * 16 + (BF16 ? 0 : 8 * e);  // of the first word
                        char* yp = reinterpret_cast<char*>(p.Y) + (off + col) * (BF16 ? 2 : 4);
                        if (decltype(wide)::value) {
                            if (col < cols) st_global_8(yp, w);
                        } else {
#pragma unroll
                            for (int g = 0; g < 2; ++g)
                                if (col + g * (BF16 ? 8 : 4) < cols)
                                    reinterpret_cast<uint4*>(yp)[g] = make_uint4(w[4 * g], w[4 * g + 1], w[4 * g + 2], w[4 * g + 3]);
                        }
                    }
                }
            };
            if (p.wide) finish(std::true_type());
            else finish(std::false_type());
            tc_fence_before();
            mbar_arrive_cluster(cluster_map(&sh->acc8_empty, 0));
        }
    }

    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // neither CTA leaves while the other may still read its shared memory or signal it
    if (threadIdx.x == 0 && sh->abort_flag) atomicOr(p.status, kStatusBitTimeout);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace

cudaError_t launch_mixed_gemm_tiles(int T, int N, int K, int r, const int8_t* x8, const int8_t* x4e,
                                    const float* s_x8, const float* s_x4, const int8_t* w8, const int8_t* w4e,
                                    const void* s_w8, const void* s_w4, bool w_scale_fp16, void* Y, int y_dtype,
                                    int32_t* dbg8, int32_t* dbg4, cudaStream_t st, const float* z_x8,
                                    const float* z_x4, const int32_t* wsum8, const int32_t* wsum4) {
    if (const cudaError_t em = launch_mixed_gemm_mid(T, N, K, r, x8, x4e, s_x8, s_x4, w8, w4e, s_w8, s_w4, w_scale_fp16, Y, y_dtype,
                                                     dbg8, dbg4, st, z_x8, z_x4, wsum8, wsum4);
        em != cudaErrorNotSupported)
        return em;
    const bool asym = z_x8 != nullptr;  // then x8 / x4e hold unsigned codes
    using Kernel = decltype(&mixed_gemm_kernel<false, false>);
    const Kernel kernels[4] = {mixed_gemm_kernel<false, false>, mixed_gemm_kernel<false, true>, mixed_gemm_kernel<true, false>,
                               mixed_gemm_kernel<true, true>};
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && !attr_set[dev]) {
        for (const Kernel k : kernels)
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemBytes))) != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    const int K4 = K - r;
    CUtensorMap tA8, tA4, tB8, tB4;
    if (!make_map_u8(&tA4, x4e, T, K4, BM) || !make_map_u8(&tB4, w4e, N, K4, BN_HALF)) return cudaErrorInvalidValue;
    if (r > 0) {
        if (!make_map_u8(&tA8, x8, T, r, BM) || !make_map_u8(&tB8, w8, N, r, BN_HALF)) return cudaErrorInvalidValue;
    } else {  // uniform INT4: no INT8 segment, its maps are never used
        tA8 = tA4;
        tB8 = tB4;
    }
    Params p;
    p.T = T; p.N = N; p.r = r; p.K4 = K4;
    int sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    p.m_tiles = (T + 2 * BM - 1) / (2 * BM);
    // The kernel takes any multiple of 16 up to BN here (B loads and TMEM offsets stay BN wide); tiles of 240 and
    // 192 columns measured 1.5-1.7 x slower per column than 256-wide ones, far more than a fuller last round saves.
    p.bn = BN;
    p.n_tiles = (N + p.bn - 1) / p.bn;
    p.kb8 = (r + BK - 1) / BK;
    p.kb4 = (K4 + BK - 1) / BK;
    p.s_x8 = s_x8; p.s_x4 = s_x4; p.s_w8 = s_w8; p.s_w4 = s_w4;
    p.w_fp16 = w_scale_fp16 ? 1 : 0;
    p.z_x8 = z_x8; p.z_x4 = z_x4; p.wsum8 = wsum8; p.wsum4 = wsum4;
    const bool bf16 = y_dtype == RESQ_Y_BF16;
    p.Y = Y; p.wide = (reinterpret_cast<uintptr_t>(Y) | static_cast<uintptr_t>(N) * (bf16 ? 2 : 4)) % 32 == 0;
    p.dbg8 = dbg8; p.dbg4 = dbg8 ? dbg4 : nullptr;
    p.status = device_status_ptr();
    const int tiles = p.m_tiles * p.n_tiles;
    const int pairs = tiles < sms / 2 ? tiles : sms / 2;
    count_launch();
    return launch_programmatic(kernels[2 * asym + bf16], 2 * pairs, kThreads, kSmemBytes, st,
                               tA8, tA4, tB8, tB4, p);
}

}  // namespace resq
