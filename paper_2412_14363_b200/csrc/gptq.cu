// GPTQ rounding of projected weights at pack time (Section 5.1: the projected weights are quantized with GPTQ).
//
// For every output channel (row of W_proj) the columns are visited in order; a weight is rounded to its code
// with the row's round-to-nearest scale of Eq. 3, and the rounding error, divided by the diagonal entry of the
// upper Cholesky factor U of the inverse Hessian, is fed back into the columns not yet visited:
//     e = (w_j - code_j * s) / U[j][j],      w[j+1:] -= e * U[j][j+1:].
// Everything is fp64 with one rounding per operation (multiply, subtract, divide written out: no contraction),
// and an element receives its K updates in the order j = 0, 1, ..: the codes are those of an fp64 reference bit
// for bit.  Rows never interact, so a CTA owns R rows for the whole sweep.
//
// What bounds it: the fp64 pipe (a row needs K^2 / 2 multiplies and as many subtractions) and the chain of K dependent
// roundings per row.  The updates of one element are a fixed sequence, but elements are independent, so the sweep is
// left-looking: the state in shared memory is the scaled error e of every column already rounded (8 bytes per weight),
// not the row.  Columns go in blocks of 256.  Eight updating warps keep one column of the next block per thread, R
// running values in registers, through all earlier columns: one coalesced read of U per column, converted once for R
// rows, e as a broadcast of two columns per load.  (A right-looking sweep reads and writes every remaining weight in
// shared memory at every step, behind two barriers.)  Meanwhile eight rounding warps take the current block through its
// chain, a group of 32 columns each: a warp feeds the errors of the groups before into its own as the updating warps do, then takes
// all R rows through the chain at once, four lanes per row, and hands the group's errors on through named barriers.
// An updated block comes back in the slots its errors will take.
// K = N = 4096: 65.1 ms right-looking, 11.5 ms left-looking with all warps waiting for the chain (two CTAs per
// SM), 7.2 ms with a rounding warp per row, 6.2 ms as it stands (3.7 ms if the fp64 pipe were always busy).  U comes from DRAM where it
// does not stay in L2 (the first call on it, K above 4096), later than the loads a thread has on their way: with few rows
// the updating warps ask L2 for it 256 rows ahead.  K = 4096, 592 rows, caches cold: 2.06 ms without, 1.16 with; K = 8192, 1184 rows: 18.9, 10.3; but
// K = N = 4096 (seven rows per CTA) 6.2, 6.4.
#include <cuda_fp16.h>

#include "internal.h"
#include "plans.h"

namespace resq {
namespace {

constexpr int kThreads = 256;  // = columns of a block
constexpr int kWarps = kThreads / 32;
constexpr int kAhead = 32;        // columns of U a thread requests ahead of their use (L2 latency)
constexpr int kCtaThreads = 2 * kThreads;  // eight updating, eight rounding warps
static_assert(kGptqMaxRows * 4 <= 32, "four lanes per row");
constexpr int kFar = 256;         // rows of U a warp asks L2 for ahead of their use (DRAM latency; a multiple of 32)
constexpr int kAskRows = 5;       // up to as many rows (K above 4800 has no more): with six and seven the updates take longer than DRAM does
constexpr int kPf = 4;            // steps by which a rounding warp requests U ahead
constexpr int kHandOver = 9, kInBlock = 10;  // named barriers behind those of the groups (1-8): a block, its groups by turns
constexpr size_t kRowLimit = 200 * 1024;   // accepted rows: 9 bytes per weight within this (the documented bound)

struct Params {
    const float* W;       // [N][K]
    const float* U;       // [K][K], upper triangular factor of H^-1
    const uint8_t* dead;  // [K] or NULL: columns whose weights are set to 0
    int N, K, r;
    int8_t* w8;
    uint8_t* w4;
    void* s8;
    void* s4;
    int fp16;
    int8_t* w4e;
};

// The chain of a group of 32 columns: lane 4 row + c holds columns c + 4 k of its row in w[k], all earlier columns applied; afterwards
// w[k] and code[k] are their scaled errors and codes.  ug: U at the group's first row and column.  yh_own + yl_own: 1 / U[j][j] of
// column `lane`.  Returns false when the short form cannot vouch for a rounding; the caller then runs the plain form.
//
// The 32 steps depend on one another, so a step's latency is what counts: seven dependent fp64 operations here against two
// divisions, a rounding, a clamp and branches in the plain form.  The next column's value comes by a shuffle before this
// step's update, and every lane of the row applies the update itself.
//  * code: fma(w, 1/s, 1.5 * 2^52) leaves rint(w (1/s)) in the low word, clamped there.  w (1/s) is within 2^-43 of
//    the rounded quotient for |quotient| <= 2^9, so the two round apart only next to a half-integer: refused (by the upper
//    word of the distance, which resolves 2^-22).
//  * x = w - code s by one fma: the product is exact (8 + 24 bits).
//  * e = x / d = fma(x, yh, x yl) with yh + yl = 1 / d to 2^-100 (N. Brisebarre and J.-M. Muller, "Correctly rounded
//    multiplication by arbitrary precision constants", 2008).  d has 24 bits, so x / d lies at least 2^-78 (relative) from the
//    midpoint of two doubles: it is (X 2^k - M D) / D beside M with whole numbers X < 2^53, D < 2^24, M < 2^54, and the
//    numerator is not 0, M D being odd and beyond 2^53.  The sum before its one rounding is within 2^-103.  x and d whose products
//    could leave the normal range are refused.
__device__ __forceinline__ bool round_group(double (&w)[8], int (&code)[8], const float* ug, int K, double yh_own, double yl_own, double s,
                                            double s_inv, bool hi_seg, int lane) {
    const int ilo = hi_seg ? -128 : -8, ihi = hi_seg ? 127 : 7, c = lane & 3, quad = lane & ~3;
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    const float* up = ug + c;
    float ub[kPf][8];  // U at rows i .. i + 3 and the lane's columns that are not behind yet
#pragma unroll
    for (int t = 0; t < kPf; ++t)
#pragma unroll
        for (int k = 0; k < 8; ++k) ub[t][k] = up[static_cast<size_t>(t) * K + 4 * k];
    uint32_t refused = 0;
    double wj = __shfl_sync(0xffffffffu, w[0], quad);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const int ki = i >> 2, kn = (i + 1) >> 2;
        float u[8];
#pragma unroll
        for (int k = ki; k < 8; ++k) u[k] = ub[i % kPf][k];
        if (i + kPf < 32) {
#pragma unroll
            for (int k = (i + kPf) >> 2; k < 8; ++k) ub[i % kPf][k] = up[static_cast<size_t>(i + kPf) * K + 4 * k];
        }
        double w_next = 0.0, u_next = 0.0;
        if (i < 31) {
            w_next = __shfl_sync(0xffffffffu, w[kn & 7], quad + ((i + 1) & 3));
            u_next = static_cast<double>(__shfl_sync(0xffffffffu, u[kn & 7], quad + ((i + 1) & 3)));
        }
        const double yh = __shfl_sync(0xffffffffu, yh_own, i), yl = __shfl_sync(0xffffffffu, yl_own, i);
        const int q = min(max(__double2loint(__fma_rn(wj, s_inv, magic)), ilo), ihi);
        const double cd = __dsub_rn(__hiloint2double(0x43380000 + (q >> 31), q), magic);
        const double x = __fma_rn(-cd, s, wj);
        const double e = __fma_rn(x, yh, __dmul_rn(x, yl));
        const uint32_t frac = static_cast<uint32_t>(__double2hiint(__fma_rn(wj, s_inv, -cd))) & 0x7FFFFFFFu;
        wj = __dsub_rn(w_next, __dmul_rn(e, u_next));
#pragma unroll
        for (int k = ki; k < 8; ++k) {
            const double v = __dsub_rn(w[k], __dmul_rn(e, static_cast<double>(u[k])));
            if (k > ki) w[k] = v;
            else w[k] = c > (i & 3) ? v : c == (i & 3) ? e : w[k];  // columns up to i are done
        }
        if (c == (i & 3)) code[ki] = q;
        // |w / s - code| next to 1/2 (beyond it only where the clamp acted), above 384 or NaN
        refused |= (frac - 0x3FDFFFFFu <= 1u) | (frac >= 0x40780000u);
        const uint32_t xh = static_cast<uint32_t>(__double2hiint(x)) & 0x7FFFFFFFu;
        refused |= (xh - (323u << 20) >= (1400u << 20)) & ((xh | static_cast<uint32_t>(__double2loint(x))) != 0u);
    }
    return !__any_sync(0xffffffffu, refused != 0u);
}

// The same in the order the definition states, divisions and all, on the row's 32 values in shared memory, which become the errors.
// Lanes that are not `active` only keep step.
__device__ __noinline__ void round_group_plain(double* val, bool active, int* code, const float* ug, int K, float d_f, double s, bool hi_seg,
                                               int lane) {
    const double lo = hi_seg ? -128.0 : -8.0, hi = hi_seg ? 127.0 : 7.0;
    const int c = lane & 3;
    for (int i = 0; i < 32; ++i) {
        const double d = __shfl_sync(0xffffffffu, static_cast<double>(d_f), i);
        const double wj = val[i];
        const double q = s > 0.0 ? fmin(fmax(rint(__ddiv_rn(wj, s)), lo), hi) : 0.0;
        const double e = __ddiv_rn(__dsub_rn(wj, __dmul_rn(q, s)), d);
        __syncwarp();
        if (active)
            for (int j = c; j < 32; j += 4) {
                if (j > i) val[j] = __dsub_rn(val[j], __dmul_rn(e, static_cast<double>(ug[static_cast<size_t>(i) * K + j])));
                if (j == i) {
                    val[j] = e;
                    code[j >> 2] = static_cast<int>(q);
                }
            }
        __syncwarp();
    }
}

// 1 / d as yh + yl, by Newton's iteration from the 23-bit approximation: residuals 1 - d y are exact (24 bits of d), so yh is
// within 2^-52 and the sum within 2^-100.  d outside 2^-100 .. 2^100 gives false.
__device__ __forceinline__ bool reciprocal_pair(float d_f, double& yh, double& yl) {
    float y_f;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y_f) : "f"(d_f));
    const double d = static_cast<double>(d_f), y0 = static_cast<double>(y_f);
    const double y1 = __fma_rn(y0, __fma_rn(-d, y0, 1.0), y0);
    yh = __fma_rn(y1, __fma_rn(-d, y1, 1.0), y1);
    yl = __dmul_rn(yh, __fma_rn(-d, yh, 1.0));
    return fabsf(d_f) >= 7.8886091e-31f && fabsf(d_f) <= 1.2676506e30f;
}

// acc[row] -= e[row][i] * u[i] for i = 0 .. n - 1 in order.
template <int R, int n>
__device__ __forceinline__ void feed_back(double (&acc)[R], const float (&u)[n], const double* e, int K) {
#pragma unroll
    for (int i = 0; i < n; i += 2) {
        const double ua = static_cast<double>(u[i]), ub = static_cast<double>(u[i + 1]);
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
            const double2 ee = *reinterpret_cast<const double2*>(e + static_cast<size_t>(rr) * K + i);
            acc[rr] = __dsub_rn(acc[rr], __dmul_rn(ee.x, ua));
            acc[rr] = __dsub_rn(acc[rr], __dmul_rn(ee.y, ub));
        }
    }
}

__device__ __forceinline__ void prefetch_l2(const float* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int R>
__global__ void __launch_bounds__(kCtaThreads, 1) gptq_rows_kernel(const Params p) {
    extern __shared__ __align__(16) unsigned char smem[];
    double* err = reinterpret_cast<double*>(smem);             // [R][K]: scaled errors of the columns visited
    __shared__ float red[2][R][2 * kWarps];
    __shared__ float scale[2][R];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n0 = blockIdx.x * R;
    const int rows = min(R, p.N - n0);
    const int K = p.K, r = p.r;
    const float* U = p.U;

    // Per-row absmax of the two segments in fp32 (dead columns zeroed), as Eq. 3 takes it.
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
        const float* src = p.W + static_cast<size_t>(n0 + min(rr, rows - 1)) * K;
        float a8 = 0.f, a4 = 0.f;
        for (int c = tid; c < K; c += kCtaThreads) {
            float w = src[c];
            if (p.dead && p.dead[c]) w = 0.f;
            if (c < r) a8 = fmaxf(a8, fabsf(w));
            else a4 = fmaxf(a4, fabsf(w));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a8 = fmaxf(a8, __shfl_xor_sync(0xffffffffu, a8, o));
            a4 = fmaxf(a4, __shfl_xor_sync(0xffffffffu, a4, o));
        }
        if (lane == 0) {
            red[0][rr][warp] = a8;
            red[1][rr][warp] = a4;
        }
    }
    __syncthreads();
    if (tid < rows) {
        float a8 = 0.f, a4 = 0.f;
        for (int w = 0; w < 2 * kWarps; ++w) {
            a8 = fmaxf(a8, red[0][tid][w]);
            a4 = fmaxf(a4, red[1][tid][w]);
        }
        float s8 = __fdiv_rn(a8, 127.f), s4 = __fdiv_rn(a4, 7.f);
        if (p.fp16) {
            s8 = __half2float(__float2half_rn(s8));
            s4 = __half2float(__float2half_rn(s4));
        }
        scale[0][tid] = s8;
        scale[1][tid] = s4;
        const size_t n = n0 + tid;
        if (p.fp16) {
            reinterpret_cast<__half*>(p.s8)[n] = __float2half_rn(s8);
            reinterpret_cast<__half*>(p.s4)[n] = __float2half_rn(s4);
        } else {
            reinterpret_cast<float*>(p.s8)[n] = s8;
            reinterpret_cast<float*>(p.s4)[n] = s4;
        }
    }
    __syncthreads();

    if (warp < kWarps) {
        // ---- updating warps: one column of the block per thread, through all columns before the block
        for (int c0 = 0; c0 < K; c0 += kThreads) {
            const int col = c0 + tid;
            const bool live = col < K;
            const float* ucol = U + (live ? col : K - 1);  // a lane past the last column reads that one, for nothing
            double acc[R];
#pragma unroll
            for (int rr = 0; rr < R; ++rr) {
                float w = live && rr < rows ? p.W[static_cast<size_t>(n0 + rr) * K + col] : 0.f;
                if (live && p.dead && p.dead[col]) w = 0.f;
                acc[rr] = static_cast<double>(w);
            }
            // Lane i asks L2 for the warp's 128 bytes of row kFar + i, then 32 rows on.  CTAs share this out: an eighth of the grid asks for a row.
            const unsigned share = gridDim.x >= 64 ? 7u : 0u;
            const float* ask = U + static_cast<size_t>(kFar + lane) * K + min(c0 + 32 * warp, K - 1);
            int ask_row = kFar + lane;
            auto request_rows = [&] {
                if constexpr (R > kAskRows) return;
                if ((((ask_row >> 5) + blockIdx.x) & share) == 0 && ask_row < K) prefetch_l2(ask);
                ask_row += 32;
                ask += static_cast<size_t>(32) * K;
            };
            const int known = max(c0 - kThreads, 0);  // columns rounded for certain: all blocks but the previous one
            float u_next[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) u_next[i] = ucol[static_cast<size_t>(i) * K];
            for (int j = 0; j < known; j += kAhead) {
                request_rows();
                float u[kAhead];
#pragma unroll
                for (int i = 0; i < kAhead; ++i) u[i] = u_next[i];
                // K >= known + kThreads: the rows requested past `known` exist
#pragma unroll
                for (int i = 0; i < kAhead; ++i) u_next[i] = ucol[static_cast<size_t>(j + kAhead + i) * K];
                feed_back<R, kAhead>(acc, u, err + j, K);
            }
            if (c0 > 0) {
                for (int g = 0; g < kWarps; ++g) {  // the previous block, group by group as it is rounded
                    const int j0 = known + 32 * g;
                    request_rows();  // the diagonal block's
                    float u[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) u[i] = ucol[static_cast<size_t>(j0 + i) * K];
                    named_sync(1 + g, kThreads + 32);
                    feed_back<R, 32>(acc, u, err + j0, K);
                }
            }
#pragma unroll
            for (int rr = 0; rr < R; ++rr)
                if (live) err[static_cast<size_t>(rr) * K + col] = acc[rr];  // handed over where its error will go
            named_arrive(kHandOver, kCtaThreads);
        }
    } else {
        // ---- rounding warps: a group of 32 columns of the block each
        const int g = warp - kWarps, row = lane >> 2, c = lane & 3;
        const bool active = row < R, stored = row < rows;
        const int rr = active ? row : R - 1;
        const double s8 = static_cast<double>(scale[0][min(rr, rows - 1)]), s4 = static_cast<double>(scale[1][min(rr, rows - 1)]);
        const double s8_inv = s8 > 0.0 ? __ddiv_rn(1.0, s8) : 0.0, s4_inv = s4 > 0.0 ? __ddiv_rn(1.0, s4) : 0.0;
        for (int c0 = 0; c0 < K; c0 += kThreads) {
            const int groups = min(kWarps, (K - c0) >> 5), j0 = c0 + 32 * g;
            if (g >= groups) {  // a last block that ends before
                named_sync(kHandOver, kCtaThreads);
                continue;
            }
            const float d_own = U[static_cast<size_t>(j0 + lane) * K + j0 + lane];
            const float* ucol = U + static_cast<size_t>(c0) * K + j0 + lane;  // the group's columns at the block's first row
            float u[32];
            if (g > 0) {
#pragma unroll
                for (int i = 0; i < 32; ++i) u[i] = ucol[static_cast<size_t>(i) * K];
            }
            double yh, yl;
            bool vouched = reciprocal_pair(d_own, yh, yl);
            named_sync(kHandOver, kCtaThreads);
            if (g > 0) {
                // ---- lane = column: the errors of the groups before
                double acc[R];
#pragma unroll
                for (int k = 0; k < R; ++k) acc[k] = err[static_cast<size_t>(k) * K + j0 + lane];
                for (int b = 0; b < g; ++b) {
                    float u_now[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) u_now[i] = u[i];
                    if (b + 1 < g) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) u[i] = ucol[static_cast<size_t>(32 * (b + 1) + i) * K];
                    }
                    named_sync(kInBlock + (b & 1), 32 * (groups - b));  // group b's errors are in place
                    feed_back<R, 32>(acc, u_now, err + c0 + 32 * b, K);
                }
#pragma unroll
                for (int k = 0; k < R; ++k) err[static_cast<size_t>(k) * K + j0 + lane] = acc[k];
                __syncwarp();
            }
            // ---- four lanes per row: the chain
            const bool hi_seg = j0 < r;
            const double s = hi_seg ? s8 : s4;
            const float* ug = U + static_cast<size_t>(j0) * K + j0;
            double* val = err + static_cast<size_t>(rr) * K + j0;
            double w[8];
            int code[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                w[k] = val[c + 4 * k];
                code[k] = 0;
            }
            vouched = __all_sync(0xffffffffu, vouched);
            vouched &= round_group(w, code, ug, K, yh, yl, s, hi_seg ? s8_inv : s4_inv, hi_seg, lane);
            if (vouched) {
                if (active) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) val[c + 4 * k] = w[k];
                }
            } else {
                int plain[8];
                round_group_plain(val, active, plain, ug, K, d_own, s, hi_seg, lane);
#pragma unroll
                for (int k = 0; k < 8; ++k) code[k] = plain[k];
            }
            __syncwarp();
            if (g + 1 < groups) named_arrive(kInBlock + (g & 1), 32 * (groups - g));
            if (c0 + kThreads < K) named_arrive(1 + g, kThreads + 32);  // K > c0 + 256: all 8 groups exist
            // ---- codes: four neighbouring columns of a row to a lane
            const size_t n = n0 + row;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                uint32_t bytes = (static_cast<uint32_t>(code[k]) & 0xFFu) << (8 * c);
                bytes |= __shfl_xor_sync(0xffffffffu, bytes, 1);
                bytes |= __shfl_xor_sync(0xffffffffu, bytes, 2);
                if (c != (k & 3) || !stored) continue;
                if (hi_seg) {
                    *reinterpret_cast<uint32_t*>(p.w8 + n * r + j0 + 4 * k) = bytes;
                } else {
                    const size_t K4 = K - r, j4 = j0 - r + 4 * k;
                    const uint32_t nib = bytes & 0x0F0F0F0Fu, two = nib | (nib >> 4);
                    *reinterpret_cast<uint16_t*>(p.w4 + (n * K4 + j4) / 2) = static_cast<uint16_t>((two & 0xFFu) | ((two >> 8) & 0xFF00u));
                    if (p.w4e) *reinterpret_cast<uint32_t*>(p.w4e + n * K4 + j4) = bytes;
                }
            }
        }
    }
}

template <int R>
cudaError_t launch_rows(const Params& p, cudaStream_t st) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(gptq_rows_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kGptqSmemPerCta));
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set[dev] = true;
    }
    const size_t smem = static_cast<size_t>(R) * p.K * 8;
    gptq_rows_kernel<R><<<(p.N + R - 1) / R, kCtaThreads, smem, st>>>(p);
    return cudaGetLastError();
}

}  // namespace

// cudaErrorNotSupported: a row (9 bytes per weight) does not fit in shared memory.
cudaError_t launch_pack_gptq(const float* W, const float* U, const uint8_t* dead, int N, int K, int r, int8_t* w8,
                             uint8_t* w4, void* s8, void* s4, bool scale_fp16, int8_t* w4e, cudaStream_t st) {
    if (static_cast<size_t>(K) * 9 > kRowLimit) return cudaErrorNotSupported;
    Params p{W, U, dead, N, K, r, w8, w4, s8, s4, scale_fp16 ? 1 : 0, w4e};
    count_launch();
    switch (gptq_rows_per_cta(N, K)) {
        case 1: return launch_rows<1>(p, st);
        case 2: return launch_rows<2>(p, st);
        case 3: return launch_rows<3>(p, st);
        case 4: return launch_rows<4>(p, st);
        case 5: return launch_rows<5>(p, st);
        case 6: return launch_rows<6>(p, st);
        case 7: return launch_rows<7>(p, st);
        default: return launch_rows<8>(p, st);
    }
}

}  // namespace resq
