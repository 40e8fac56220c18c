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
// shared memory at every step, behind two barriers.)  Meanwhile one rounding warp per row takes the current block through
// its chain, 32 columns at a time with the values exchanged by shuffles, and hands each 32 over to the updating
// warps through a named barrier; an updated block comes back in the slots its errors will take.
// K = N = 4096: 65.1 ms right-looking, 11.5 ms left-looking with all warps waiting for the chain (two CTAs per
// SM), 7.2 ms as it stands, the fp64 pipe 52 % busy (3.7 ms if it were always).
#include <cuda_fp16.h>

#include "internal.h"
#include "plans.h"

namespace resq {
namespace {

constexpr int kThreads = 256;  // = columns of a block
constexpr int kWarps = kThreads / 32;
constexpr int kAhead = 32;        // columns of U a thread requests ahead of their use (L2 latency)
static_assert(kGptqMaxRows <= kWarps, "one warp per row rounds");
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

// One group of 32 columns of one row, lane l holding column l's value w (all earlier columns applied): rounds the
// columns in order and feeds each error back into the ones after it.  u[i]: U[i] of the group at this lane's column.
// Returns false when the short form cannot vouch for a rounding; the caller then runs the plain form on the same input.
//
// The 32 steps depend on one another, so a step's latency is what counts: nine dependent fp64 operations here (about
// 370 cycles) against two divisions, a rounding, a clamp and branches (about 740) in the plain form.
//  * code: fma(w, 1/s, 1.5 * 2^52) leaves rint(w (1/s)) in the low word, clamped there.  w (1/s) is within 2^-44 of
//    the rounded quotient for |quotient| <= 2^9, so the two round apart only next to a half-integer: refused.
//  * x = w - code s by one fma: the product is exact (8 + 24 bits).
//  * e = x / d: q0 = w / d - code (s / d) is formed beside x from products with y = RN(1 / d), two corrections
//    q += (x - d q) y follow, of which the last rounds correctly by Markstein's theorem (P. Markstein, "Computation of
//    elementary functions on the IBM RISC System/6000 processor", 1990) when y is the rounded reciprocal and the
//    quotient before it faithful.  q0 is off by a few 2^-53 |w / d|, so a tiny x / w (below 2^-40), where one
//    correction would not make it faithful, is refused; so are x and d whose products could leave the normal range.
__device__ __forceinline__ bool round_group(double w, const float (&u)[32], float d_f, double s, bool hi_seg, int lane,
                                            double& e_own, int& code_own) {
    const double d_own = static_cast<double>(d_f);
    const int ilo = hi_seg ? -128 : -8, ihi = hi_seg ? 127 : 7;
    const double s_inv = s > 0.0 ? __ddiv_rn(1.0, s) : 0.0;
    const double y_own = __ddiv_rn(1.0, d_own);
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    bool refused = !(fabsf(d_f) >= 1.17549435e-38f && fabsf(d_f) <= 3.402823466e38f);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const double d = __shfl_sync(0xffffffffu, d_own, i), y = __shfl_sync(0xffffffffu, y_own, i);
        const double wj = __shfl_sync(0xffffffffu, w, i);
        const int k = min(max(__double2loint(__fma_rn(wj, s_inv, magic)), ilo), ihi);
        const double c = __dsub_rn(__hiloint2double(0x43380000 + (k >> 31), k), magic);
        const double x = __fma_rn(-c, s, wj);
        double q = __fma_rn(-c, __dmul_rn(s, y), __dmul_rn(wj, y));
        q = __fma_rn(__fma_rn(-q, d, x), y, q);
        const double e = __fma_rn(__fma_rn(-q, d, x), y, q);
        w = __dsub_rn(w, __dmul_rn(e, static_cast<double>(u[i])));  // lanes <= i hold finished columns
        const double t = __dmul_rn(wj, s_inv);
        const double frac = fabs(__dsub_rn(t, c));  // beyond 1/2 only where the clamp acted
        const uint32_t ex = static_cast<uint32_t>(__double2hiint(x)) & 0x7FF00000u;
        const bool x_ok = ex - (300u << 20) < (1500u << 20) && fabs(x) > 9.094947017729282e-13 * fabs(wj);
        refused |= (frac > 0.5 - 1e-9 && frac < 0.5 + 1e-9) || fabs(t) > 512.0 || !(x_ok || wj == 0.0);
        if (lane == i) {
            e_own = e;
            code_own = k;
        }
    }
    return !__any_sync(0xffffffffu, refused);
}

// The same in the order the definition states, divisions and all.  ug: U at the group's first row, this lane's column.
__device__ __noinline__ double round_group_plain(double w, const float* ug, int K, float d_f, double s, bool hi_seg,
                                                 int lane, int* code_own) {
    const double lo = hi_seg ? -128.0 : -8.0, hi = hi_seg ? 127.0 : 7.0;
    double e_own = 0.0;
    for (int i = 0; i < 32; ++i) {
        const double d = __shfl_sync(0xffffffffu, static_cast<double>(d_f), i);
        const double wj = __shfl_sync(0xffffffffu, w, i);
        const double c = s > 0.0 ? fmin(fmax(rint(__ddiv_rn(wj, s)), lo), hi) : 0.0;
        const double e = __ddiv_rn(__dsub_rn(wj, __dmul_rn(c, s)), d);
        w = __dsub_rn(w, __dmul_rn(e, static_cast<double>(ug[static_cast<size_t>(i) * K])));
        if (lane == i) {
            e_own = e;
            *code_own = static_cast<int>(c);
        }
    }
    return e_own;
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

__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int R>
__global__ void __launch_bounds__(kThreads + 32 * R, 1) gptq_rows_kernel(const Params p) {
    extern __shared__ __align__(16) unsigned char smem[];
    double* err = reinterpret_cast<double*>(smem);             // [R][K]: scaled errors of the columns visited
    __shared__ float red[2][R][kWarps + R];
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
        for (int c = tid; c < K; c += kThreads + 32 * R) {
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
        for (int w = 0; w < kWarps + R; ++w) {
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
            const int known = max(c0 - kThreads, 0);  // columns rounded for certain: all blocks but the previous one
            float u_next[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) u_next[i] = ucol[static_cast<size_t>(i) * K];
            for (int j = 0; j < known; j += kAhead) {
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
                    float u[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) u[i] = ucol[static_cast<size_t>(j0 + i) * K];
                    named_sync(1 + g, kThreads + 32 * R);
                    feed_back<R, 32>(acc, u, err + j0, K);
                }
            }
#pragma unroll
            for (int rr = 0; rr < R; ++rr)
                if (live) err[static_cast<size_t>(rr) * K + col] = acc[rr];  // handed over where its error will go
            named_arrive(1 + kWarps, kThreads + 32 * R);
        }
    } else {
        // ---- rounding warps: one row each; the block's columns c0 + 32 m + lane in w[m]
        const int rr = warp - kWarps;
        for (int c0 = 0; c0 < K; c0 += kThreads) {
            named_sync(1 + kWarps, kThreads + 32 * R);
            const int groups = min(kWarps, (K - c0) >> 5);
            double w[kWarps];
#pragma unroll
            for (int m = 0; m < kWarps; ++m)
                w[m] = m < groups ? err[static_cast<size_t>(rr) * K + c0 + 32 * m + lane] : 0.0;
            __syncwarp();
#pragma unroll
            for (int g = 0; g < kWarps; ++g) {
                if (g < groups) {
                    const int j0 = c0 + 32 * g;
                    const float* ug = U + static_cast<size_t>(j0) * K + j0 + lane;
                    float u[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) u[i] = ug[static_cast<size_t>(i) * K];
                    const float d = ug[static_cast<size_t>(lane) * K];
                    const double s = static_cast<double>(scale[j0 < r ? 0 : 1][rr]);
                    double e_own = 0.0;
                    int code = 0;
                    if (rr < rows) {  // the whole warp
                        if (!round_group(w[g], u, d, s, j0 < r, lane, e_own, code))
                            e_own = round_group_plain(w[g], ug, K, d, s, j0 < r, lane, &code);
                        const size_t n = n0 + rr;
                        const int nib = __shfl_down_sync(0xffffffffu, code, 1);
                        if (j0 < r) {
                            p.w8[n * r + j0 + lane] = static_cast<int8_t>(code);
                        } else {
                            const int K4 = K - r;
                            if ((lane & 1) == 0)
                                p.w4[n * (K4 / 2) + (j0 - r + lane) / 2] =
                                    static_cast<uint8_t>((code & 0xF) | ((nib & 0xF) << 4));
                            if (p.w4e) p.w4e[n * K4 + j0 - r + lane] = static_cast<int8_t>(code);
                        }
                    }
                    err[static_cast<size_t>(rr) * K + j0 + lane] = e_own;
                    __syncwarp();
                    if (c0 + kThreads < K) named_arrive(1 + g, kThreads + 32 * R);  // K > c0 + 256: all 8 groups exist
#pragma unroll
                    for (int m = g + 1; m < kWarps; ++m) {
                        if (m < groups) {
                            float um[32];
#pragma unroll
                            for (int i = 0; i < 32; ++i) um[i] = ug[static_cast<size_t>(i) * K + 32 * (m - g)];
                            double one[1] = {w[m]};
                            feed_back<1, 32>(one, um, err + static_cast<size_t>(rr) * K + j0, K);
                            w[m] = one[0];
                        }
                    }
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
    gptq_rows_kernel<R><<<(p.N + R - 1) / R, kThreads + 32 * R, smem, st>>>(p);
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
