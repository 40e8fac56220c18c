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
// not the row.  Columns go in blocks of 512.  Eight updating warps keep two columns of the next block per thread, 2 R
// running values in registers, through all earlier columns: one coalesced read of U per row and thread, converted once for R
// rows, e as a broadcast of two columns per load.  (A right-looking sweep reads and writes every remaining weight in
// shared memory at every step, behind two barriers.)  Meanwhile eight rounding warps take the current block through its
// chain, two groups of 32 columns each: a warp feeds the errors of the groups before into its own as the updating warps do, then takes
// all R rows through the chain at once, four lanes per row, and hands the group's errors on.
// An updated block comes back in the slots its errors will take.
//
// Beside an fp64 instruction, which holds a scheduler for two cycles, every other one costs a cycle, a conversion of U about five.  Cycles that
// 512 columns of U take in the updating warps alone, R = 7 (112 in the fp64 pipe): 165 with one column per thread, 135 with two
// (half the broadcasts and loads), 131 with four or eight rows of U asked for again where they were used instead of copied.
// K = N = 4096: 65.1 ms right-looking, 11.5 ms left-looking with all warps waiting for the chain (two CTAs per
// SM), 7.2 ms with a rounding warp per row, 6.2 with blocks of 256 and one column per thread, 5.5 ms as it stands (3.7 ms if the fp64 pipe
// were always busy).  Of its 10300 cycles alone a group of 32 columns spent 8500 in the chain, 270 a step; now 4200 of 6100
// (512 columns, 256 rows: 105 -> 78 us).  U comes from DRAM where it
// does not stay in L2 (the first call on it, K above 4096), later than the loads a thread has on their way: the updating warps ask L2
// for it 256 rows ahead.  Caches cold, ms without / with: K = 4096, 592 rows 2.06 / 1.16 (blocks of 256), 888 rows 1.35 / 1.25 (warm 1.21 / 1.22),
// 4096 rows 5.52 / 5.47; K = 8192, 1184 rows 18.9 / 10.3 (blocks of 256).
#include <cuda_fp16.h>

#include "internal.h"
#include "plans.h"
#include "ptx.cuh"

namespace resq {
namespace {

constexpr int kThreads = 256;     // updating threads, two columns of a block each
constexpr int kWarps = kThreads / 32;
constexpr int kBlock = 2 * kThreads, kGroups = kBlock / 32;
constexpr int kCtaThreads = 2 * kThreads;  // eight updating, eight rounding warps
static_assert(kGptqMaxRows * 4 <= 32, "four lanes per row");
constexpr int kFar = 256;         // rows of U a warp asks L2 for ahead of their use (DRAM latency; a multiple of 32)
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
    int* status;
    int diag_pitch;  // of the diagonal blocks in the errors' slots; 0: they have room of their own behind the errors
};

// U's diagonal block of a group in doubles, above the diagonal only, row behind row: (i, j) at tri(i) + j.  Read at j <= i (lanes that
// then drop what they read) it stays within the kTri slots.
constexpr int kTri = 512;
__host__ __device__ constexpr int tri(int i) { return 30 * i - i * (i - 1) / 2; }
static_assert(tri(0) >= 0 && tri(30) + 31 < kTri, "packed diagonal block");

// One rounding: the code of w, its error x = w - code s, and e = x / U[j][j] (y: 1 / U[j][j] in two parts).
//  * code: fma(w, 1/s, 1.5 * 2^52) leaves rint(w (1/s)) in the low word, clamped there.  w (1/s) is within 2^-43 of
//    the rounded quotient for |quotient| <= 2^9, so the two round apart only next to a half-integer: refused (by the upper
//    word of the distance, which resolves 2^-22).
//  * x by one fma: the product is exact (8 + 24 bits).
//  * e = fma(x, yh, x yl) with yh + yl = 1 / d to 2^-100 (N. Brisebarre and J.-M. Muller, "Correctly rounded
//    multiplication by arbitrary precision constants", 2008).  d has 24 bits, so x / d lies at least 2^-78 (relative) from the
//    midpoint of two doubles: it is (X 2^k - M D) / D beside M with whole numbers X < 2^53, D < 2^24, M < 2^54, and the
//    numerator is not 0, M D being odd and beyond 2^53.  The sum before its one rounding is within 2^-103.  x and d whose products
//    could leave the normal range are refused.
struct Rounding {
    int q;
    double cd, x, e;
};
__device__ __forceinline__ Rounding round_short(double w, double s, double s_inv, int ilo, int ihi, double2 y) {
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    Rounding o;
    o.q = min(max(__double2loint(__fma_rn(w, s_inv, magic)), ilo), ihi);
    o.cd = __dsub_rn(__hiloint2double(0x43380000 + (o.q >> 31), o.q), magic);
    o.x = __fma_rn(-o.cd, s, w);
    o.e = __fma_rn(o.x, y.x, __dmul_rn(o.x, y.y));
    return o;
}
__device__ __forceinline__ bool refused(const Rounding& o, double w, double s_inv) {
    const uint32_t frac = static_cast<uint32_t>(__double2hiint(__fma_rn(w, s_inv, -o.cd))) & 0x7FFFFFFFu;
    const uint32_t xh = static_cast<uint32_t>(__double2hiint(o.x)) & 0x7FFFFFFFu;
    // |w / s - code| next to 1/2 (beyond it only where the clamp acted), above 384 or NaN
    return (frac - 0x3FDFFFFFu <= 1u) | (frac >= 0x40780000u) |
           ((xh - (323u << 20) >= (1400u << 20)) & ((xh | static_cast<uint32_t>(__double2loint(o.x))) != 0u));
}

// The chain of a group of 32 columns: lane 4 row + c holds columns c + 4 k of its row in w[k], all earlier columns applied; afterwards
// w[k] has the group's earlier columns applied too: the value that is rounded.  ud: U's diagonal block, y: 1 / U[j][j] in two parts.
//
// The 32 steps depend on one another, so a step's latency counts (seven dependent fp64 operations against two divisions, a rounding,
// a clamp and branches in the plain form), and, beside two updating warps, its instructions.  So the next column's value comes by a
// shuffle before this step's update and every lane of the row applies the update itself; U waits in shared memory, in
// doubles (a conversion takes a scheduler as long as three fp64 operations, a shuffle as long as two); and codes, errors and the tests of what the short form
// can vouch for are taken from the values afterwards, eight columns of a lane side by side.
__device__ __forceinline__ void round_group(double (&w)[8], const double* ud, const double2* y, double s, double s_inv, int ilo, int ihi, int lane) {
    const int c = lane & 3, quad = lane & ~3;
    double wj = __shfl_sync(0xffffffffu, w[0], quad);
#pragma unroll
    for (int i = 0; i < 31; ++i) {
        const int ki = i >> 2, kn = (i + 1) >> 2;
        const double w_next = __shfl_sync(0xffffffffu, w[kn], quad + ((i + 1) & 3));
        const double e = round_short(wj, s, s_inv, ilo, ihi, y[i]).e;
        wj = __dsub_rn(w_next, __dmul_rn(e, ud[tri(i) + i + 1]));
#pragma unroll
        for (int k = kn; k < 8; ++k) {
            const double v = __dsub_rn(w[k], __dmul_rn(e, ud[tri(i) + 4 * k + c]));
            w[k] = k > ki || c > (i & 3) ? v : w[k];  // columns up to i are done
        }
    }
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

// acc[c][row] -= e[row][i] * u[c][i] for i = 0 .. n - 1 in order.
template <int R, int C, int n>
__device__ __forceinline__ void feed_back(double (&acc)[C][R], const float (&u)[C][n], const double* e, int K) {
#pragma unroll
    for (int i = 0; i < n; i += 2) {
        double ua[C], ub[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            ua[c] = static_cast<double>(u[c][i]);
            ub[c] = static_cast<double>(u[c][i + 1]);
        }
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
            const double2 ee = *reinterpret_cast<const double2*>(e + static_cast<size_t>(rr) * K + i);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                acc[c][rr] = __dsub_rn(acc[c][rr], __dmul_rn(ee.x, ua[c]));
                acc[c][rr] = __dsub_rn(acc[c][rr], __dmul_rn(ee.y, ub[c]));
            }
        }
    }
}

__device__ __forceinline__ void prefetch_l2(const float* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// A block takes a millisecond at most (K = 14336: 0.5), so the caller's limit counts from a second on.  Polling instead of sleeping
// takes issue slots from the updating warps (3 %).
constexpr uint64_t kBlockNs = 1000000000;

template <int R>
__global__ void __launch_bounds__(kCtaThreads, 1) gptq_rows_kernel(const Params p) {
    // Rows of U per set that an updating thread has on their way, two sets.  As many as the registers hold: K = 4096, ms with 4 / 8 / 16: R = 7
    // 5.41 / 5.64 / spills; R = 4 - / 0.96 / 1.08; K = 8192, R = 2 - / 2.47 / 2.34.
    constexpr int kAhead = R >= 6 ? 4 : R >= 3 ? 8 : 16;
    extern __shared__ __align__(16) unsigned char smem[];
    double* err = reinterpret_cast<double*>(smem);             // [R][K]: scaled errors of the columns visited
    float* red = reinterpret_cast<float*>(smem);               // [2][R][warps], over the errors
    __shared__ float scale[2][R];
    __shared__ double2 inv_d[2][32];                           // 1 / U[j][j] in two parts, of two groups by turns
    __shared__ uint64_t ready, done[kGroups];  // a block's columns are updated; a group of it is rounded
    __shared__ int abort_flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n0 = blockIdx.x * R;
    const int rows = min(R, p.N - n0);
    const int K = p.K, r = p.r;
    const float* U = p.U;
    // Blocks are kBlock wide but for the first, which takes what is left: a narrow last one would keep threads idle through all columns.
    const int first_width = (K - 1) % kBlock + 1, first_groups = first_width >> 5;
    if (tid == 0) {
        mbar_init(&ready, kWarps + max(kWarps - first_groups, 0));  // and the rounding warps without a group in the first block
        for (int g = 0; g < kGroups; ++g) mbar_init(&done[g], 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) { return mbar_wait_asleep(bar, parity, &abort_flag, p.status, kBlockNs); };
    // parity of group g's phase in block b (groups beyond the first block's start a block later)
    auto done_parity = [&](int g, int b) { return static_cast<uint32_t>(b + (g >= first_groups ? 1 : 0)) & 1u; };

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
            red[rr * 2 * kWarps + warp] = a8;
            red[(R + rr) * 2 * kWarps + warp] = a4;
        }
    }
    __syncthreads();
    if (tid < rows) {
        float a8 = 0.f, a4 = 0.f;
        for (int w = 0; w < 2 * kWarps; ++w) {
            a8 = fmaxf(a8, red[tid * 2 * kWarps + w]);
            a4 = fmaxf(a4, red[(R + tid) * 2 * kWarps + w]);
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
        // ---- updating warps: two columns of the block per thread, through all columns before the block
        int prev0 = 0, c0 = 0;  // first column of the block before, of this one
        const uint32_t pitch = K * 4u;
        for (int b = 0; c0 < K; ++b) {
            const int width = b == 0 ? first_width : kBlock;
            const int col = c0 + 2 * tid;
            const bool live = 2 * tid < width;
            uint32_t at = (live ? col : K - 2) * 4u;  // of the next row's two columns in U; a lane past the first block's last column reads the last two, for nothing
            double acc[2][R];
#pragma unroll
            for (int rr = 0; rr < R; ++rr) {
                float2 w = make_float2(0.f, 0.f);
                if (live && rr < rows) {
                    w = *reinterpret_cast<const float2*>(p.W + static_cast<size_t>(n0 + rr) * K + col);
                    if (p.dead && p.dead[col]) w.x = 0.f;
                    if (p.dead && p.dead[col + 1]) w.y = 0.f;
                }
                acc[0][rr] = static_cast<double>(w.x);
                acc[1][rr] = static_cast<double>(w.y);
            }
            // Lane i asks L2 for the warp's 256 bytes of row kFar + i, then 32 rows on.  CTAs share this out: an eighth of the grid asks for a row.
            const unsigned share = gridDim.x >= 64 ? 7u : 0u;
            const float* ask = U + static_cast<size_t>(kFar + lane) * K + min(c0 + 64 * warp, K - 1);
            int ask_row = kFar + lane;
            auto request_rows = [&] {
                if ((((ask_row >> 5) + blockIdx.x) & share) == 0 && ask_row < K) {
                    prefetch_l2(ask);
                    if (c0 + 64 * warp + 32 < K) prefetch_l2(ask + 32);
                }
                ask_row += 32;
                ask += static_cast<size_t>(32) * K;
            };
            // Two sets of rows by turns, each asked for again behind its use (copies between sets would cost an issue slot a value).
            float u0[2][kAhead], u1[2][kAhead];
            auto load_rows = [&](float (&u)[2][kAhead]) {
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    const float2 v = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(U) + at);
                    at += pitch;
                    u[0][i] = v.x;
                    u[1][i] = v.y;
                }
            };
            load_rows(u0);
            load_rows(u1);
            // 32 columns; the rows asked for behind the last of them are the block's own: it has 32
            auto feed_32 = [&](int j) {
                request_rows();
#pragma unroll 1
                for (int t = 0; t < 32; t += 2 * kAhead) {
                    feed_back<R, 2, kAhead>(acc, u0, err + j + t, K);
                    load_rows(u0);
                    feed_back<R, 2, kAhead>(acc, u1, err + j + t + kAhead, K);
                    load_rows(u1);
                }
            };
            for (int j = 0; j < prev0; j += 32) feed_32(j);
            for (int j = prev0; j < c0; j += 32) {  // the block before, group by group as it is rounded
                if (!warp_wait(&done[(j - prev0) >> 5], done_parity((j - prev0) >> 5, b - 1))) goto failed;
                feed_32(j);
            }
            if (live) {  // handed over where its errors will go
#pragma unroll
                for (int rr = 0; rr < R; ++rr)
                    *reinterpret_cast<double2*>(err + static_cast<size_t>(rr) * K + col) = make_double2(acc[0][rr], acc[1][rr]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ready);
            prev0 = c0;
            c0 += width;
        }
    } else {
        // ---- rounding warps: groups of 32 columns of the block by turns
        const int row = lane >> 2, c = lane & 3;
        const bool active = row < R, stored = row < rows;
        const int rr = active ? row : R - 1;
        const double s8 = static_cast<double>(scale[0][min(rr, rows - 1)]), s4 = static_cast<double>(scale[1][min(rr, rows - 1)]);
        const double s8_inv = s8 > 0.0 ? __ddiv_rn(1.0, s8) : 0.0, s4_inv = s4 > 0.0 ? __ddiv_rn(1.0, s4) : 0.0;
        // A warp without a group in the first block has no say in its phase of `ready`, and two could complete while it sleeps in its wait.
        // So it arrives too: at its start, then for the next phase when it has seen this one.
        const bool onlooker = warp - kWarps >= first_groups;
        if (onlooker && lane == 0) mbar_arrive(&ready);
        auto block_ready = [&](int b) {
            if (!warp_wait(&ready, b & 1)) return false;
            if (onlooker && lane == 0) mbar_arrive(&ready);
            return true;
        };
        for (int b = 0, c0 = 0; c0 < K; c0 += b == 0 ? first_width : kBlock, ++b) {
            const int groups = b == 0 ? first_groups : kGroups;
            if (warp - kWarps >= groups && !block_ready(b)) goto failed;
            // Diagonal blocks, two by turns: behind the errors where that fits, else in slots of two rows that wait for nothing now: the next
            // block's, which is handed over when this one is rounded, or behind the last block the second one's, whose errors nobody reads any more.
            double* diag = p.diag_pitch ? err + static_cast<size_t>(c0 + kBlock < K ? c0 + (b == 0 ? first_width : kBlock) : first_width)
                                        : err + static_cast<size_t>(R) * K;
            const int diag_pitch = p.diag_pitch ? p.diag_pitch : kTri;
            for (int g = warp - kWarps; g < groups; g += kWarps) {
                const int j0 = c0 + 32 * g;
                const float* ucol = U + static_cast<size_t>(c0) * K + j0 + lane;  // the group's columns at the block's first row
                float ud[32], u[32];  // of the diagonal block; of the rows of a group before
#pragma unroll
                for (int i = 0; i < 32; ++i) ud[i] = ucol[static_cast<size_t>(32 * g + i) * K];
                if (g > 0) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) u[i] = ucol[static_cast<size_t>(i) * K];
                }
                const float d_own = U[static_cast<size_t>(j0 + lane) * K + j0 + lane];
                double* tri_ud = diag + (g & 1) * static_cast<size_t>(diag_pitch);
                double2 y;
                bool vouched = reciprocal_pair(d_own, y.x, y.y);
                if (g < kWarps && !block_ready(b)) goto failed;
                auto keep_diagonal = [&] {  // once the group before the last has left its place
#pragma unroll
                    for (int i = 0; i < 31; ++i)
                        if (lane > i) tri_ud[tri(i) + lane] = static_cast<double>(ud[i]);
                    inv_d[g & 1][lane] = y;
                };
                if (g < 2) keep_diagonal();
                if (g > 0) {
                    // ---- lane = column: the errors of the groups before
                    double acc[1][R];
#pragma unroll
                    for (int k = 0; k < R; ++k) acc[0][k] = err[static_cast<size_t>(k) * K + j0 + lane];
                    for (int before = 0; before < g; ++before) {
                        if (!warp_wait(&done[before], done_parity(before, b))) goto failed;
#pragma unroll
                        for (int part = 0; part < 2; ++part) {
                            float u_now[1][16];
#pragma unroll
                            for (int i = 0; i < 16; ++i) u_now[0][i] = u[16 * part + i];
                            feed_back<R, 1, 16>(acc, u_now, err + c0 + 32 * before + 16 * part, K);
                            if (before + 1 < g) {
#pragma unroll
                                for (int i = 0; i < 16; ++i) u[16 * part + i] = ucol[static_cast<size_t>(32 * (before + 1) + 16 * part + i) * K];
                            }
                        }
                        if (before == g - 2) keep_diagonal();
                    }
#pragma unroll
                    for (int k = 0; k < R; ++k) err[static_cast<size_t>(k) * K + j0 + lane] = acc[0][k];
                }
                __syncwarp();
                // ---- four lanes per row: the chain
                const bool hi_seg = j0 < r;
                const double s = hi_seg ? s8 : s4, s_inv = hi_seg ? s8_inv : s4_inv;
                const int ilo = hi_seg ? -128 : -8, ihi = hi_seg ? 127 : 7;
                double* val = err + static_cast<size_t>(rr) * K + j0;
                double w[8];
                int code[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) w[k] = val[c + 4 * k];
                round_group(w, tri_ud, inv_d[g & 1], s, s_inv, ilo, ihi, lane);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const Rounding o = round_short(w[k], s, s_inv, ilo, ihi, inv_d[g & 1][c + 4 * k]);
                    vouched = vouched && !refused(o, w[k], s_inv);
                    code[k] = o.q;
                    w[k] = o.e;
                }
                vouched = __all_sync(0xffffffffu, vouched);
                if (vouched) {
                    if (active) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) val[c + 4 * k] = w[k];
                    }
                } else {
                    int plain[8];
                    round_group_plain(val, active, plain, U + static_cast<size_t>(j0) * K + j0, K, d_own, s, hi_seg, lane);
#pragma unroll
                    for (int k = 0; k < 8; ++k) code[k] = plain[k];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&done[g]);
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
    return;
failed:  // the shared flag is set: every other warp leaves at its next wait
    if (lane == 0) atomicOr(p.status, kStatusBitTimeout);
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
    // Room for two diagonal blocks, or none: then K is above 3300, of seven blocks and more, and R at least 2 (gptq_rows_per_cta).
    const size_t smem = static_cast<size_t>(R) * p.K * 8, diag = 2 * kTri * sizeof(double);
    const bool apart = smem + diag <= kGptqSmemPerCta;
    Params q = p;
    q.diag_pitch = apart ? 0 : p.K;
    gptq_rows_kernel<R><<<(p.N + R - 1) / R, kCtaThreads, smem + (apart ? diag : 0), st>>>(q);
    return cudaGetLastError();
}

}  // namespace

// cudaErrorNotSupported: a row (9 bytes per weight) does not fit in shared memory.
cudaError_t launch_pack_gptq(const float* W, const float* U, const uint8_t* dead, int N, int K, int r, int8_t* w8,
                             uint8_t* w4, void* s8, void* s4, bool scale_fp16, int8_t* w4e, cudaStream_t st) {
    if (static_cast<size_t>(K) * 9 > kRowLimit) return cudaErrorNotSupported;
    Params p{W, U, dead, N, K, r, w8, w4, s8, s4, scale_fp16 ? 1 : 0, w4e, device_status_ptr(), 0};
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
