// Rules on the host that pick a kernel form from the sizes of a call.  Plain arithmetic, no CUDA: the launchers use them, and
// the tests ask them which form a shape takes.
#pragma once
#include <cstddef>
#include <cstdint>

namespace resq {

// ---- mixed GEMM beyond 16 tokens: which kernel (mixed_gemm_mid.cu; mixed_gemm.cu: the large tiles), token tile, split
struct MidPlan {
    int ntok, tok_tiles, splits;
    bool use;  // false: the large tiles
};

// Which (token tile, split) and whether at all.  Modelled times in ns:
//   this kernel  waves * (k-blocks per pair * c(N) + 3200 + 27 N - 1500) + 1500, c = 214 up to N = 128, 297 at 256 (fewer
//                stages fit), plus the exchange: 1200 + 5 N (S = 2), 2200 + 6 N (S = 3); one wave is 74 pairs; clusters of
//                four fit one wave up to 128 CTAs, clusters of six up to 96 (144 took two), eight never paid;
//   tile kernel  rounds * (k-blocks * 295 + 4100) + 5800, a round being 74 tiles of 256 x 256 (within a tenth of 1214 times
//                over 22 layer shapes, 1024 x 2048 to 28672 x 8192, and 17 to 4096 tokens, weights in L2 and not).
// Where several waves follow one another the first line is short by 12 % and 1500 ns a wave, for the ends that the persistent
// kernel overlaps.  All of this was measured with the epilogues that both kernels had before the present ones: over those 1214 calls
// the choice was 0.1 % slower than the better kernel of each, at most 4 %.  With the present epilogues (both kernels over 240
// shapes, 917 runs) it is 0.4 %, a new fit of the same form 0.15 %.
inline MidPlan mid_plan(int T, int N, int kbt) {
    constexpr int kTile = 256;  // tokens and channels of a large tile
    const long ch = (N + kTile - 1) / kTile;
    const long tile_rounds = (ch * ((T + kTile - 1) / kTile) + 73) / 74;
    long best = tile_rounds * (kbt * 295L + 4100) + 5800;
    MidPlan pl = {0, 0, 0, false};
    for (int ntok = 256; ntok >= 32; ntok -= 32) {
        const int nt = (T + ntok - 1) / ntok;
        if (ntok > 32 && (T + ntok - 33) / (ntok - 32) == nt) continue;  // a narrower tile covers T with as many
        const long c = ntok <= 128 ? 214 : ntok == 160 ? 222 : ntok == 192 ? 231 : ntok == 224 ? 250 : 297;
        for (int s = 1; s <= 3; ++s) {
            const long ctas = ch * nt * 2 * s;
            if (s > 1 && (ctas > (s == 2 ? 128 : 96) || kbt < 4 * s)) break;
            const long waves = s > 1 ? 1 : (ch * nt + 73) / 74;
            const long one = (kbt + s - 1) / s * c + 3200 + 27L * ntok + (s == 2 ? 1200 + 5L * ntok : s == 3 ? 2200 + 6L * ntok : 0);
            long t = waves * (one - 1500) + 1500;
            if (waves > 1) t += t * 12 / 100 + waves * 1500;
            if (t < best) {
                best = t;
                pl = {ntok, nt, s, true};
            }
        }
    }
    return pl;
}

// ---- products of up to eight tokens (decode_stream.cu): whether every CTA quantizes the rows itself.  A row's share of the CTA's threads keeps
// its values in registers: up to 64 each, where all or half of the threads share a row, else 32.  us on the device, a quantizer before / in the
// product (K x N, symmetric): one row 1024 x 1024 6.8 / 4.8, 2048 x 3072 6.6 / 5.4, 4096 x 28672 14.1 / 13.2, 14336 x 4096 12.1 / 10.7; two rows
// 2048 x 3072 6.9 / 6.0, 8192 x 8192 12.2 / 11.9; four rows 2048 x 3072 7.3 / 6.7, but 4096 x 6144 9.0 / 9.8; six rows 1024 x 1024 6.6 / 6.4, but
// 2048 x 3072 7.4 / 8.2.  Weights from memory, 130 calls within the rule, both forms of codes: 0.73 to 1.00 of the time, but two rows of
// 6144 x 6144 and 8192 x 8192 and three of 2048 x 16384 1.03 to 1.04, one of 12288 x 4096 1.02 (the host's 2.4 us less beside it).
inline bool quantizes_rows(int T, int K) {
    const int threads = T > 4 ? 32 : T > 2 ? 64 : T > 1 ? 128 : 256;  // of a row
    return T <= 8 && K <= (T > 2 ? 32 : 64) * threads;
}

// Not where Y lies over some of X: every CTA reads all rows, while others store already.  A quantizer of its own has read X by then.
inline bool ranges_meet(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y ? y - x < a_bytes : x - y < b_bytes;
}

// ---- GPTQ packing (gptq.cu): rows per CTA, one CTA per SM.  As many as fit its shared memory (8 bytes per weight), then no
// more than spread the rows evenly over the rounds this takes.
constexpr int kGptqMaxRows = 8;                 // one rounding warp each
constexpr size_t kGptqSmemPerCta = 225 * 1024;  // dynamic shared memory of a CTA

inline int gptq_rows_per_cta(int N, int K) {
    int R = static_cast<int>(kGptqSmemPerCta / (static_cast<size_t>(K) * 8));
    if (R > kGptqMaxRows) R = kGptqMaxRows;
    const int rounds = (N + 148 * R - 1) / (148 * R);
    return (N + 148 * rounds - 1) / (148 * rounds);
}

// ---- query projection and cache append (kv_cache.cu), tiles of 16 head vectors: whether the warps of a CTA go through tiles together
constexpr long long kAppendWarps = 148 * 2 * 8;  // of the grid: tiles of a round
// Each kind of tile is tens of KB of straight code, and an SM whose warps are at different places of it waits for instructions.  As
// long as each kind is within a round the warps keep pace by themselves.  us, d = 128, 16 heads each, apart / together: 2600 tokens (2.2
// rounds of keys and values) 57.6 / 34.5, 3000 75 / 41 and without a query 46 / 31 (four of five cycles of a warp's wait);
// 32 / 8 heads, 2600 tokens (1.1) 36.3 / 32.4, 2048 (0.9) 27.2 / 29.0.  One round of keys and values and no second one beside: 1500
// tokens of 16 heads (1.3 + 0.6) 24.7 / 29.0.  d = 64, half the code: 2600 tokens of 16 heads 23.8 / 17.7, 2300 (1.95) 15.4 / 15.8.
inline bool append_tiles_together(int d, long long kv_tiles, long long tiles) {
    return kv_tiles > (d == 128 ? 1 : 2) * kAppendWarps && tiles >= 2 * kAppendWarps;
}

// ---- causal run (kv_prefill.cu): tiles of 128 rows per CTA, CTAs of a cluster that split the steps of 64 positions
struct PrefillPlan {
    int tiles_per_cta, splits;
    bool pair;             // the CTA's two tiles walk together, not one after the other
    long long row_groups;  // groups of tiles_per_cta tiles; the grid is row_groups * Hkv * splits
};  // d_head = 64 has no form for two tiles together (a thread would hold 32 outputs beside its scores)

// Between one and two rounds of tiles a CTA takes two of them, d_head = 128 in one of two forms.  In turn, a long and a short one:
// all CTAs are equally long, but each walks what both tiles see twice.  Together, two neighbours: they share the expanded codes and
// fill each other's waits.  So in turn is better for a prompt and together behind a prefix of about its length.  Measured (32 / 8 heads, 608
// to 1184 tokens behind 0 to 8 times as many, within 3 % but for one round more), ns: in turn 1330 a step and 13500, together 2080
// a step of two tiles and 10000; CTAs beyond 148 are a part of the last row group and follow another part of it.  1024 tokens, us in
// turn / together: at 0 36 / 44, behind 512 57 / 60, 1024 79 / 77, 4096 205 / 176, 8192 376 / 310.  Beyond two rounds
// together: 2048 tokens 114 / 82, behind 4096 447 / 349.  Measured while all scores of a pair came behind its output product; now a
// step of it takes 2030, which would take one of those 35 shapes to the other form (1184 tokens behind 592).
inline bool prefill_together(int pos0, int T, int g, int Hkv, long long single) {
    auto steps = [=](long long tile) -> long long {  // of 64 positions, up to the last one that the tile's rows see
        const long long last = (tile * 128 + 127) / g;
        return (pos0 + (last < T ? last + 1 : T) + 63) / 64;
    };
    const bool behind = (single + 1) / 2 * Hkv > 148;  // a CTA of the last row group follows another one
    const long long one = 2 * (1330 * steps(single / 2) + 8500), turn = 1330 * (steps(single - 1) + steps(0)) + 13500;
    const long long two = 2 * (2080 * steps(1) + 10000), pair = 2080 * steps(single - 1) + 10000;
    return (behind && two > pair ? two : pair) < (behind && one > turn ? one : turn);
}

inline PrefillPlan prefill_plan(int pos0, int T, int g, int Hkv, int d_head) {
    constexpr int kRows = 128, kStep = 64;
    PrefillPlan pl;
    const long long single = (static_cast<long long>(T) * g + kRows - 1) / kRows;
    const bool fits = single * Hkv <= 148, two_rounds = !fits && single * Hkv <= 2 * 148;
    pl.pair = d_head == 128 && !fits && (!two_rounds || prefill_together(pos0, T, g, Hkv, single));
    pl.tiles_per_cta = pl.pair || two_rounds ? 2 : 1;
    pl.row_groups = (single + pl.tiles_per_cta - 1) / pl.tiles_per_cta;
    const int steps = (pos0 + T + kStep - 1) / kStep;
    // One CTA per SM is in flight; at least four steps per CTA of a cluster pay for the merge.  15 clusters of eight run at the same time; one
    // more makes a second round.  At d_head = 64 that is what the tiles of 64 rows before took (32 / 8 heads, 64 tokens behind 4000: 39.2
    // us, 40.1 with eight CTAs each, 32.8 with four); at 128 (74 before, 42 and 31) the limit is still that of single CTAs.
    const int eights = d_head == 128 ? 148 : 15 * 8;
    pl.splits = 1;
    while (pl.splits < 8 && pl.row_groups * Hkv * pl.splits * 2 <= (pl.splits == 4 ? eights : 148) && steps >= 8 * pl.splits) pl.splits *= 2;
    return pl;
}

// ---- attention at d_head = 64, rows that are alone (kv_d64.cu)
enum Pack { kPackNever = 0, kPackIfShort = 1, kPackAlways = 2 };  // whether a CTA takes as many items as it has warps
struct Attn64Plan {
    int warps;        // per CTA
    int splits;       // CTAs of a cluster that share an item
    int pack;         // Pack
    int short_steps;  // kPackIfShort: items of up to as many steps of 32 positions are packed
    long long ctas;   // grid
};

// Query rows that are alone: one item per (row, KV head).  The lengths are on the device; the capacity stands in for them.
inline Attn64Plan attention64_rows_plan(int rows, int Hkv, int capacity) {
    const long long items = static_cast<long long>(rows) * Hkv;
    if (items >= 2 * 3 * 148) {
        // four rounds of full CTAs, three per SM: packed whatever the lengths
        const int pack = items >= 4LL * 3 * 148 * 4 ? kPackAlways : kPackIfShort;
        return {4, 1, pack, 4, pack == kPackAlways ? (items + 3) / 4 : items};
    }
    // twelve warps, one CTA per SM.  A round of CTAs with an item each takes about as long as one and a half steps of a
    // packed CTA; three packed steps lost where lengths differ (512 items of 64 to 128 positions: 15 -> 19 us).
    Attn64Plan pl{12, 1, items > 148 ? kPackIfShort : kPackNever, items > 2 * 148 ? 2 : 1, 0};
    // at least two steps per warp
    while (pl.splits < 8 && items * pl.splits * 2 <= 148 && capacity / 32 >= 4 * 12 * pl.splits) pl.splits *= 2;
    pl.ctas = items * pl.splits;
    return pl;
}

}  // namespace resq
