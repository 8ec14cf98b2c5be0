// How the wide GEMM (gemm_wide.cuh) cuts its output into tiles.  Host code only, free of CUDA.
//
// What bounds it: a prompt's or an unpadded batch's token count is new on nearly every call, and a forward or backward of a
// few hundred tokens asks for up to seven plans before its first launch, while the GPU waits.  The search therefore costs
// about a microsecond a plan: three evaluations of a candidate instead of one per CTA pair, and most candidates dropped
// before that by the average of their tiles' cycles over the pairs.  (The ten plans that one new token count can ask for on
// the 4096 x 11008 layer, slowest of 64 counts, one core: 12 us; every pair of every candidate: 870.)
#pragma once

#include <algorithm>
#include <cstdint>
#include <mutex>

namespace moc {
namespace tc {

constexpr int WIDE_N = 512, WIDE_STEP = 64, WIDE_SKEW = 2;

// How the output is cut.  Rows: 256-row blocks of all problems.  The first `t1` tiles are w1 columns wide, the others w2.
//   by_columns == 0: rows one after the other, their tiles from left to right; the first `split` rows have wide tiles
//   by_columns == 1: column by column, all rows in turn (few rows and a large B: B is read once); the first `split` columns
//                    have wide tiles
struct TilePlan {
    int rows, by_columns, split, w1, nt1, w2, nt2, t1, total;
    double cycles;  // of the pair that finishes last, by the model below
};

// SM cycles a pair needs for one contraction block of a tile of w columns: its MMAs, or the loads at what an SM gets from L2
constexpr double WIDE_MMA_CYCLES = 2.06;  // per column
inline double wide_block_cycles(int w) { return std::max(WIDE_MMA_CYCLES * w, (16384.0 + 64.0 * w) / 58.0); }

// Cycles that an accumulator of 256 columns costs (bf16 outputs; fp32 ones among them): what the epilogue keeps it from the MMAs,
// of which the skew covers a part, and what its stores take of the loads' way to L2.  Measured, a tile of two accumulators and 32
// blocks is 250 cycles longer than its MMAs with bf16 outputs and 2700 with fp32 gate values in every other tile.  Larger than
// that, because they also keep the search from tiles of 256 + 64 columns, whose MMAs of 64 columns take what 128 do (62 blocks: 890
// cycles each instead of the 659 of wide_block_cycles): with 1024 and 2000, 16544 x 3960 x 10560 took such tiles throughout
// and its gate + up 2.77 ms instead of 2.42.
constexpr int WIDE_DRAIN_BF16 = 2000, WIDE_DRAIN_F32 = 3500;

// No plan of `rows` x N over kb blocks is shorter: its MMAs spread evenly.
inline double plan_cycles_at_least(int rows, int64_t N, int kb, int pairs) { return WIDE_MMA_CYCLES * rows * (double)N * kb / pairs; }

// Tiles of `rows` x N for `pairs` CTA pairs: wide ones for as many whole waves as there are (or one fewer), the rest in the
// one width that finishes first; or that width throughout.  (Measured at d_model 2048, d_ff 5504: down projection of 1111
// tokens, 40 tiles of 256 columns for 74 pairs, 36.8 us; 55 of 192.)
// drain: one of the two above.  Of a tile with two accumulators the part of it that the skew does not cover is lost; with
// one, the other is worked in meanwhile.
// any_first: the first tiles may have any width, not 512 alone (few columns: one tile as wide as they are spans them).
inline TilePlan search_tiles(int rows, int N, int kb, int pairs, bool by_columns, int drain, bool any_first) {
    constexpr int kWidths = WIDE_N / WIDE_STEP;
    const int n_up = (N + WIDE_STEP - 1) / WIDE_STEP * WIDE_STEP;
    double cycles_of[kWidths + 1];  // of a tile, by its width in steps
    int across[kWidths + 1];        // tiles across all columns
    for (int i = 1; i <= kWidths; ++i) {
        const int w = std::min(i * WIDE_STEP, n_up);
        const double mma = kb * wide_block_cycles(w) + 350.0;
        cycles_of[i] = w > WIDE_N / 2 ? mma + std::max(0, drain - WIDE_SKEW * 512) : std::max(mma, drain * w / 256.0);
        across[i] = (N + i * WIDE_STEP - 1) / (i * WIDE_STEP);
    }
    TilePlan best{};
    const auto consider = [&](int i1, int split, int i2) {
        const int w1 = i1 * WIDE_STEP, w2 = i2 * WIDE_STEP;
        const double c1 = cycles_of[i1], c2 = cycles_of[i2];
        const int nt2 = !by_columns || split == 0 ? across[i2] : split < N ? (N - split + w2 - 1) / w2 : 0;
        const int t1 = by_columns ? split / w1 * rows : split * across[i1];
        const int total = t1 + (by_columns ? nt2 * rows : (rows - split) * nt2);
        // (the slowest pair has at least the average: nothing that could win is dropped here, whatever the roundings)
        if (best.total && t1 * c1 + (total - t1) * c2 > best.cycles * pairs * (1 + 1e-9)) return;
        // Tiles go round the pairs in turn: pair j has every pairs-th one from j on.  Both counts fall by one at most once as
        // j grows, at their remainders, so the slowest pair is the first one, or the first behind either step.
        double cycles = 0.0;
        for (const int j : {0, t1 % pairs, total % pairs}) {
            const int n1 = t1 > j ? (t1 - 1 - j) / pairs + 1 : 0, n = total > j ? (total - 1 - j) / pairs + 1 : 0;
            cycles = std::max(cycles, n1 * c1 + (n - n1) * c2);
        }
        if (best.total == 0 || cycles < best.cycles) best = TilePlan{rows, by_columns ? 1 : 0, split, w1, across[i1], w2, nt2, t1, total, cycles};
    };
    const int most = any_first ? std::min(kWidths, n_up / WIDE_STEP) : kWidths;
    for (int i1 = most; i1 >= (any_first ? 1 : kWidths); --i1) {
        const int w1 = i1 * WIDE_STEP;
        const int units = by_columns ? N / w1 : rows;          // what is split off as wide: columns' tiles or rows
        const int per_unit = by_columns ? rows : across[i1];   // tiles of one
        const int waves = (int)((int64_t)units * per_unit / pairs);
        int splits[4], n = 0;
        for (int f = waves; f >= std::max(1, waves - 1); --f) {
            const int u = (int)std::min<int64_t>(units, (int64_t)f * pairs / per_unit);
            for (int v = u; v >= std::max(1, u - 1); --v) splits[n++] = by_columns ? v * w1 : v;
        }
        for (int i2 = most; i2 >= 1; --i2) {
            if (i1 == most) consider(i1, 0, i2);
            for (int i = 0; i < n; ++i) consider(i1, splits[i], i2);
        }
    }
    return best;
}

// The same, remembered by problem size.  The memory is bounded and allocates nothing: a new size takes the place of the
// oldest of the four that share its set.
inline TilePlan plan_tiles(int rows, int N, int kb, int pairs, bool by_columns, int drain, bool any_first = false) {
    struct Entry {
        int key[6];
        uint32_t age;  // 0: empty
        TilePlan plan;
    };
    constexpr int kSets = 256, kWays = 4;
    static std::mutex mu;
    static Entry known[kSets][kWays];
    static uint32_t clock = 0;
    const int key[6] = {rows, N, kb, pairs, (by_columns ? 1 : 0) + (any_first ? 2 : 0), drain};
    uint64_t h = 0x9e3779b97f4a7c15ull;
    for (const int v : key) h = (h ^ (uint64_t)(uint32_t)v) * 0xff51afd7ed558ccdull;
    Entry *const set = known[h >> 56];
    {
        std::lock_guard<std::mutex> lock(mu);
        for (int i = 0; i < kWays; ++i)
            if (set[i].age && std::equal(key, key + 6, set[i].key)) return set[i].plan;
    }
    const TilePlan plan = search_tiles(rows, N, kb, pairs, by_columns, drain, any_first);
    std::lock_guard<std::mutex> lock(mu);
    Entry *oldest = set;
    for (int i = 1; i < kWays; ++i)
        if (set[i].age < oldest->age) oldest = set + i;
    std::copy(key, key + 6, oldest->key);
    clock += clock == UINT32_MAX ? 0u : 1u;
    oldest->age = clock;
    oldest->plan = plan;
    return plan;
}

}  // namespace tc
}  // namespace moc
