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

// SM cycles of one contraction block in a tile of w columns, operands in L2.  Measured (74 tiles at a time, the difference of
// contractions of 8, 16 and 32 blocks, sm__cycles_elapsed) when lane 0 issued the MMAs, 480 cycles for a block's four and its commit: 64 to
// 256 columns, one accumulator, 540 to 570, whatever they are; 320 columns 770 to 820 and 384 780 to 800 (MMAs of 64 columns take
// what those of 128 do), 448 985, 512 1100.  The constants are older than the kernel: issued by an elected thread a block of 64 or 128
// columns takes 350, 256 610.  They stay because a fit to those (335 up to 128 columns, 560 at 256, 70 bytes a cycle) made 1111
// tokens of 2048 x 5461 246 -> 240 us, but 33736 of 1696 x 6784 6104 -> 6368 and 615 of 2184 x 5824 195 -> 206.
constexpr double WIDE_MMA_CYCLES = 2.06;  // per column
inline double wide_block_cycles(int w) { return w <= WIDE_N / 2 ? 528.0 + w / 8.0 : WIDE_MMA_CYCLES * std::max(w, 3 * WIDE_N / 4); }

// What a tile's outputs cost: cycles that a tile of two accumulators loses (measured with 32 blocks); cycles that the epilogue
// takes for 256 columns, which a tile of one accumulator cannot be shorter than; bytes of an element, whose stores share
// the SM's way to L2 with the loads (with both at 58 bytes a cycle 256 columns of gate + up over 12 blocks take 8.8 thousand cycles,
// 8.9 measured, and not the 6.7 of their MMAs).  us, by 2.06 cycles a column, the loads and larger losses instead | by this: steps
// of 8126 tokens, 2720 x 7232, 2714 | 2524 (tiles of 320 columns throughout before), 9154, 4784 x 12736, 8611 | 8128, 777, 2048 x 5504,
// 194 | 186; forwards of 400 tokens, 4096 x 11008, 127 | 118, 2506, 4416 x 11776, 736 | 688; other sizes within 2 %.
struct WideOutputs {
    int lost, epilogue, bytes;
};
constexpr WideOutputs WIDE_OUT_BF16 = {250, 2000, 2}, WIDE_OUT_GATE_UP = {2700, 3500, 3}, WIDE_OUT_F32 = {2700, 3500, 4};
constexpr double WIDE_L2_BYTES = 58.0;  // a cycle, per SM
inline double wide_tile_cycles(int w, int kb, const WideOutputs &out) {
    const double l2 = (kb * (16384.0 + 64.0 * w) + 128.0 * out.bytes * w) / WIDE_L2_BYTES;
    const double cycles = std::max(kb * wide_block_cycles(w), l2) + 350.0;
    return w > WIDE_N / 2 ? cycles + out.lost : std::max(cycles, out.epilogue * w / 256.0);
}

// No plan of `rows` x N over kb blocks is shorter: its MMAs spread evenly.
inline double plan_cycles_at_least(int rows, int64_t N, int kb, int pairs) { return WIDE_MMA_CYCLES * rows * (double)N * kb / pairs; }

// Tiles of `rows` x N for `pairs` CTA pairs: wide ones for as many whole waves as there are (or one fewer), the rest in the
// one width that finishes first; or that width throughout.  (Measured at d_model 2048, d_ff 5504: down projection of 1111
// tokens, 40 tiles of 256 columns for 74 pairs, 36.8 us; 55 of 192.)
// any_first: the first tiles may have any width, not 512 alone (few columns: one tile as wide as they are spans them).
inline TilePlan search_tiles(int rows, int N, int kb, int pairs, bool by_columns, const WideOutputs &out, bool any_first) {
    constexpr int kWidths = WIDE_N / WIDE_STEP;
    const int n_up = (N + WIDE_STEP - 1) / WIDE_STEP * WIDE_STEP;
    double cycles_of[kWidths + 1];  // of a tile, by its width in steps
    int across[kWidths + 1];        // tiles across all columns
    for (int i = 1; i <= kWidths; ++i) {
        const int w = std::min(i * WIDE_STEP, n_up);
        cycles_of[i] = wide_tile_cycles(w, kb, out);
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
inline TilePlan plan_tiles(int rows, int N, int kb, int pairs, bool by_columns, const WideOutputs &out, bool any_first = false) {
    struct Entry {
        int key[6];
        uint32_t age;  // 0: empty
        TilePlan plan;
    };
    constexpr int kSets = 256, kWays = 4;
    static std::mutex mu;
    static Entry known[kSets][kWays];
    static uint32_t clock = 0;
    const int key[6] = {rows, N, kb, pairs, (by_columns ? 1 : 0) + (any_first ? 2 : 0), out.lost * 8 + out.bytes};
    uint64_t h = 0x9e3779b97f4a7c15ull;
    for (const int v : key) h = (h ^ (uint64_t)(uint32_t)v) * 0xff51afd7ed558ccdull;
    Entry *const set = known[h >> 56];
    {
        std::lock_guard<std::mutex> lock(mu);
        for (int i = 0; i < kWays; ++i)
            if (set[i].age && std::equal(key, key + 6, set[i].key)) return set[i].plan;
    }
    const TilePlan plan = search_tiles(rows, N, kb, pairs, by_columns, out, any_first);
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
