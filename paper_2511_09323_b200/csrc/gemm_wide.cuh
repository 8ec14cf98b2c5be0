// The dense bf16 GEMM of the tensor-core plan: CTA pairs on tiles of 256 rows and up to 512 columns.
//
// What bounds it: a pair's MMA (cta_group::2, M = 256) works 2 cycles per column and 64-element contraction block; the two
// CTAs' operands have to arrive from L2 meanwhile.  On 256 x 256 tiles those are 32 KiB per CTA and block of 512 cycles,
// 64 bytes a cycle, and the SMs together get some 58 (measured with the MMAs left out: 550 to 615 cycles a block; the kernel
// of such tiles that this one replaced needed 700, 65536 x 2048 x 11008 in 2.13 ms; now 1.90).  Twice the columns per tile share the rows' half of that: 48 KiB per 1024 cycles.  The tile then fills
// tensor memory (two accumulators of 256 columns), so nothing is left to work in while the epilogue drains it; instead the
// two accumulators run a few blocks apart: the first is ahead at both ends of the contraction, so that its epilogue overlaps
// the second's last blocks and its next tile starts while the second is being drained.
//
// The tiles need not have one width.  With few tiles, or a last wave that few of them fill, the remaining rows (or columns)
// are cut into narrower ones, in steps of 64 columns, so that all pairs finish together: plan_tiles() (tile_plan.h) chooses.
//
// Roles: warp 0 TMA loads, warp 1 MMAs (leading CTA) and the TMEM allocation, warps 2..9 epilogue, two per TMEM lane quarter.
// Barriers as in the pair kernel of tc_gemm.cuh.
#pragma once

#include "tc_gemm.cuh"
#include "tile_plan.h"

namespace moc {
namespace tc {

constexpr int WIDE_THREADS = 320, WIDE_EPI_WARPS = 8, WIDE_STAGES_MAX = 6;
constexpr uint32_t WIDE_B_BYTES = (BN / 2) * BK * 2;  // one accumulator's half of B in a stage, at most
constexpr uint32_t WIDE_RING_BYTES = 192 * 1024;      // 4 stages of A | B | B, or 6 of A | B where no tile is wider than 256
constexpr size_t WIDE_SMEM_BYTES = 1024 + WIDE_RING_BYTES + BAR_REGION_BYTES + WIDE_EPI_WARPS * EPI_BOX_BYTES;

struct WideParams {
    Params g;
    CUtensorMap b_rem[3];  // K-major B: boxes for the accumulator of fewer than 256 columns of the narrower tiles
    CUtensorMap b_rem1[2]; // TRANSPOSED: the same for the first tiles
    TilePlan t;
    int m_blocks;          // 256-row blocks of one problem
    int stages;
    uint32_t stage_bytes;
    uint32_t f32_outputs;  // bit i: problem i's output is fp32, not bf16
    // TRANSPOSED: the problems are `k_split` parts of one contraction, of its `k_operands` pairs of operands in turn (k_blocks
    // blocks each; blocks past an operand's end are zeros), their fp32 outputs c_step elements apart
    int k_split, k_operands;
    int64_t c_step;
};

// one tile
struct WideTile {
    int m_blk, prob, n0;
    int s0, s1;           // columns of the two accumulators (multiples of 64; s1 may be 0)
    uint32_t box0, box1;  // K-major B: rows of the boxes loaded for them (the box of a clipped tile keeps its height)
};
__device__ __forceinline__ WideTile wide_tile(const WideParams &p, int tile) {
    WideTile t;
    int row, w;
    const bool first = tile < p.t.t1;
    const int i = first ? tile : tile - p.t.t1;
    w = first ? p.t.w1 : p.t.w2;
    if (p.t.by_columns) {
        const int c = i / p.t.rows;
        row = i - c * p.t.rows;
        t.n0 = (first ? 0 : p.t.split) + c * w;
    } else {
        const int nt = first ? p.t.nt1 : p.t.nt2, r = i / nt;
        row = r + (first ? 0 : p.t.split);
        t.n0 = (i - r * nt) * w;
    }
    if (p.g.problem_major) {
        t.prob = row / p.m_blocks;
        t.m_blk = row - t.prob * p.m_blocks;
    } else {
        t.m_blk = row / p.g.num_problems;
        t.prob = row - t.m_blk * p.g.num_problems;
    }
    const int valid = min(w, (p.g.N - t.n0 + WIDE_STEP - 1) / WIDE_STEP * WIDE_STEP);
    t.s0 = min(valid, BN);
    t.s1 = valid - t.s0;
    const int full0 = min(w, BN);
    t.box0 = (uint32_t)full0 / 2;
    t.box1 = (uint32_t)(w - full0) / 2;
    return t;
}

// The epilogues read an accumulator into registers and hand it back to the MMAs (release) before they store it: what the
// stores take is then hidden behind the next tile's MMAs.  (Released after its last store, by an arrival that also waited for
// the stores to arrive, an accumulator was held for 4000 cycles (bf16) to 7000 (fp32) and the MMAs stood still for a
// quarter of gate + up and a fifth of dZ; held for 570 and 2600, 65536 x 2048 x 5504, thousands of SM cycles: gate + up 2 x
// 1602 -> 2 x 1422, dZ 1508 -> 1320, down 1314 -> 1250, grad_x 2531 -> 2469; 16384 x 768 x 2048, dZ 67.3 -> 56.1.)

// An output that is stored column by column (TRANSPOSED): the lanes are consecutive elements of a stored row, so
// a column leaves as one contiguous store of the warp.
template <int EPI, class Release>
__device__ __forceinline__ void transposed_epilogue(const WideParams &w, int prob, int row0, int n0, int cols, int half, uint32_t taddr,
                                                    Release release) {
    const Params &p = w.g;
    const int lane = threadIdx.x & 31, row = row0 + lane;
    const bool f32_out = EPI == EPI_F32 || (EPI == EPI_GATE_UP && prob == 0);
    const int out = w.k_split > 1 ? 0 : prob;
    const int64_t ld = p.ldc[out], at = (int64_t)n0 * ld + row + (w.k_split > 1 ? prob * w.c_step : 0);
    cols = min(cols, p.N - n0);
    if (row0 >= p.M) cols = 0;
    uint32_t r[4][32];
    const auto column = [&](int i) { return 32 * half + 64 * i; };
#pragma unroll
    for (int i = 0; i < 4; ++i) tmem_ld32(taddr + (uint32_t)column(i), r[i]);  // (all 256 columns exist, whatever the tile's width)
    tmem_ld_wait();
    release();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c0 = column(j);
        if (c0 >= cols) break;
        const int valid = row < p.M ? min(32, cols - c0) : 0;
        if (f32_out) {
            float *dst = static_cast<float *>(p.c[out]) + at + c0 * ld;
#pragma unroll
            for (int i = 0; i < 32; ++i, dst += ld)
                if (i < valid) *dst = __uint_as_float(r[j][i]);
        } else {
            __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(p.c[out]) + at + c0 * ld;
#pragma unroll
            for (int i = 0; i < 32; ++i, dst += ld)
                if (i < valid) *dst = __float2bfloat16_rn(__uint_as_float(r[j][i]));
        }
    }
}

// Every thread stores its own row (outputs without 16-byte rows, accumulation).
template <int EPI, class Release>
__device__ __forceinline__ void direct_epilogue(const Params &p, int prob, int row0, int n0, int cols, int half, uint32_t taddr,
                                                Release release) {
    const int row = row0 + (int)(threadIdx.x & 31);
    const bool f32_out = EPI == EPI_F32 || (EPI == EPI_GATE_UP && prob == 0);
    cols = row0 < p.M ? min(cols, p.N - n0) : 0;
#pragma unroll 1
    for (int c0 = 32 * half; c0 < cols; c0 += 64) {
        uint32_t r[32];
        __syncwarp();
        tmem_ld32(taddr + (uint32_t)c0, r);
        tmem_ld_wait();
        const int valid = cols - c0;
        if (row >= p.M) continue;
        if (f32_out) {
            store_row_f32(static_cast<float *>(p.c[prob]) + (int64_t)row * p.ldc[prob] + n0 + c0, r, valid);
        } else {
            __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(p.c[prob]) + (int64_t)row * p.ldc[prob] + n0 + c0;
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
            if (EPI == EPI_BF16 && p.accumulate) {
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (i < valid) v[i] += __bfloat162float(dst[i]);
            }
            store_row_bf16(dst, v, valid);
        }
    }
    release();
}

// Where a warp's 32 rows of the output go.  A chunk of 32 rows x 128 bytes passes through the warp's box in shared memory (16-byte
// pieces XOR-swizzled, free of bank conflicts both ways) and leaves as stores of whole 128-byte lines, eight lanes to a row.
// (Bulk tensor stores queue behind the loads in flight: some 3000 cycles until such a store has read its box.  Every thread
// storing 32-byte sectors of its own row, without the box: gate + up at 65536 x 2048 x 11008 1.24 -> 1.37 ms a chunk.)
struct RowChunks {
    uint8_t *out;     // first of this lane's pieces
    int64_t pitch4;   // bytes from a row to the fourth after it
    int rows_left;    // rows from this lane's first on
    bool whole;       // all 32 rows exist
    uint32_t box;

    __device__ __forceinline__ void store(int byte, int bytes, const uint32_t (&w)[32]) const {  // `bytes` of each row exist from `byte` on
        const uint32_t lane = threadIdx.x & 31, r_sub = lane >> 3, piece = lane & 7;
        uint8_t *dst = out + byte;
        const uint32_t my_row = box + lane * 128u;
#pragma unroll
        for (int i = 0; i < 8; ++i) st_shared_v4(my_row + (((uint32_t)i ^ piece) << 4), w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
        __syncwarp();
        const auto staged = [&](int i) {
            const uint32_t rr = (uint32_t)(4 * i) + r_sub;
            return ld_shared_v4(box + rr * 128u + ((piece ^ (rr & 7u)) << 4));
        };
        if (whole && bytes >= 128) {
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                uint4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = staged(h + i);
#pragma unroll
                for (int i = 0; i < 4; ++i, dst += pitch4) *reinterpret_cast<uint4 *>(dst) = v[i];
            }
        } else {
            const int left = bytes - 16 * (int)piece;  // from this lane's piece on
#pragma unroll 1
            for (int i = 0; i < 8; ++i, dst += pitch4) {
                const uint4 v = staged(i);
                if (4 * i >= rows_left) continue;
                if (left >= 16) {
                    *reinterpret_cast<uint4 *>(dst) = v;
                } else {
                    const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (2 * e < left) reinterpret_cast<uint16_t *>(dst)[e] = (uint16_t)(x[e >> 1] >> (16 * (e & 1)));
                }
            }
        }
        __syncwarp();
    }
};

// A tile's one or two accumulators, as the epilogue sees them: address in tensor memory, barriers that say "complete" and (in the
// leading CTA) "read".
struct TileAccumulators {
    uint32_t taddr, full, empty;  // of the accumulators in the order of tensor memory
    uint32_t used;                // accumulators handed out before this tile: they alternate
    int cols0, cols1;             // that exist in the output; 0: none
    bool two;
    volatile int *abort_flag;
    int *status;

    __device__ __forceinline__ uint32_t slot(int j) const { return (used + (uint32_t)j) & 1u; }
    __device__ __forceinline__ uint32_t at(int j) const { return taddr + slot(j) * BN; }
    __device__ __forceinline__ int cols(int j) const { return j ? cols1 : cols0; }
    __device__ __forceinline__ bool wait(int j) const {
        const bool ok = __all_sync(0xffffffffu, mbar_wait(full + 8u * slot(j), ((used + (uint32_t)j) >> 1) & 1u, abort_flag, status));
        tc_fence_after();
        return ok;
    }
    __device__ __forceinline__ void release(int j) const {  // (nothing but the reads of tensor memory is ordered by this arrival)
        tc_fence_before();
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive_cluster_relaxed(empty + 8u * slot(j));
    }
};

// A warp's share of a tile: every other 128-byte chunk (`half` says which) of its 32 rows, in registers as it will be stored: 32 fp32
// columns a chunk, or 64 rounded to bf16.  Three chunks are held at a time, so that an accumulator is read ahead of the
// stores as far as the registers go.  (All four of an fp32 accumulator: the registers spill, into an L1 that shared memory has
// left no room: gate + up 1620 thousand cycles again.)  The second accumulator of a tile is complete a thousand cycles after the first.
// Between a tcgen05.ld and its wait the destination registers may not be touched.  So no load stands in a branch that joins
// before its wait, where a compiler could copy them: chunks that the tile or the output does not have are loaded all the same
// (an accumulator's 256 columns always exist), and the two element types and one and two accumulators part for good.
__device__ __forceinline__ bool wide_epilogue(const TileAccumulators &acc, const RowChunks &rows, bool f32, int half) {
    uint32_t v0[32], v1[32], v2[32];
    const int width = f32 ? 32 : 64, shift = f32 ? 2 : 1;  // columns of a chunk; bytes of an element, as a power of two
    const auto column = [&](int i) { return width * (half + 2 * i); };
    const auto load = [&](int j, int i, uint32_t (&h)[32]) __attribute__((always_inline)) {  // (fp32; complete after a wait)
        tmem_ld32(acc.at(j) + (uint32_t)(32 * (half + 2 * i)), h);
    };
    const auto round = [&](int j, int i, uint32_t (&h)[32]) __attribute__((always_inline)) {  // (bf16; complete)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t r[2][16];
            tmem_ld16(acc.at(j) + (uint32_t)(64 * (half + 2 * i) + 32 * c), r[0]);
            tmem_ld16(acc.at(j) + (uint32_t)(64 * (half + 2 * i) + 32 * c + 16), r[1]);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 16; ++q)
                h[16 * c + q] = pack_bf16(__uint_as_float(r[q >> 3][2 * (q & 7)]), __uint_as_float(r[q >> 3][2 * (q & 7) + 1]));
        }
    };
    const auto store = [&](int j, int i, const uint32_t (&h)[32]) __attribute__((always_inline)) {
        if (column(i) < acc.cols(j)) rows.store((j * BN + column(i)) << shift, (acc.cols(j) - column(i)) << shift, h);
    };
    if (!acc.wait(0)) return false;
    if (f32) {
        load(0, 0, v0);
        load(0, 1, v1);
        load(0, 2, v2);
        tmem_ld_wait();
        store(0, 0, v0);
        load(0, 3, v0);
        tmem_ld_wait();
        acc.release(0);
        store(0, 1, v1);
        if (!acc.two) {
            store(0, 2, v2);
            store(0, 3, v0);
            return true;
        }
        if (!acc.wait(1)) return false;
        load(1, 0, v1);
        store(0, 2, v2);
        load(1, 1, v2);
        store(0, 3, v0);
        load(1, 2, v0);
        tmem_ld_wait();
        store(1, 0, v1);
        load(1, 3, v1);
        tmem_ld_wait();
        acc.release(1);
        store(1, 2, v0);
        store(1, 3, v1);
        store(1, 1, v2);
    } else {
        round(0, 0, v0);
        round(0, 1, v1);
        acc.release(0);
        store(0, 0, v0);
        if (!acc.two) {
            store(0, 1, v1);
            return true;
        }
        if (!acc.wait(1)) return false;
        round(1, 0, v2);
        round(1, 1, v0);
        acc.release(1);
        store(0, 1, v1);
        store(1, 0, v2);
        store(1, 1, v0);
    }
    return true;
}

// TRANSPOSED: the caller has exchanged the operands (see swapped_gemm_pays) and every output is stored as its transpose
template <bool A_MN, bool B_MN, int EPI, bool TRANSPOSED = false>
__global__ void __launch_bounds__(WIDE_THREADS, 1) gemm_wide_kernel(const __grid_constant__ WideParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // 128-byte swizzle atoms need 1024-byte alignment
    uint8_t *smem = smem_raw + (base - raw);
    const uint32_t bar_base = base + WIDE_RING_BYTES;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (WIDE_STAGES_MAX + s); };
    auto tfull_bar = [&](uint32_t a) { return bar_base + 8u * (2 * WIDE_STAGES_MAX + a); };
    auto tempty_bar = [&](uint32_t a) { return bar_base + 8u * (2 * WIDE_STAGES_MAX + ACC_STAGES + a); };
    volatile uint32_t *tmem_holder =
        reinterpret_cast<volatile uint32_t *>(smem + WIDE_RING_BYTES + 8 * (2 * WIDE_STAGES_MAX + 2 * ACC_STAGES));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();  // 0: the pair's leading CTA
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    const int kb_total = p.g.k_blocks * p.g.k_segments;
    int *const status = p.g.status;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (uint32_t a = 0; a < ACC_STAGES; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), 2 * WIDE_EPI_WARPS);  // one arrival per epilogue warp of the pair
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc_pair(smem_u32(const_cast<uint32_t *>(tmem_holder)), TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // the partner's barriers exist before anything signals them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();  // (for the kernel in front)

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (one per CTA).  One thread's
        // instructions per block have to stay well below a block's MMAs: everything that a tile fixes is worked out ahead.
        if (elect_one()) {
            for (int i = 0; i < 3; ++i) {
                prefetch_tmap(&p.g.a_map[i]);
                prefetch_tmap(&p.g.b_map[i]);
            }
            const uint32_t lead_bars = map_to_cta(bar_base, 0), ring_end = base + (uint32_t)p.stages * p.stage_bytes;
            uint32_t sa = base, bar = 0, phase = 0;  // stage: its A operand, its barriers' offset
            bool ok = true;
            for (int tile = pair; tile < p.t.total && ok; tile += num_pairs) {
                const WideTile t = wide_tile(p, tile);
                const int m0 = t.m_blk * (2 * BM) + (int)rank * BM;  // this CTA's rows of A
                const int h0 = t.s0 / 2, h1 = t.s1 / 2;              // its share of the accumulators' columns of B
                const int nb0 = t.n0 + (int)rank * h0, nb1 = t.n0 + BN + (int)rank * h1;
                const bool two0 = h0 > 64, any1 = h1 > 0, two1 = h1 > 64;  // MN-major B: boxes of 64 columns
                const uint32_t b_bytes = B_MN ? (uint32_t)(1 + (two0 ? 1 : 0) + (any1 ? 1 : 0) + (two1 ? 1 : 0)) * 8192u
                                              : (t.box0 + (any1 ? t.box1 : 0u)) * (uint32_t)(BK * 2);
                const uint32_t tx = 2 * (A_STAGE_BYTES + b_bytes);
                for (int seg = 0; seg < p.g.k_segments && ok; ++seg) {
                    const bool part = TRANSPOSED && p.k_split > 1;
                    const int pair_of = part ? t.prob % p.k_operands : 0;
                    const CUtensorMap *am = &p.g.a_map[part ? pair_of : p.g.a_idx[t.prob][seg]];
                    const int bi = part ? pair_of : p.g.b_idx[t.prob][seg];
                    const CUtensorMap *rem = TRANSPOSED && tile < p.t.t1 ? &p.b_rem1[bi] : &p.b_rem[bi];
                    const CUtensorMap *bm0 = !B_MN && t.box0 < BN / 2 ? rem : &p.g.b_map[bi];
                    const CUtensorMap *bm1 = !B_MN && t.box1 < BN / 2 ? rem : &p.g.b_map[bi];
                    const int k_begin = part ? t.prob / p.k_operands * p.g.k_blocks * BK : 0, k_end = k_begin + p.g.k_blocks * BK;
                    for (int kk = k_begin; kk < k_end; kk += BK) {
                        if (!mbar_wait(bar_base + bar + 8u * WIDE_STAGES_MAX, phase ^ 1u, abort_flag, status)) {
                            ok = false;
                            break;
                        }
                        const uint32_t full = lead_bars + bar, sb = sa + A_STAGE_BYTES;
                        if (rank == 0) mbar_expect_tx(bar_base + bar, tx);
                        if (A_MN) {
                            tma_load_2d_pair(sa, am, full, m0, kk);
                            tma_load_2d_pair(sa + 64 * BK * 2, am, full, m0 + 64, kk);
                        } else {
                            tma_load_2d_pair(sa, am, full, kk, m0);
                        }
                        if (B_MN) {
                            tma_load_2d_pair(sb, bm0, full, nb0, kk);
                            if (two0) tma_load_2d_pair(sb + 64 * BK * 2, bm0, full, nb0 + 64, kk);
                            if (any1) tma_load_2d_pair(sb + WIDE_B_BYTES, bm1, full, nb1, kk);
                            if (two1) tma_load_2d_pair(sb + WIDE_B_BYTES + 64 * BK * 2, bm1, full, nb1 + 64, kk);
                        } else {
                            tma_load_2d_pair(sb, bm0, full, kk, nb0);
                            if (any1) tma_load_2d_pair(sb + WIDE_B_BYTES, bm1, full, kk, nb1);
                        }
                        bar += 8u;
                        sa += p.stage_bytes;
                        if (sa == ring_end) {
                            sa = base;
                            bar = 0;
                            phase ^= 1u;
                        }
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leading CTA only)
        if (rank == 0 && elect_one()) {
            // one instruction consumes 16 contraction elements: 32 bytes along a K-major row, or 16 rows of 128 bytes in
            // an MN-major box (descriptor addresses are in units of 16 bytes)
            constexpr uint32_t a_step = A_MN ? 128u : 2u, b_step = B_MN ? 128u : 2u;
            constexpr uint32_t idesc0 = make_idesc<A_MN, B_MN, 2 * BM>() & ~(0x3fu << 17);
            const uint64_t a_desc = make_smem_desc(base, A_MN ? BK * 128 : 16, 1024);
            const uint64_t b_desc = make_smem_desc(base + A_STAGE_BYTES, B_MN ? BK * 128 : 16, 1024);
            const uint32_t hi = (uint32_t)(a_desc >> 32), a_lo = (uint32_t)a_desc, b_lo = (uint32_t)b_desc;
            // a stage: its barriers' offset, its operands' offset in the descriptors' units, the barriers' phase
            struct Cursor {
                uint32_t bar, off, phase;
            } at = {0, 0, 0};
            const uint32_t off_step = p.stage_bytes >> 4, off_end = (uint32_t)p.stages * off_step;
            auto next = [&](Cursor &c) {
                c.bar += 8u;
                c.off += off_step;
                if (c.off == off_end) {
                    c.bar = c.off = 0;
                    c.phase ^= 1u;
                }
            };
            auto arrived = [&](const Cursor &c) {
                if (!mbar_wait(bar_base + c.bar, c.phase, abort_flag, status)) return false;
                tc_fence_after();
                return true;
            };
            auto release = [&](const Cursor &c) { umma_commit_pair(bar_base + c.bar + 8u * WIDE_STAGES_MAX); };  // in both CTAs
            auto mma = [&](const Cursor &c, uint32_t j, uint32_t d, uint32_t idesc, bool first) {
                const uint32_t a = a_lo + c.off, b = b_lo + c.off + j * (WIDE_B_BYTES >> 4);
                umma_bf16_pair_lohi(d, a, b, hi, idesc, first ? 0u : 1u);
#pragma unroll
                for (uint32_t k = 1; k < BK / 16; ++k) umma_bf16_pair_lohi(d, a + k * a_step, b + k * b_step, hi, idesc, 1u);
            };
            uint32_t used = 0;  // accumulators handed out so far: they alternate
            bool ok = true;
            for (int tile = pair; tile < p.t.total && ok; tile += num_pairs) {
                const WideTile t = wide_tile(p, tile);
                const uint32_t r0 = used & 1u, r1 = r0 ^ 1u;
                const uint32_t id0 = idesc0 | ((uint32_t)(t.s0 >> 3) << 17), id1 = idesc0 | ((uint32_t)(t.s1 >> 3) << 17);
                const uint32_t d0 = tmem_base + r0 * BN, d1 = tmem_base + r1 * BN;
                if (!mbar_wait(tempty_bar(r0), ((used >> 1) & 1u) ^ 1u, abort_flag, status)) break;
                tc_fence_after();
                if (t.s1 == 0) {
                    for (int kb = 0; kb < kb_total && ok; ++kb) {
                        if (!(ok = arrived(at))) break;
                        mma(at, 0, d0, id0, kb == 0);
                        release(at);
                        next(at);
                    }
                    if (!ok) break;
                    umma_commit_pair(tfull_bar(r0));  // accumulator complete, in both CTAs
                    ++used;
                    continue;
                }
                const int skew = min(WIDE_SKEW, kb_total / 2);
                // `skew` blocks of one accumulator, then the same blocks of the other; the stages go back with the second
                auto first_pass = [&](bool begin) {
                    Cursor c = at;
                    for (int i = 0; i < skew && ok; ++i) {
                        if (!(ok = arrived(c))) break;
                        mma(c, 0, d0, id0, begin && i == 0);
                        next(c);
                    }
                };
                auto second_pass = [&](bool begin) {
                    for (int i = 0; i < skew; ++i) {
                        mma(at, 1, d1, id1, begin && i == 0);
                        release(at);
                        next(at);
                    }
                };
                first_pass(true);
                if (!ok || !(ok = mbar_wait(tempty_bar(r1), (((used + 1) >> 1) & 1u) ^ 1u, abort_flag, status))) break;
                tc_fence_after();
                if (skew > 0) second_pass(true);
                for (int kb = skew; kb < kb_total - skew; ++kb) {
                    if (!(ok = arrived(at))) break;
                    mma(at, 0, d0, id0, kb == 0);
                    mma(at, 1, d1, id1, kb == 0);
                    release(at);
                    next(at);
                }
                if (!ok) break;
                first_pass(false);
                if (!ok) break;
                umma_commit_pair(tfull_bar(r0));
                second_pass(false);
                umma_commit_pair(tfull_bar(r1));
                used += 2;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9 of each CTA)
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        uint32_t used = 0;
        bool ok = true;
        for (int tile = pair; tile < p.t.total && ok; tile += num_pairs) {
            const WideTile t = wide_tile(p, tile);
            const int row0 = t.m_blk * (2 * BM) + (int)rank * BM + quarter * 32;
            TileAccumulators acc;
            acc.taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
            acc.full = tfull_bar(0);
            acc.empty = map_to_cta(tempty_bar(0), 0);
            acc.used = used;
            acc.cols0 = row0 < p.g.M ? min(t.s0, p.g.N - t.n0) : 0;
            acc.cols1 = row0 < p.g.M ? min(t.s1, p.g.N - t.n0 - BN) : 0;
            acc.two = t.s1 > 0;
            acc.abort_flag = abort_flag;
            acc.status = status;
            used += acc.two ? 2u : 1u;
            if (TRANSPOSED || p.g.direct_store != 0 || (EPI == EPI_BF16 && p.g.accumulate)) {
#pragma unroll 1
                for (int j = 0; j < (acc.two ? 2 : 1); ++j) {
                    if (!(ok = acc.wait(j))) break;
                    const auto done = [&]() { acc.release(j); };
                    if constexpr (TRANSPOSED)
                        transposed_epilogue<EPI>(p, t.prob, row0, t.n0 + j * BN, j ? t.s1 : t.s0, half, acc.at(j), done);
                    else
                        direct_epilogue<EPI>(p.g, t.prob, row0, t.n0 + j * BN, j ? t.s1 : t.s0, half, acc.at(j), done);
                }
            } else {
                const bool f32_out = (p.f32_outputs >> t.prob) & 1u;  // (not from EPI: as a constant it leaves a register allocation that spills)
                const int esz = f32_out ? 4 : 2, r_sub = lane >> 3;
                const int64_t pitch = (int64_t)p.g.ldc[t.prob] * esz;
                RowChunks rows;
                rows.out = static_cast<uint8_t *>(p.g.c[t.prob]) + (row0 + r_sub) * pitch + t.n0 * esz + (lane & 7) * 16;
                rows.pitch4 = 4 * pitch;
                rows.rows_left = p.g.M - row0 - r_sub;
                rows.whole = row0 + 32 <= p.g.M;
                rows.box = bar_base + BAR_REGION_BYTES + (uint32_t)(warp - 2) * EPI_BOX_BYTES;
                ok = wide_epilogue(acc, rows, f32_out, half);
            }
        }
    }

    // ---------------------------------------------------------------------- teardown
    // The next kernel of the stream may be launched once every CTA has come here with one of its warps: a pair's second CTA at its
    // start, where the warp of the MMAs has nothing to do, the leading one when its loader has requested the last tile's operands.  The
    // next kernel then does its set-up beside the last MMAs and stores, and waits for this one to complete before it touches what
    // this one wrote, as the element-wise kernel and the sum of partial outputs do.  Those give no such sign themselves, and the leading
    // CTAs not at their start: what is launched early takes its place on the first SMs that are free.  us a call in a row over three
    // sets of operands, no sign | all CTAs at their start | this: forward of 307 tokens, 4096 x 11008, 117.6 | 120.6 | 110.2; step of 1111
    // tokens, 2048 x 5461, 265 | 253 | 247; of 16384, 768 x 2048, 524 | 515 | 510.  (The row selector is launched the ordinary way: waiting
    // like this took it 2 us of 72 at 16384 x 2048, its loads no longer being known constant, and 4 us of that step.)
    pdl_launch_dependents();
    __syncwarp();
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // neither CTA leaves while the partner may still read its shared memory or signal it
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

}  // namespace tc
}  // namespace moc
