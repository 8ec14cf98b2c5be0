// Decode for one or two tokens as ONE cooperative kernel (bf16, d_model <= 4096).
//
// The four-kernel decode plan reads the right bytes (Section 5: the gate matrix once, then only the selected rows of
// W_up and W_down) but spends two thirds of its time on the hand-overs between kernels.  Here every SM keeps a fixed
// share of the CHANNELS for the whole call, so that nothing but a few words per token has to cross between SMs:
//
//   phase 1   the CTA streams its channels' rows of W_gate and keeps their gate values g[t][j] in shared memory
//             (Eq. (Moc-1)); it adds them to a global histogram of the order-preserving keys, and to one of finer parts
//   select    grid barrier; every CTA scans the histogram for the bin that holds the K-th largest key, and that bin's
//             parts; where those leave it open, it appends its own keys of that bin (with their channels) to a
//             global list; grid barrier; every CTA ranks its own candidates against the list: a channel is kept
//             when fewer than K channels precede it in (value descending, channel ascending) order -- the mask
//             definition of Section 3.2 with the tie rule of the library, decided without any single SM ever seeing
//             the whole row
//   phase 3   the CTA streams the rows of W_up and W_down of ITS kept channels only, forms z = SiLU(g) u (Eq. (MoC-2))
//             and its partial output, adds it to a global fp32 accumulator; grid barrier; the CTAs round slices of
//             the accumulator to bf16.
//
// What bounds it (one token of 4096 x 11008, us from the first CTA's start, medians, stamps of a measuring build): the gate rows have passed at 16.7 (90 MB at
// 7.2 TB/s from 4 on), the histogram is complete at 19.2, the kept channels are known at 21.6, W_up's rows have passed at 24.8,
// W_down's at 26.2, those of the CTA with the most kept channels (15 against 9 on average) at 27.8, the last barrier at 29.9; 4.5 more
// until the next call's start.  us per call, a row to a warp, its products by one FMA each with x read from shared memory for every
// row, and both barriers of the selection in every call | now: 4096 x 11008, one token 38.2 | 34.4, block form 40.7 | 36.4, two
// tokens 50.0 | 38.9; 2048 x 5504, one 24.6 | 19.7, two 32.5 | 20.5.
//
// Grid barriers are cooperative-groups grid syncs (the launch is cooperative: all CTAs are resident, or the launch
// fails).  No CTA ever leaves before the last barrier: a bounded wait that runs out raises MOC_ERR_TIMEOUT, stops the
// CTA's streaming, and the CTA still walks through every barrier.
#pragma once

#include <cooperative_groups.h>

#include "grouped_select.cuh"
#include "moc_common.cuh"
#include "tc_gemm.cuh"

namespace moc {
namespace dc {

constexpr int kMaxTokens = 2;         // (four tokens in registers take four rows' sums over a warp at a time: 52 and 55 us at three and four,
                                      // 4096 x 11008, against the four-kernel plan's 57 and 59, but 35.5 against 33.9 at 2048 x 5504)
constexpr int kMaxD = 4096;          // a thread owns 8 output columns
constexpr int kConsumerWarps = 16;
constexpr int kThreads = (kConsumerWarps + 2) * 32;  // + one producer warp, and one in which a thread sees to the grid's barriers
constexpr int kMaxRows = 256;        // channels per CTA
// Bins of the order-preserving keys: 128 to an octave of 2^-5 <= g < 2^4, where a threshold usually lies, 4 to an octave of every
// other 2^-24 <= |g| < 2^14, one to an octave beyond.  The keys of the threshold's bin go through one counter and are ranked
// against one another: of 11008 gate values of deviation 1.3 some 480 share a bin of 4 to an octave and 20 one of 128
// (two tokens, K = F / 8: 2048 x 8192 40.4 -> 39.6, 4096 x 11008 54.2 -> 53.0 us).  With one bin to an octave from 2^-6 down
// gates of deviation 0.013 took 46.0 us against 40.1 at one token and 66.2 against 54 at two; with 4096 bins, of which none is
// wider than a quarter of an octave, one token takes 0.3 us more to clear and scan them.
constexpr int kBins = 2048;
__host__ __device__ constexpr uint32_t bins_below(uint32_t key, uint32_t from, uint32_t to, int shift) {
    return ((key < from ? from : key < to ? key : to) - from) >> shift;
}
__host__ __device__ constexpr uint32_t key_bin(uint32_t key) {
    return (key >> 23) + bins_below(key, 0x39800000u, 0x4c800000u, 21) +  // -2^14 < g <= -2^-24
           bins_below(key, 0xb3800000u, 0xc6800000u, 21) +                // 2^-24 <= g < 2^14
           bins_below(key, 0xbd000000u, 0xc1800000u, 16);                 // 2^-5 <= g < 2^4
}
static_assert(key_bin(0xffffffffu) < (uint32_t)kBins, "the bins cover every key");
// Counters of equal parts of each of the narrow bins, of 2^-5 <= g < 2^4: as many parts as the workspace has room for (256 at one
// token of 11008 channels, 128 at two), four bits each, eight to a word.  Where the part that holds the K-th largest key holds no more
// keys than are kept of it, it decides alone, and the exchange of the bin's keys, a barrier of the grid and 3 us in all, does not
// take place.  A counter that overflows lowers the sum of its bin's counters, which then differs from the bin's own.
constexpr uint32_t kFineFrom = 0xbd000000u, kFineTo = 0xc1800000u;  // keys
constexpr int kNarrowBins = (int)((kFineTo - kFineFrom) >> 16), kMostParts = 256;
// Which of the narrow bins (0: the lowest) a bin is.  The wider steps of key_bin fall on a narrow bin's edge and leave numbers out:
// one behind each 32 of them, another behind each 128.
__host__ __device__ constexpr uint32_t narrow_bin(uint32_t bin) {
    const uint32_t x = bin - key_bin(kFineFrom), y = x % 133u;
    return x / 133u * 128u + y - y / 33u;
}
__host__ __device__ constexpr bool narrow_bins_follow() {
    for (uint32_t i = 0; i < (uint32_t)kNarrowBins; ++i)
        if (narrow_bin(key_bin(kFineFrom + (i << 16))) != i || narrow_bin(key_bin(kFineFrom + (i << 16) + 0xffffu)) != i) return false;
    return true;
}
static_assert(narrow_bins_follow(), "narrow_bin undoes key_bin");
constexpr int kMaxStages = 32;
constexpr size_t kStaticReserve = 8 * 1024;  // of shared memory, for the kernel's static part
constexpr int kFirstStages = 2;  // requested before the shared arrays are cleared
struct Params {
    const __nv_bfloat16 *x, *wg, *wu, *wd;
    __nv_bfloat16 *out;
    int d, F, K, grouped;
    int unit;            // channels are dealt to the CTAs in units of this many (8 with the 2-of-8 mask, else 1)
    int stages, of_stage;  // ring stages of `of_stage` weight rows each
    int col_groups;        // parts of the columns that the consumer warps share out (a power of two)
    int rp;              // channels of a CTA, at most, rounded up to 8
    int parts, part_shift;  // of a narrow bin (a power of two, at least 8; or 0: none), and log2 of the keys in one
    // workspace
    uint32_t *hist;      // [T][kBins]
    uint32_t *fine;      // [T][kNarrowBins][parts / 8]
    uint32_t *cand_n;    // [T]
    uint2 *cand;         // [T][F]  (key, channel)
    float *acc;          // [T][d]
    int *status;
    // the block form (Section 2, "LLM structure"): x holds the residual stream h, the layer reads RMSNorm(h) with
    // weight rms_w and adds h to its output; rms_w == nullptr: the plain layer on x
    const __nv_bfloat16 *rms_w;
    float rms_eps;
    // test hook: when not null, [T][F] bytes that receive 1 for every channel a token keeps and 0 for the others
    uint8_t *kept_out;
};

__host__ __device__ inline uint32_t row_pitch(int d) { return ((uint32_t)d * 2u + 127u) & ~127u; }  // of a row in the ring
// ring | partial sums [col_groups][T][rp] | g [T][rp] | z [rp][T]
inline size_t smem_bytes(int T, int d, int rp, int col_groups, int of_stage, int stages) {
    return (size_t)stages * of_stage * row_pitch(d) + (size_t)(std::max(col_groups, 4) + 2) * T * rp * 4;
}

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float sum2(uint64_t v) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return lo + hi;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ void fma2(uint64_t &c, uint64_t a, uint64_t b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b)); }
// eight bf16 values as four pairs of fp32
__device__ __forceinline__ void unpack8(const uint4 &q, uint64_t (&v)[4]) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
}
// Sums over the warp of N values a lane (a power of two): lane l has that of value l * N / 32.
template <int N>
__device__ __forceinline__ float warp_sums(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int m = 16;
#pragma unroll
    for (int n = N / 2; n > 0; n /= 2, m /= 2) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float other = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + n], m);
            v[i] = (up ? v[i + n] : v[i]) + other;
        }
    }
    for (; m > 0; m /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], m);
    return v[0];
}

template <int T>  // tokens: 1 or 2
__global__ void __launch_bounds__(kThreads, 1) decode_coop_kernel(const __grid_constant__ Params p) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ uint64_t bars[2 * kMaxStages];
    __shared__ __align__(16) uint4 s_zero;
    __shared__ int s_abort;
    __shared__ uint32_t s_scan[kConsumerWarps];
    __shared__ uint32_t s_bin[T], s_above[T], s_count[T];
    __shared__ uint32_t s_least[T];         // the least key that is kept; 0: not settled by the parts of its bin
    __shared__ uint16_t s_list[kMaxRows];   // the CTA's kept channels (offsets in its range), kept by any token
    __shared__ __align__(4) uint8_t s_mask[kMaxRows];  // per channel of the range: which tokens keep it (bit t)
    __shared__ int s_nsel;
    // Thread 0 is the one that signals and awaits a barrier of the grid, some 2 us each, while the others go on to what does not depend
    // on it: its warp is the last one here and streams nothing.
    const int lane = threadIdx.x & 31, warp = threadIdx.x < 32 ? kThreads / 32 - 1 : (int)threadIdx.x / 32 - 1, tid = 32 * warp + lane;
    const bool producer = warp == kConsumerWarps, consumer = warp < kConsumerWarps;
    const int d = p.d, F = p.F, rp = p.rp;
    const uint32_t pitch = row_pitch(d), stage_bytes = (uint32_t)p.of_stage * pitch;
    uint8_t *const ring = dsm;
    float *const part = reinterpret_cast<float *>(ring + (size_t)p.stages * stage_bytes);  // [col_groups][T][rp]
    float *const sg = part + max(p.col_groups, 4) * T * rp, *const sz = sg + T * rp;
    const uint32_t row_bytes = (uint32_t)d * 2u;
    auto full_bar = [&](int s) { return tc::smem_u32(&bars[s]); };
    auto empty_bar = [&](int s) { return tc::smem_u32(&bars[kMaxStages + s]); };
    auto consumer_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kConsumerWarps * 32) : "memory"); };

    // the CTA's channels: units [u0, u1) of `unit` channels each
    const int units = (F + p.unit - 1) / p.unit;
    const int u0 = (int)(((int64_t)blockIdx.x * units) / gridDim.x);
    const int u1 = (int)(((int64_t)(blockIdx.x + 1) * units) / gridDim.x);
    const int c0 = u0 * p.unit, c1 = min(F, u1 * p.unit);
    const int rows = max(0, c1 - c0);  // <= kMaxRows (the host checks)

    if (tid == 0) {
        for (int s = 0; s < p.stages; ++s) {
            tc::mbar_init(full_bar(s), 1);
            tc::mbar_init(empty_bar(s), kConsumerWarps);
        }
        s_abort = 0;
        s_nsel = 0;
        s_zero = make_uint4(0, 0, 0, 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // ---- ring: the producer, an elected thread (tc::elect_one), issues a bulk copy per weight row; stages are consumed in the order
    //      issued, each by all consumer warps.
    int p_stage = 0, c_stage = 0;
    uint32_t p_phase = 0, c_phase = 0;
    auto slot = [&](int s) { return ring + (size_t)s * stage_bytes; };
    auto request = [&](const __nv_bfloat16 *w, const uint16_t *list, int from, int to) -> bool {  // rows [from, to) of a phase
#pragma unroll 1
        for (int i = from; i < to; i += p.of_stage) {
            if (!tc::mbar_wait(empty_bar(p_stage), p_phase ^ 1u, &s_abort, p.status)) return false;
            const int here = min(p.of_stage, to - i);
            const uint32_t bar = full_bar(p_stage);
            uint32_t dst = tc::smem_u32(slot(p_stage));
            tc::mbar_expect_tx(bar, row_bytes * (uint32_t)here);
#pragma unroll 1
            for (int j = i; j < i + here; ++j, dst += pitch) tc::bulk_copy_g2s(dst, w + (int64_t)(c0 + (list ? (int)list[j] : j)) * d, row_bytes, bar);
            if (++p_stage == p.stages) {
                p_stage = 0;
                p_phase ^= 1u;
            }
        }
        return true;
    };
    auto wait_stage = [&]() { return __all_sync(0xffffffffu, tc::mbar_wait(full_bar(c_stage), c_phase, &s_abort, p.status)); };
    auto leave_stage = [&]() {
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(empty_bar(c_stage));
        if (++c_stage == p.stages) {
            c_stage = 0;
            c_phase ^= 1u;
        }
    };
    // Products of a phase's rows with the tokens.  The warps share out the columns, in `col_groups` parts, and the rows of a stage: so
    // few columns to a warp that it can hold them of all tokens in registers, as fp32 (read anew for each phase).  Plain FMAs, two to
    // an instruction: with mma.sync, a token a row, a call at one token of 4096 x 11008 took 53 us with 8 weight rows to an
    // MMA and 70 with 4.
    constexpr int NV = 4 / T, BR = T;  // 8-column vectors of a lane; rows at a time
    const int group = warp & (p.col_groups - 1), row_part = consumer ? warp / p.col_groups : 0, row_parts = kConsumerWarps / p.col_groups;
    const int v0 = (d >> 3) * group / p.col_groups + lane, v1 = (d >> 3) * (group + 1) / p.col_groups;  // this lane's: v0, v0 + 32 ...
    float scale[T];  // RMSNorm's
#pragma unroll
    for (int t = 0; t < T; ++t) scale[t] = 1.f;
    auto consume_dots = [&](int n) {
        uint64_t x[NV][T][4];
#pragma unroll
        for (int j = 0; j < NV; ++j)
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const int v = v0 + 32 * j;
                uint4 q = make_uint4(0, 0, 0, 0);
                if (v < v1) {
                    q = reinterpret_cast<const uint4 *>(p.x + (int64_t)t * d)[v];
                    if (p.rms_w) {  // y = h / sqrt(mean(h^2) + eps) . weight, rounded to bf16 as the layer's input
                        float h8[8], w8[8];
                        const uint32_t hw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                        for (int e = 0; e < 8; ++e) h8[e] = __uint_as_float(e % 2 ? hw[e / 2] & 0xffff0000u : hw[e / 2] << 16);
                        Vec8<__nv_bfloat16>::load(p.rms_w + 8 * v, w8);
#pragma unroll
                        for (int e = 0; e < 8; ++e) h8[e] = h8[e] * scale[t] * w8[e];
                        q = make_uint4(tc::pack_bf16(h8[0], h8[1]), tc::pack_bf16(h8[2], h8[3]), tc::pack_bf16(h8[4], h8[5]), tc::pack_bf16(h8[6], h8[7]));
                    }
                }
                unpack8(q, x[j][t]);
            }
#pragma unroll 1
        for (int i = 0; i < n; i += p.of_stage) {
            if (!wait_stage()) break;
            const int here = min(p.of_stage, n - i);
#pragma unroll 1
            for (int b = row_part * BR; b < here; b += row_parts * BR) {
                uint64_t acc[BR][T];
#pragma unroll
                for (int r = 0; r < BR; ++r) {
                    const uint4 *row = reinterpret_cast<const uint4 *>(slot(c_stage) + (uint32_t)min(b + r, here - 1) * pitch);
#pragma unroll
                    for (int j = 0; j < NV; ++j) {
                        uint64_t w[4];
                        unpack8(*(v0 + 32 * j < v1 ? row + v0 + 32 * j : &s_zero), w);
#pragma unroll
                        for (int t = 0; t < T; ++t) {
                            if (j == 0) acc[r][t] = mul2(x[0][t][0], w[0]);
                            else fma2(acc[r][t], x[j][t][0], w[0]);
#pragma unroll
                            for (int e = 1; e < 4; ++e) fma2(acc[r][t], x[j][t][e], w[e]);
                        }
                    }
                }
                float sums[BR * T];
#pragma unroll
                for (int r = 0; r < BR; ++r)
#pragma unroll
                    for (int t = 0; t < T; ++t) sums[r * T + t] = sum2(acc[r][t]);
                const float sum = warp_sums<BR * T>(sums);
                const int at = lane * (BR * T) / 32, r = at / T, t = at - r * T;
                if (lane % (32 / (BR * T)) == 0 && b + r < here) part[(group * T + t) * rp + i + b + r] = sum;
            }
            leave_stage();
        }
    };
    auto dot = [&](int t, int i) {  // of the phase's i-th row with token t
        float sum = 0.f;
#pragma unroll 4
        for (int c = 0; c < p.col_groups; ++c) sum += part[(c * T + t) * rp + i];
        return sum;
    };

    // ---- start: the first gate rows leave at once (the ring is empty: nothing to wait for); the CTA clears its slices of the
    //      arrays that all CTAs share
    const int first = min(min(p.stages, kFirstStages) * p.of_stage, rows);  // (the producer joins the barrier below: it must not be late)
    tc::pdl_wait();  // (weights, too, may come from the kernel in front; requested ahead of this they are not there any earlier)
    // Released behind that wait: the next kernel may fetch weights ahead of its own wait, and what wrote them may be the kernel in front
    // of this one.  (Nothing is lost: the CTAs hold their SM for some 30 us yet.)
    tc::pdl_launch_dependents();
    if (producer && tc::elect_one()) request(p.wg, nullptr, 0, first);
    {
        if (p.rms_w) {
            // RMSNorm of the rows: y = h / sqrt(mean(h^2) + eps) . weight, rounded to bf16 as the layer's input (every CTA
            // normalises all rows); d <= 8 kThreads, so that a thread has at most one vector of a row
            constexpr int kWarps = kThreads / 32;
            float *const warp_ss = part;  // [T][kWarps] (not in use yet)
#pragma unroll
            for (int t = 0; t < T; ++t) {
                float ss = 0.f;
                if (tid * 8 < d) {
                    float h8[8];
                    Vec8<__nv_bfloat16>::load(p.x + (int64_t)t * d + tid * 8, h8);
#pragma unroll
                    for (int e = 0; e < 8; ++e) ss = fmaf(h8[e], h8[e], ss);
                }
                ss = warp_sum(ss);
                if (lane == 0) warp_ss[t * kWarps + warp] = ss;
            }
            __syncthreads();
#pragma unroll
            for (int t = 0; t < T; ++t) {
                float tot = 0.f;
                for (int w = 0; w < kWarps; ++w) tot += warp_ss[t * kWarps + w];
                scale[t] = rsqrtf(tot / (float)d + p.rms_eps);
            }
            __syncthreads();  // (the partial sums are the consumers' from here on)
        }
        for (int i = tid; i < kMaxRows; i += kThreads) s_mask[i] = 0;
        const int nthr = (int)gridDim.x * kThreads, gtid = (int)blockIdx.x * kThreads + tid;
        if (!p.grouped) {
#pragma unroll 1
            for (int i = gtid; i < T * kBins; i += nthr) p.hist[i] = 0u;
#pragma unroll 1
            for (int i = gtid; i < T * kNarrowBins * p.parts / 32; i += nthr) reinterpret_cast<uint4 *>(p.fine)[i] = make_uint4(0, 0, 0, 0);
#pragma unroll 1
            for (int i = gtid; i < T; i += nthr) p.cand_n[i] = 0u;
        }
#pragma unroll 1
        for (int i = gtid; i < T * d; i += nthr) p.acc[i] = 0.f;
    }
    // #0, split: the CTA announces that its slices are clear now and waits for the others only when it is about to
    // touch the shared arrays, after phase 1 (the arrival is a block-wide barrier too)
    auto clear_token = grid.barrier_arrive();

    // ---- phase 1: gate values of the CTA's channels, histogram of their keys
    if (producer) {
        if (tc::elect_one()) request(p.wg, nullptr, first, rows);
    } else if (consumer) {
        consume_dots(rows);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < T * rows; i += kThreads) {
        const int t = i / rows, r = i - t * rows;
        sg[t * rp + r] = dot(t, r);
    }
    grid.barrier_wait(std::move(clear_token));  // every CTA's slices of the shared arrays are clear
    __syncthreads();

    // ---- selection
    if (!p.grouped) {
#pragma unroll 1
        for (int i = tid; i < T * rows; i += kThreads) {
            const int t = i / rows, r = i - t * rows;
            const uint32_t key = gate_key(sg[t * rp + r]);
            atomicAdd(&p.hist[t * kBins + key_bin(key)], 1u);
            if (p.parts > 0 && key >= kFineFrom && key < kFineTo) {
                const uint32_t f = (key - kFineFrom) >> p.part_shift;
                atomicAdd(&p.fine[t * (kNarrowBins * p.parts / 8) + (f >> 3)], 1u << (4u * (f & 7u)));
            }
        }
        grid.sync();  // #1 (the barrier's release / acquire pair orders the CTAs' writes before the others' reads): every CTA's keys are in the histogram
        // the bin of the K-th largest key and the number of keys above that bin (suffix sums over the bins, the consumer warps
        // of a token one after the other)
        {
            constexpr int kWarpsOf = kConsumerWarps / T, N = kBins / (kWarpsOf * 32);
            static_assert(N % 4 == 0, "16-byte loads");
            const int t = warp / kWarpsOf, j = tid - t * kWarpsOf * 32;
            uint32_t h[N] = {}, s = 0u, own = 0u;
            if (consumer) {
#pragma unroll
                for (int i = 0; i < N / 4; ++i) {
                    const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(p.hist + t * kBins) + j * (N / 4) + i);
                    h[4 * i] = q.x, h[4 * i + 1] = q.y, h[4 * i + 2] = q.z, h[4 * i + 3] = q.w;
                }
#pragma unroll
                for (int i = 0; i < N; ++i) s += h[i];
                own = s;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_down_sync(0xffffffffu, s, o);
                    if (lane + o < 32) s += v;
                }
                if (lane == 0) s_scan[warp] = s;
            }
            __syncthreads();
            if (consumer) {
                uint32_t after = 0u;
                for (int w = warp + 1; w < (t + 1) * kWarpsOf; ++w) after += s_scan[w];
                uint32_t above = s + after - own;  // keys in strictly higher bins than this thread's
#pragma unroll
                for (int i = N - 1; i >= 0; --i) {
                    if (above < (uint32_t)p.K && above + h[i] >= (uint32_t)p.K) {
                        s_bin[t] = (uint32_t)(N * j + i);
                        s_above[t] = above;
                        s_count[t] = h[i];
                    }
                    above += h[i];
                }
            }
            __syncthreads();
        }
        // its parts, by a warp for each token
        if (warp < T) {
            constexpr uint32_t kFirst = key_bin(kFineFrom), kLast = key_bin(kFineTo - 1u);
            const uint32_t bin = s_bin[warp], need = (uint32_t)p.K - s_above[warp];
            uint32_t least = 0u;
            if (p.parts > 0 && bin >= kFirst && bin <= kLast) {
                const uint32_t narrow = narrow_bin(bin), words = (uint32_t)p.parts / 8u;
                const uint32_t q = lane < (int)words ? __ldcg(p.fine + (warp * kNarrowBins + narrow) * words + lane) : 0u;
                uint32_t n[8], s = 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    n[i] = (q >> (4 * i)) & 15u;
                    s += n[i];
                }
                const uint32_t own = s;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_down_sync(0xffffffffu, s, o);
                    if (lane + o < 32) s += v;
                }
                const bool all_counted = __shfl_sync(0xffffffffu, s, 0) == s_count[warp];
                uint32_t above = s - own;
#pragma unroll
                for (int i = 7; i >= 0; --i) {  // one part in all has the K-th key; where it is kept whole, its least key is the limit
                    above += n[i];
                    if (n[i] != 0u && above == need && all_counted) least = kFineFrom + ((narrow * p.parts + 8u * lane + i) << p.part_shift);
                }
                least = __reduce_max_sync(0xffffffffu, least);
            }
            if (lane == 0) s_least[warp] = least;
        }
        __syncthreads();
        bool open = false;  // (the same in every CTA: all have read the same counts)
#pragma unroll
        for (int t = 0; t < T; ++t) open = open || s_least[t] == 0u;
        const auto keep = [&](int t, int r) { atomicOr(reinterpret_cast<unsigned int *>(s_mask) + (r >> 2), (1u << t) << (8 * (r & 3))); };
#pragma unroll 1
        for (int i = tid; i < T * rows; i += kThreads) {
            const int t = i / rows, r = i - t * rows;
            const uint32_t key = gate_key(sg[t * rp + r]), bin = key_bin(key);
            if (s_least[t] != 0u ? key >= s_least[t] : bin > s_bin[t]) keep(t, r);
            // the CTA's keys of a bin that is not settled join the global candidate list
            if (s_least[t] == 0u && bin == s_bin[t]) {
                const uint32_t pos = atomicAdd(&p.cand_n[t], 1u);
                p.cand[(int64_t)t * F + pos] = make_uint2(key, (uint32_t)(c0 + r));
            }
        }
        if (open) {
            grid.sync();  // #2: the candidate lists are complete
            // rank the CTA's own candidates: one warp per candidate, the lanes share the list -- which is first copied to
            // shared memory (the ring is idle between the phases) when it fits, so that the ranking loops do not pay a
            // trip to L2 per step
            uint32_t n_of[T], off_of[T], total = 0;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                n_of[t] = min(__ldcg(&p.cand_n[t]), (uint32_t)F);
                off_of[t] = total;
                total += n_of[t];
            }
            uint2 *scand = reinterpret_cast<uint2 *>(ring);
            const bool staged = (size_t)total * sizeof(uint2) <= (size_t)p.stages * stage_bytes;
            if (staged) {
#pragma unroll
                for (int t = 0; t < T; ++t)
                    for (uint32_t j = tid; j < n_of[t]; j += kThreads) scand[off_of[t] + j] = __ldcg(&p.cand[(int64_t)t * F + j]);
            }
            __syncthreads();
            for (int i = warp; i < T * rows; i += kThreads / 32) {
                const int t = i / rows, r = i - t * rows;
                const uint32_t key = gate_key(sg[t * rp + r]);
                if (s_least[t] == 0u && key_bin(key) == s_bin[t]) {
                    uint32_t n = 0, ot = 0;
#pragma unroll
                    for (int tt = 0; tt < T; ++tt)
                        if (tt == t) {
                            n = n_of[tt];
                            ot = off_of[tt];
                        }
                    const uint32_t ch = (uint32_t)(c0 + r);
                    uint32_t before = 0;
                    for (uint32_t j = lane; j < n; j += 32) {
                        const uint2 o = staged ? scand[ot + j] : __ldcg(&p.cand[(int64_t)t * F + j]);
                        before += (o.x > key || (o.x == key && o.y < ch)) ? 1u : 0u;
                    }
                    before = __reduce_add_sync(0xffffffffu, before);
                    if (lane == 0 && s_above[t] + before < (uint32_t)p.K) keep(t, r);
                }
            }
            tc::fence_async_smem();  // (the list was written with ordinary stores, bulk copies write there next)
        }
    } else {
        // MoC 2:8 (Section 4): the CTA's range is made of whole groups of eight channels; the mask is local
#pragma unroll 1
        for (int i = tid; i < T * (rows >> 3); i += kThreads) {
            const int t = i / (rows >> 3), q = i - t * (rows >> 3);
            uint32_t key[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) key[e] = gate_key(sg[t * rp + 8 * q + e]);
            int lo, hi;
            top2_of_8(key, lo, hi);
            atomicOr(reinterpret_cast<unsigned int *>(s_mask) + ((8 * q + lo) >> 2), (1u << t) << (8 * ((8 * q + lo) & 3)));
            atomicOr(reinterpret_cast<unsigned int *>(s_mask) + ((8 * q + hi) >> 2), (1u << t) << (8 * ((8 * q + hi) & 3)));
        }
    }
    __syncthreads();  // (and the ring is the producer's again)
    if (p.kept_out)
#pragma unroll 1
        for (int i = tid; i < T * rows; i += kThreads) {
            const int t = i / rows, r = i - t * rows;
            p.kept_out[(int64_t)t * F + c0 + r] = (uint8_t)((s_mask[r] >> t) & 1);
        }
    if (warp == 0) {  // the kept channels in ascending order
        int n = 0;
        for (int base = 0; base < rows; base += 32) {
            const int r = base + lane;
            const bool f = r < rows && s_mask[r] != 0;
            const uint32_t b = __ballot_sync(0xffffffffu, f);
            if (f) s_list[n + __popc(b & ((1u << lane) - 1u))] = (uint16_t)r;
            n += __popc(b);
        }
        if (lane == 0) s_nsel = n;
    }
    __syncthreads();
    const int nsel = s_nsel;

    // ---- phase 3: up rows (u, z = SiLU(g) u), then down rows (every thread owns 8 columns)
    uint64_t acc[T][4];  // pairs of columns
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][e] = 0ull;
    if (producer) {
        if (tc::elect_one() && request(p.wu, s_list, 0, nsel)) request(p.wd, s_list, 0, nsel);
    } else if (consumer) {
        consume_dots(nsel);
        consumer_sync();
        for (int i = tid; i < nsel * T; i += kConsumerWarps * 32) {
            const int k = i / T, t = i - k * T, r = s_list[k];
            sz[i] = ((s_mask[r] >> t) & 1) ? silu_f(sg[t * rp + r]) * dot(t, k) : 0.f;
        }
        consumer_sync();  // every z is in shared memory
        const int col = tid * 8;
#pragma unroll 1
        for (int i = 0; i < nsel; i += p.of_stage) {
            if (wait_stage() && col < d) {
                const uint8_t *row = slot(c_stage) + col * 2;
                const int here = min(p.of_stage, nsel - i);
#pragma unroll 1
                for (int j = 0; j < here; ++j, row += pitch) {
                    uint64_t w[4];
                    unpack8(*reinterpret_cast<const uint4 *>(row), w);
#pragma unroll
                    for (int t = 0; t < T; ++t) {
                        const float z = sz[(i + j) * T + t];
#pragma unroll
                        for (int e = 0; e < 4; ++e) fma2(acc[t][e], pack2(z, z), w[e]);
                    }
                }
            }
            leave_stage();
        }
        if (col < d && nsel > 0) {
#pragma unroll
            for (int t = 0; t < T; ++t) {
                float *dst = p.acc + (int64_t)t * d + col;
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    asm volatile("{\n\t.reg .f32 a, b, c, d;\n\tmov.b64 {a, b}, %1;\n\tmov.b64 {c, d}, %2;\n\tred.global.add.v4.f32 [%0], {a, b, c, d};\n\t}" ::"l"(dst + 4 * h),
                                 "l"(acc[t][2 * h]), "l"(acc[t][2 * h + 1])
                                 : "memory");
            }
        }
    }
    __syncthreads();
    grid.sync();  // #3: every CTA's partial output is in the accumulator

    // ---- out = bf16(accumulator), a slice per CTA
    {
        const int vecs = T * d / 8;
#pragma unroll 1
        for (int v = (int)blockIdx.x * kThreads + tid; v < vecs; v += (int)gridDim.x * kThreads) {
            float4 a = __ldcg(reinterpret_cast<const float4 *>(p.acc) + 2 * v);
            float4 b = __ldcg(reinterpret_cast<const float4 *>(p.acc) + 2 * v + 1);
            if (p.rms_w) {  // the residual connection: out = h + D
                float h8[8];
                Vec8<__nv_bfloat16>::load(p.x + (size_t)v * 8, h8);
                a.x += h8[0], a.y += h8[1], a.z += h8[2], a.w += h8[3];
                b.x += h8[4], b.y += h8[5], b.z += h8[6], b.w += h8[7];
            }
            reinterpret_cast<uint4 *>(p.out)[v] =
                make_uint4(tc::pack_bf16(a.x, a.y), tc::pack_bf16(a.z, a.w), tc::pack_bf16(b.x, b.y), tc::pack_bf16(b.z, b.w));
        }
    }
    if (s_abort) {  // copies still in flight must land before shared memory goes away
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) __nanosleep(1000);
    }
}

}  // namespace dc
}  // namespace moc
