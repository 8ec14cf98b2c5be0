// Row Top-K selector of the tensor-core plan for rows of up to 14336 channels: a team of W warps per token, the gate row
// held in registers (VPL values per lane).
//
//   G [rows, ldg] fp32, U [rows, ldu] bf16: the dense projections of the token chunk.
//   Emits idx / g / u of the K kept channels (when saving) and rewrites the token's U row IN PLACE into the masked hidden
//   Z' = SiLU(g) u on the kept channels, 0 elsewhere -- the A operand of the down projection.  Exact: the K largest signed
//   gate values, indices ascending, equal values to the lower channel, NaN as -inf, -0 equal to +0.
//
// What bounds it: 8 bytes per channel have to move (G, U in, Z' out), and the instructions of the search have to stay
// below what the SM issues meanwhile.  A row is therefore read once, into registers, and walked three times in straight
// lines of predicated instructions (as branches, which is what plain code compiles to, each walk costs twice as much):
//   1. histogram: every value is mapped to one of 256, 512 or 1024 equal bins (row_bins.h: as many as K needs) of a window around the expected
//      threshold (multiply-add with saturation, so that what lies outside falls into the end bins) and counted with one
//      shared-memory atomic;
//   2. every warp scans the counts: bin b of the K-th largest value.  Everything from (just below) bin b on is a candidate
//      set of K + a few values: counted per group of 128 channels, one packed prefix sum over the lanes;
//   3. the candidate set goes to shared memory in ascending channel order, {value, channel} each.
//   4. The few entries of bin b are ranked exactly (value descending, channel ascending); those beyond rank K are dropped.
//   5. The K kept entries -- dense work now -- get their u, SiLU and product and are scattered into a zeroed row, which
//      leaves as one bulk store, while the next row's values are on their way into the registers.
// The window comes from a sample of the row itself (mean and mean absolute deviation of 128 of its values) and the normal
// quantile of K / F: nothing depends on other rows or earlier calls.  It decides the speed only: a row whose threshold lies
// outside, or whose bin b holds too many values, is searched over the whole key range, 256 bins at a time (exact for any
// values).  The team meets at five barriers a row and shares nothing with other teams.
#pragma once

#include "row_bins.h"
#include "tc_gemm.cuh"
#include "topk_select.cuh"

namespace moc {
namespace rs {

constexpr uint32_t kMaxRanked = 32;     // candidates ranked by one lane each

// CTAs (= teams) of W warps that an SM should hold: registers for VPL values per lane plus some 60.  More warps with fewer
// registers spill the values that are on their way, which stalls the walk they should overlap (16384 rows of 5504
// channels: 178 us with 128 registers, 251 with 96).
constexpr int ctas_per_sm(int W, int VPL) { return (VPL > 32 ? 16 : 20) / W; }

// normal_quantile on the device, with the fast functions (it only places a window)
__device__ __forceinline__ float normal_quantile_fast(int F, int K) {
    const float q = ((float)K - 0.5f) / (float)F, p = fminf(q, 1.0f - q), t = sqrtf(-2.0f * __logf(fmaxf(p, 1e-6f)));
    const float z = t - (2.515517f + t * (0.802853f + t * 0.010328f)) / (1.0f + t * (1.432788f + t * (0.189269f + t * 0.001308f)));
    return q > 0.5f ? -z : z;
}

struct Layout {
    uint32_t z, kept, hist, xch, bar, total;  // byte offsets (the up row is at 0)
};
__host__ __device__ inline Layout layout(int W, int bins, int ldu, int K) {
    Layout L{};
    uint32_t o = (uint32_t)ldu * 2u;
    L.z = o;
    o += (uint32_t)ldu * 2u;
    L.kept = o;  // {gate value, channel} in ascending channel order
    o += (((uint32_t)K + kMaxRanked) * 8u + 15u) & ~15u;
    L.hist = o;
    o += (uint32_t)bins * 4u;
    L.xch = o;  // number of ranked entries, pad[3] | ranked entries {value, list index} | two words per warp
    o += (4u + 2u * kMaxRanked + 2u * (uint32_t)W) * 4u;
    L.bar = (o + 7u) & ~7u;
    L.total = (L.bar + 8u + 15u) & ~15u;
    return L;
}

// One predicated 8-byte store, no branch; the address moves on by ordinary arithmetic, which the compiler can spread out.
__device__ __forceinline__ void keep_if_ge(float x, float tau, int ch, uint32_t &at) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ge.f32 p, %1, %2;\n\t@p st.shared.v2.b32 [%0], {%4, %3};\n\t}" ::"r"(at), "f"(x), "f"(tau), "r"(ch),
        "r"(__float_as_uint(x))
        : "memory");
    at += x >= tau ? 8u : 0u;
}
// four times the bin of a value: non-decreasing in x, NaN and everything below the window in bin 0, above it in the last
template <int BINS>
__device__ __forceinline__ uint32_t bin4(float x, float scale, float offset) {
    constexpr int bits = BINS == 1024 ? 10 : BINS == 512 ? 9 : 8;
    const float q = __saturatef(fmaf(x, scale, offset));
    return (__float_as_uint(fmaf(q, 1.0f - 0.5f / BINS, 1.0f)) >> (23 - bits - 2)) & (4u * BINS - 4u);
}

// where the want-th largest of the counted values lies
struct BinRank {
    uint32_t total;  // values counted
    uint32_t bin;    // its bin (valid when total >= want)
    uint32_t above;  // values in higher bins
    uint32_t count;  // values in the bin
};
template <int BINS>
__device__ __forceinline__ BinRank scan_bins(const uint32_t *hist, uint32_t want) {
    constexpr int N = BINS / 32;  // bins of a lane
    const int lane = threadIdx.x & 31;
    // values counted by this lane and by those above it
    const auto from_lane_up = [&](uint32_t v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t nb = __shfl_down_sync(0xffffffffu, v, o);
            if (lane + o < 32) v += nb;
        }
        return v;
    };
    BinRank r;
    uint32_t tot = 0, bin = 0, above = 0, cnt = 0;
    int src;
    if constexpr (N <= 8) {
        uint32_t h[N];
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const uint4 q = reinterpret_cast<const uint4 *>(hist)[N / 4 * lane + i];
            h[4 * i] = q.x;
            h[4 * i + 1] = q.y;
            h[4 * i + 2] = q.z;
            h[4 * i + 3] = q.w;
        }
#pragma unroll
        for (int i = 0; i < N; ++i) tot += h[i];
        const uint32_t suf = from_lane_up(tot);
        r.total = __shfl_sync(0xffffffffu, suf, 0);
        uint32_t gt = suf - tot;
        const bool here = gt < want && want <= suf;
#pragma unroll
        for (int i = N - 1; i >= 0; --i) {
            if (gt < want && want <= gt + h[i]) {
                bin = (uint32_t)(lane * N + i);
                above = gt;
                cnt = h[i];
            }
            gt += h[i];
        }
        src = max(0, __ffs(__ballot_sync(0xffffffffu, here)) - 1);
    } else {
        // Many bins beside a row that fills the registers: a lane's sum first (its 16-byte pieces in an order that keeps the
        // lanes off each other's banks), then the bins of the lane that holds the one looked for, one to a lane.
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const uint4 q = reinterpret_cast<const uint4 *>(hist)[N / 4 * lane + ((i + lane * N / 32) & (N / 4 - 1))];
            tot += q.x + q.y + q.z + q.w;
        }
        uint32_t suf = from_lane_up(tot);
        r.total = __shfl_sync(0xffffffffu, suf, 0);
        above = suf - tot;
        src = max(0, __ffs(__ballot_sync(0xffffffffu, above < want && want <= suf)) - 1);
        const uint32_t over = __shfl_sync(0xffffffffu, above, src);
        bin = (uint32_t)(N * src + lane);
        cnt = lane < N ? hist[bin] : 0u;
        suf = from_lane_up(cnt) + over;
        above = suf - cnt;
        src = max(0, __ffs(__ballot_sync(0xffffffffu, above < want && want <= suf)) - 1);
    }
    r.bin = __shfl_sync(0xffffffffu, bin, src);
    r.above = __shfl_sync(0xffffffffu, above, src);
    r.count = __shfl_sync(0xffffffffu, cnt, src);
    return r;
}

// A row whose threshold the window missed (or whose bin holds too many values): 8 bits of the threshold's key per pass over
// the row in global memory, then the kept channels in order.  The whole team; leaves the list complete behind a barrier of
// its own.  (A function: in line, its registers and its branches cost the common path a quarter.)
template <int W, int BINS>
__device__ __noinline__ void search_whole_range(const float *g, int F, int K, uint32_t *hist, uint2 *kept, volatile uint32_t *xw) {
    constexpr int TT = 32 * W;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    auto sync = [&]() {
        if (W == 1) __syncwarp();
        else __syncthreads();
    };
    uint32_t base = 0u, want = (uint32_t)K;
    for (int shift = 24; shift >= 0; shift -= 8) {
        sync();
        for (int i = tid; i < 256; i += TT) hist[i] = 0u;
        sync();
        const uint32_t limit = shift == 24 ? 0xffffffffu : (1u << (shift + 8)) - 1u;
#pragma unroll 8
        for (int c = tid; c < F; c += TT) {
            const uint32_t d = gate_key(__ldg(g + c)) - base;
            if (d <= limit) atomicAdd(&hist[d >> shift], 1u);
        }
        sync();
        const BinRank k = scan_bins<256>(hist, want);
        base += k.bin << shift;
        want -= k.above;
    }
    sync();
    // key `base` is the threshold; `want` of the values equal to it are kept, the first ones.  Warp w takes every 32-channel
    // group of its W-th of the row: first it counts, then it writes behind what the warps before it count.
    const int groups = (F + 31) >> 5, g0 = groups * w / W, g1 = groups * (w + 1) / W;
    uint32_t n_gt = 0, n_eq = 0;
#pragma unroll 4
    for (int v = g0; v < g1; ++v) {
        const int c = v * 32 + lane;
        const uint32_t key = c < F ? gate_key(__ldg(g + c)) : 0u;
        n_gt += (uint32_t)__popc(__ballot_sync(0xffffffffu, c < F && key > base));
        n_eq += (uint32_t)__popc(__ballot_sync(0xffffffffu, c < F && key == base));
    }
    if (lane == 0) {
        xw[w] = n_gt;
        xw[W + w] = n_eq;
    }
    sync();
    uint32_t gt = 0, eq = 0;
    for (int i = 0; i < w; ++i) {
        gt += xw[i];
        eq += xw[W + i];
    }
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll 4
    for (int v = g0; v < g1; ++v) {
        const int c = v * 32 + lane;
        const float x = c < F ? __ldg(g + c) : 0.f;
        const uint32_t key = c < F ? gate_key(x) : 0u;
        const bool is_gt = c < F && key > base, is_eq = c < F && key == base;
        const uint32_t bg = __ballot_sync(0xffffffffu, is_gt), be = __ballot_sync(0xffffffffu, is_eq);
        const uint32_t e = eq + (uint32_t)__popc(be & lt);
        if (is_gt || (is_eq && e < want)) kept[gt + (uint32_t)__popc(bg & lt) + min(e, want)] = make_uint2(__float_as_uint(x), (uint32_t)c);
        gt += (uint32_t)__popc(bg);
        eq += (uint32_t)__popc(be);
    }
    sync();
    for (int i = tid; i < BINS; i += TT) hist[i] = 0u;
    sync();
}

template <int W, int VPL, int BINS>
__global__ void __launch_bounds__(32 * W, ctas_per_sm(W, VPL)) select_rows_reg_kernel(
    const float *__restrict__ G, int ldg, __nv_bfloat16 *__restrict__ U, int ldu, int64_t rows, int F, int K, float quantile,
    int16_t *__restrict__ idx_out, __nv_bfloat16 *__restrict__ g_out, __nv_bfloat16 *__restrict__ u_out, int *status) {
    using namespace tc;
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr int TT = 32 * W;         // threads of the team (= of the CTA)
    constexpr int GPW = VPL / 4;       // 128-channel groups per warp: lane l of a group holds channels 4 l .. 4 l + 3
    constexpr int NP = (GPW + 3) / 4;  // words of packed per-group counts
    const Layout L = layout(W, BINS, ldu, K);
    const __nv_bfloat16 *su = reinterpret_cast<const __nv_bfloat16 *>(smem);
    __nv_bfloat16 *sz = reinterpret_cast<__nv_bfloat16 *>(smem + L.z);
    uint2 *kept = reinterpret_cast<uint2 *>(smem + L.kept);
    const uint32_t kept_at = smem_u32(kept);
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem + L.hist);
    const uint32_t hist_at = smem_u32(hist);
    volatile uint32_t *xch = reinterpret_cast<volatile uint32_t *>(smem + L.xch);
    uint2 *ranked = reinterpret_cast<uint2 *>(smem + L.xch + 16);
    volatile uint32_t *xw = xch + 4 + 2 * kMaxRanked;
    const uint32_t bar = smem_u32(smem + L.bar);
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int c0 = w * GPW * 128 + lane * 4;  // this lane's first channel
    auto sync = [&]() {
        if (W == 1) __syncwarp();
        else __syncthreads();
    };
    const uint32_t u_bytes = (uint32_t)ldu * 2u;
    auto clear_hist = [&]() {
        for (int i = tid; i < BINS / 4; i += TT) reinterpret_cast<uint4 *>(hist)[i] = make_uint4(0, 0, 0, 0);
    };
    float x[VPL];
    // the sample: a quad per lane, spread over the row (every warp of the team reads the same 128 values)
    const bool sampled = F >= 128;
    const int sample_c = sampled ? (int)((uint32_t)lane * (uint32_t)(F >> 2) >> 5) * 4 : 0;
    float4 sample = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_row = [&](int64_t r) {
        const float *g = G + r * (int64_t)ldg;
        const int full = F / 128 - w * GPW;  // this warp's groups that lie inside the row
#pragma unroll
        for (int v = 0; v < GPW; ++v) {
            const int c = c0 + v * 128;
            float4 q;
            if (v < full) {  // (the same for the whole warp)
                q = __ldcs(reinterpret_cast<const float4 *>(g + c));
            } else {  // (ldg is a multiple of 8: a quad that begins inside the row ends inside it)
                q = c < F ? __ldcs(reinterpret_cast<const float4 *>(g + c)) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                if (c + 1 >= F) q.y = -INFINITY;
                if (c + 2 >= F) q.z = -INFINITY;
                if (c + 3 >= F) q.w = -INFINITY;
            }
            x[4 * v] = q.x;
            x[4 * v + 1] = q.y;
            x[4 * v + 2] = q.z;
            x[4 * v + 3] = q.w;
        }
        if (sampled) sample = *reinterpret_cast<const float4 *>(g + sample_c);
    };
    auto request_u = [&](int64_t r) {  // (one thread)
        mbar_expect_tx(bar, u_bytes);
        bulk_copy_g2s(smem_u32(smem), U + r * (int64_t)ldu, u_bytes, bar);
    };

    // The last rows first: the GEMM that wrote G and U ended with them, so they are what the L2 still holds; and the down
    // projection, which walks the tokens upwards, then begins with the Z' rows that were written last.
    const int64_t r0 = rows - 1 - (int64_t)blockIdx.x;
    if (r0 < 0) return;
    load_row(r0);
    if (tid == 0) {
        s_abort = 0;
        xch[0] = 0u;
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        request_u(r0);
    }
    clear_hist();
    sync();
    uint32_t phase = 0;

    for (int64_t r = r0; r >= 0; r -= gridDim.x) {
        if (tid == 0) bulk_store_wait_read<0>();  // the previous row's Z' has left shared memory
        // ---- the window
        const float mean = warp_sum(sample.x + sample.y + sample.z + sample.w) * (1.0f / 128.0f);
        const float mad = warp_sum(fabsf(sample.x - mean) + fabsf(sample.y - mean) + fabsf(sample.z - mean) + fabsf(sample.w - mean)) *
                          (1.0f / 128.0f);
        // (with the mean within 128 deviations, the roundings of the bins' edges stay below a hundredth of a bin)
        const bool window = sampled && mad > 1e-30f && mad < 1e30f && fabsf(mean) < 128.f * mad;
        const float lo = fmaf(mad, 1.2533f * quantile - kWindowMad, mean);  // sigma of normal values = 1.2533 mad
        const float scale = window ? 0.5f / (kWindowMad * mad) : 0.f, offset = -lo * scale;
        // ---- 1. histogram
        bool fast = window;
        BinRank b = {};
        float from = 0.f, below = 0.f;  // the candidate set; entries under `below` are ranked
        if (window) {
#pragma unroll
            for (int i = 0; i < VPL; ++i)
                asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(hist_at + bin4<BINS>(x[i], scale, offset)) : "memory");
            sync();
            b = scan_bins<BINS>(hist, (uint32_t)K);
            fast = b.bin >= 1u && b.bin < BINS - 1u && b.count <= kMaxRanked - 4u;
            const float width = 2.f * kWindowMad * mad / (BINS - 0.5f);
            from = fmaf((float)b.bin - 0.05f, width, lo);   // a little below and above the bin: rounding decides into which
            below = fmaf((float)b.bin + 1.05f, width, lo);  // bin a value at its edge falls
        }
        uint32_t n_list = (uint32_t)K;
        if (fast) {
            // ---- 2. the candidate set: counts of every group, packed four to a word (a group holds at most 128)
            uint32_t pk[NP] = {}, inc[NP], tot[NP], wsum = 0;
#pragma unroll
            for (int i = 0; i < VPL; ++i)
                if (x[i] >= from) pk[i >> 4] += 1u << (8 * ((i >> 2) & 3));
#pragma unroll
            for (int j = 0; j < NP; ++j) inc[j] = pk[j];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const uint32_t nb = __shfl_up_sync(0xffffffffu, inc[j], o);
                    if (lane >= o) inc[j] += nb;
                }
            }
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                tot[j] = __shfl_sync(0xffffffffu, inc[j], 31);
                inc[j] -= pk[j];
#pragma unroll
                for (int q = 0; q < 4; ++q) wsum += (tot[j] >> (8 * q)) & 255u;
            }
            if (W > 1 && lane == 0) xw[w] = wsum;
            sync();  // (also: every warp has scanned the histogram)
            clear_hist();
            uint32_t before = 0;
            n_list = W > 1 ? 0u : wsum;
            if (W > 1) {
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const uint32_t t = xw[i];
                    before += i < w ? t : 0u;
                    n_list += t;
                }
            }
            fast = n_list - b.above <= kMaxRanked;  // (else: too many values at the bin's edges)
            if (fast) {
                // ---- 3. the list
                uint32_t first = kept_at + 8u * before;
#pragma unroll
                for (int v = 0; v < GPW; ++v) {
                    uint32_t at = first + 8u * ((inc[v >> 2] >> (8 * (v & 3))) & 255u);
#pragma unroll
                    for (int e = 0; e < 4; ++e) keep_if_ge(x[4 * v + e], from, c0 + v * 128 + e, at);
                    first += 8u * ((tot[v >> 2] >> (8 * (v & 3))) & 255u);
                }
            }
        }
        if (!fast) {
            search_whole_range<W, BINS>(G + r * (int64_t)ldg, F, K, hist, kept, xw);
            n_list = (uint32_t)K;
        }
        for (int i = tid; i < (ldu >> 3); i += TT) reinterpret_cast<uint4 *>(sz)[i] = make_uint4(0, 0, 0, 0);
        sync();
        const int64_t next = r - gridDim.x;
        if (next >= 0) load_row(next);  // travels while the list is worked on
        // ---- 4. the entries of bin b
        if (fast) {
            for (uint32_t i = tid; i < n_list; i += TT)
                if (__uint_as_float(kept[i].x) < below) {
                    const uint32_t at = atomicAdd(const_cast<uint32_t *>(xch), 1u);
                    if (at < kMaxRanked) ranked[at] = make_uint2(kept[i].x, i);
                }
        }
        // a wait that gave up ends the team
        const bool ok = mbar_wait(bar, phase, &s_abort, status);
        const bool dead = W == 1 ? __any_sync(0xffffffffu, !ok) : __syncthreads_or(!ok ? 1 : 0) != 0;
        if (W == 1) __syncwarp();
        if (dead) break;
        phase ^= 1u;
        uint32_t drop_at = 0xffffffffu;  // list index of the entry this lane found to be dropped
        if (fast) {
            const uint32_t n_ranked = xch[0];
            if (n_ranked <= kMaxRanked) {
                // everything else in the list is larger: an entry is kept when fewer than K come before it
                const uint2 e = (uint32_t)lane < n_ranked ? ranked[lane] : make_uint2(0xff800000u, 0xffffffffu);
                const float v = __uint_as_float(e.x);
                uint32_t rank = n_list - n_ranked;
                for (uint32_t i = 0; i < n_ranked; ++i) {
                    const uint2 q = ranked[i];
                    const float ov = __uint_as_float(q.x);
                    rank += ov > v || (ov == v && q.y < e.y) ? 1u : 0u;
                }
                if ((uint32_t)lane < n_ranked && rank >= (uint32_t)K) {
                    drop_at = e.y;
                    kept[drop_at].y = 0xffffffffu;  // (every warp marks the same entries, for itself)
                }
                __syncwarp();
            } else {  // too many values at the bin's edges
                search_whole_range<W, BINS>(G + r * (int64_t)ldg, F, K, hist, kept, xw);
                n_list = (uint32_t)K;
            }
        }
        // ---- 5. values of the kept channels: two entries of the list per lane
        int16_t *const ri = idx_out ? idx_out + r * K : nullptr;
        __nv_bfloat16 *const rg = g_out + r * K, *const ru = u_out + r * K;
        for (uint32_t i0 = (uint32_t)w * 64u; i0 < n_list; i0 += 2 * TT) {
            const uint32_t before = (uint32_t)__popc(__ballot_sync(0xffffffffu, drop_at < i0));  // dropped ahead of these 64
            const uint32_t i = i0 + 2u * lane;
            const uint4 e = i < n_list ? *reinterpret_cast<const uint4 *>(kept + i) : make_uint4(0u, 0xffffffffu, 0u, 0xffffffffu);
            const bool in0 = e.y != 0xffffffffu, in1 = e.w != 0xffffffffu && i + 1u < n_list;
            const uint32_t m0 = __ballot_sync(0xffffffffu, in0), m1 = __ballot_sync(0xffffffffu, in1), lt = (1u << lane) - 1u;
            const uint32_t at0 = i0 - before + (uint32_t)__popc(m0 & lt) + (uint32_t)__popc(m1 & lt), at1 = at0 + (in0 ? 1u : 0u);
            const uint32_t ch0 = in0 ? e.y : 0u, ch1 = in1 ? e.w : 0u;
            const float g0 = __uint_as_float(e.x), g1 = __uint_as_float(e.z);
            const __nv_bfloat16 u0 = su[ch0], u1 = su[ch1];
            const __nv_bfloat16 z0 = __float2bfloat16_rn(silu_f(g0) * __bfloat162float(u0)), z1 = __float2bfloat16_rn(silu_f(g1) * __bfloat162float(u1));
            if (in0) sz[ch0] = z0;
            if (in1) sz[ch1] = z1;
            if (ri) {
                if (in0) {
                    ri[at0] = (int16_t)ch0;
                    rg[at0] = __float2bfloat16_rn(g0);
                    ru[at0] = u0;
                }
                if (in1) {
                    ri[at1] = (int16_t)ch1;
                    rg[at1] = __float2bfloat16_rn(g1);
                    ru[at1] = u1;
                }
            }
        }
        fence_async_smem();
        sync();
        if (tid == 0) {
            xch[0] = 0u;
            bulk_copy_s2g(U + r * (int64_t)ldu, smem_u32(sz), u_bytes);
            if (next >= 0) request_u(next);
        }
    }
    if (tid == 0) bulk_store_wait_all();  // shared memory must outlive the stores that read it
    if (s_abort) {                        // ... and the copies into it that a wait gave up on
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) __nanosleep(1000);
    }
}

}  // namespace rs
}  // namespace moc
