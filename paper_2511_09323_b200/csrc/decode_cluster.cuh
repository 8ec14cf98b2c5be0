// Decode on small layers: one cluster of 16 CTAs per token or two, no grid barrier, no workspace (bf16).
//
// What bounds the one-kernel form of decode_coop.cuh on a small layer is not its rows (768 x 2048: 3.1 MB of W_gate, a few
// hundred kept rows) but three barriers of all SMs, a cooperative launch that waits for the whole GPU, and two exchanges
// through L2.  Sixteen SMs read such a matrix in the time of one of those barriers, and a cluster exchanges through shared
// memory.  The CTAs split the CHANNELS as there:
//
//   phase 1   the CTA's rows of W_gate, requested before the wait for the kernel in front (weights do not depend on it); two warps
//             per 16 rows form the gate values of all the group's tokens (Eq. (Moc-1)); their keys go to all 16 CTAs
//   select    cluster barrier; every CTA has the whole rows of keys: histogram, bin of the K-th largest, exact ranks
//             inside the bin (value descending, channel ascending) -- the mask definition of Section 3.2
//   phase 2   the rows of W_up and W_down of the CTA's kept channels, z = SiLU(g) u (Eq. (MoC-2)), a partial output per CTA
//   output    every CTA sends the partial sums of a slice of columns to the CTA that owns the slice; cluster barrier; the
//             owners add 16 of them in a fixed order, add the residual and round
//
// All three products run on mma.sync (rows are the 16 of m16n8k16, tokens the 8).  z is held in fp32 and multiplied as the sum of
// three bf16 numbers, 24 bits.  Shared memory of another CTA is written 16 bytes at a time: 4-byte stores take five cycles each
// (768 x 2048: the keys alone 5 us).
//
// What is left (768 x 2048, one token, 24 thousand cycles from the token's arrival): gate values 5.5, exchange of keys 1.6, selection
// 5, kept rows 2.1 until they are there and 5 until they are multiplied, exchange of the partial sums 1.9; each of them is a short
// piece of code that is fetched anew in every launch.  The gate rows do not appear: that is in a row of these calls,
// 13.7 us each, where a launch begins before the one in front has ended and requests them then.  Behind a kernel that does not
// release its dependents early they stand in the call, 18.6 us: a cluster's way to L2 is what bounds it there, about 0.7 TB/s for
// 16 SMs of one GPC, and on larger layers a form on all SMs is faster (cluster_pays).
//
// Clusters share nothing, so it does not matter how many run at a time.  A cluster barrier cannot fail; a wait for a copy that
// runs out raises MOC_ERR_TIMEOUT and the CTA walks on through both barriers.
#pragma once

#include "decode_coop.cuh"

namespace moc {
namespace dcl {

constexpr int kCluster = 16;
constexpr int kWarps = 16;                   // consumers
constexpr int kThreads = (kWarps + 1) * 32;  // + one producer warp
constexpr int kMaxTokens = 2;                // per cluster
constexpr int kMaxD = 2048;
constexpr int kMaxStages = 16;               // of 16 rows
constexpr int kMaxRows = 512;                // channels per CTA
constexpr int kBins = dc::kBins;

// Rows in shared memory are 64 bytes (mod 128) apart, so that the 64-byte pieces of two rows that a quarter of a warp reads lie on
// different banks; the rows of W_down, of which 16-byte pieces of eight rows are read at a time, 80 bytes.
__host__ __device__ inline uint32_t row_pitch(int d) { return (uint32_t)d * 2u + ((64u - (uint32_t)d * 2u) & 127u); }
__host__ __device__ inline uint32_t down_pitch(int d) { return (uint32_t)d * 2u + ((80u - (uint32_t)d * 2u) & 127u); }
inline int slice_vecs(int d) { return (d / 8 + kCluster - 1) / kCluster; }  // 8-column pieces a CTA owns
// channels of the CTA that has most, rounded up to whole 16-byte pieces of keys
inline int rows_of(int F, int unit) { return (((F + unit - 1) / unit + kCluster - 1) / kCluster * unit + 7) & ~7; }

// shared memory, byte offsets (the weight rows' ring is at 0; between the phases it holds histograms and candidates)
struct Layout {
    uint32_t x, keys, own, g, zp, part, out, recv, total;
};
inline Layout layout(int T, int d, int F, int unit, int stages) {
    const auto up = [](uint32_t v) { return (v + 127u) & ~127u; };
    const uint32_t rp = (uint32_t)rows_of(F, unit), n = (uint32_t)T;
    const uint32_t ring = (uint32_t)stages * 8u * (row_pitch(d) + (row_pitch(d) > down_pitch(d) ? row_pitch(d) : down_pitch(d))), search = n * ((uint32_t)kBins * 4u + kCluster * rp * 2u);
    Layout L{};
    L.x = up(ring > search ? ring : search);
    L.keys = up(L.x + n * row_pitch(d));                     // [T][16][rp]
    L.own = up(L.keys + n * kCluster * rp * 4u);             // [T][rp] keys of this CTA
    L.g = up(L.own + n * rp * 4u);                           // [2][T][rp] gate values, in two parts of the contraction
    L.zp = up(L.g + 2u * n * rp * 4u);                       // [8][8 * stages + 8] bf16 parts of z
    L.part = up(L.zp + 8u * (8u * (uint32_t)stages + 8u) * 2u);  // [4][8][16 rows][T] parts of u
    L.out = up(L.part + 4u * 8u * 16u * n * 4u);                 // [T][d] partial output
    L.recv = up(L.out + n * (uint32_t)d * 4u);               // [16][T][slice]
    L.total = up(L.recv + kCluster * n * (uint32_t)slice_vecs(d) * 32u);
    return L;
}

struct Params {
    const __nv_bfloat16 *x, *wg, *wu, *wd;
    __nv_bfloat16 *out;
    int tokens, d, F, K, grouped;
    int unit;    // channels are dealt to the CTAs in units of this many (8 when F % 8 == 0, else 1)
    int stages;  // of 16 weight rows each
    int rp, own_vecs;  // rows_of(F, unit), slice_vecs(d)
    Layout at;
    int *status;
    const __nv_bfloat16 *rms_w;  // the block form: x is the residual stream h (see decode_coop.cuh); null: the plain layer
    float rms_eps;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void store_cluster_v4(uint32_t dst, const uint4 &v) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Products of 16 staged rows with the tokens over the 32-element blocks b0 .. b1 of the contraction, by one warp: a lane holds
// rows lane / 4 and that plus 8, tokens 2 (lane % 4) and the next.  Inside a block the contraction is permuted, in both
// operands alike, so that a lane's elements are 16 consecutive bytes.  (One function for both phases: instructions are fetched
// anew in every launch, some hundred cycles per 128 bytes, and that is most of what a short phase takes.)
template <int T>
__device__ __noinline__ float4 products_of_16_rows(const uint8_t *rows, uint32_t eight_rows, const uint8_t *tokens, int b0, int b1, int left) {
    float c[2][4] = {};
    const bool token = (int)((threadIdx.x & 31) >> 2) < T;
#pragma unroll 2
    for (int b = b0; b < b1; ++b) {
        uint4 a = make_uint4(0, 0, 0, 0), e = a, x = a;
        if (b * 32 < left) {
            a = *reinterpret_cast<const uint4 *>(rows + b * 64);
            e = *reinterpret_cast<const uint4 *>(rows + eight_rows + b * 64);
            if (token) x = *reinterpret_cast<const uint4 *>(tokens + b * 64);
        }
        mma_16816(c[0], a.x, e.x, a.y, e.y, x.x, x.y);
        mma_16816(c[1], a.z, e.z, a.w, e.w, x.z, x.w);
    }
    return make_float4(c[0][0] + c[1][0], c[0][1] + c[1][1], c[0][2] + c[1][2], c[0][3] + c[1][3]);
}

template <int T>  // tokens of a cluster: one or two
__global__ void __launch_bounds__(kThreads, 1) decode_cluster_kernel(const __grid_constant__ Params p) {
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ __align__(16) uint4 s_zero;
    __shared__ uint64_t full[kMaxStages], empty[kMaxStages], s_up, s_down;
    __shared__ int s_abort, s_nsel;
    __shared__ uint32_t s_scan[T][kWarps], s_bin[T], s_above[T], s_ncand[T], s_count[kWarps];
    __shared__ uint16_t s_list[kMaxRows];              // the CTA's kept channels (offsets in its range), kept by any token
    __shared__ __align__(4) uint8_t s_mask[kMaxRows];  // per channel of the range: which tokens keep it (bit t)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lane_g = lane >> 2, lane_q = lane & 3;
    const bool producer = warp == kWarps;
    const uint32_t rank = tc::cluster_ctarank();
    const int d = p.d, F = p.F, t0 = (int)(blockIdx.x / kCluster) * T, nt = min(T, p.tokens - t0);
    const int rp = p.rp;
    const Layout &L = p.at;
    const uint32_t row_bytes = (uint32_t)d * 2u, pitch = row_pitch(d), dpitch = down_pitch(d), stage_bytes = 16u * pitch;
    uint32_t *const keys = reinterpret_cast<uint32_t *>(dsm + L.keys), *const own = reinterpret_cast<uint32_t *>(dsm + L.own);
    uint32_t *const hist = reinterpret_cast<uint32_t *>(dsm);
    uint16_t *const cand = reinterpret_cast<uint16_t *>(dsm + T * kBins * 4);
    float *const sg = reinterpret_cast<float *>(dsm + L.g), *const part = reinterpret_cast<float *>(dsm + L.part);
    __nv_bfloat16 *const zp = reinterpret_cast<__nv_bfloat16 *>(dsm + L.zp);
    float *const s_out = reinterpret_cast<float *>(dsm + L.out);
    const uint32_t smem = tc::smem_u32(dsm);

    // the CTA's channels
    const int units = (F + p.unit - 1) / p.unit;
    const int c0 = (int)((int64_t)rank * units / kCluster) * p.unit;
    const int c1 = min(F, (int)((int64_t)(rank + 1) * units / kCluster) * p.unit);
    const int rows = max(0, c1 - c0);  // <= rp
    const int groups = (rows + 15) / 16;

    if (tid == 0) {
        for (int s = 0; s < p.stages; ++s) {
            tc::mbar_init(tc::smem_u32(&full[s]), 1);
            tc::mbar_init(tc::smem_u32(&empty[s]), kWarps);
        }
        tc::mbar_init(tc::smem_u32(&s_up), 1);
        tc::mbar_init(tc::smem_u32(&s_down), 1);
        s_abort = 0;
        s_zero = make_uint4(0, 0, 0, 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cluster_arrive();  // #0: the CTA's shared memory exists (waited for before the first store into another CTA's)
    tc::pdl_launch_dependents();
    // (the producer warp) 16 rows, or what is left of them, to stage s; by one elected thread (a lane for each row: four tokens of
    // 768 x 2048 15.2 us instead of 14.3)
    const auto request = [&](int g, int s) {
        const int n = min(16, rows - g * 16);
        const uint32_t bar = tc::smem_u32(&full[s]);
        if (tc::elect_one()) {
            tc::mbar_expect_tx(bar, (uint32_t)n * row_bytes);
            for (int i = 0; i < n; ++i)
                tc::bulk_copy_g2s(smem + (uint32_t)s * stage_bytes + (uint32_t)i * pitch, p.wg + (int64_t)(c0 + g * 16 + i) * d, row_bytes, bar);
        }
        __syncwarp();
    };
    if (producer)
        for (int g = 0; g < min(groups, p.stages); ++g) request(g, g);
    for (int i = tid; i < kMaxRows / 4; i += kThreads) reinterpret_cast<uint32_t *>(s_mask)[i] = 0u;
    if (tid < T) s_ncand[tid] = 0u;

    // ---- the tokens (of a group that is not full, the last one again; its output is not stored)
    tc::pdl_wait();
    const auto token_row = [&](int t) { return (int64_t)(t0 + min(t, nt - 1)) * d; };
    const auto sx = [&](int t) { return reinterpret_cast<__nv_bfloat16 *>(dsm + L.x + (uint32_t)t * pitch); };
#pragma unroll
    for (int t = 0; t < T; ++t)
        for (int i = tid * 8; i < d; i += kThreads * 8) *reinterpret_cast<uint4 *>(sx(t) + i) = *reinterpret_cast<const uint4 *>(p.x + token_row(t) + i);
    if (p.rms_w) {
        // (the arithmetic of decode_coop.cuh: every CTA normalises the rows it has staged, in place)
        __syncthreads();
        float ss[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            ss[t] = 0.f;
            for (int i = tid; i < d; i += kThreads) {
                const float v = __bfloat162float(sx(t)[i]);
                ss[t] = fmaf(v, v, ss[t]);
            }
            ss[t] = warp_sum(ss[t]);
        }
        if (lane == 0)
#pragma unroll
            for (int t = 0; t < T; ++t) part[t * 32 + warp] = ss[t];  // (not in use yet)
        __syncthreads();
#pragma unroll
        for (int t = 0; t < T; ++t) {
            float tot = 0.f;
            for (int w = 0; w < kThreads / 32; ++w) tot += part[t * 32 + w];
            const float scale = rsqrtf(tot / (float)d + p.rms_eps);
            for (int i = tid; i < d; i += kThreads)
                sx(t)[i] = __float2bfloat16_rn(__bfloat162float(sx(t)[i]) * scale * __bfloat162float(p.rms_w[i]));
        }
    }
    __syncthreads();

    const int blocks = (d + 31) / 32;
    const auto row_products = [&](uint32_t base, int b0, int b1, float (&sum)[4]) {
        const float4 c = products_of_16_rows<T>(dsm + base + (uint32_t)lane_g * pitch + (uint32_t)lane_q * 16u, 8u * pitch,
                                                dsm + L.x + (uint32_t)(lane_g < T ? lane_g : 0) * pitch + (uint32_t)lane_q * 16u, b0, b1,
                                                d - lane_q * 8);
        sum[0] = c.x, sum[1] = c.y, sum[2] = c.z, sum[3] = c.w;
    };
    // element (row, token) of such a result
    const auto each = [&](const float (&sum)[4], auto put) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (2 * lane_q + (i & 1) < T) put(lane_g + 8 * (i >> 1), 2 * lane_q + (i & 1), sum[i]);
    };

    // ---- phase 1: 16 rows by two warps, half of the contraction each (a warp per row with FMAs, its share of the token in registers:
    // 10 thousand cycles at 768 x 2048 instead of 5.5).  When the stages are used more than once, every warp sees every
    // round of theirs (a parity test only tells an odd from an even number of completed rounds).
    const bool once = groups <= p.stages;
    if (producer) {
        uint32_t phase = 0;
        for (int g = p.stages, s = 0; g < groups; ++g) {
            if (!__all_sync(0xffffffffu, tc::mbar_wait(tc::smem_u32(&empty[s]), phase, &s_abort, p.status))) break;
            request(g, s);
            if (++s == p.stages) s = 0, phase ^= 1u;
        }
    } else {
        uint32_t phase = 0;
#pragma unroll 1
        for (int g = 0, s = 0; g < groups; ++g) {
            const bool mine = (g & 7) == warp >> 1;
            if (mine || !once) {
                if (!__all_sync(0xffffffffu, tc::mbar_wait(tc::smem_u32(&full[s]), phase, &s_abort, p.status))) break;
                if (mine) {
                    const int h = warp & 1;
                    float sum[4];
                    row_products((uint32_t)s * stage_bytes, h ? blocks / 2 : 0, h ? blocks : blocks / 2, sum);
                    each(sum, [&](int r, int t, float v) {
                        if (g * 16 + r < rp) sg[(h * T + t) * rp + g * 16 + r] = v;
                    });
                }
                __syncwarp();
                if (lane == 0 && !once) tc::mbar_arrive(tc::smem_u32(&empty[s]));
            }
            if (++s == p.stages) s = 0, phase ^= 1u;
        }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < T; ++t)
        for (int r = tid; r < rp; r += kThreads) {
            const float v = sg[t * rp + r] + sg[(T + t) * rp + r];
            sg[t * rp + r] = v;
            own[t * rp + r] = r < rows ? gate_key(v) : 0u;  // (0: below every key)
        }
    if (!p.grouped)
        for (int i = tid; i < T * kBins / 4; i += kThreads) reinterpret_cast<uint4 *>(hist)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    cluster_wait();  // #0

    // ---- selection
    if (!p.grouped) {
        if (!producer) {  // the keys to all CTAs, one a warp
            const uint32_t dst = tc::map_to_cta(tc::smem_u32(keys + rank * rp), (uint32_t)warp);
#pragma unroll 1
            for (int t = 0; t < T; ++t)
                for (int i = lane * 4; i < rp; i += 128)
                    store_cluster_v4(dst + (uint32_t)(t * kCluster * rp + i) * 4u, *reinterpret_cast<const uint4 *>(own + t * rp + i));
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();  // #1: the rows of keys are complete
        const int n_keys = kCluster * rp;  // of a token: slots in ascending channel order, some of them empty
#pragma unroll 1
        for (int t = 0; t < T; ++t)
            for (int i = tid; i < n_keys; i += kThreads) {
                const uint32_t key = keys[t * n_keys + i];
                if (key) atomicAdd(&hist[t * kBins + dc::key_bin(key)], 1u);
            }
        __syncthreads();
        // the bin of the K-th largest key and the number of keys above that bin: suffix sums, four bins to a thread
        static_assert(kBins == 4 * kWarps * 32, "");
        uint32_t suf[T];
        if (!producer) {
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const uint4 q = reinterpret_cast<const uint4 *>(hist + t * kBins)[tid];
                uint32_t s = q.x + q.y + q.z + q.w;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_down_sync(0xffffffffu, s, o);
                    if (lane + o < 32) s += v;
                }
                if (lane == 0) s_scan[t][warp] = s;
                suf[t] = s;
            }
        }
        __syncthreads();
        if (!producer) {
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const uint4 q = reinterpret_cast<const uint4 *>(hist + t * kBins)[tid];
                const uint32_t h[4] = {q.x, q.y, q.z, q.w};
                uint32_t above = suf[t] - (q.x + q.y + q.z + q.w);
                above += __reduce_add_sync(0xffffffffu, lane > warp && lane < kWarps ? s_scan[t][lane] : 0u);
#pragma unroll
                for (int i = 3; i >= 0; --i) {
                    if (above < (uint32_t)p.K && above + h[i] >= (uint32_t)p.K) {
                        s_bin[t] = (uint32_t)(4 * tid + i);
                        s_above[t] = above;
                    }
                    above += h[i];
                }
            }
        }
        __syncthreads();
        // the keys of that bin (in any order: they are ranked by value and slot), and the CTA's own above it
        const int first = (int)rank * rp;
        const auto keep = [&](int r, int t) { atomicOr(reinterpret_cast<unsigned int *>(s_mask) + (r >> 2), (1u << t) << (8 * (r & 3))); };
#pragma unroll 1
        for (int t = 0; t < T; ++t) {
            const uint32_t bin = s_bin[t];
            for (int i = tid; i < n_keys; i += kThreads) {
                const uint32_t key = keys[t * n_keys + i], b = dc::key_bin(key);
                if (b < bin || !key) continue;
                if (b == bin) cand[t * n_keys + atomicAdd(&s_ncand[t], 1u)] = (uint16_t)i;
                else if (i >= first && i < first + rows) keep(i - first, t);
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int t = 0; t < T; ++t) {
            const int n = (int)s_ncand[t];
            for (int j = warp; j < n; j += kWarps + 1) {
                const int i = cand[t * n_keys + j];
                if (i < first || i >= first + rows) continue;
                const uint32_t key = keys[t * n_keys + i];
                uint32_t before = 0;
                for (int l = lane; l < n; l += 32) {
                    const int o = cand[t * n_keys + l];
                    const uint32_t ok = keys[t * n_keys + o];
                    before += ok > key || (ok == key && o < i) ? 1u : 0u;
                }
                before = __reduce_add_sync(0xffffffffu, before);
                if (lane == 0 && s_above[t] + before < (uint32_t)p.K) keep(i - first, t);
            }
        }
    } else {
        // MoC 2:8 (Section 4): the CTA's range is made of whole groups of eight channels; the mask is local
        for (int i = tid; i < T * (rows >> 3); i += kThreads) {
            const int t = i / (rows >> 3), q = i - t * (rows >> 3);
            uint32_t key[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) key[e] = own[t * rp + 8 * q + e];
            int lo, hi;
            top2_of_8(key, lo, hi);
            atomicOr(reinterpret_cast<unsigned int *>(s_mask) + ((8 * q + lo) >> 2), (1u << t) << (8 * ((8 * q + lo) & 3)));
            atomicOr(reinterpret_cast<unsigned int *>(s_mask) + ((8 * q + hi) >> 2), (1u << t) << (8 * ((8 * q + hi) & 3)));
        }
    }
    tc::fence_async_smem();  // (histogram and candidates were written with ordinary stores, bulk copies write there next)
    __syncthreads();
    // the kept channels in ascending order (a row of the range per consumer thread)
    static_assert(kMaxRows <= kWarps * 32, "");
    uint32_t ballot = 0;
    if (!producer) {
        ballot = __ballot_sync(0xffffffffu, tid < rows && s_mask[tid] != 0);
        if (lane == 0) s_count[warp] = (uint32_t)__popc(ballot);
    }
    __syncthreads();
    if (!producer) {
        const int at = (int)__reduce_add_sync(0xffffffffu, lane < warp ? s_count[lane] : 0u);
        if ((ballot >> lane) & 1u) s_list[at + __popc(ballot & ((1u << lane) - 1u))] = (uint16_t)tid;
        if (tid == kWarps * 32 - 1) s_nsel = at + __popc(ballot);
    }
    __syncthreads();
    const int nsel = s_nsel;

    // ---- phase 2: the kept rows, as many at a time as half the ring holds
    constexpr int kSlots = 2;  // columns of the products that a part of z takes, whether there are one or two tokens
    constexpr int kParts = 3;  // bf16 numbers that add up to a z
    const int batch = p.stages * 8, zpitch = batch + 8;
    const uint32_t down0 = smem + (uint32_t)batch * pitch;
    for (int b0 = 0, turn = 0; b0 < nsel; b0 += batch, ++turn) {
        const int n = min(batch, nsel - b0), n16 = (n + 15) / 16;
        if (producer) {
            if (lane == 0) {
                tc::mbar_expect_tx(tc::smem_u32(&s_up), (uint32_t)n * row_bytes);
                tc::mbar_expect_tx(tc::smem_u32(&s_down), (uint32_t)n * row_bytes);
            }
            __syncwarp();
            for (int i = lane; i < n; i += 32)
                tc::bulk_copy_g2s(smem + (uint32_t)i * pitch, p.wu + (int64_t)(c0 + s_list[b0 + i]) * d, row_bytes, tc::smem_u32(&s_up));
            for (int i = lane; i < n; i += 32)
                tc::bulk_copy_g2s(down0 + (uint32_t)i * dpitch, p.wd + (int64_t)(c0 + s_list[b0 + i]) * d, row_bytes, tc::smem_u32(&s_down));
        } else {
            const bool up = __all_sync(0xffffffffu, tc::mbar_wait(tc::smem_u32(&s_up), (uint32_t)turn & 1u, &s_abort, p.status));
            // u: 16 rows by one to four warps, a part of the contraction each (n16 <= 8: at most 16 stages)
            const int splits = n16 <= 4 ? 4 : 2, share = n16 <= 4 ? warp >> 2 : warp >> 3, mine = warp & (n16 <= 4 ? 3 : 7);
            if (mine < n16) {
                const int per = (blocks + splits - 1) / splits;
                float sum[4];
                row_products((uint32_t)mine * stage_bytes, per * share, min(blocks, per * (share + 1)), sum);
                each(sum, [&](int r, int t, float v) { part[((share * 8 + mine) * 16 + r) * T + t] = v; });
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kWarps * 32) : "memory");
            // z and its parts (columns that no part fills hold anything: their products are not used)
            for (int i = tid; i < n16 * 16 * T; i += kWarps * 32) {
                const int t = i & (T - 1), j = i / T;
                float z = 0.f;
                if (j < n && up) {
                    const int r = s_list[b0 + j];
                    if ((s_mask[r] >> t) & 1) {
                        float u = 0.f;
                        for (int s = 0; s < splits; ++s) u += part[((s * 8 + (j >> 4)) * 16 + (j & 15)) * T + t];
                        z = silu_f(sg[t * rp + r]) * u;
                    }
                }
                float left = z;
                const bool finite = fabsf(z) <= 3.4e38f;
#pragma unroll
                for (int k = 0; k < kParts; ++k) {
                    __nv_bfloat16 b = k + 1 < kParts ? __float2bfloat16_rz(left) : __float2bfloat16_rn(left);
                    left -= __bfloat162float(b);
                    // (of an infinite or NaN z the first part says so.  A part that is zero would make a product with an infinite
                    // weight NaN: the smallest number of z's sign instead)
                    if (k > 0 && !finite) b = __ushort_as_bfloat16(0);
                    if (k > 0 && z != 0.f && __bfloat162float(b) == 0.f) b = __ushort_as_bfloat16(z < 0.f ? 0x8001 : 0x0001);
                    zp[(k * kSlots + t) * zpitch + j] = b;
                }
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kWarps * 32) : "memory");
            const bool down = __all_sync(0xffffffffu, tc::mbar_wait(tc::smem_u32(&s_down), (uint32_t)turn & 1u, &s_abort, p.status));
            // 16 columns at a time are the rows of the product: transposed 8 x 8 blocks (columns + 8 in blocks 1 and 3, rows + 8 in 2
            // and 3); the parts of z are added up behind it
            const int right = (lane >> 3) & 1, row = (lane & 7) + ((lane >> 4) << 3);
#pragma unroll 1
            for (int col = warp * 16; col < d; col += kWarps * 16) {
                float acc[4] = {};
#pragma unroll 1
                for (int k = 0; k < n16; ++k) {
                    const uint32_t *zb = reinterpret_cast<const uint32_t *>(zp + lane_g * zpitch + k * 16) + lane_q;
                    const int r = k * 16 + row;
                    const uint32_t src = down && r < n && col + 8 * right < d ? down0 + (uint32_t)r * dpitch + (uint32_t)(col + 8 * right) * 2u
                                                                              : tc::smem_u32(&s_zero);
                    uint32_t a0, a1, a2, a3;
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3)
                                 : "r"(src)
                                 : "memory");
                    mma_16816(acc, a0, a1, a2, a3, zb[0], zb[4]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float v = lane_q < kParts ? acc[e] : 0.f;  // (part lane % 4 of token e % 2)
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    const int t = e & 1, c = col + lane_g + 8 * (e >> 1);
                    if (lane_q == 0 && t < T && c < d) s_out[t * d + c] = turn ? s_out[t * d + c] + v : v;
                }
                __syncwarp();
            }
        }
        __syncthreads();
    }

    // ---- output: the partial sums to the owners of their columns
    if (nsel == 0)
        for (int i = tid; i < T * d; i += kThreads) s_out[i] = 0.f;
    __syncthreads();
    const int own_vecs = p.own_vecs;
    if (!producer) {  // (a warp per owner)
        const uint32_t dst = tc::map_to_cta(tc::smem_u32(dsm + L.recv), (uint32_t)warp) + (uint32_t)((int)rank * T * own_vecs) * 32u;
        const int first = warp * own_vecs * 8, cols = min(own_vecs * 8, d - first);
#pragma unroll 1
        for (int t = 0; t < T; ++t)
            for (int c = lane * 4; c < cols; c += 128)
                store_cluster_v4(dst + (uint32_t)(t * own_vecs * 8 + c) * 4u, *reinterpret_cast<const uint4 *>(s_out + t * d + first + c));
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();  // #2 (and nobody touches another CTA's shared memory any more)
    {
        const float *recv = reinterpret_cast<const float *>(dsm + L.recv);
        const int cols = own_vecs * 8, first = (int)rank * cols;
#pragma unroll 1
        for (int t = 0; t < nt; ++t)
            for (int i = tid; i < cols && first + i < d; i += kThreads) {
                float sum = 0.f;
#pragma unroll
                for (int s = 0; s < kCluster; ++s) sum += recv[(s * T + t) * cols + i];
                const int64_t at = (int64_t)(t0 + t) * d + first + i;
                if (p.rms_w) sum += __bfloat162float(p.x[at]);  // the residual connection: out = h + D
                p.out[at] = __float2bfloat16_rn(sum);
            }
    }
    if (s_abort) {  // copies still in flight must land before shared memory goes away
        const long long begin = clock64();
        while (clock64() - begin < 2000000LL) __nanosleep(1000);
    }
}

}  // namespace dcl
}  // namespace moc
