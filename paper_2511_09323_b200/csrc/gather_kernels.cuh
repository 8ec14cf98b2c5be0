// Gathered (ALU) kernels of the MoC FFN: exact fp32-accumulate implementations of every step of
// the operator that touch only the selected channels.  They serve the fp32 storage type, shapes
// the tensor-core path does not take, and small batches, where reading only the K selected rows
// of W_up / W_down is the whole point (Section 5 of the paper).
//
// All weights are channel-major [F_ld, d]: a selected channel is one contiguous d-vector, read
// with 16-byte (bf16) / 32-byte (fp32) vector loads by consecutive threads.
#pragma once

#include "moc_common.cuh"
#include "topk_select.cuh"

namespace moc {

constexpr int kTokenThreads = 256;

// ------------------------------------------------------------------------------------------------
// Dense gate projection on the ALUs:  C[M,N] (fp32) = A[M,Kd] * B[N,Kd]^T, both operands K-major, Kd a multiple of 8.
// (Eq. (Moc-1), G = X W_gate.)  (BM / TM) x (BN / TN) threads, TM x TN outputs per thread.
//
// Large problems are bound by the FMA pipe if the operands come out of shared memory fast enough: 8 x 8 outputs read 64 bytes
// per 64 FMAs (with 4 x 4: 32 per 16).  The next slab is loaded to registers while one is multiplied and goes into the other
// buffer: one barrier per slab.  Small ones are bound by the chain of slabs, so they take small tiles (more CTAs) of long slabs.
// 4096 x 2048 x 768: one buffer, 4 x 4 outputs and scalar loads took 541 us (24 TFLOP/s), now 341 (38); 256 x 512 x 128
// 11.2 -> 5.3.
// Every output is one chain of FMAs in ascending k, whatever the tile.
template <typename T>
__device__ __forceinline__ float4 load4_f32(const T *p);
template <>
__device__ __forceinline__ float4 load4_f32<float>(const float *p) { return *reinterpret_cast<const float4 *>(p); }
template <>
__device__ __forceinline__ float4 load4_f32<__nv_bfloat16>(const __nv_bfloat16 *p) {
    const uint2 w = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xffff0000u));
}

template <typename T, int BM, int BN, int TM, int TN, int BK>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), 2) gemm_nt_alu_kernel(const T *__restrict__ A, const T *__restrict__ B,
                                                                           float *__restrict__ C, int M, int N, int Kd, int ldc) {
    constexpr int THREADS = (BM / TM) * (BN / TN), Q = BK / 4;  // Q: 4-element pieces of a row's slab
    constexpr int NA = BM * Q / THREADS, NB = BN * Q / THREADS;
    static_assert(BM * Q % THREADS == 0 && BN * Q % THREADS == 0 && TM % 4 == 0 && TN % 4 == 0, "tile");
    __shared__ __align__(16) float As[2][BK][BM + 4], Bs[2][BK][BN + 4];
    const int tid = threadIdx.x, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    // a thread's outputs: groups of four rows (columns) BM / (TM / 4) apart, so that a warp's reads do not collide
    constexpr int GM = BM / (TM / 4), GN = BN / (TN / 4);
    const int tx = tid % (BN / TN), ty = tid / (BN / TN);
    float acc[TM][TN] = {};
    float4 ra[NA], rb[NB];
    const auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int e = tid + i * THREADS, row = m0 + e / Q, k = k0 + e % Q * 4;
            ra[i] = row < M && k < Kd ? load4_f32<T>(A + (int64_t)row * Kd + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = tid + i * THREADS, row = n0 + e / Q, k = k0 + e % Q * 4;
            rb[i] = row < N && k < Kd ? load4_f32<T>(B + (int64_t)row * Kd + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    const auto put = [&](int buf) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int e = tid + i * THREADS, row = e / Q, k = e % Q * 4;
            As[buf][k][row] = ra[i].x;
            As[buf][k + 1][row] = ra[i].y;
            As[buf][k + 2][row] = ra[i].z;
            As[buf][k + 3][row] = ra[i].w;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = tid + i * THREADS, row = e / Q, k = e % Q * 4;
            Bs[buf][k][row] = rb[i].x;
            Bs[buf][k + 1][row] = rb[i].y;
            Bs[buf][k + 2][row] = rb[i].z;
            Bs[buf][k + 3][row] = rb[i].w;
        }
    };
    load(0);
    put(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < Kd; k0 += BK, buf ^= 1) {
        const bool more = k0 + BK < Kd;
        if (more) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; i += 4) *reinterpret_cast<float4 *>(&a[i]) = *reinterpret_cast<const float4 *>(&As[buf][kk][i / 4 * GM + ty * 4]);
#pragma unroll
            for (int j = 0; j < TN; j += 4) *reinterpret_cast<float4 *>(&b[j]) = *reinterpret_cast<const float4 *>(&Bs[buf][kk][j / 4 * GN + tx * 4]);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if (more) put(buf ^ 1);
        __syncthreads();
    }
    const bool vec = (ldc & 3) == 0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + i / 4 * GM + ty * 4 + i % 4;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            const int n = n0 + j / 4 * GN + tx * 4;
            float *c = C + (int64_t)m * ldc + n;
            if (vec && n + 4 <= N) {
                *reinterpret_cast<float4 *>(c) = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (n + e < N) c[e] = acc[i][j + e];
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Row selector fused with the gather of the gate values: one CTA per token of the chunk.
//   G [rows, ldg] fp32 (transient) -> idx [rows,K] int16 ascending, and optionally the saved gate
//   values topk_gate [rows,K] in the storage type.
template <typename T>
__global__ void __launch_bounds__(kSelectThreads) select_rows_kernel(const float *__restrict__ G, int64_t rows,
                                                                      int F, int ldg, int K,
                                                                      int16_t *__restrict__ idx_out,
                                                                      T *__restrict__ topk_gate, int post_silu) {
    extern __shared__ __align__(16) uint32_t select_keys[];
    __shared__ SelectSmem sm;
    SelectGuess guess;
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const float *g = G + r * (int64_t)ldg;
        uint32_t tau;
        int need;
        block_select_row<kSelectThreads>(g, F, K, select_keys, sm, guess, tau, need, post_silu != 0);
        int16_t *o = idx_out + r * (int64_t)K;
        T *og = topk_gate ? topk_gate + r * (int64_t)K : nullptr;
        block_ordered_emit<kSelectThreads>(select_keys, F, tau, need, sm, [&](int pos, int j) {
            o[pos] = (int16_t)j;
            // the value comes back from the key in shared memory: a global load inside the ordered walk
            // would cost a memory round trip per chunk
            // (keys of SiLU(g) do not give g back: the post-SiLU variant reads it)
            if (og) og[pos] = from_f32<T>(post_silu ? g[j] : key_to_float(select_keys[j]));
        });
        __syncthreads();
    }
}

// Accumulates  acc[v-th 8-vector] += sum_k coef[k] * W[rowidx[k], 8v..8v+7]  over the token's K rows,
// with the CTA's threads laid out as (row-group g) x (vector lane vl); partial sums of the groups
// are combined through shared memory.  Used by the down projection and by grad_x.
// red: shared scratch of at least THREADS/min(nvec,THREADS) * d floats when more than one group exists.
template <typename T, int NSRC, typename RowW, typename Coef>
__device__ __forceinline__ void token_row_combine(int d, int K, const int *rowidx, RowW roww, Coef coef,
                                                  float *red, T *__restrict__ dst) {
    const int tid = threadIdx.x;
    const int nvec = d >> 3;
    const int lanes_v = nvec < kTokenThreads ? nvec : kTokenThreads;
    const int G = kTokenThreads / lanes_v;
    const int g = tid / lanes_v, vl = tid % lanes_v;
    for (int v = vl; v < nvec; v += lanes_v) {
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (g < G) {
            // four rows' loads are in flight together (an L2 round trip per row otherwise); the sum stays in the order of k
            constexpr int ROWS = 4 / NSRC;
            for (int k0 = g; k0 < K; k0 += ROWS * G) {
                float w[ROWS][NSRC][8];
                int j[ROWS];
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    const int k = k0 + i * G;
                    j[i] = k < K ? rowidx[k] : -1;  // (negative: an invalid saved index, status already raised)
                    if (j[i] >= 0) {
#pragma unroll
                        for (int s = 0; s < NSRC; ++s) Vec8<T>::load(roww(s) + (int64_t)j[i] * d + 8 * v, w[i][s]);
                    }
                }
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    if (j[i] < 0) continue;
#pragma unroll
                    for (int s = 0; s < NSRC; ++s) {
                        const float c = coef(s, k0 + i * G);
#pragma unroll
                        for (int e = 0; e < 8; ++e) acc[e] = fmaf(c, w[i][s][e], acc[e]);
                    }
                }
            }
        }
        if (G == 1) {
            Vec8<T>::store(dst + 8 * v, acc);
        } else {
            // G > 1 only when nvec < THREADS, i.e. this loop body runs once per thread
            if (g < G) {
#pragma unroll
                for (int e = 0; e < 8; ++e) red[g * d + 8 * v + e] = acc[e];
            }
            __syncthreads();
            if (g == 0) {
                for (int gg = 1; gg < G; ++gg)
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[e] += red[gg * d + 8 * v + e];
                Vec8<T>::store(dst + 8 * v, acc);
            }
            __syncthreads();
        }
    }
}

// A warp's dot products of the vector in shared memory with DOT_ROWS rows k0, k0 + step, ... of W (negative index: none), their
// loads in flight together; the product of row i comes back in lane i.
// (100 tokens of 512 x 1365: step 168 -> 119 us with this, the rows taken together below and the gate projection; many tokens
// are bound by L2, 4096 of 768 x 2048 read 6.4 GB in 597 us.)
constexpr int DOT_ROWS = 4;
template <typename T>
__device__ __forceinline__ float warp_row_dots(const float *xs, const T *__restrict__ W, const int (&j)[DOT_ROWS], int d) {
    const int lane = threadIdx.x & 31;
    float acc[DOT_ROWS] = {};
    for (int v = lane; v < (d >> 3); v += 32) {
        float w[DOT_ROWS][8];
#pragma unroll
        for (int i = 0; i < DOT_ROWS; ++i)
            if (j[i] >= 0) Vec8<T>::load(W + (int64_t)j[i] * d + 8 * v, w[i]);
#pragma unroll
        for (int i = 0; i < DOT_ROWS; ++i)
            if (j[i] >= 0) {
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[i] = fmaf(xs[8 * v + e], w[i][e], acc[i]);
            }
    }
    float mine = 0.f;
#pragma unroll
    for (int i = 0; i < DOT_ROWS; ++i) {
        const float s = warp_sum(acc[i]);
        if (lane == i) mine = s;
    }
    return mine;
}

// ------------------------------------------------------------------------------------------------
// Forward, per token (grid.x = tokens of the chunk):
//   u_k = x . W_up[idx_k,:]        (Eq. (Moc-1) on the mask only)
//   z_k = SiLU(g_k) * u_k          (Eq. (MoC-2))
//   out = sum_k z_k W_down[idx_k,:]
// gate values come from the transient fp32 gate projection G (unrounded).
// Dynamic shared memory: d floats (x) + K floats (z) + K ints (idx) + reduction scratch.
template <typename T>
__global__ void __launch_bounds__(kTokenThreads) forward_token_kernel(
    const T *__restrict__ x, const T *__restrict__ w_up, const T *__restrict__ w_down,
    const float *__restrict__ G, int ldg, const int16_t *__restrict__ idx, int d, int K, T *__restrict__ out,
    T *__restrict__ topk_up, int red_floats) {
    extern __shared__ __align__(16) float fsm[];
    float *xs = fsm;
    float *zs = xs + d;
    int *js = reinterpret_cast<int *>(zs + K);
    float *red = reinterpret_cast<float *>(js + K);
    (void)red_floats;
    const int64_t t = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T *xt = x + t * d;
    for (int v = tid; v < (d >> 3); v += kTokenThreads) {
        float f[8];
        Vec8<T>::load(xt + 8 * v, f);
#pragma unroll
        for (int e = 0; e < 8; ++e) xs[8 * v + e] = f[e];
    }
    for (int k = tid; k < K; k += kTokenThreads) js[k] = idx[t * K + k];
    __syncthreads();
    const float *gt = G + t * (int64_t)ldg;
    constexpr int NW = kTokenThreads / 32;
    for (int k0 = warp; k0 < K; k0 += DOT_ROWS * NW) {
        int j[DOT_ROWS];
#pragma unroll
        for (int i = 0; i < DOT_ROWS; ++i) j[i] = k0 + i * NW < K ? js[k0 + i * NW] : -1;
        const int k = k0 + lane * NW;
        const bool mine = lane < DOT_ROWS && k < K;
        const float g = mine ? gt[js[k]] : 0.f;  // (its load is in flight beside the rows')
        const float u = warp_row_dots<T>(xs, w_up, j, d);
        if (mine) {
            zs[k] = silu_f(g) * u;
            if (topk_up) topk_up[t * K + k] = from_f32<T>(u);
        }
    }
    __syncthreads();
    token_row_combine<T, 1>(
        d, K, js, [&](int) { return w_down; }, [&](int, int k) { return zs[k]; }, red, out + t * d);
}

// ------------------------------------------------------------------------------------------------
// Backward, per token (grid.x = tokens):  Eqs. (bp-1)..(bp-3) on the mask and Eq. (bp-5).
//   dz_k = grad_out . W_down[idx_k,:];  s = SiLU(g);  z = s u;  dU = s dz;  dG = u dz SiLU'(g)
//   grad_x = sum_k dG_k W_gate[idx_k,:] + dU_k W_up[idx_k,:]
// The compact coefficients z, dU, dG go to coef [3, T*K] fp32 for the weight-gradient kernels.
template <typename T>
__global__ void __launch_bounds__(kTokenThreads) backward_token_kernel(
    const T *__restrict__ w_gate, const T *__restrict__ w_up, const T *__restrict__ w_down,
    const int16_t *__restrict__ idx, const T *__restrict__ topk_gate, const T *__restrict__ topk_up,
    const T *__restrict__ grad_out, int d, int F, int K, int64_t TK, T *__restrict__ grad_x,
    float *__restrict__ coef, int *__restrict__ status) {
    extern __shared__ __align__(16) float fsm[];
    float *ds = fsm;
    float *dgs = ds + d;
    float *dus = dgs + K;
    int *js = reinterpret_cast<int *>(dus + K);
    float *red = reinterpret_cast<float *>(js + K);
    const int64_t t = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T *dt = grad_out + t * d;
    for (int v = tid; v < (d >> 3); v += kTokenThreads) {
        float f[8];
        Vec8<T>::load(dt + 8 * v, f);
#pragma unroll
        for (int e = 0; e < 8; ++e) ds[8 * v + e] = f[e];
    }
    for (int k = tid; k < K; k += kTokenThreads) {
        int j = idx[t * K + k];
        if (j < 0 || j >= F) {
            raise_status(status, MOC_ERR_BAD_INDEX);
            j = -1;
        }
        js[k] = j;
    }
    __syncthreads();
    constexpr int NW = kTokenThreads / 32;
    for (int k0 = warp; k0 < K; k0 += DOT_ROWS * NW) {
        int j[DOT_ROWS];
#pragma unroll
        for (int i = 0; i < DOT_ROWS; ++i) j[i] = k0 + i * NW < K ? js[k0 + i * NW] : -1;
        const int k = k0 + lane * NW;
        const bool mine = lane < DOT_ROWS && k < K;
        const float g = mine ? to_f32<T>(topk_gate[t * K + k]) : 0.f, u = mine ? to_f32<T>(topk_up[t * K + k]) : 0.f;
        const float dz = warp_row_dots<T>(ds, w_down, j, d);
        if (mine) {
            float z = 0.f, dU = 0.f, dG = 0.f;
            if (js[k] >= 0) {
                const float s = silu_f(g);
                z = s * u;
                dU = s * dz;
                dG = u * dz * dsilu_f(g);
            }
            dgs[k] = dG;
            dus[k] = dU;
            if (coef) {
                coef[t * K + k] = z;
                coef[TK + t * K + k] = dU;
                coef[2 * TK + t * K + k] = dG;
            }
        }
    }
    __syncthreads();
    if (grad_x) {
        token_row_combine<T, 2>(
            d, K, js, [&](int s) { return s == 0 ? w_gate : w_up; },
            [&](int s, int k) { return s == 0 ? dgs[k] : dus[k]; }, red, grad_x + t * d);
    }
}

// ------------------------------------------------------------------------------------------------
// Per-channel token lists (a CSR transpose of idx), built deterministically so that every weight
// gradient row is a sum over its tokens in ascending token order.
//   counts [nb, F]  : per token-block, per channel occurrence counts, then exclusive offsets
//   row_start [F+1] : list start of each channel
//   pairs [T*K]     : pair id p = t*K + k, grouped by channel, tokens ascending
// Token block b covers tokens [b*tb, min(T,(b+1)*tb)).
__global__ void __launch_bounds__(256) csr_count_kernel(const int16_t *__restrict__ idx, int64_t T, int K, int F,
                                                        int tb, uint32_t *__restrict__ counts, unsigned int *done) {
    extern __shared__ __align__(16) uint32_t cnt[];
    if (blockIdx.x == 0 && threadIdx.x == 0) *done = 0;
    for (int j = threadIdx.x; j < F; j += 256) cnt[j] = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * tb;
    const int64_t t1 = t0 + tb < T ? t0 + tb : T;
    const int64_t e0 = t0 * K, e1 = t1 * K;
    for (int64_t e = e0 + threadIdx.x; e < e1; e += 256) {
        const int j = idx[e];
        if (j >= 0 && j < F) atomicAdd(&cnt[j], 1u);
    }
    __syncthreads();
    uint32_t *o = counts + (int64_t)blockIdx.x * F;
    for (int j = threadIdx.x; j < F; j += 256) o[j] = cnt[j];
}

// A CTA for 32 channels: exclusive prefix over the token blocks, a warp for each 32nd of them (the loads of a channel's counts
// one after the other took 66 us for 512 blocks); totals[j] = list length.  The last CTA to finish scans the totals:
// row_start[F + 1].  done: zeroed by csr_count_kernel.
__global__ void __launch_bounds__(1024) csr_scan_kernel(uint32_t *__restrict__ counts, int nb, int F, uint32_t *totals,
                                                        uint32_t *__restrict__ row_start, unsigned int *done) {
    __shared__ uint32_t part[32][33];
    __shared__ uint32_t wtot[32];
    __shared__ uint32_t carry;
    __shared__ unsigned int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = blockIdx.x * 32 + lane, per = (nb + 31) / 32;
    const int b0 = min(warp * per, nb), b1 = min(b0 + per, nb);
    uint32_t sum = 0;
    if (j0 < F) {
        const uint32_t *c = counts + j0;
#pragma unroll 8
        for (int b = b0; b < b1; ++b) sum += c[(int64_t)b * F];
    }
    part[warp][lane] = sum;
    __syncthreads();
    uint32_t run = 0;
    for (int w = 0; w < warp; ++w) run += part[w][lane];
    if (j0 < F) {
        uint32_t *c = counts + j0;
        for (int b = b0; b < b1; b += 8) {
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = b + i < b1 ? c[(int64_t)(b + i) * F] : 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (b + i < b1) c[(int64_t)(b + i) * F] = run;
                run += v[i];
            }
        }
        if (warp == 31) __stcg(&totals[j0], run);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        s_last = atomicAdd(done, 1u) == gridDim.x - 1 ? 1u : 0u;
        carry = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int base = 0; base < F; base += 1024) {
        const int j = base + tid;
        const uint32_t v = j < F ? __ldcg(&totals[j]) : 0u;
        uint32_t s = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t n = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += n;
        }
        if (lane == 31) wtot[warp] = s;
        __syncthreads();
        uint32_t before = carry;
        for (int w = 0; w < warp; ++w) before += wtot[w];
        if (j < F) row_start[j] = before + s - v;
        __syncthreads();
        if (tid == 1023) carry = before + s;
        __syncthreads();
    }
    if (tid == 0) row_start[F] = carry;
}

__global__ void __launch_bounds__(256) csr_fill_kernel(const int16_t *__restrict__ idx, int64_t T, int K, int F,
                                                       int tb, const uint32_t *__restrict__ counts,
                                                       const uint32_t *__restrict__ row_start,
                                                       uint32_t *__restrict__ pairs) {
    extern __shared__ __align__(16) uint32_t cursor[];
    const uint32_t *c = counts + (int64_t)blockIdx.x * F;
    for (int j = threadIdx.x; j < F; j += 256) cursor[j] = row_start[j] + c[j];
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * tb;
    const int64_t t1 = t0 + tb < T ? t0 + tb : T;
    for (int64_t t = t0; t < t1; ++t) {
        // channels of one token are distinct, so the order inside a list is the token order
        for (int k = threadIdx.x; k < K; k += 256) {
            const int j = idx[t * K + k];
            if (j >= 0 && j < F) {
                const uint32_t pos = atomicAdd(&cursor[j], 1u);
                pairs[pos] = (uint32_t)(t * K + k);
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------------
// Weight gradients, one CTA per channel row j (Eqs. (bp-1) and (bp-4) restricted to the mask):
//   grad_w_down[j,:] = sum_p z_p  * grad_out[t_p,:]
//   grad_w_up  [j,:] = sum_p dU_p * x[t_p,:]
//   grad_w_gate[j,:] = sum_p dG_p * x[t_p,:]          p over the channel's (token, slot) pairs
// Rows no token selected (and padding rows) are written as exact zeros.
//
// FIND: every CTA finds its channel's pairs in idx itself (list_scans_pay: while all CTAs together read little), and no lists are
// built.  256 tokens, K = 64, 512 channels: 512 x 32 KiB out of L2, and three launches fewer in front of 11 us of work
// (step 95.8 -> 88; 100 tokens of 512 x 1365: 116 -> 108).
constexpr int kFindTokens = 4096;
constexpr int64_t kFindBytes = 64 << 20;  // some 8 us of L2 reads, against the 16 or more of the kernels that build the lists
inline bool list_scans_pay(int64_t tokens, int K, int rows) {
    return tokens <= kFindTokens && tokens * K * 2 * rows <= kFindBytes;
}
// list[0..n) = the pairs of channel j, tokens ascending; slot: scratch, one entry per token.  Returns n.
__device__ __forceinline__ int find_pairs(const int16_t *__restrict__ idx, int tokens, int K, int j, int16_t *slot, uint32_t *list) {
    __shared__ int s_warp[kTokenThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, TK = tokens * K;
    for (int t = tid; t < tokens; t += kTokenThreads) slot[t] = -1;
    __syncthreads();
    // (channels of one token are distinct: at most one match each)
    const auto check = [&](int e, int v) {
        if (v == j) slot[e / K] = (int16_t)(e % K);
    };
    const int whole = (reinterpret_cast<uintptr_t>(idx) & 15u) == 0 ? TK / 8 : 0;
#pragma unroll 4
    for (int q = tid; q < whole; q += kTokenThreads) {
        const uint4 v = reinterpret_cast<const uint4 *>(idx)[q];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            check(8 * q + 2 * i, (int)(int16_t)(w[i] & 0xffffu));
            check(8 * q + 2 * i + 1, (int)(int16_t)(w[i] >> 16));
        }
    }
#pragma unroll 4
    for (int e = 8 * whole + tid; e < TK; e += kTokenThreads) check(e, idx[e]);
    __syncthreads();
    int n = 0;
    for (int base = 0; base < tokens; base += kTokenThreads) {
        const int t = base + tid, k = t < tokens ? slot[t] : -1;
        const uint32_t hits = __ballot_sync(0xffffffffu, k >= 0);
        if (lane == 0) s_warp[warp] = __popc(hits);
        __syncthreads();
        int at = n;
        for (int w = 0; w < kTokenThreads / 32; ++w) {
            if (w < warp) at += s_warp[w];
            n += s_warp[w];
        }
        if (k >= 0) list[at + __popc(hits & ((1u << lane) - 1u))] = (uint32_t)(t * K + k);
        __syncthreads();
    }
    return n;
}

template <typename T, bool FIND>
__global__ void __launch_bounds__(kTokenThreads) wgrad_rows_kernel(
    const T *__restrict__ x, const T *__restrict__ grad_out, const float *__restrict__ coef, int64_t TK,
    const uint32_t *__restrict__ row_start, const uint32_t *__restrict__ pairs, const int16_t *__restrict__ idx, int tokens, int d,
    int F, int K, T *__restrict__ gw_gate, T *__restrict__ gw_up, T *__restrict__ gw_down, int accumulate) {
    extern __shared__ __align__(16) float red[];  // [G][3][d] when G > 1; FIND: the list and the slots behind it
    const int j = blockIdx.x;
    const int tid = threadIdx.x;
    const int nvec = d >> 3;
    const int lanes_v = nvec < kTokenThreads ? nvec : kTokenThreads;
    const int G = kTokenThreads / lanes_v;
    const int g = tid / lanes_v, vl = tid % lanes_v;
    uint32_t p0 = 0, p1 = 0;
    if constexpr (FIND) {
        uint32_t *list = reinterpret_cast<uint32_t *>(red + (G > 1 ? 3 * G * d : 0));
        if (j < F) p1 = (uint32_t)find_pairs(idx, tokens, K, j, reinterpret_cast<int16_t *>(list + tokens), list);
        pairs = list;
    } else if (j < F) {
        p0 = row_start[j];
        p1 = row_start[j + 1];
    }
    for (int v = vl; v < nvec; v += lanes_v) {
        float a_dn[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        float a_up[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        float a_gt[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (g < G) {
            for (uint32_t q = p0 + g; q < p1; q += G) {
                const uint32_t p = pairs[q];
                const int64_t t = p / (uint32_t)K;
                float xv[8], dv[8];
                if (gw_down) {
                    Vec8<T>::load(grad_out + t * d + 8 * v, dv);
                    const float z = coef[p];
#pragma unroll
                    for (int e = 0; e < 8; ++e) a_dn[e] = fmaf(z, dv[e], a_dn[e]);
                }
                if (gw_up || gw_gate) {
                    Vec8<T>::load(x + t * d + 8 * v, xv);
                    const float dU = coef[TK + p], dG = coef[2 * TK + p];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        a_up[e] = fmaf(dU, xv[e], a_up[e]);
                        a_gt[e] = fmaf(dG, xv[e], a_gt[e]);
                    }
                }
            }
        }
        if (G > 1) {
            if (g < G) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    red[(g * 3 + 0) * d + 8 * v + e] = a_dn[e];
                    red[(g * 3 + 1) * d + 8 * v + e] = a_up[e];
                    red[(g * 3 + 2) * d + 8 * v + e] = a_gt[e];
                }
            }
            __syncthreads();
            if (g == 0) {
                for (int gg = 1; gg < G; ++gg)
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        a_dn[e] += red[(gg * 3 + 0) * d + 8 * v + e];
                        a_up[e] += red[(gg * 3 + 1) * d + 8 * v + e];
                        a_gt[e] += red[(gg * 3 + 2) * d + 8 * v + e];
                    }
            }
        }
        if (g == 0) {
            const int64_t o = (int64_t)j * d + 8 * v;
            T *dst[3] = {gw_down, gw_up, gw_gate};
            float *src[3] = {a_dn, a_up, a_gt};
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                if (!dst[s]) continue;
                float r[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) r[e] = src[s][e];
                if (accumulate) {
                    float old[8];
                    Vec8<T>::load(dst[s] + o, old);
#pragma unroll
                    for (int e = 0; e < 8; ++e) r[e] += old[e];
                }
                Vec8<T>::store(dst[s] + o, r);
            }
        }
        if (G > 1) __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------- up values again
// topk_up[t, k] = U[t, idx[t, k]] from a dense U [T, ldu] (the tensor-core plan recomputes U with its GEMM), or, with
// U == nullptr, the dot product x[t, :] . w_up[idx[t, k], :] itself in fp32 (one warp per kept channel).
// An index outside [0, F) is skipped (its output is set to zero) and reported.
template <typename T>
__global__ void __launch_bounds__(256) recompute_up_kernel(const T *__restrict__ x, const T *__restrict__ w_up,
                                                           const __nv_bfloat16 *__restrict__ U, int ldu,
                                                           const int16_t *__restrict__ idx, int64_t tokens, int K, int F,
                                                           int d, T *__restrict__ up_out, int *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int64_t total = tokens * K;
    if (U) {
        for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < total; i += (int64_t)gridDim.x * 256) {
            const int64_t t = i / K;
            const int j = idx[i];
            if (j < 0 || j >= F) {
                raise_status(status, MOC_ERR_BAD_INDEX);
                up_out[i] = from_f32<T>(0.f);
            } else {
                up_out[i] = from_f32<T>(__bfloat162float(U[t * ldu + j]));
            }
        }
        return;
    }
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); i < total; i += warps) {
        const int64_t t = i / K;
        const int j = idx[i];
        if (j < 0 || j >= F) {
            if (lane == 0) {
                raise_status(status, MOC_ERR_BAD_INDEX);
                up_out[i] = from_f32<T>(0.f);
            }
            continue;
        }
        const T *xr = x + t * d, *wr = w_up + (int64_t)j * d;
        float sum = 0.f;
        for (int c = lane * 8; c < d; c += 256) {
            float a[8], b[8];
            Vec8<T>::load(xr + c, a);
            Vec8<T>::load(wr + c, b);
#pragma unroll
            for (int e = 0; e < 8; ++e) sum = fmaf(a[e], b[e], sum);
        }
        sum = warp_sum(sum);
        if (lane == 0) up_out[i] = from_f32<T>(sum);
    }
}

}  // namespace moc
