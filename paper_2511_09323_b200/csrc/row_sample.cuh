// Backward element-wise step (Eqs. (bp-1)..(bp-3) on the mask, with S' and Z' recomputed from the saved values), a team of W
// warps per token:
//   dz = dZ[t, j] for each saved channel j, s = SiLU(g), z = s u, dU = s dz, dG = u dz SiLU'(g);
// the dZ row is overwritten IN PLACE by the masked Z', dU' and dG' rows are written masked (zeros elsewhere).  A saved index
// outside [0, F) is skipped and raises MOC_ERR_BAD_INDEX.
//
// What bounds it: 8 bytes per channel (dZ in, three rows out) and 6 per saved entry.  The rows are staged in shared memory:
// dZ and the saved entries arrive by bulk copies, the three masked rows are built in zeroed buffers and leave as bulk
// stores, so all global traffic is coalesced and the scattered accesses stay on chip.  An entry is read, worked on and
// scattered in one go (three barriers a token); shared memory bounds the tokens in flight, four at 5504 channels, so the
// teams grow with the row.  With two warps a token and a list of entries between two passes: 16384 x 5504, K = 1376,
// 250 us, now
// 176; 65536 x 5504, K = 688, 711 us, now 540 (440 at the copy rate).
#pragma once

#include "tc_gemm.cuh"

namespace moc {
namespace rs {

struct SampleLayout {
    uint32_t z, du, dg, saved, bar, total;  // byte offsets (the dZ row is at 0); saved: idx | g | u, K8 entries each
};
__host__ __device__ inline SampleLayout sample_layout(int ld, int K) {
    SampleLayout L{};
    const uint32_t row = (uint32_t)ld * 2u;
    L.z = row;
    L.du = 2 * row;
    L.dg = 3 * row;
    L.saved = 4 * row;
    L.bar = L.saved + 3u * 2u * (((uint32_t)K + 7u) & ~7u);
    L.total = L.bar + 16u;
    return L;
}
constexpr int sample_warps(int F) { return F <= 1024 ? 1 : F <= 3072 ? 2 : F <= 8192 ? 4 : 8; }

template <int W>
__global__ void __launch_bounds__(32 * W) sample_rows_kernel(const int16_t *idx_in, const __nv_bfloat16 *gval_in,
                                                            const __nv_bfloat16 *uval_in, int64_t T, int K, int F, int ld,
                                                            __nv_bfloat16 *__restrict__ dz_z, __nv_bfloat16 *__restrict__ du,
                                                            __nv_bfloat16 *__restrict__ dg, int *__restrict__ status) {
    using namespace tc;
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ int s_abort;
    pdl_wait();
    const int16_t *const idx = after_pdl_wait(idx_in);
    const __nv_bfloat16 *const gval = after_pdl_wait(gval_in), *const uval = after_pdl_wait(uval_in);
    constexpr int TT = 32 * W;
    const SampleLayout L = sample_layout(ld, K);
    const int tid = threadIdx.x, K8 = (K + 7) & ~7;
    const __nv_bfloat16 *sdz = reinterpret_cast<const __nv_bfloat16 *>(smem);
    __nv_bfloat16 *sz = reinterpret_cast<__nv_bfloat16 *>(smem + L.z), *su = reinterpret_cast<__nv_bfloat16 *>(smem + L.du),
                  *sg = reinterpret_cast<__nv_bfloat16 *>(smem + L.dg);
    const uint16_t *saved = reinterpret_cast<const uint16_t *>(smem + L.saved);
    const uint32_t bar = smem_u32(smem + L.bar), row_bytes = (uint32_t)ld * 2u, saved_bytes = (uint32_t)K * 2u;
    const bool staged = (K & 7) == 0;  // the saved rows are multiples of 16 bytes: bulk copies (else plain loads)
    auto sync = [&]() {
        if (W == 1) __syncwarp();
        else __syncthreads();
    };
    auto request = [&](int64_t t) {  // (one thread)
        mbar_expect_tx(bar, row_bytes + (staged ? 3u * saved_bytes : 0u));
        bulk_copy_g2s(smem_u32(smem), dz_z + t * (int64_t)ld, row_bytes, bar);
        if (staged) {
            const uint32_t s = smem_u32(saved);
            bulk_copy_g2s(s, idx + t * K, saved_bytes, bar);
            bulk_copy_g2s(s + 2u * K8, gval + t * K, saved_bytes, bar);
            bulk_copy_g2s(s + 4u * K8, uval + t * K, saved_bytes, bar);
        }
    };
    auto entry = [&](int j, __nv_bfloat16 gb, __nv_bfloat16 ub) {
        if (j < 0 || j >= F) {
            raise_status(status, MOC_ERR_BAD_INDEX);
            return;
        }
        const float dz = __bfloat162float(sdz[j]), g = __bfloat162float(gb), u = __bfloat162float(ub), s = silu_f(g);
        sz[j] = __float2bfloat16_rn(s * u);
        su[j] = __float2bfloat16_rn(s * dz);
        sg[j] = __float2bfloat16_rn(u * dz * dsilu_f(g));
    };

    // the last tokens first: the GEMM that wrote dZ ended with them
    const int64_t t0 = T - 1 - (int64_t)blockIdx.x;
    if (t0 < 0) return;
    if (tid == 0) {
        s_abort = 0;
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        request(t0);
    }
    uint32_t phase = 0;
    for (int64_t t = t0; t >= 0; t -= gridDim.x) {
        if (tid == 0) bulk_store_wait_read<0>();  // the previous token's rows have left shared memory
        sync();
        {
            uint4 *rows = reinterpret_cast<uint4 *>(smem + L.z);  // the three rows lie one behind the other
            const uint4 zero = make_uint4(0, 0, 0, 0);
            for (int v = tid; v < 3 * (ld >> 3); v += TT) rows[v] = zero;
        }
        // a wait that gave up ends the team
        const bool ok = mbar_wait(bar, phase, &s_abort, status);
        const bool dead = W == 1 ? __any_sync(0xffffffffu, !ok) : __syncthreads_or(!ok ? 1 : 0) != 0;
        if (W == 1) __syncwarp();
        if (dead) break;
        phase ^= 1u;
        if (staged) {
            const uint32_t *si = reinterpret_cast<const uint32_t *>(saved);
            const __nv_bfloat162 *sgv = reinterpret_cast<const __nv_bfloat162 *>(saved + K8), *suv = reinterpret_cast<const __nv_bfloat162 *>(saved + 2 * K8);
#pragma unroll 2
            for (int i = tid; i < (K >> 1); i += TT) {
                const uint32_t j = si[i];
                const __nv_bfloat162 g = sgv[i], u = suv[i];
                entry((int16_t)(j & 0xffffu), g.x, u.x);
                entry((int16_t)(j >> 16), g.y, u.y);
            }
        } else {
            for (int k = tid; k < K; k += TT) entry(idx[t * K + k], gval[t * K + k], uval[t * K + k]);
        }
        fence_async_smem();
        sync();
        if (tid == 0) {
            bulk_copy_s2g(dz_z + t * (int64_t)ld, smem_u32(sz), row_bytes);
            bulk_copy_s2g(du + t * (int64_t)ld, smem_u32(su), row_bytes);
            bulk_copy_s2g(dg + t * (int64_t)ld, smem_u32(sg), row_bytes);
            if (t - gridDim.x >= 0) request(t - gridDim.x);
        }
    }
    if (tid == 0) bulk_store_wait_all();  // shared memory must outlive the stores that read it
    if (s_abort) {                        // ... and the copies into it that a wait gave up on
        const long long c0 = clock64();
        while (clock64() - c0 < 2000000LL) __nanosleep(1000);
    }
}

}  // namespace rs
}  // namespace moc
