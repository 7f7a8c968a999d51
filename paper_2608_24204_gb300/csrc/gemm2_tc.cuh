// Prefill GEMM on pairs of SMs (tcgen05 cta_group::2), for chunks with tiles enough
// for every pair.
//
// gemm_tc.cuh's kernel on 128 x BN tiles is bound by shared-memory ports, not by the
// tensor cores: per k-block it writes the activation terms and the weight rows once
// and every MMA reads both operands again, 1157 cycles for 128 x 192 x 64 with two
// terms where the MMAs take 768 (115 to 120 bytes a cycle).  A pair shares one
// 256 x BN tile: each CTA holds its own 128 rows of A and half of the weight rows, and
// the tensor cores of both read the halves of B from both shared memories, so the
// weight bytes written and read per FLOP halve.  Numerics, pipeline, roles and epilogues are
// those of gemm_tc.cuh: the products of an MMA and their order of accumulation in a
// group of k-blocks are the same, so the results are bit for bit the same.
//
// Roles per CTA: warp 0 loads this CTA's rows of A and its half of B and signals the
// leader's (rank 0) "full" barrier, whose expected bytes count both CTAs; warp 1
// allocates TMEM and, in the leader, issues the MMAs of the pair; each commit arrives at
// the "empty" (or "accumulator full") barriers of both CTAs; warps 2..9 fold and
// store this CTA's 128 rows and free the accumulator at the leader.
//
// Measured, 2048 tokens at 8B widths, one CTA per tile and pairs: gate/up 602 and 532 us a
// layer (962 GFLOP of MMAs: 1.8 PFLOP/s), QKV 242 and 215, O 103 and 100, down 286 and 270.
#pragma once
#include "gemm_tc.cuh"

namespace wici {

// geometry of a pair's 256 x BN tile, per CTA
template <int BN, int AT>
struct TcPairTile {
    static_assert(BN % 32 == 0 && BN <= 256, "BN: a multiple of 32 up to 256");
    static constexpr uint32_t B_BYTES = BN / 2 * TC_BK * 2;                // half of the weight rows
    static constexpr uint32_t STAGE_BYTES = AT * TC_A_BYTES + B_BYTES;
    static constexpr int STAGES = (int)(TC_SMEM_BUDGET / STAGE_BYTES);
    static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024;
    static constexpr int EPI_COLS = BN / 2;                                // columns per epilogue warp
    static constexpr uint32_t ACC_STRIDE = TC_TMEM_COLS / 2;
    static_assert(STAGES >= 3 && STAGE_BYTES % 1024 == 0, "ring stages");
};

__host__ __device__ constexpr uint32_t tc_pair_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(2 * TC_BM >> 4) << 24);
}

// a box into this CTA's shared memory, its bytes counted on the barrier of the pair's
// leader (the CTA-rank bit of a shared::cluster address cleared)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
        "%3}], [%4];" ::"r"(dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar & 0xFEFFFFFFu)
        : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrives at the barrier at this address in both CTAs when the MMAs issued so far are done
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .u32 ra;\n\tmapa.shared::cluster.u32 ra, %0, 0;\n\t"
        "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}" ::"r"(bar)
        : "memory");
}

template <int BN, int WT, class Epi>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, 1)
    gemm2_tc_kernel(const __grid_constant__ GemmMaps maps, int T, int N, int K, int *err, const Epi epi) {
    static_assert(WT == 1 || WT == kTerms, "one exact bf16 weight term, or three");
    constexpr int AT = Epi::kATerms;
    constexpr int WU = WT == 1 ? 1 : AT;
    using G = TcPairTile<BN, AT>;
    constexpr int S = G::STAGES;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], acc_full[2], acc_free[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_issued;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)blockIdx.x & 1;
    const int ntm = (T + 2 * TC_BM - 1) / (2 * TC_BM), ntn = (N + BN - 1) / BN;
    const int ntiles = ntm * ntn;
    const int tile0 = (int)blockIdx.x >> 1, tile_step = (int)gridDim.x >> 1;
    const int nk = (K + TC_BK - 1) / TC_BK, nkk = nk * WU;
    const int ngroups = (nkk + TC_GROUP - 1) / TC_GROUP;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_free[b]), 2 * TC_EPI_WARPS);
        }
        fence_barrier_init();
        s_issued = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // both CTAs' barriers and tensor memory are ready
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    griddep_launch_dependents();
    if (warp != 0) griddep_wait();   // warp 0 waits behind its first weight copies

    if (warp == 0) {
        if (lane == 0) {  // ------------------------------------------- TMA producer
            int it = 0;
            bool ok = true;
            // as in gemm_tc_kernel: the first bf16 weight copies precede the wait
            const int early = WT == 1 && tile0 < ntiles ? min(S, nkk) : 0;
            for (int s = 0; s < early; ++s) {
                const uint32_t fb = smem_u32(&full_bar[s]);
                if (rank == 0) mbar_arrive_expect_tx(fb, 2u * (AT * TC_A_BYTES + G::B_BYTES));
                tma_load_2d_pair(base + (uint32_t)s * G::STAGE_BYTES + AT * TC_A_BYTES, &maps.w[0], s * TC_BK,
                                 (tile0 / ntm) * BN + rank * (BN / 2), fb);
            }
            griddep_wait();
            for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
                const int m0 = (tile % ntm) * 2 * TC_BM + rank * TC_BM, n0 = (tile / ntm) * BN + rank * (BN / 2);
                for (int kk = 0; kk < nkk; ++kk, ++it) {
                    const int s = it % S;
                    if (it >= S && !(ok = mbar_wait(smem_u32(&empty_bar[s]), ((it / S) + 1) & 1, err, SITE_TC_EMPTY)))
                        break;
                    const int j = WT == 1 ? 0 : kk / nk, kb = kk - j * nk;     // weight term, k-block
                    const uint32_t st = base + (uint32_t)s * G::STAGE_BYTES;
                    const uint32_t fb = smem_u32(&full_bar[s]);
                    const int na = AT - j;   // term j meets the activation terms i < AT - j only
                    if (rank == 0) {
                        if (it >= early) mbar_arrive_expect_tx(fb, 2u * ((uint32_t)na * TC_A_BYTES + G::B_BYTES));
                        s_issued = it + 1;
                    }
#pragma unroll
                    for (int t = 0; t < AT; ++t)
                        if (t < na) tma_load_2d_pair(st + t * TC_A_BYTES, &maps.a[t], kb * TC_BK, m0, fb);
                    if (it >= early) tma_load_2d_pair(st + AT * TC_A_BYTES, &maps.w[j], kb * TC_BK, n0, fb);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {  // ------------------------------- MMA issuer of the pair
            constexpr uint32_t idesc = tc_pair_idesc(BN);
            bool ok = true;
            int it = 0, gg = 0;
            for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
                for (int gi = 0; gi < ngroups && ok; ++gi, ++gg) {
                    const int b = gg & 1;
                    if (gg >= 2 && !(ok = mbar_wait(smem_u32(&acc_free[b]), ((gg / 2) + 1) & 1, err, SITE_TC_FREE)))
                        break;
                    tc_fence_after();
                    const uint32_t acc = tmem + (uint32_t)b * G::ACC_STRIDE;
                    const int kk0 = gi * TC_GROUP, kk1 = min(nkk, kk0 + TC_GROUP);
                    for (int kk = kk0; kk < kk1; ++kk, ++it) {
                        const int s = it % S;
                        ok = mbar_wait(smem_u32(&full_bar[s]), (it / S) & 1, err, SITE_TC_FULL);
                        if (!ok) break;
                        tc_fence_after();
                        const int nt = WT == 1 ? AT : AT - kk / nk;
                        const uint32_t st = base + (uint32_t)s * G::STAGE_BYTES;
                        const uint64_t bd0 = tc_desc_sw128(st + AT * TC_A_BYTES);
                        const uint64_t ad0 = tc_desc_sw128(st);
#pragma unroll
                        for (int k = 0; k < TC_BK / 16; ++k)
#pragma unroll
                            for (int t = 0; t < AT; ++t)
                                if (t < nt)
                                    tc_mma_pair(acc, ad0 + (uint64_t)((t * TC_A_BYTES + 32 * k) >> 4),
                                                bd0 + (uint64_t)(2 * k), idesc, (kk != kk0 || k != 0 || t != 0));
                        tc_commit_pair(smem_u32(&empty_bar[s]));
                    }
                    if (ok) tc_commit_pair(smem_u32(&acc_full[b]));
                }
            }
        }
    } else {  // ------------------------------------------------------- epilogue
        const int q = warp & 3;                          // TMEM lane quadrant of this warp
        const int half = (warp - 2) >> 2;                // which half of the tile's columns
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        bool ok = true;
        int gg = 0;
        for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
            const int m0 = (tile % ntm) * 2 * TC_BM + rank * TC_BM, n0 = (tile / ntm) * BN;
            const int t = m0 + q * 32 + lane;
            float sum[G::EPI_COLS];
#pragma unroll
            for (int c = 0; c < G::EPI_COLS; ++c) sum[c] = 0.f;
            for (int gi = 0; gi < ngroups; ++gi, ++gg) {
                const int b = gg & 1;
                ok = mbar_wait(smem_u32(&acc_full[b]), (gg / 2) & 1, err, SITE_TC_ACCUM);
                if (!ok) break;
                tc_fence_after();
                const uint32_t ta = tmem + lane_base + (uint32_t)b * G::ACC_STRIDE + (uint32_t)(half * G::EPI_COLS);
#pragma unroll
                for (int c0 = 0; c0 < G::EPI_COLS; c0 += 16) {
                    float v[16];
                    tc_ld16(ta + (uint32_t)c0, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) sum[c0 + i] += v[i];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_leader(smem_u32(&acc_free[b]));
            }
            const int c0 = n0 + half * G::EPI_COLS;
            if (ok && t < T) epi.row(t, c0, sum, N - c0);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0 && lane == 0 && rank == 0) {
        // nothing may still land in the pair's shared memory after exit (all stages were
        // consumed on the normal path; this only matters after a wait gave up)
        const int issued = s_issued;
        for (int kb = issued - S < 0 ? 0 : issued - S; kb < issued; ++kb)
            mbar_wait(smem_u32(&full_bar[kb % S]), (kb / S) & 1, err, SITE_TC_DRAIN);
    }
    __syncwarp();
    cluster_sync_all();   // neither CTA leaves while the other may still signal its barriers
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS)
                     : "memory");
    }
}

}  // namespace wici
