// The convolution layer of conv_tc.cuh on pairs of SMs (tcgen05 cta_group::2): a pair
// shares a 256 x 256 tile, each CTA holds its own 128 rows of A and half of B's 256
// columns, and the tensor cores of both read the halves from both shared memories.
// Per FLOP that is half of B's copies and of its shared-memory reads: a reduction
// block of the filter gradient takes four boxes per CTA instead of six, and stages are
// 32 KB instead of 48, so the ring holds six.  Same products in the same order as
// conv_tc.cuh.  Barriers and roles as in gemm2_tc.cuh.
//
// Measured at the paper's sample (4 x 1024 x 224 x 224, 1024 filters; 947 GFLOP each), us a
// call, one CTA per tile (with 16-byte stores) and pairs (with 32-byte ones): forward 587 and
// 540, data gradient (with the filter's transposition) 845 and 637, filter gradient 716 and 655.
#pragma once
#include "conv_tc.cuh"
#include "gemm2_tc.cuh"

namespace wici {

constexpr int CV2_STAGES = 6;
constexpr uint32_t CV2_B_BYTES = CV_B_BYTES / 2;
constexpr uint32_t CV2_STAGE_BYTES = CV_A_BYTES + CV2_B_BYTES;
constexpr size_t CV2_SMEM = (size_t)CV2_STAGES * CV2_STAGE_BYTES + 1024;

__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                                 uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
        "%4, %5}], [%6];" ::"r"(dst),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar & 0xFEFFFFFFu)
        : "memory");
}

// tiles of one launch: pairs of M tiles (the last one's second may lie past the images:
// its image index is a.n or more, its loads fill with zeros and nothing is stored)
template <int MODE>
__host__ __device__ __forceinline__ int cv_pair_tiles(const ConvArgs &a) {
    const int mpairs = (a.n * a.pt * a.qt + 1) / 2;
    if (MODE == CONV_FWD) return mpairs * (a.k / CV_BN);
    if (MODE == CONV_DGRAD) return 4 * mpairs * (a.c / CV_BN);
    return 9 * (a.k / (2 * CV_BM)) * (a.c / CV_BN);
}

// coordinates of CTA `rank`'s half of pair tile t
template <int MODE>
__device__ __forceinline__ CvTile cv_pair_tile(const ConvArgs &a, int t, int rank) {
    CvTile s = {};
    const int ntn = (MODE == CONV_FWD ? a.k : a.c) / CV_BN;
    s.nt = t % ntn;
    t /= ntn;
    if constexpr (MODE == CONV_WGRAD) {
        const int ntm = a.k / (2 * CV_BM);
        s.mt = 2 * (t % ntm) + rank;
        s.tap = t / ntm;
        s.nkb = a.n * ((a.p + 3) / 4) * a.qt;
        return s;
    }
    if constexpr (MODE == CONV_DGRAD) {
        const int mpairs = (a.n * a.pt * a.qt + 1) / 2;
        s.cls = t / mpairs;
        t %= mpairs;
        cv_class(s.cls, s.ph, s.pw);
        s.nkb = cv_ntaps_1d(s.ph) * cv_ntaps_1d(s.pw) * (a.k / CV_BK);
    } else {
        s.nkb = 9 * (a.c / CV_BK);
    }
    int m = 2 * t + rank;
    s.q0 = (m % a.qt) * 16;
    m /= a.qt;
    s.p0 = (m % a.pt) * 8;
    s.n = m / a.pt;
    return s;
}

// this CTA's loads of reduction block kb: its A rows, its half of B
template <int MODE>
__device__ __forceinline__ void cv_pair_load(const ConvArgs &a, const CvTile &s, int rank, int kb, const CUtensorMap *ma,
                                             const CUtensorMap *mb, uint32_t sa, uint32_t sb, uint32_t bar) {
    const int nb = s.nt * CV_BN + rank * (CV_BN / 2);
    if constexpr (MODE == CONV_FWD) {
        const int cbs = a.c / CV_BK, tap = kb / cbs, c0 = (kb % cbs) * CV_BK, r = tap / 3, ss = tap % 3;
        tma_load_4d_pair(sa, ma, c0, 2 * s.q0 + ss - 1, 2 * s.p0 + r - 1, s.n, bar);
        tma_load_2d_pair(sb, mb, tap * a.c + c0, nb, bar);
    } else if constexpr (MODE == CONV_DGRAD) {
        const int kbs = a.k / CV_BK, ti = kb / kbs, k0 = (kb % kbs) * CV_BK;
        const int nts = cv_ntaps_1d(s.pw);
        const int r = cv_tap_1d(s.ph, ti / nts), ss = cv_tap_1d(s.pw, ti % nts);
        tma_load_4d_pair(sa, ma, k0, s.q0 + (s.pw + 1 - ss) / 2, s.p0 + (s.ph + 1 - r) / 2, s.n, bar);
        tma_load_2d_pair(sb, mb, k0, (r * 3 + ss) * a.c + nb, bar);
    } else {
        const int pbs = (a.p + 3) / 4, pb = kb % (pbs * a.qt);
        const int n = kb / (pbs * a.qt), p0 = (pb / a.qt) * 4, q0 = (pb % a.qt) * 16;
        const int r = s.tap / 3, ss = s.tap % 3;
#pragma unroll
        for (int i = 0; i < CV_BM / 64; ++i)
            tma_load_4d_pair(sa + i * CV_BOX_BYTES, ma, s.mt * CV_BM + 64 * i, q0, p0, n, bar);
#pragma unroll
        for (int i = 0; i < CV_BN / 2 / 64; ++i)
            tma_load_4d_pair(sb + i * CV_BOX_BYTES, mb, nb + 64 * i, 2 * q0 + ss - 1, 2 * p0 + r - 1, n, bar);
    }
}

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(CV_THREADS, 1)
    conv2_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                    const ConvArgs a) {
    constexpr bool MN = MODE == CONV_WGRAD;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[CV2_STAGES], empty_bar[CV2_STAGES], acc_full[2], acc_free[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_issued;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)blockIdx.x & 1;
    const int tile0 = (int)blockIdx.x >> 1, tile_step = (int)gridDim.x >> 1;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < CV2_STAGES; ++s) {
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
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // both CTAs' barriers and tensor memory are ready
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    griddep_launch_dependents();
    griddep_wait();

    if (warp == 0) {
        if (lane == 0) {  // ------------------------------------------- TMA producer
            int it = 0;
            bool ok = true;
            for (int t = tile0; t < a.ntiles && ok; t += tile_step) {
                const CvTile s = cv_pair_tile<MODE>(a, t, rank);
                for (int kb = 0; kb < s.nkb; ++kb, ++it) {
                    const int st = it % CV2_STAGES;
                    if (it >= CV2_STAGES &&
                        !(ok = mbar_wait(smem_u32(&empty_bar[st]), ((it / CV2_STAGES) + 1) & 1, a.err, SITE_CV_EMPTY)))
                        break;
                    const uint32_t sa = base + (uint32_t)st * CV2_STAGE_BYTES;
                    const uint32_t fb = smem_u32(&full_bar[st]);
                    if (rank == 0) {
                        mbar_arrive_expect_tx(fb, 2 * CV2_STAGE_BYTES);
                        s_issued = it + 1;
                    }
                    cv_pair_load<MODE>(a, s, rank, kb, &map_a, &map_b, sa, sa + CV_A_BYTES, fb);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {  // ------------------------------- MMA issuer of the pair
            constexpr uint32_t idesc = (cv_idesc(MN) & ~(0x1Fu << 24)) | ((uint32_t)(2 * CV_BM >> 4) << 24);
            bool ok = true;
            int it = 0, tt = 0;
            for (int t = tile0; t < a.ntiles && ok; t += tile_step, ++tt) {
                const int nkb = cv_pair_tile<MODE>(a, t, 0).nkb;
                const int b = tt & 1;
                if (tt >= 2 && !(ok = mbar_wait(smem_u32(&acc_free[b]), ((tt / 2) + 1) & 1, a.err, SITE_CV_FREE)))
                    break;
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * CV_BN);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int st = it % CV2_STAGES;
                    ok = mbar_wait(smem_u32(&full_bar[st]), (it / CV2_STAGES) & 1, a.err, SITE_CV_FULL);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sa = base + (uint32_t)st * CV2_STAGE_BYTES, sb = sa + CV_A_BYTES;
#pragma unroll
                    for (int k = 0; k < CV_BK / 16; ++k) {
                        uint64_t ad, bd;
                        if constexpr (MN) {   // 16 pixels = 16 rows of 128 B further
                            ad = cv_desc_mn(sa + 2048u * k, CV_BOX_BYTES);
                            bd = cv_desc_mn(sb + 2048u * k, CV_BOX_BYTES);
                        } else {              // 16 channels = 32 B further inside the swizzled rows
                            ad = tc_desc_sw128(sa + 32u * k);
                            bd = tc_desc_sw128(sb + 32u * k);
                        }
                        tc_mma_pair(acc, ad, bd, idesc, (kb | k) != 0);
                    }
                    tc_commit_pair(smem_u32(&empty_bar[st]));
                }
                if (!ok) break;
                tc_commit_pair(smem_u32(&acc_full[b]));
            }
        }
    } else {  // ------------------------------------------------------- epilogue
        const int qd = warp & 3, half = (warp - 2) >> 2;
        const int m = qd * 32 + lane;                   // tile row = TMEM lane
        const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
        int tt = 0;
        for (int t = tile0; t < a.ntiles; t += tile_step, ++tt) {
            const CvTile s = cv_pair_tile<MODE>(a, t, rank);
            const int b = tt & 1;
            if (!mbar_wait(smem_u32(&acc_full[b]), (tt / 2) & 1, a.err, SITE_CV_ACCUM)) break;
            tc_fence_after();
            float *row = cv_row<MODE>(a, s, m);
#pragma unroll
            for (int c0 = 0; c0 < CV_BN / 2; c0 += 32) {
                float v[32];
                tc_ld32(tmem + lane_base + (uint32_t)(b * CV_BN + half * (CV_BN / 2) + c0), v);
                if (row) {
#pragma unroll
                    for (int i = 0; i < 32; i += 8) st_global_8(row + half * (CV_BN / 2) + c0 + i, v + i, a.wide);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_leader(smem_u32(&acc_free[b]));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0 && lane == 0 && rank == 0) {
        const int issued = s_issued;
        for (int kb = issued - CV2_STAGES < 0 ? 0 : issued - CV2_STAGES; kb < issued; ++kb)
            mbar_wait(smem_u32(&full_bar[kb % CV2_STAGES]), (kb / CV2_STAGES) & 1, a.err, SITE_CV_DRAIN);
    }
    __syncwarp();
    cluster_sync_all();   // neither CTA leaves while the other may still signal its barriers
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

}  // namespace wici
