// One 3x3, stride-2, padding-1 convolution layer on the tensor cores, forward
// and both gradients of backpropagation, as implicit GEMMs (the paper's second
// evaluated application, NVIDIA's CNN-training sample, Sec. 5.4).  Channels
// last: x [N][H][W][C], w [K][3][3][C], y and dy [N][P][Q][K], P = H/2, Q = W/2,
// all bf16 except the fp32 outputs.  bf16 operands are exact, products are
// exact, and each output accumulates in fp32 in TMEM over its whole reduction.
//
//   forward    y[pix][k]  = sum_{tap, c} X_tap[pix][c] w[k][tap][c]
//              M = output pixels (tiles of 8 rows x 16 columns), N = K, reduction
//              9 taps x C.  X_tap is x at (2p + r - 1, 2q + s - 1): one TMA box
//              with element strides 2 in h and w, zero outside the image.
//   data grad  dx[h][v][c] = sum dy[p][q][k] w[k][r][s][c] over 2p + r - 1 = h,
//              2q + s - 1 = v.  The output pixels split into four parity classes
//              (h even/odd x v even/odd); in each, a tap (r, s) reads dy at a
//              fixed offset (p = i + (ph + 1 - r) / 2 for h = 2i + ph), so every
//              class is a plain implicit GEMM over its 1, 2, 2 or 4 taps with the
//              filter transposed to [tap][c][k] (K-major B).
//   filter grad dw[k][tap][c] = sum_pix dy[pix][k] X_tap[pix][c]: per tap a GEMM
//              M = K, N = C, reduction over the N P Q pixels in blocks of 64
//              (4 output rows x 16 columns).  Both operands are pixel-by-channel
//              tiles, i.e. MN-major for tcgen05.
//
// Few tiles (small layers): with SPLIT = 2, 4 or 8 a cluster of CTAs shares one tile,
// each over a range of the reduction blocks; the CTAs then exchange column slices of
// their sums through shared memory, add them in rank order and store their slices.
// Large layers run on pairs of SMs (conv2_tc.cuh).
// Persistent, one CTA per SM, three warp roles as in the prefill GEMM: warp 0
// issues the TMA loads into a 4-stage ring (16 KB A + 32 KB B a stage), warp 1
// allocates 512 TMEM columns (two 256-column accumulators) and issues
// tcgen05.mma, warps 2..9 read a finished accumulator (lane quadrant x column
// half) and store fp32 rows while the next tile accumulates.  Waits are bounded.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "gemm_tc.cuh"

namespace wici {

enum ConvMode : int { CONV_FWD = 0, CONV_DGRAD = 1, CONV_WGRAD = 2 };

constexpr int CV_BM = 128, CV_BN = 256, CV_BK = 64, CV_STAGES = 4, CV_THREADS = 320;
constexpr uint32_t CV_A_BYTES = CV_BM * CV_BK * 2;        // 16 KB
constexpr uint32_t CV_B_BYTES = CV_BN * CV_BK * 2;        // 32 KB
constexpr uint32_t CV_STAGE_BYTES = CV_A_BYTES + CV_B_BYTES;
constexpr size_t CV_SMEM = (size_t)CV_STAGES * CV_STAGE_BYTES + 1024;
constexpr uint32_t CV_BOX_BYTES = 64 * 64 * 2;            // one 64-pixel x 64-channel box (filter grad)

enum : int { SITE_CV_EMPTY = 71, SITE_CV_FULL = 72, SITE_CV_ACCUM = 73, SITE_CV_FREE = 74, SITE_CV_DRAIN = 75 };

struct ConvArgs {
    int n, c, h, w, k, p, q;
    int pt, qt;          // output-row tiles (8 rows) and column tiles (16 columns)
    int ntiles;
    bool wide;           // out is 32-byte aligned
    float *out;          // y [N][P][Q][K], dx [N][H][W][C] or dw [K][3][3][C]
    int *err;
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(dst),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

// MN-major operand, 128-byte swizzle: rows are reduction indices (pixels) of 64
// consecutive M/N values; 8-row groups 1024 B apart, the next 64 values `lbo` further
__device__ __forceinline__ uint64_t cv_desc_mn(uint32_t saddr, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// kind::f16: D fp32, A and B bf16, M = 128, N = 256; MN-major A and B when mn
__host__ __device__ constexpr uint32_t cv_idesc(bool mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((mn ? 1u : 0u) << 15) | ((mn ? 1u : 0u) << 16) |
           ((uint32_t)(CV_BN >> 3) << 17) | ((uint32_t)(CV_BM >> 4) << 24);
}

// the data-gradient parity classes, heaviest first: (ph, pw) and their tap count
__device__ __forceinline__ void cv_class(int cls, int &ph, int &pw) {
    ph = cls == 0 || cls == 1 ? 1 : 0;     // classes: (1,1) 4 taps, (1,0) 2, (0,1) 2, (0,0) 1
    pw = cls == 0 || cls == 2 ? 1 : 0;
}
__device__ __forceinline__ int cv_ntaps_1d(int ph) { return ph ? 2 : 1; }
// i-th tap index along one axis of a class: even phase -> r = 1; odd -> r = 0, 2
__device__ __forceinline__ int cv_tap_1d(int ph, int i) { return ph ? 2 * i : 1; }

// Eight consecutive fp32.  Lanes hold rows far apart, so one 32-byte store per lane writes
// whole sectors where two 16-byte ones write halves; `wide`: the output is 32-byte
// aligned (callers promise 16).
__device__ __forceinline__ void st_global_8(float *p, const float *v, bool wide) {
    if (!wide) {
        reinterpret_cast<float4 *>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4 *>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
        return;
    }
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

// tile -> (mode-specific) coordinates; the reduction length in 64-wide blocks
struct CvTile {
    int n, p0, q0, nt;     // forward / data grad: image, first output row / column, N tile
    int cls, ph, pw;       // data grad
    int tap, mt;           // filter grad: tap, M (k) tile
    int nkb;               // reduction blocks
};

template <int MODE>
__device__ __forceinline__ CvTile cv_tile(const ConvArgs &a, int t) {
    CvTile s = {};
    if constexpr (MODE == CONV_FWD) {
        const int ntn = a.k / CV_BN;
        s.nt = t % ntn;
        int m = t / ntn;
        s.q0 = (m % a.qt) * 16;
        m /= a.qt;
        s.p0 = (m % a.pt) * 8;
        s.n = m / a.pt;
        s.nkb = 9 * (a.c / CV_BK);
    } else if constexpr (MODE == CONV_DGRAD) {
        const int ntn = a.c / CV_BN, per_class = a.n * a.pt * a.qt * ntn;
        s.cls = t / per_class;
        int m = t % per_class;
        s.nt = m % ntn;
        m /= ntn;
        s.q0 = (m % a.qt) * 16;
        m /= a.qt;
        s.p0 = (m % a.pt) * 8;
        s.n = m / a.pt;
        cv_class(s.cls, s.ph, s.pw);
        s.nkb = cv_ntaps_1d(s.ph) * cv_ntaps_1d(s.pw) * (a.k / CV_BK);
    } else {
        const int ntn = a.c / CV_BN, ntm = a.k / CV_BM;
        s.nt = t % ntn;
        s.mt = (t / ntn) % ntm;
        s.tap = t / (ntn * ntm);
        s.nkb = a.n * ((a.p + 3) / 4) * a.qt;
    }
    return s;
}

// TMA loads of reduction block kb of a tile into stage buffers (A at sa, B at sb)
template <int MODE>
__device__ __forceinline__ void cv_load(const ConvArgs &a, const CvTile &s, int kb, const CUtensorMap *ma,
                                        const CUtensorMap *mb, uint32_t sa, uint32_t sb, uint32_t bar) {
    if constexpr (MODE == CONV_FWD) {
        const int cbs = a.c / CV_BK, tap = kb / cbs, c0 = (kb % cbs) * CV_BK, r = tap / 3, ss = tap % 3;
        // x at rows 2p + r - 1, columns 2q + s - 1 (element strides 2): 8 x 16 pixels x 64 channels
        tma_load_4d(sa, ma, c0, 2 * s.q0 + ss - 1, 2 * s.p0 + r - 1, s.n, bar);
        tma_load_2d(sb, mb, tap * a.c + c0, s.nt * CV_BN, bar);                 // w[k][tap][c]
    } else if constexpr (MODE == CONV_DGRAD) {
        const int kbs = a.k / CV_BK, ti = kb / kbs, k0 = (kb % kbs) * CV_BK;
        const int nts = cv_ntaps_1d(s.pw);
        const int r = cv_tap_1d(s.ph, ti / nts), ss = cv_tap_1d(s.pw, ti % nts);
        const int dp = (s.ph + 1 - r) / 2, dq = (s.pw + 1 - ss) / 2;
        tma_load_4d(sa, ma, k0, s.q0 + dq, s.p0 + dp, s.n, bar);              // dy at (i + dp, j + dq)
        tma_load_2d(sb, mb, k0, (r * 3 + ss) * a.c + s.nt * CV_BN, bar);       // w^T[tap][c][k]
    } else {
        const int pbs = (a.p + 3) / 4, pb = kb % (pbs * a.qt);
        const int n = kb / (pbs * a.qt), p0 = (pb / a.qt) * 4, q0 = (pb % a.qt) * 16;
        const int r = s.tap / 3, ss = s.tap % 3;
        // A: dy pixels x 128 channels k (two 64-channel boxes); B: x pixels x 256 channels c
#pragma unroll
        for (int i = 0; i < CV_BM / 64; ++i) tma_load_4d(sa + i * CV_BOX_BYTES, ma, s.mt * CV_BM + 64 * i, q0, p0, n, bar);
#pragma unroll
        for (int i = 0; i < CV_BN / 64; ++i)
            tma_load_4d(sb + i * CV_BOX_BYTES, mb, s.nt * CV_BN + 64 * i, 2 * q0 + ss - 1, 2 * p0 + r - 1, n, bar);
    }
}

// this thread's output row of tile s (tile row m), its columns from the tile's first;
// nullptr outside the image
template <int MODE>
__device__ __forceinline__ float *cv_row(const ConvArgs &a, const CvTile &s, int m) {
    if constexpr (MODE == CONV_WGRAD) return a.out + ((size_t)(s.mt * CV_BM + m) * 9 + s.tap) * a.c + s.nt * CV_BN;
    const int i = s.p0 + m / 16, j = s.q0 + m % 16;
    if (s.n >= a.n || i >= a.p || j >= a.q) return nullptr;
    if constexpr (MODE == CONV_FWD)
        return a.out + (((size_t)s.n * a.p + i) * a.q + j) * a.k + s.nt * CV_BN;
    else
        return a.out + (((size_t)s.n * a.h + 2 * i + s.ph) * a.w + 2 * j + s.pw) * a.c + s.nt * CV_BN;
}

template <int MODE, int SPLIT>
__global__ void __launch_bounds__(CV_THREADS, 1)
    conv_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                   const ConvArgs a) {
    constexpr bool MN = MODE == CONV_WGRAD;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[CV_STAGES], empty_bar[CV_STAGES], acc_full[2], acc_free[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_issued;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // this CTA's tiles, and its range of a tile's reduction blocks
    const int rank = (int)blockIdx.x % SPLIT, tile0 = (int)blockIdx.x / SPLIT, tile_step = (int)gridDim.x / SPLIT;

    if (threadIdx.x == 0) {
        for (int s = 0; s < CV_STAGES; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_free[b]), TC_EPI_WARPS);
        }
        fence_barrier_init();
        s_issued = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    griddep_launch_dependents();
    griddep_wait();

    if (warp == 0) {
        if (lane == 0) {  // ------------------------------------------- TMA producer
            int it = 0;
            bool ok = true;
            for (int t = tile0; t < a.ntiles && ok; t += tile_step) {
                const CvTile s = cv_tile<MODE>(a, t);
                const int kb1 = (rank + 1) * s.nkb / SPLIT;
                for (int kb = rank * s.nkb / SPLIT; kb < kb1; ++kb, ++it) {
                    const int st = it % CV_STAGES;
                    if (it >= CV_STAGES &&
                        !(ok = mbar_wait(smem_u32(&empty_bar[st]), ((it / CV_STAGES) + 1) & 1, a.err, SITE_CV_EMPTY)))
                        break;
                    const uint32_t sa = base + (uint32_t)st * CV_STAGE_BYTES;
                    const uint32_t fb = smem_u32(&full_bar[st]);
                    mbar_arrive_expect_tx(fb, CV_STAGE_BYTES);
                    cv_load<MODE>(a, s, kb, &map_a, &map_b, sa, sa + CV_A_BYTES, fb);
                    s_issued = it + 1;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {  // ------------------------------------------- MMA issuer
            constexpr uint32_t idesc = cv_idesc(MN);
            bool ok = true;
            int it = 0, tt = 0;
            for (int t = tile0; t < a.ntiles && ok; t += tile_step, ++tt) {
                const CvTile s = cv_tile<MODE>(a, t);
                const int b = tt & 1;
                if (tt >= 2 && !(ok = mbar_wait(smem_u32(&acc_free[b]), ((tt / 2) + 1) & 1, a.err, SITE_CV_FREE)))
                    break;
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * CV_BN);
                const int kb0 = rank * s.nkb / SPLIT, kb1 = (rank + 1) * s.nkb / SPLIT;
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const int st = it % CV_STAGES;
                    ok = mbar_wait(smem_u32(&full_bar[st]), (it / CV_STAGES) & 1, a.err, SITE_CV_FULL);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sa = base + (uint32_t)st * CV_STAGE_BYTES, sb = sa + CV_A_BYTES;
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
                        tc_mma(acc, ad, bd, idesc, kb != kb0 || k != 0);
                    }
                    tc_commit(smem_u32(&empty_bar[st]));
                }
                if (!ok) break;
                tc_commit(smem_u32(&acc_full[b]));
            }
        }
    } else {  // ------------------------------------------------------- epilogue
        const int qd = warp & 3, half = (warp - 2) >> 2;
        const int m = qd * 32 + lane;                   // tile row = TMEM lane
        const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
        int tt = 0;
        bool ok = true;
        for (int t = tile0; t < a.ntiles && ok; t += tile_step, ++tt) {
            const CvTile s = cv_tile<MODE>(a, t);
            const int b = tt & 1;
            ok = mbar_wait(smem_u32(&acc_full[b]), (tt / 2) & 1, a.err, SITE_CV_ACCUM);
            tc_fence_after();
            float *row = cv_row<MODE>(a, s, m);
            const uint32_t ta = tmem + lane_base + (uint32_t)(b * CV_BN + half * (CV_BN / 2));
            if constexpr (SPLIT == 1) {
                if (!ok) break;
#pragma unroll
                for (int c0 = 0; c0 < CV_BN / 2; c0 += 32) {
                    float v[32];
                    tc_ld32(ta + (uint32_t)c0, v);
                    if (row) {
#pragma unroll
                        for (int i = 0; i < 32; i += 8) st_global_8(row + half * (CV_BN / 2) + c0 + i, v + i, a.wide);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&acc_free[b]));
            } else {
                // one tile per CTA: every CTA of the cluster has finished with its ring, so the
                // sums' column slices cross through it, as [source rank][4 columns][row]: the 32 rows
                // of a warp are 512 consecutive bytes
                constexpr int SL = CV_BN / SPLIT;
                constexpr uint32_t SRC = CV_BM * SL * 4;
                static_assert(SPLIT * SRC <= CV_STAGES * CV_STAGE_BYTES, "slices fit the ring");
                const bool some = (rank + 1) * s.nkb / SPLIT > rank * s.nkb / SPLIT;   // else nothing was accumulated
                cluster_sync_all();
#pragma unroll
                for (int c0 = 0; c0 < CV_BN / 2; c0 += 32) {
                    float v[32];
                    tc_ld32(ta + (uint32_t)c0, v);
#pragma unroll
                    for (int i = 0; i < 32; i += 4) {
                        const int col = half * (CV_BN / 2) + c0 + i;
                        st_cluster_v4(base + (uint32_t)rank * SRC + (uint32_t)((col % SL) / 4 * CV_BM + m) * 16, col / SL,
                                      some ? v[i] : 0.f, some ? v[i + 1] : 0.f, some ? v[i + 2] : 0.f,
                                      some ? v[i + 3] : 0.f);
                    }
                }
                cluster_sync_all();
                constexpr int NC = SL / 2;   // columns of the slice per warp of a pair
                const uint8_t *src = smem_raw + (base - smem_u32(smem_raw)) + (size_t)(half * NC / 4 * CV_BM + m) * 16;
                if (ok && row) {
#pragma unroll
                    for (int c = 0; c < NC; c += 8) {
                        float v[8] = {};
#pragma unroll
                        for (int r = 0; r < SPLIT; ++r) {
                            const float4 x = *reinterpret_cast<const float4 *>(src + r * SRC + c / 4 * CV_BM * 16);
                            const float4 y = *reinterpret_cast<const float4 *>(src + r * SRC + (c / 4 + 1) * CV_BM * 16);
                            v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
                            v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
                        }
                        st_global_8(row + rank * SL + half * NC + c, v, a.wide);
                    }
                }
            }
        }
    }
    if constexpr (SPLIT > 1) {
        if (warp < 2) {   // the epilogue warps' two cluster barriers count every thread
            __syncwarp();
            cluster_sync_all();
            cluster_sync_all();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0 && lane == 0) {
        const int issued = s_issued;
        for (int kb = issued - CV_STAGES < 0 ? 0 : issued - CV_STAGES; kb < issued; ++kb)
            mbar_wait(smem_u32(&full_bar[kb % CV_STAGES]), (kb / CV_STAGES) & 1, a.err, SITE_CV_DRAIN);
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// w [K][9][C] -> w^T [9][C][K] (the data gradient's K-major B operand), 32 x 32 tiles, 8 warps
__global__ void conv_transpose_filter_kernel(const uint16_t *w, uint16_t *wt, int K, int C) {
    __shared__ uint16_t tile[32][33];
    griddep_launch_dependents();
    griddep_wait();   // an earlier data gradient may still read wt
    const int lane = threadIdx.x & 31, tap = blockIdx.z, k0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    for (int i = threadIdx.x >> 5; i < 32; i += 8) {
        const int k = k0 + i, c = c0 + lane;
        tile[i][lane] = (k < K && c < C) ? w[((size_t)k * 9 + tap) * C + c] : 0;
    }
    __syncthreads();
    for (int i = threadIdx.x >> 5; i < 32; i += 8) {
        const int c = c0 + i, k = k0 + lane;
        if (c < C && k < K) wt[((size_t)tap * C + c) * K + k] = tile[lane][i];
    }
}

}  // namespace wici
