// Prefill GEMM on the 5th-generation tensor cores (tcgen05 + TMEM + TMA).
//
//   C[T][N] = (A_0 + A_1 + A_2)[T][K] . W[N][K]^T,  fp32 accumulation in TMEM
//
// A is an fp32 activation carried as kTerms = 3 bf16 terms (split_bf16x3); W is
// bf16 and exact.  The three products accumulate into one fp32 TMEM
// accumulator, so the activations keep fp32 precision on bf16 MMAs (the bf16x3
// scheme of Henry, Tang & Heinecke, ARITH 2019, applied to one operand).
//
// Accumulation: one tcgen05 accumulator that absorbs the whole K dimension adds
// each MMA's result with the tensor core's internal alignment, and over K/16
// k-steps x 3 terms that error grows well past fp32 summation (measured: 4x the
// logits error of the fp32 CUDA-core path at the Llama-3-8B shape).  So the MMAs
// accumulate only TC_GROUP k-blocks into one of two TMEM buffers; the epilogue
// warps fold each finished group into fp32 registers (round-to-nearest adds)
// while the next group accumulates into the other buffer.
//
// Weights in the 8-bit block format arrive dequantised as WT = 3 bf16 terms
// W = W_0 + W_1 + W_2 (exact: a code times an fp16 scale has at most 18
// significant bits).  The K loop then runs once per weight term j < AT, issuing
// the products A_i W_j with i + j < AT, AT the activation terms of the GEMM:
// with AT = 3 that is 3 + 2 + 1 MMAs per k-step (the dropped products lie below
// 2^-24 of the result); with AT = 2 it is 2 + 1, the weight then carried at the
// activations' own 16 significant bits.
//
// Persistent: one CTA per SM walks the output tiles (M tiles fastest, so the
// CTAs that run together share a weight tile through L2) with three warp roles:
//   warp 0      TMA producer: 2-D tiled loads (128-byte swizzle) of the three A
//               terms and the W k-block into a shared-memory ring;
//   warp 1      allocates 512 TMEM columns and issues tcgen05.mma (one thread);
//               each stage is released by tcgen05.commit to its "empty" barrier;
//   warps 2..9  tcgen05.ld of one TMEM lane quadrant and half of the tile's
//               columns each (one output row per thread), group sums in
//               registers, then the fused epilogue on column pairs.  The
//               epilogue of one tile overlaps the MMAs of the next.
//
// Few tiles (short chunks): the tiles of a 128-row chunk of a 4096-column matrix
// are 32, on 152 SMs, and streaming the weights is what costs.  With SPLIT = 2 or 4
// a cluster of SPLIT CTAs shares one tile: each takes a range of the k-blocks, then
// the CTAs exchange column slices of their sums through shared memory (every CTA
// adds the slices of its BN / SPLIT columns in rank order) and run the epilogue on
// their slices.
//
// Chunks of at most 64 tokens (STACK, two activation terms): the two terms of the 64 rows
// are the 128 rows of one tile, so each weight k-step is read by one MMA instead of two
// (shared-memory ports bound these, too: 96 KB a k-block of 128 columns, 64 KB stacked).
// Rows r and r + 64 of the accumulator are the two terms' sums; they meet in shared
// memory on the way to the epilogue.
// Every mbarrier wait is bounded; a wait that gives up records its site in
// *err and the CTA still drains its copies, frees TMEM and exits.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace wici {

constexpr int TC_BM = 128, TC_BK = 64, TC_THREADS = 320, TC_EPI_WARPS = 8;
constexpr int TC_GROUP = 4;                                             // k-blocks per TMEM accumulation
constexpr uint32_t TC_A_BYTES = TC_BM * TC_BK * 2;                      // 16 KB per term
constexpr uint32_t TC_TMEM_COLS = 512;                                  // two accumulator buffers
constexpr size_t TC_SMEM_BUDGET = 216 * 1024;                           // ring bytes

// geometry of a 128 x BN output tile whose stages hold AT activation terms
template <int BN, int AT = kTerms>   // AT: 128-row blocks of activations per stage
struct TcTile {
    static_assert(BN % 32 == 0 && BN <= 256, "BN: a multiple of 32 up to 256");
    static constexpr uint32_t B_BYTES = BN * TC_BK * 2;
    static constexpr uint32_t STAGE_BYTES = AT * TC_A_BYTES + B_BYTES;
    static constexpr int STAGES = (int)(TC_SMEM_BUDGET / STAGE_BYTES);
    static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024;
    static constexpr int EPI_COLS = BN / 2;                               // columns per epilogue warp
    static constexpr uint32_t ACC_STRIDE = TC_TMEM_COLS / 2;              // TMEM columns between the two buffers
    static_assert(STAGES >= 3, "at least three ring stages");
};

// Tensor maps of one GEMM, all with boxes 64 elements wide and 128-byte swizzle.  One
// copy per operand and k-block: boxes of 64 rows of W, three to a 192-column tile,
// cost 17% of a long chunk's gate/up GEMM.
struct GemmMaps {
    CUtensorMap a[kTerms];   // activation terms, boxes of a_rows rows
    CUtensorMap w[kTerms];   // weight terms, boxes of BN rows
    int a_rows;              // 128, or what a chunk shorter than a tile needs
};

// everything the cluster's CTAs wrote before is visible to all of them after
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// 16 bytes into the shared memory of CTA `rank` of the cluster, at the address that `addr` has here
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t rank, float a, float b, float c, float d) {
    asm volatile(
        "{\n\t.reg .u32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "st.shared::cluster.v4.f32 [ra], {%2, %3, %4, %5};\n\t}" ::"r"(addr),
        "r"(rank), "f"(a), "f"(b), "f"(c), "f"(d)
        : "memory");
}

enum : int { SITE_TC_EMPTY = 21, SITE_TC_FULL = 22, SITE_TC_ACCUM = 23, SITE_TC_DRAIN = 24, SITE_TC_FREE = 25 };

// instruction descriptor of tcgen05.mma.kind::f16: D fp32, A and B bf16, both
// K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t tc_idesc(int n) {
    return (1u << 4)                      // D format: f32
           | (1u << 7)                    // A format: bf16
           | (1u << 10)                   // B format: bf16
           | ((uint32_t)(n >> 3) << 17)
           | ((uint32_t)(TC_BM >> 4) << 24);
}

// shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of
// 128 bytes, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t tc_desc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address
    d |= (uint64_t)1 << 16;                     // leading byte offset (unused with this swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;                     // descriptor version for tcgen05
    d |= (uint64_t)2 << 61;                     // swizzle mode: 128 B
    return d;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float *v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// the epilogue warps of a cluster's CTAs (and their other warps), or those of a CTA by itself
template <int SPLIT>
__device__ __forceinline__ void exchange_sync() {
    if constexpr (SPLIT > 1)
        cluster_sync_all();
    else
        asm volatile("bar.sync 2, 256;" ::: "memory");
}

// Epi::row(t, c, v, n): output row t, the thread's span of columns from c on, of
// which n are inside the matrix
template <int BN, int SPLIT, bool STACK, int WT, class Epi>
__global__ void __launch_bounds__(TC_THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ GemmMaps maps, int T, int N, int K, int *err, const Epi epi) {
    static_assert(WT == 1 || WT == kTerms, "one exact bf16 weight term, or three");
    static_assert(SPLIT == 1 || SPLIT == 2 || SPLIT == 4, "CTAs of a tile");
    constexpr int AT = Epi::kATerms;   // activation terms multiplied (and loaded)
    static_assert(AT >= 1 && AT <= kTerms, "activation terms");
    static_assert(!STACK || AT == 2, "two terms stacked");
    using G = TcTile<BN, STACK ? 1 : AT>;
    constexpr uint32_t A_TERM = STACK ? TC_A_BYTES / 2 : TC_A_BYTES;   // stacked: boxes of 64 rows
    constexpr uint32_t A_STAGE = STACK ? TC_A_BYTES : AT * TC_A_BYTES;
    constexpr int S = G::STAGES;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], acc_full[2], acc_free[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_issued;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntm = (T + TC_BM - 1) / TC_BM, ntn = (N + BN - 1) / BN;
    const int ntiles = ntm * ntn;
    const int nk = (K + TC_BK - 1) / TC_BK;
    constexpr int WU = WT == 1 ? 1 : Epi::kATerms;  // weight terms used
    // this CTA's tiles, and its range of the k-blocks of all weight terms
    const int rank = (int)blockIdx.x % SPLIT;
    const int tile0 = (int)blockIdx.x / SPLIT, tile_step = (int)gridDim.x / SPLIT;
    const int kk_begin = rank * nk * WU / SPLIT, kk_end = (rank + 1) * nk * WU / SPLIT;
    const int ngroups = (kk_end - kk_begin + TC_GROUP - 1) / TC_GROUP;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_bytes = (uint32_t)maps.a_rows * (TC_BK * 2);   // loaded per term

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
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
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    griddep_launch_dependents();
    if (warp != 0) griddep_wait();   // warp 0 waits behind its first weight copies

    if (warp == 0) {
        if (lane == 0) {  // ------------------------------------------- TMA producer
            int it = 0, s = 0;   // k-blocks issued over all tiles; the next one's stage
            uint32_t ph = 0;     // and its phase
            bool ok = true;
            // a bf16 weight does not depend on the kernels before this one: its first k-blocks
            // are on their way while those finish (8-bit: dequantised by the kernel before)
            const int early = WT == 1 && tile0 < ntiles ? min(S, kk_end - kk_begin) : 0;
            for (int e = 0; e < early; ++e) {
                const uint32_t fb = smem_u32(&full_bar[e]);
                mbar_arrive_expect_tx(fb, AT * a_bytes + G::B_BYTES);
                tma_load_2d(base + (uint32_t)e * G::STAGE_BYTES + A_STAGE, &maps.w[0], (kk_begin + e) * TC_BK,
                            (tile0 / ntm) * BN, fb);
            }
            griddep_wait();
            for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
                const int m0 = (tile % ntm) * TC_BM, n0 = (tile / ntm) * BN;
                for (int kk = kk_begin; kk < kk_end; ++kk, ++it) {
                    if (it >= S && !(ok = mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u, err, SITE_TC_EMPTY))) break;
                    const int j = WT == 1 ? 0 : kk / nk, kb = kk - j * nk;     // weight term, k-block
                    const uint32_t st = base + (uint32_t)s * G::STAGE_BYTES;
                    const uint32_t fb = smem_u32(&full_bar[s]);
                    // term j meets the activation terms i <= 2 - j only
                    const int na = STACK ? AT : AT - j;   // stacked: both terms, their MMAs are one
                    if (it >= early) mbar_arrive_expect_tx(fb, (uint32_t)na * a_bytes + G::B_BYTES);
#pragma unroll
                    for (int t = 0; t < AT; ++t)
                        if (t < na) tma_load_2d(st + t * A_TERM, &maps.a[t], kb * TC_BK, m0, fb);
                    if (it >= early) tma_load_2d(st + A_STAGE, &maps.w[j], kb * TC_BK, n0, fb);
                    s_issued = it + 1;
                    if (++s == S) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {  // ------------------------------------------- MMA issuer
            constexpr uint32_t idesc = tc_idesc(BN);
            bool ok = true;
            int gg = 0, s = 0;   // groups over all tiles, the next k-block's stage
            uint32_t ph = 0;     // and its phase
            for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
                for (int gi = 0; gi < ngroups && ok; ++gi, ++gg) {
                    const int b = gg & 1;
                    // the epilogue must have read this buffer's previous group
                    if (gg >= 2 && !(ok = mbar_wait(smem_u32(&acc_free[b]), ((gg / 2) + 1) & 1, err, SITE_TC_FREE)))
                        break;
                    tc_fence_after();
                    const uint32_t acc = tmem + (uint32_t)b * G::ACC_STRIDE;
                    const int kk0 = kk_begin + gi * TC_GROUP, kk1 = min(kk_end, kk0 + TC_GROUP);
                    for (int kk = kk0; kk < kk1; ++kk) {
                        ok = mbar_wait(smem_u32(&full_bar[s]), ph, err, SITE_TC_FULL);
                        if (!ok) break;
                        tc_fence_after();
                        const int nt = STACK ? 1 : WT == 1 ? AT : AT - kk / nk;   // activation terms meeting this weight term
                        const uint32_t st = base + (uint32_t)s * G::STAGE_BYTES;
                        // descriptors of k-step 0; each k-step of 16 elements is 32 bytes further
                        const uint64_t bd0 = tc_desc_sw128(st + A_STAGE);
                        const uint64_t ad0 = tc_desc_sw128(st);
#pragma unroll
                        for (int k = 0; k < TC_BK / 16; ++k)
#pragma unroll
                            for (int t = 0; t < kTerms; ++t)
                                if (t < nt)
                                    tc_mma(acc, ad0 + (uint64_t)((t * TC_A_BYTES + 32 * k) >> 4),
                                           bd0 + (uint64_t)(2 * k), idesc, (kk != kk0 || k != 0 || t != 0));
                        tc_commit(smem_u32(&empty_bar[s]));
                        if (++s == S) {
                            s = 0;
                            ph ^= 1u;
                        }
                    }
                    tc_commit(smem_u32(&acc_full[b]));  // fires when this group's MMAs have completed
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
            const int m0 = (tile % ntm) * TC_BM, n0 = (tile / ntm) * BN;
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
                for (int c0 = 0; c0 + 32 <= G::EPI_COLS; c0 += 32) {
                    float v[32];
                    tc_ld32(ta + (uint32_t)c0, v);
#pragma unroll
                    for (int i = 0; i < 32; ++i) sum[c0 + i] += v[i];
                }
                if constexpr (G::EPI_COLS % 32 != 0) {   // a last 16 columns
                    constexpr int c0 = G::EPI_COLS - 16;
                    float v[16];
                    tc_ld16(ta + (uint32_t)c0, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) sum[c0 + i] += v[i];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&acc_free[b]));
            }
            if constexpr (SPLIT == 1 && !STACK) {
                const int c0 = n0 + half * G::EPI_COLS;
                if (ok && t < T) epi.row(t, c0, sum, N - c0);
            } else {
                // one tile per CTA: every CTA of the cluster has finished with its ring, so the
                // sums' column slices cross through it, as [source rank][4 columns][row]: the 32 rows
                // of a warp are 512 consecutive bytes (row-major slices took 4 to 7 us to cross)
                constexpr int SL = BN / SPLIT;
                constexpr uint32_t SRC = TC_BM * SL * 4;
                static_assert(SPLIT * SRC <= G::STAGES * G::STAGE_BYTES && SL % 16 == 0, "slices fit the ring");
                const int row = q * 32 + lane;
                exchange_sync<SPLIT>();
#pragma unroll
                for (int c = 0; c < G::EPI_COLS; c += 4) {
                    const int col = half * G::EPI_COLS + c;
                    st_cluster_v4(base + (uint32_t)rank * SRC + (uint32_t)((col % SL) / 4 * TC_BM + row) * 16, col / SL,
                                  sum[c], sum[c + 1], sum[c + 2], sum[c + 3]);
                }
                exchange_sync<SPLIT>();
                // this CTA's slice: half of it per warp of a pair, or all of it in the first
                constexpr int NC = SL % 32 == 0 ? SL / 2 : SL;
                if ((SL % 32 == 0 || half == 0) && (!STACK || q < 2)) {   // stacked: 64 rows of output
                    const int part = SL % 32 == 0 ? half * NC : 0;
                    const uint8_t *src = smem_raw + (base - smem_u32(smem_raw)) + (size_t)(part / 4 * TC_BM + row) * 16;
                    float v[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) v[c] = 0.f;
#pragma unroll
                    for (int r = 0; r < SPLIT; ++r)
#pragma unroll
                        for (int c = 0; c < NC; c += 4) {
                            const float4 x = *reinterpret_cast<const float4 *>(src + r * SRC + c / 4 * TC_BM * 16);
                            v[c] += x.x; v[c + 1] += x.y; v[c + 2] += x.z; v[c + 3] += x.w;
                            if constexpr (STACK) {   // the second term's sums
                                const float4 y =
                                    *reinterpret_cast<const float4 *>(src + r * SRC + (c / 4 * TC_BM + TC_BM / 2) * 16);
                                v[c] += y.x; v[c + 1] += y.y; v[c + 2] += y.z; v[c + 3] += y.w;
                            }
                        }
                    const int c0 = n0 + rank * SL + part;
                    if (ok && t < T && c0 < N) epi.row(t, c0, v, N - c0);
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
        // nothing may still land in shared memory after exit (all stages were
        // consumed on the normal path; this only matters after a wait gave up)
        const int issued = s_issued;
        for (int kb = issued - S < 0 ? 0 : issued - S; kb < issued; ++kb)
            mbar_wait(smem_u32(&full_bar[kb % S]), (kb / S) & 1, err, SITE_TC_DRAIN);
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS)
                     : "memory");
    }
}

}  // namespace wici
