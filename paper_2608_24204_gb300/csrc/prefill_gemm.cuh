// The prefill GEMMs: tile choice, epilogues and launches.  The kernels of one epilogue are
// instantiated in a file of their own (prefill_gemm_*.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "gemm2_tc.cuh"
#include "gemm_tc.cuh"
#include "kernels.h"

namespace wici {

// The tile of one GEMM: its width, the CTAs that share one by splitting the k-blocks, or
// a pair of CTAs on a tile of 256 rows.
struct TileChoice {
    int bn, split;
    bool pair;
    bool stack;   // both activation terms of at most 64 rows in one tile
};

// Chosen per call from the chunk's own length, by modelled SM cycles: waves of tiles x
// (k-blocks of a CTA x cycles of a k-block + fixed).  A k-block takes its MMAs (bn / 2
// cycles per 128 (256 for a pair) x bn x 16 one) or its shared-memory traffic at 115 bytes
// a cycle (the operands written once, A and B read by every MMA; half of B per CTA of a
// pair), whichever is longer; measured at 2048 tokens, 8B widths: 1157 cycles for 192
// columns and two terms (1214 modelled).  fixed is the pipeline's fill and the epilogue,
// plus the exchange of a split tile.  Split tiles run as one wave only; how many clusters
// fit at once the driver says (SMs come in groups that they may not divide).  224 columns without a pair only for
// GEMMs of two activation terms (three leave too few ring stages).
// The choice used to be made for the largest chunk: a 61-token chunk at 8B widths then
// ran its O and down projections on 19 CTAs, 41 and 108 us against 26 and 46 now, and a
// 512-token one at 1B widths took 3731 us instead of 3023.
inline TileChoice pick_tile(int T, int N, int K, int at, int wu, const PrefillMaps &mp) {
    const int nk = (K + TC_BK - 1) / TC_BK * wu;
    const double mmas = wu == 1 ? at : (at + 1) * 0.5;   // per k-block and k-step
    TileChoice best = {0, 0, false, false};
    double best_cost = 0.0;
    auto consider = [&](TileChoice c, int units, int slots, double rows, double b_rows, double port) {
        const double n = c.stack ? 1.0 : mmas;
        const double mma = 2.0 * c.bn * n;
        const double smem = ((n * rows + b_rows) * 128.0 + 4.0 * n * (4096.0 + 32.0 * b_rows)) / port;
        const double cost = (double)((units + slots - 1) / slots) *
                            ((double)((nk + c.split - 1) / c.split) * (mma > smem ? mma : smem) + 2500.0 +
                             (c.split > 1 ? 2500.0 : 0.0));
        if (best.bn == 0 || cost < best_cost) {
            best = c;
            best_cost = cost;
        }
    };
    const int tm = (T + TC_BM - 1) / TC_BM, tm2 = (T + 2 * TC_BM - 1) / (2 * TC_BM);
    const int rows = T < TC_BM ? (T + 31) / 32 * 32 : TC_BM;
    for (int bn : {128, 192, 224})
        for (int split : {1, 2, 4}) {
            if (bn == 224 && (at != 2 || split != 1)) continue;
            const int units = tm * ((N + bn - 1) / bn) * split;
            if (split > 1 && units > (split == 2 ? 2 * mp.pairs : 4 * mp.quads)) continue;
            // 192 columns and three terms leave three ring stages: 8% more per k-block than the ports ask for
            if (at == 2 && T <= TC_BM / 2 && (bn == 128 || (bn == 192 && split == 1)) && units <= mp.sms)
                consider({bn, split, false, true}, units, mp.sms, TC_BM, bn, 115.0);
            consider({bn, split, false, false}, units, mp.sms, rows, bn, at == 3 && bn == 192 ? 106.0 : 115.0);
        }
    if (T > TC_BM && mp.pairs > 0)
        for (int bn : {192, 224, 256})
            consider({bn, 1, true, false}, tm2 * ((N + bn - 1) / bn), mp.pairs, TC_BM, bn / 2, 115.0);
    return best;
}

// store a as its three bf16 terms
__device__ __forceinline__ void split_store(uint16_t *const *t, size_t i, float a) {
    uint16_t t0, t1, t2;
    split_bf16x3(a, t0, t1, t2);
    t[0][i] = t0;
    t[1][i] = t1;
    t[2][i] = t2;
}

struct Terms {   // kTerms pointers passed by value to kernels
    uint16_t *p[kTerms];
};

// --------------------------------------------------------------- epilogues ----
// pair(t, c, a, b): GEMM output row t, columns (c, c + 1)
struct PEpiQKV {  // packed QKV columns -> Q (three bf16 terms) and K/V pages (bf16)
    static constexpr int kATerms = kTerms;   // activation terms the GEMM multiplies
    Terms Q;
    uint16_t *kv;
    const int *pages;
    const float2 *rope;
    const uint16_t *bias;
    int P, qdim, kvdim, d, nkv;
    size_t page_elems;
    float *raw;      // qk_norm: q | k of row t land here as they are ([t][qdim + kvdim], natural order)
    __device__ void pair(int t, int c, float a, float b) const {
        if (bias) {
            a += bf16_to_f32(bias[c]);
            b += bf16_to_f32(bias[c + 1]);
        }
        const int pos = P + t;
        uint16_t *page = kv + (size_t)pages[pos / kPage] * page_elems;
        const int slot = pos % kPage;
        if (raw && c < qdim + kvdim) {
            const int hd = c / d, i = (c % d) >> 1, half = d >> 1;
            float *dst = raw + (size_t)t * (qdim + kvdim) + hd * d;
            dst[i] = a;
            dst[i + half] = b;
        } else if (c < qdim + kvdim) {
            const int hd = c / d, i = (c % d) >> 1, half = d >> 1;
            const float2 cs = rope[(size_t)pos * half + i];
            const float ra = a * cs.x - b * cs.y;
            const float rb = b * cs.x + a * cs.y;
            if (c < qdim) {
                const size_t qo = (size_t)t * qdim + hd * d + i;
                split_store(Q.p, qo, ra);
                split_store(Q.p, qo + half, rb);
            } else {
                uint16_t *kr = page + ((size_t)(hd - qdim / d) * kPage + slot) * d;
                kr[i] = f32_to_bf16(ra);
                kr[i + half] = f32_to_bf16(rb);
            }
        } else {
            const int j = c - qdim - kvdim, vh = j / d, e = j % d;
            uint16_t *vr = page + (size_t)nkv * kPage * d + ((size_t)vh * kPage + slot) * d;
            vr[e] = f32_to_bf16(a);
            vr[e + 1] = f32_to_bf16(b);
        }
    }
    // 16 columns at a time: one head and one of q / k / v (head_dim, qdim and
    // kvdim are multiples of 64), 16-byte stores
    template <int NC>
    __device__ __forceinline__ void row(int t, int c0, const float (&v)[NC], int n) const {
        const int pos = P + t;
        uint16_t *page = kv + (size_t)pages[pos / kPage] * page_elems;
        const int slot = pos % kPage, half = d >> 1;
#pragma unroll
        for (int g = 0; g < NC; g += 16) {
            const int c = c0 + g;
            if (g + 16 > n) {
#pragma unroll
                for (int k = 0; k < 16; k += 2)
                    if (g + k + 1 < n) pair(t, c + k, v[g + k], v[g + k + 1]);
                continue;
            }
            float x[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) x[k] = v[g + k] + (bias ? bf16_to_f32(bias[c + k]) : 0.f);
            if (raw && c < qdim + kvdim) {
                // 8 RoPE pairs (i0 + k, i0 + k + d/2) of one head, unnormalised
                const int hd = c / d, i0 = (c % d) >> 1;
                float *dst = raw + (size_t)t * (qdim + kvdim) + hd * d + i0;
                *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[2], x[4], x[6]);
                *reinterpret_cast<float4 *>(dst + 4) = make_float4(x[8], x[10], x[12], x[14]);
                *reinterpret_cast<float4 *>(dst + half) = make_float4(x[1], x[3], x[5], x[7]);
                *reinterpret_cast<float4 *>(dst + half + 4) = make_float4(x[9], x[11], x[13], x[15]);
            } else if (c < qdim + kvdim) {
                const int hd = c / d, i0 = (c % d) >> 1;
                float ra[8], rb[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 cs = rope[(size_t)pos * half + i0 + k];
                    ra[k] = x[2 * k] * cs.x - x[2 * k + 1] * cs.y;
                    rb[k] = x[2 * k + 1] * cs.x + x[2 * k] * cs.y;
                }
                if (c < qdim) {
                    const size_t qo = (size_t)t * qdim + hd * d + i0;
                    uint32_t wa[kTerms][4], wb[kTerms][4];
#pragma unroll
                    for (int k = 0; k < 8; k += 2) {
                        uint16_t a0[kTerms], a1[kTerms], b0[kTerms], b1[kTerms];
                        split_bf16x3(ra[k], a0[0], a0[1], a0[2]);
                        split_bf16x3(ra[k + 1], a1[0], a1[1], a1[2]);
                        split_bf16x3(rb[k], b0[0], b0[1], b0[2]);
                        split_bf16x3(rb[k + 1], b1[0], b1[1], b1[2]);
#pragma unroll
                        for (int q = 0; q < kTerms; ++q) {
                            wa[q][k >> 1] = (uint32_t)a0[q] | ((uint32_t)a1[q] << 16);
                            wb[q][k >> 1] = (uint32_t)b0[q] | ((uint32_t)b1[q] << 16);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < kTerms; ++q) {
                        *reinterpret_cast<uint4 *>(Q.p[q] + qo) = make_uint4(wa[q][0], wa[q][1], wa[q][2], wa[q][3]);
                        *reinterpret_cast<uint4 *>(Q.p[q] + qo + half) =
                            make_uint4(wb[q][0], wb[q][1], wb[q][2], wb[q][3]);
                    }
                } else {
                    uint16_t *kr = page + ((size_t)(hd - qdim / d) * kPage + slot) * d + i0;
                    uint32_t wa[4], wb[4];
#pragma unroll
                    for (int k = 0; k < 8; k += 2) {
                        wa[k >> 1] = (uint32_t)f32_to_bf16(ra[k]) | ((uint32_t)f32_to_bf16(ra[k + 1]) << 16);
                        wb[k >> 1] = (uint32_t)f32_to_bf16(rb[k]) | ((uint32_t)f32_to_bf16(rb[k + 1]) << 16);
                    }
                    *reinterpret_cast<uint4 *>(kr) = make_uint4(wa[0], wa[1], wa[2], wa[3]);
                    *reinterpret_cast<uint4 *>(kr + half) = make_uint4(wb[0], wb[1], wb[2], wb[3]);
                }
            } else {
                const int j = c - qdim - kvdim, vh = j / d, e0 = j % d;
                uint16_t *vr = page + (size_t)nkv * kPage * d + ((size_t)vh * kPage + slot) * d + e0;
                uint32_t w[8];
#pragma unroll
                for (int k = 0; k < 16; k += 2)
                    w[k >> 1] = (uint32_t)f32_to_bf16(x[k]) | ((uint32_t)f32_to_bf16(x[k + 1]) << 16);
                *reinterpret_cast<uint4 *>(vr) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4 *>(vr + 8) = make_uint4(w[4], w[5], w[6], w[7]);
            }
        }
    }
};

// row(t, c0, v, n): output row t, columns c0 .. c0 + n of one thread's span
// (NC consecutive columns, c0 a multiple of 32), written with 16-byte stores
struct PEpiResidual {  // X[t][c] += v
    float *X;
    int ld;
    // the O and down GEMMs multiply two terms of their activations (o, m): with
    // gate/up also at two terms, measured at 1.36e-2 max-abs against the fp64
    // oracle at the Qwen2.5-14B shape (1.30e-2 with three); the QKV GEMM keeps
    // three terms (two there fail the 2e-2 tolerance)
    static constexpr int kATerms = 2;
    __device__ void pair(int t, int c, float a, float b) const {
        float2 *p = reinterpret_cast<float2 *>(X + (size_t)t * ld + c);
        float2 v = *p;
        v.x += a;
        v.y += b;
        *p = v;
    }
    template <int NC>
    __device__ __forceinline__ void row(int t, int c0, const float (&v)[NC], int n) const {
        float *x = X + (size_t)t * ld + c0;
#pragma unroll
        for (int j = 0; j < NC; j += 4) {
            if (j + 4 <= n) {
                float4 *p = reinterpret_cast<float4 *>(x + j);
                float4 a = *p;
                a.x += v[j]; a.y += v[j + 1]; a.z += v[j + 2]; a.w += v[j + 3];
                *p = a;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (j + e < n) x[j + e] += v[j + e];
            }
        }
    }
};

struct PEpiSwiGLU {  // interleaved (gate, up) columns -> M[t][c/2] = silu(g) * u as three terms
    Terms M;
    int ld;
    // the gate/up GEMM multiplies two terms of its activation (16 significant bits):
    // measured against the fp64 oracle at the 8B and 14B shapes, it moves the
    // logits by less than 1e-4, where two terms in every GEMM fail the tolerance
    static constexpr int kATerms = 2;
    __device__ void pair(int t, int c, float a, float b) const {
        split_store(M.p, (size_t)t * ld + (c >> 1), a / (1.0f + expf(-a)) * b);
    }
    template <int NC>
    __device__ __forceinline__ void row(int t, int c0, const float (&v)[NC], int n) const {
        const size_t o = (size_t)t * ld + (c0 >> 1);
#pragma unroll
        for (int j = 0; j < NC; j += 16) {   // 8 outputs: one 16-byte store per term
            if (j + 16 <= n) {
                uint32_t w[kTerms][4];
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const float g0 = v[j + 2 * k], u0 = v[j + 2 * k + 1];
                    const float g1 = v[j + 2 * k + 2], u1 = v[j + 2 * k + 3];
                    uint16_t a[kTerms], b[kTerms];
                    split_bf16x3(g0 / (1.0f + expf(-g0)) * u0, a[0], a[1], a[2]);
                    split_bf16x3(g1 / (1.0f + expf(-g1)) * u1, b[0], b[1], b[2]);
#pragma unroll
                    for (int q = 0; q < kTerms; ++q) w[q][k >> 1] = (uint32_t)a[q] | ((uint32_t)b[q] << 16);
                }
#pragma unroll
                for (int q = 0; q < kTerms; ++q)
                    *reinterpret_cast<uint4 *>(M.p[q] + o + (j >> 1)) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
            } else {
#pragma unroll
                for (int k = 0; k < 16; k += 2)
                    if (j + k + 1 < n) pair(t, c0 + j + k, v[j + k], v[j + k + 1]);
            }
        }
    }
};

// --------------------------------------------------------------- launches ----
// the weight operand of one GEMM: one exact bf16 matrix, or three terms
struct WOperand {
    const MatrixMaps *w[kTerms];
    int terms;
};

template <int BN, int SPLIT, bool STACK = false, class Epi>
cudaError_t launch_gemm(const Plan &p, const GemmMaps &maps, int terms, int T, int N, int K, int *err,
                               const Epi &epi, cudaStream_t st) {
    const int tiles = ((T + TC_BM - 1) / TC_BM) * ((N + BN - 1) / BN);
    // persistent, at most one CTA per SM; a split tile's CTAs are one cluster
    const dim3 grid(SPLIT > 1 ? tiles * SPLIT : tiles < p.num_sms ? tiles : p.num_sms);
    constexpr size_t smem = TcTile<BN, STACK ? 1 : Epi::kATerms>::SMEM;
    if (terms == 1)
        return launch_kernel(gemm_tc_kernel<BN, SPLIT, STACK, 1, Epi>, grid, TC_THREADS, smem, st, SPLIT, p.pdl, maps, T, N, K, err,
                             epi);
    return launch_kernel(gemm_tc_kernel<BN, SPLIT, STACK, kTerms, Epi>, grid, TC_THREADS, smem, st, SPLIT, p.pdl, maps, T, N, K,
                         err, epi);
}

template <int BN, class Epi>
cudaError_t launch_gemm_pair(const Plan &p, int pairs, const GemmMaps &maps, int terms, int T, int N, int K, int *err,
                                    const Epi &epi, cudaStream_t st) {
    const int tiles = ((T + 2 * TC_BM - 1) / (2 * TC_BM)) * ((N + BN - 1) / BN);
    const int grid = 2 * (tiles < pairs ? tiles : pairs);
    constexpr size_t smem = TcPairTile<BN, Epi::kATerms>::SMEM;
    // __cluster_dims__ gives the pairs
    if (terms == 1)
        return launch_kernel(gemm2_tc_kernel<BN, 1, Epi>, dim3(grid), TC_THREADS, smem, st, 1, p.pdl, maps, T, N, K, err,
                             epi);
    return launch_kernel(gemm2_tc_kernel<BN, kTerms, Epi>, dim3(grid), TC_THREADS, smem, st, 1, p.pdl, maps, T, N, K, err,
                         epi);
}

template <class Epi>
cudaError_t gemm(const Plan &p, const PrefillMaps &mp, const MatrixMaps (&a)[kTerms], const WOperand &w,
                        int T, int N, int K, int *err, const Epi &epi, cudaStream_t st, LaunchHook *hook,
                        const char *name) {
    const TileChoice c = pick_tile(T, N, K, Epi::kATerms, w.terms == 1 ? 1 : Epi::kATerms, mp);
    GemmMaps maps;
    // rows of a tile past the chunk are not loaded; a stacked tile is two boxes of 64
    maps.a_rows = c.stack ? 64 : T < TC_BM ? (T + 31) / 32 * 32 : TC_BM;
    for (int t = 0; t < kTerms; ++t) {
        const CUtensorMap *ma = matrix_map(a[t], maps.a_rows), *mw = matrix_map(*w.w[t], c.pair ? c.bn / 2 : c.bn);
        if (!ma || !mw) return cudaErrorInvalidValue;
        maps.a[t] = *ma;
        maps.w[t] = *mw;
    }
    if (hook) hook->before(name);
    cudaError_t e;
    auto shared = [&](auto bn, auto stack) {   // 128 columns, or 192 unstacked
        constexpr int BN = decltype(bn)::value;
        constexpr bool ST = decltype(stack)::value;
        return c.split == 1   ? launch_gemm<BN, 1, ST>(p, maps, w.terms, T, N, K, err, epi, st)
               : c.split == 2 ? launch_gemm<BN, 2, ST>(p, maps, w.terms, T, N, K, err, epi, st)
                              : launch_gemm<BN, 4, ST>(p, maps, w.terms, T, N, K, err, epi, st);
    };
    using std::integral_constant;
    if (c.pair)
        e = c.bn == 256   ? launch_gemm_pair<256>(p, mp.pairs, maps, w.terms, T, N, K, err, epi, st)
            : c.bn == 224 ? launch_gemm_pair<224>(p, mp.pairs, maps, w.terms, T, N, K, err, epi, st)
                          : launch_gemm_pair<192>(p, mp.pairs, maps, w.terms, T, N, K, err, epi, st);
    else if (c.bn == 128 && !c.stack)
        e = shared(integral_constant<int, 128>(), std::false_type());
    else if (c.bn == 192 && !c.stack)
        e = shared(integral_constant<int, 192>(), std::false_type());
    else if constexpr (Epi::kATerms == 2)
        e = c.bn == 224   ? launch_gemm<224, 1>(p, maps, w.terms, T, N, K, err, epi, st)
            : c.bn == 128 ? shared(integral_constant<int, 128>(), std::true_type())
                          : launch_gemm<192, 1, true>(p, maps, w.terms, T, N, K, err, epi, st);
    else
        e = cudaErrorInvalidValue;   // pick_tile picks 224 and stacked tiles for two terms only
    if (hook) hook->after(name);
    return e;
}

// shared-memory limits of every kernel that gemm<Epi> launches
template <class Epi>
cudaError_t setup_gemm() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *f, size_t bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    constexpr int AT = Epi::kATerms;
#define WICI_GEMM_SET(BN, SPLIT, ST, WT) \
    set((const void *)gemm_tc_kernel<BN, SPLIT, ST, WT, Epi>, TcTile<BN, ST ? 1 : AT>::SMEM);
#define WICI_GEMM_SETS(WT)                                                                                            \
    WICI_GEMM_SET(128, 1, false, WT) WICI_GEMM_SET(128, 2, false, WT) WICI_GEMM_SET(128, 4, false, WT)               \
    WICI_GEMM_SET(192, 1, false, WT) WICI_GEMM_SET(192, 2, false, WT) WICI_GEMM_SET(192, 4, false, WT)               \
    set((const void *)gemm2_tc_kernel<192, WT, Epi>, TcPairTile<192, AT>::SMEM);                                     \
    set((const void *)gemm2_tc_kernel<224, WT, Epi>, TcPairTile<224, AT>::SMEM);                                     \
    set((const void *)gemm2_tc_kernel<256, WT, Epi>, TcPairTile<256, AT>::SMEM);
    WICI_GEMM_SETS(1)
    WICI_GEMM_SETS(kTerms)
    if constexpr (AT == 2) {
#define WICI_GEMM_SETS2(WT)                                                                                           \
    WICI_GEMM_SET(224, 1, false, WT) WICI_GEMM_SET(128, 1, true, WT) WICI_GEMM_SET(128, 2, true, WT)                 \
    WICI_GEMM_SET(128, 4, true, WT) WICI_GEMM_SET(192, 1, true, WT)
        WICI_GEMM_SETS2(1)
        WICI_GEMM_SETS2(kTerms)
#undef WICI_GEMM_SETS2
    }
#undef WICI_GEMM_SETS
#undef WICI_GEMM_SET
    return e;
}

// clusters of `size` (2: the pair kernel) that run at once on the current device
template <class Epi>
cudaError_t resident_clusters(int size, int *n) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(size * 1024));
    cfg.blockDim = dim3(TC_THREADS);
    cfg.dynamicSmemBytes = size == 2 ? TcPairTile<256, 2>::SMEM : TcTile<128, 2>::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return size == 2 ? cudaOccupancyMaxActiveClusters(n, gemm2_tc_kernel<256, 1, Epi>, &cfg)
                     : cudaOccupancyMaxActiveClusters(n, gemm_tc_kernel<128, 4, false, 1, Epi>, &cfg);
}

#define WICI_GEMM_INSTANCE(EXTERN, Epi)                                                                               \
    EXTERN template cudaError_t gemm<Epi>(const Plan &, const PrefillMaps &, const MatrixMaps (&)[kTerms],       \
                                          const WOperand &, int, int, int, int *, const Epi &, cudaStream_t,         \
                                          LaunchHook *, const char *);                                               \
    EXTERN template cudaError_t setup_gemm<Epi>();                                                                   \
    EXTERN template cudaError_t resident_clusters<Epi>(int, int *);

}  // namespace wici
