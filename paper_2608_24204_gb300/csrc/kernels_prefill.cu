// Prefill: a chunk of T prompt tokens at positions P..P+T-1 through every
// layer.  The four linear maps of a layer run on the tcgen05 GEMM (gemm_tc.cuh)
// with fused epilogues (bias + RoPE + paged KV append, residual add, SwiGLU)
// and the causal attention on the tcgen05 attention kernel (attn_tc.cuh); the
// kernels around them produce the tensor-core operands as bf16 terms (split_bf16x3).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "common.cuh"
#include "attn_tc.cuh"
#include "device_table.h"
#include "kernels.h"
#include "prefill_gemm.cuh"

namespace wici {

WICI_GEMM_INSTANCE(extern, PEpiQKV)
WICI_GEMM_INSTANCE(extern, PEpiResidual)
WICI_GEMM_INSTANCE(extern, PEpiSwiGLU)

// ----------------------------------------------------------- embed / norm ----
__global__ void embed_rows_kernel(const uint16_t *E, const int *tok, float *X, int H) {
    griddep_launch_dependents();
    griddep_wait();
    const int t = blockIdx.x;
    const uint16_t *row = E + (size_t)tok[t] * H;
    for (int i = threadIdx.x; i < H; i += blockDim.x) X[(size_t)t * H + i] = bf16_to_f32(row[i]);
}

// A[t] = X[t] / sqrt(mean(X[t]^2) + eps) * g, stored as three bf16 terms
// One CTA per row t: RMSNorm of x_t with gain g, stored as the first `nterms`
// bf16 terms of the next GEMM's operand (its kATerms).  H % 8 == 0: 8-element
// chunks, one 16-byte store per term.
__global__ void rmsnorm_rows_kernel(const float *X, const uint16_t *g, const Terms A, int H, float eps,
                                    int nterms) {
    __shared__ float s_part[32];
    griddep_launch_dependents();
    griddep_wait();
    const int t = blockIdx.x;
    const float4 *x = reinterpret_cast<const float4 *>(X + (size_t)t * H);
    const int nc = H >> 3;
    float ss = 0.f;
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        const float4 u = x[2 * c], v = x[2 * c + 1];
        ss = fmaf(u.x, u.x, ss); ss = fmaf(u.y, u.y, ss); ss = fmaf(u.z, u.z, ss); ss = fmaf(u.w, u.w, ss);
        ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss); ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss);
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_part[w];
    const float rinv = 1.0f / sqrtf(tot / (float)H + eps);
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        const float4 u = x[2 * c], v = x[2 * c + 1];
        const uint4 gw = reinterpret_cast<const uint4 *>(g)[c];
        const float y[8] = {u.x * rinv * bf16lo(gw.x), u.y * rinv * bf16hi(gw.x), u.z * rinv * bf16lo(gw.y),
                            u.w * rinv * bf16hi(gw.y), v.x * rinv * bf16lo(gw.z), v.y * rinv * bf16hi(gw.z),
                            v.z * rinv * bf16lo(gw.w), v.w * rinv * bf16hi(gw.w)};
        uint32_t w[kTerms][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint16_t a0[kTerms], a1[kTerms];
            split_bf16x3(y[2 * e], a0[0], a0[1], a0[2]);
            split_bf16x3(y[2 * e + 1], a1[0], a1[1], a1[2]);
#pragma unroll
            for (int q = 0; q < kTerms; ++q) w[q][e] = (uint32_t)a0[q] | ((uint32_t)a1[q] << 16);
        }
        const size_t o = (size_t)t * H + 8 * (size_t)c;
#pragma unroll
        for (int q = 0; q < kTerms; ++q)
            if (q < nterms) *reinterpret_cast<uint4 *>(A.p[q] + o) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
    }
}

// ------------------------------------------------- Qwen3 q/k norm (prefill) --
// One warp per (row t, head): the head of raw q (or k) RMS-normalised over
// head_dim with its gain, RoPE at position P + t, then q as three bf16 terms in
// Q[t] or k as bf16 in its page slot.  Lane l holds elements l*EPL ..; the RoPE
// partner of element i < d/2 is i + d/2, in lane l + 16.
template <int D>
__global__ void qk_norm_rope_kernel(const float *raw, const uint16_t *qn, const uint16_t *kn, const float2 *rope,
                                    Terms Q, uint16_t *kv, const int *pages, size_t page_elems, int P, int nq,
                                    int nkv, float eps) {
    constexpr int EPL = D / 32, HALF = D / 2;
    griddep_launch_dependents();
    griddep_wait();
    const int t = blockIdx.x, lane = threadIdx.x & 31;
    const int hd = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (hd >= nq + nkv) return;
    const int qdim = nq * D, kvdim = nkv * D;
    const float *src = raw + (size_t)t * (qdim + kvdim) + (size_t)hd * D + lane * EPL;
    const uint16_t *gain = hd < nq ? qn : kn;
    float v[EPL];
    float ss = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        v[e] = src[e];
        ss = fmaf(v[e], v[e], ss);
    }
    const float rinv = 1.0f / sqrtf(warp_sum(ss) / (float)D + eps);
    const int pos = P + t;
#pragma unroll
    for (int e = 0; e < EPL; ++e) v[e] = v[e] * rinv * bf16_to_f32(gain[lane * EPL + e]);
    float r[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        const float other = __shfl_xor_sync(0xffffffffu, v[e], 16);
        const float2 cs = rope[(size_t)pos * HALF + (lane * EPL + e) % HALF];
        r[e] = lane < 16 ? v[e] * cs.x - other * cs.y : v[e] * cs.x + other * cs.y;
    }
    if (hd < nq) {
        const size_t o = (size_t)t * qdim + (size_t)hd * D + lane * EPL;
#pragma unroll
        for (int e = 0; e < EPL; ++e) split_store(Q.p, o + e, r[e]);
    } else {
        uint16_t *kr = kv + (size_t)pages[pos / kPage] * page_elems + ((size_t)(hd - nq) * kPage + pos % kPage) * D +
                       lane * EPL;
#pragma unroll
        for (int e = 0; e < EPL; ++e) kr[e] = f32_to_bf16(r[e]);
    }
}

// ------------------------------------------------ 8-bit block format (prefill) --
// W[r][c] = d[r][c / 32] * code[r][c] of `rows` arena rows (int8 codes, then
// the row's fp16 block scales), written as three bf16 terms of a
// row-major [rows][K] matrix.  The product is exact in fp32 (at most 18
// significant bits), and so is its split into three terms.  8 elements per
// thread: one 8-byte code load, one scale, one 16-byte store per term.
__global__ void q8_dequant_terms_kernel(const uint8_t *src, int rows, int K, const Terms out, int nterms) {
    griddep_launch_dependents();
    griddep_wait();   // the GEMM before still reads the terms of its matrix
    const int per_row = K / 8;
    const size_t rb = (size_t)K + (size_t)K / 16;
    const long long n = (long long)rows * per_row;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / per_row;
        const int c = (int)(i - r * per_row);
        const uint8_t *row = src + (size_t)r * rb;
        const uint2 w = *reinterpret_cast<const uint2 *>(row + (size_t)c * 8);
        const float d = __half2float(__ushort_as_half(*reinterpret_cast<const unsigned short *>(row + K + (c >> 2) * 2)));
        uint32_t t[kTerms][4];
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            const uint32_t word = k < 4 ? w.x : w.y;
            const float a = d * (float)(int8_t)(word >> (8 * (k & 3)));
            const float b = d * (float)(int8_t)(word >> (8 * ((k & 3) + 1)));
            uint16_t ta[kTerms], tb[kTerms];
            split_bf16x3(a, ta[0], ta[1], ta[2]);
            split_bf16x3(b, tb[0], tb[1], tb[2]);
#pragma unroll
            for (int q = 0; q < kTerms; ++q) t[q][k >> 1] = (uint32_t)ta[q] | ((uint32_t)tb[q] << 16);
        }
        const size_t o = (size_t)r * K + (size_t)c * 8;
#pragma unroll
        for (int q = 0; q < kTerms; ++q)
            if (q < nterms) *reinterpret_cast<uint4 *>(out.p[q] + o) = make_uint4(t[q][0], t[q][1], t[q][2], t[q][3]);
    }
}

static cudaError_t dequant_terms(const Plan &p, const Bufs &b, const uint16_t *W, int rows, int K, int nterms,
                                 cudaStream_t st, LaunchHook *hook) {
    const long long n = (long long)rows * (K / 8);
    const int grid = (int)((n + 255) / 256 < 8 * p.num_sms ? (n + 255) / 256 : 8 * p.num_sms);
    if (hook) hook->before("prefill_q8_dequant");
    const cudaError_t e =
        launch_kernel(q8_dequant_terms_kernel, dim3(grid), 256, 0, st, 1, p.pdl, reinterpret_cast<const uint8_t *>(W), rows,
                      K, Terms{{b.Wt[0], b.Wt[1], b.Wt[2]}}, nterms);
    if (hook) hook->after("prefill_q8_dequant");
    return e;
}

// --------------------------------------------------------------- RoPE table --
__global__ void rope_table_kernel(float2 *rope, int n_pos, int half, double theta) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_pos * half) return;
    const int p = idx / half, i = idx % half;
    const double freq = pow(theta, -2.0 * (double)i / (double)(2 * half));
    double s, c;
    sincos((double)p * freq, &s, &c);
    rope[idx] = make_float2((float)c, (float)s);
}

// ================================================================ host =======

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

bool encode_tiled(CUtensorMap *m, int rank, const void *ptr, const uint64_t *dims, const uint64_t *strides_bytes,
                  const uint32_t *box, const uint32_t *elem_strides) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t d[5], st[4];
    cuuint32_t b[5], e[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        b[i] = box[i];
        e[i] = elem_strides[i];
        if (i + 1 < rank) st[i] = strides_bytes[i];
    }
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(ptr), d, st, b, e,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D map over a row-major bf16 matrix [rows][K]; boxes of 64 x box_rows, 128 B swizzle
static bool encode_2d(CUtensorMap *m, const void *ptr, int rows, int K, int box_rows) {
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)rows}, strides[1] = {(uint64_t)K * 2};
    const uint32_t box[2] = {(uint32_t)TC_BK, (uint32_t)box_rows}, es[2] = {1, 1};
    return encode_tiled(m, 2, ptr, dims, strides, box, es);
}

const CUtensorMap *matrix_map(const MatrixMaps &m, int box) {
    for (int i = 0; i < kMapBoxes; ++i) {
        if (kMapBox[i] != box) continue;
        if (!m.ready[i]) m.ready[i] = encode_2d(&m.map[i], m.ptr, m.rows, m.K, box);
        return m.ready[i] ? &m.map[i] : nullptr;
    }
    return nullptr;
}

static MatrixMaps matrix(const void *ptr, int rows, int K) {
    MatrixMaps m;
    m.ptr = ptr;
    m.rows = rows;
    m.K = K;
    return m;
}

// the KV pool of every layer as [page (layer-major)][K|V][kv head][16 slots][d]:
// boxes of 64 d x 16 slots of one (page, K|V, head)
static bool encode_kv(CUtensorMap *m, const void *ptr, const Plan &p) {
    const uint64_t dims[5] = {(uint64_t)p.d, (uint64_t)kPage, (uint64_t)p.nkv, 2, (uint64_t)p.L * (uint64_t)p.max_pages};
    const uint64_t strides[4] = {(uint64_t)p.d * 2, (uint64_t)kPage * p.d * 2, (uint64_t)p.nkv * kPage * p.d * 2,
                                 (uint64_t)2 * p.nkv * kPage * p.d * 2};
    const uint32_t box[5] = {64, (uint32_t)kPage, 1, 1, 1}, es[5] = {1, 1, 1, 1, 1};
    return encode_tiled(m, 5, ptr, dims, strides, box, es);
}

const char *make_prefill_maps(const Plan &p, const Bufs &b, PrefillMaps *m) {
    const int T = p.max_chunk;
    for (int t = 0; t < kTerms; ++t) {
        m->a[t] = matrix(b.A[t], T, p.H);
        m->o[t] = matrix(b.O[t], T, p.qdim);
        m->m[t] = matrix(b.M[t], T, p.F);
        if (p.q8) {   // the 8-bit format: every GEMM reads the one dequantised matrix in the workspace
            m->wt_qkv[t] = matrix(b.Wt[t], p.nqkv, p.H);
            m->wt_o[t] = matrix(b.Wt[t], p.H, p.qdim);
            m->wt_gu[t] = matrix(b.Wt[t], 2 * p.F, p.H);
            m->wt_d[t] = matrix(b.Wt[t], p.H, p.F);
        }
    }
    if (!encode_kv(&m->kv, b.KV, p)) return "cuTensorMapEncodeTiled failed for the attention operands";
    for (int l = 0; l < (p.q8 ? 0 : p.L); ++l) {
        const LayerOffsets &lo = p.layer[l];
        m->wqkv.push_back(matrix(b.W + lo.wqkv, p.nqkv, p.H));
        m->wo.push_back(matrix(b.W + lo.wo, p.H, p.qdim));
        m->wgu.push_back(matrix(b.W + lo.wgu, 2 * p.F, p.H));
        m->wd.push_back(matrix(b.W + lo.wd, p.H, p.F));
    }
    m->sms = p.num_sms;
    // kernel limits and resident clusters (there may be none): once per device
    struct Clusters {
        int pairs = 0, quads = 0;
    };
    static DeviceTable<Clusters> devices;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return "no CUDA device";
    Clusters n;
    const char *refused = devices.get(dev, &n, [](Clusters *d) -> const char * {
        const auto limit = [](const void *f, size_t bytes) {
            return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
        };
        if (setup_gemm<PEpiQKV>() != cudaSuccess || setup_gemm<PEpiResidual>() != cudaSuccess ||
            setup_gemm<PEpiSwiGLU>() != cudaSuccess ||
            !limit((const void *)attn_tc_kernel<128>, AttnSmem<128>::TOTAL + 1024) ||
            !limit((const void *)attn_tc_kernel<64>, AttnSmem<64>::TOTAL + 1024))
            return "cannot raise the shared-memory limits of the prefill kernels";
        if (resident_clusters<PEpiSwiGLU>(2, &d->pairs) != cudaSuccess ||
            resident_clusters<PEpiSwiGLU>(4, &d->quads) != cudaSuccess)
            return "cannot query the resident clusters of the tensor-core GEMM";
        return nullptr;
    });
    if (refused) return refused;
    m->pairs = n.pairs < p.num_sms / 2 ? n.pairs : p.num_sms / 2;
    m->quads = n.quads < p.num_sms / 4 ? n.quads : p.num_sms / 4;
    return nullptr;
}

// causal GQA attention of chunk rows [0, T) at positions P.. on the tensor cores
cudaError_t launch_attn_tc(const Plan &p, const Bufs &b, const PrefillMaps &mp, int layer, int P, int T,
                           cudaStream_t st) {
    AttnArgs a;
    for (int t = 0; t < AT_TERMS; ++t) a.Q[t] = b.Q[t];
    for (int t = 0; t < kTerms; ++t) a.O[t] = b.O[t];
    a.pages = b.pages;
    a.err = b.ctrl + CTRL_ERR;
    a.P = P;
    a.T = T;
    a.nq = p.nq;
    a.group = p.group;
    a.tpt = attn_tokens_per_tile(p.group);
    a.layer = layer;
    a.max_pages = p.max_pages;
    a.scale_log2 = 1.4426950408889634f / sqrtf((float)p.d);
    dim3 grid(((T + a.tpt - 1) / a.tpt) * p.nkv);
    if (p.d == 128)
        return launch_kernel(attn_tc_kernel<128>, grid, AT_THREADS, AttnSmem<128>::TOTAL + 1024, st, 1, p.pdl, mp.kv, a);
    return launch_kernel(attn_tc_kernel<64>, grid, AT_THREADS, AttnSmem<64>::TOTAL + 1024, st, 1, p.pdl, mp.kv, a);
}

// bf16: the layer's own matrix; 8-bit format: dequantise the layer's rows into
// the workspace terms first (stream order makes the previous GEMM finish reading them)
template <class Epi>
static cudaError_t weight_operand(const Plan &p, const Bufs &b, const MatrixMaps &bf16_map,
                                  const MatrixMaps *terms, const uint16_t *rows, int n_rows, int K, cudaStream_t st,
                                  LaunchHook *hook, WOperand *w) {
    if (!p.q8) {
        *w = WOperand{{&bf16_map, &bf16_map, &bf16_map}, 1};
        return cudaSuccess;
    }
    *w = WOperand{{&terms[0], &terms[1], &terms[2]}, kTerms};
    return dequant_terms(p, b, rows, n_rows, K, Epi::kATerms, st, hook);   // the weight terms the GEMM uses
}

cudaError_t enqueue_prefill_chunk(const Plan &p, const Bufs &b, const PrefillMaps &mp, cudaStream_t st, int P,
                                  int T, int lm_pos_add, LaunchHook *hook) {
    cudaError_t e;
    int *err = b.ctrl + CTRL_ERR;
    if ((e = launch_kernel(embed_rows_kernel, dim3(T), 256, 0, st, 1, p.pdl, b.W + p.w_embed, b.tok, b.X, p.H)) !=
        cudaSuccess)
        return e;
    for (int l = 0; l < p.L; ++l) {
        const LayerOffsets &lo = p.layer[l];
        uint16_t *kvl = b.KV + (size_t)l * p.kv_layer_elems;
        // A3 + A4: RMSNorm, QKV (+bias), RoPE, paged KV append
        const Terms A = {{b.A[0], b.A[1], b.A[2]}};
        if ((e = launch_kernel(rmsnorm_rows_kernel, dim3(T), 256, 0, st, 1, p.pdl, b.X, b.W + lo.attn_norm, A, p.H,
                               p.cfg.rms_eps, PEpiQKV::kATerms)) != cudaSuccess)
            return e;
        PEpiQKV eq = {{{b.Q[0], b.Q[1], b.Q[2]}}, kvl, b.pages, b.rope, p.cfg.qkv_bias ? b.W + lo.bqkv : nullptr, P, p.qdim,
                      p.kvdim, p.d, p.nkv, p.kv_page_elems, p.qk_norm ? b.QKraw : nullptr};
        WOperand w;
        if ((e = weight_operand<PEpiQKV>(p, b, p.q8 ? mp.wt_qkv[0] : mp.wqkv[l], mp.wt_qkv, b.W + lo.wqkv, p.nqkv, p.H, st,
                                hook, &w)) != cudaSuccess)
            return e;
        if ((e = gemm(p, mp, mp.a, w, T, p.nqkv, p.H, err, eq, st, hook, "prefill_qkv")) != cudaSuccess)
            return e;
        if (p.qk_norm) {
            // Qwen3 block: per-head q/k norm, then RoPE and the operand / page stores
            const Terms Qt = {{b.Q[0], b.Q[1], b.Q[2]}};
            const dim3 grid(T, (p.nq + p.nkv + 7) / 8);
            if (hook) hook->before("prefill_qk_norm_rope");
            e = launch_kernel(p.d == 128 ? qk_norm_rope_kernel<128> : qk_norm_rope_kernel<64>, grid, 256, 0, st, 1, p.pdl,
                              b.QKraw, b.W + lo.qn, b.W + lo.kn, b.rope, Qt, kvl, b.pages, p.kv_page_elems, P, p.nq,
                              p.nkv, p.cfg.rms_eps);
            if (hook) hook->after("prefill_qk_norm_rope");
            if (e != cudaSuccess) return e;
        }
        // A5: causal attention over the cache (earlier chunks + this one), tensor cores
        if (hook) hook->before("prefill_attention");
        e = launch_attn_tc(p, b, mp, l, P, T, st);
        if (hook) hook->after("prefill_attention");
        if (e != cudaSuccess) return e;
        // A6: O projection + residual
        if ((e = weight_operand<PEpiResidual>(p, b, p.q8 ? mp.wt_o[0] : mp.wo[l], mp.wt_o, b.W + lo.wo, p.H, p.qdim, st, hook,
                                &w)) != cudaSuccess)
            return e;
        if ((e = gemm(p, mp, mp.o, w, T, p.H, p.qdim, err, PEpiResidual{b.X, p.H}, st, hook,
                      "prefill_o_proj")) != cudaSuccess)
            return e;
        // A7: RMSNorm + gate/up + SwiGLU
        if ((e = launch_kernel(rmsnorm_rows_kernel, dim3(T), 256, 0, st, 1, p.pdl, b.X, b.W + lo.ffn_norm, A, p.H,
                               p.cfg.rms_eps, PEpiSwiGLU::kATerms)) != cudaSuccess)
            return e;
        const Terms M = {{b.M[0], b.M[1], b.M[2]}};
        if ((e = weight_operand<PEpiSwiGLU>(p, b, p.q8 ? mp.wt_gu[0] : mp.wgu[l], mp.wt_gu, b.W + lo.wgu, 2 * p.F, p.H, st,
                                hook, &w)) != cudaSuccess)
            return e;
        if ((e = gemm(p, mp, mp.a, w, T, 2 * p.F, p.H, err, PEpiSwiGLU{M, p.F}, st, hook,
                      "prefill_gate_up")) != cudaSuccess)
            return e;
        // A8: down projection + residual
        if ((e = weight_operand<PEpiResidual>(p, b, p.q8 ? mp.wt_d[0] : mp.wd[l], mp.wt_d, b.W + lo.wd, p.H, p.F, st, hook,
                                &w)) != cudaSuccess)
            return e;
        if ((e = gemm(p, mp, mp.m, w, T, p.H, p.F, err, PEpiResidual{b.X, p.H}, st, hook,
                      "prefill_down")) != cudaSuccess)
            return e;
    }
    if (lm_pos_add > 0) {
        // A9 on the chunk's last row only
        return enqueue_lm_head(p, b, b.X + (size_t)(T - 1) * p.H, st, p.pdl, lm_pos_add, hook);
    }
    return cudaSuccess;
}

cudaError_t enqueue_rope_table(const Plan &p, const Bufs &b, cudaStream_t st) {
    const int half = p.d / 2;
    const int n = p.cfg.max_tokens * half;
    rope_table_kernel<<<(n + 255) / 256, 256, 0, st>>>(b.rope, p.cfg.max_tokens, half, p.cfg.rope_theta);
    return cudaGetLastError();
}

}  // namespace wici
