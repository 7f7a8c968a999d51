// Host side of the decode step and of the LM head: shapes, launches and kernel attributes.
#include "decode_step.cuh"

namespace wici {

enum : int { SITE_PROBE = 99 };

// ------------------------------------------------------------ probe kernel ----
__global__ void bounded_wait_probe_kernel(int *err, long long limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(smem_u32(&bar), 0, err, SITE_PROBE, (uint64_t)limit_ns);
}
// ============================================================ host side ====

size_t mega_part_words(int nkv, int group, int d) { return (size_t)nkv * kMaxSplits * group * (d + 2); }

// the (NCH, RPS, FULL) shapes of every supported K (K % 8 == 0, K <= 16384)
#define WICI_GEMV_SHAPES(X)                                                                     \
    X(1, 8, true) X(1, 8, false) X(2, 4, true) X(2, 4, false) X(3, 2, true) X(3, 2, false)     \
    X(4, 2, true) X(4, 2, false) X(5, 1, true) X(5, 1, false) X(6, 1, true) X(6, 1, false)     \
    X(7, 1, true) X(7, 1, false) X(8, 1, true) X(8, 1, false)

template <class Epi>
static void *gemv_fn(int K) {
    const int nch = gemv_nch(K), rps = gemv_rps(K);
    const bool full = (K / 8) == nch * kGemvConsumers;
#define WICI_PICK(N, R, F) \
    if (nch == N && rps == R && full == F) return (void *)gemv_kernel<N, R, F, Epi>;
    WICI_GEMV_SHAPES(WICI_PICK)
#undef WICI_PICK
    return nullptr;
}

template <class Epi>
static cudaError_t set_gemv_attrs() {
#define WICI_ATTR(N, R, F)                                                                              \
    {                                                                                                   \
        cudaError_t e = cudaFuncSetAttribute(gemv_kernel<N, R, F, Epi>,                                \
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,              \
                                             (int)gemv_smem_bytes(1, kGemvRingBytes));                 \
        if (e != cudaSuccess) return e;                                                                 \
    }
    WICI_GEMV_SHAPES(WICI_ATTR)
#undef WICI_ATTR
    return cudaSuccess;
}

// The instantiated shapes: (head dim, GEMV shape of K = hidden, GEMV shape of K = ffn)
using MegaH4096 = GShape<2, 4, true>;     // Llama-3-8B widths: hidden 4096, ffn 14336
using MegaF14336 = GShape<7, 1, true>;
using MegaH2048 = GShape<1, 8, true>;     // Llama-3.2-1B widths: hidden 2048, ffn 8192
using MegaF8192 = GShape<4, 2, true>;
using MegaH5120 = GShape<3, 2, false>;    // Qwen2.5-14B widths: hidden 5120, ffn 13824
using MegaF13824 = GShape<7, 1, false>;
using MegaSmall = GShape<1, 8, false>;    // hidden and ffn below 2048 (e.g. 256 / 688)
using MegaF12288 = GShape<6, 1, true>;    // Qwen3-8B widths: hidden 4096, ffn 12288
// 8-bit block format: 16-element chunks per thread (NCH = ceil(K / 4096)), and
// rows of q8_row_bytes(K) bytes per 32 KB slot: as many as fit, even where a
// unit is a row pair
using Q8H4096 = GShape<1, 7, true>;       // 7 x 4352 B
using Q8F14336 = GShape<4, 2, false>;     // 2 x 15232 B; 896 chunks
using Q8Small = GShape<1, 8, false>;      // 8 x <= 1904 B (K < 2048)
using Q8F12288 = GShape<3, 2, true>;      // 2 x 13056 B
// (head dim, bf16 shape K = hidden, bf16 shape K = ffn, 8-bit format, its shapes)
#define WICI_MEGA_SHAPES(X)                                       \
    X(128, MegaH4096, MegaF14336, false, MegaH4096, MegaF14336)   \
    X(64, MegaH2048, MegaF8192, false, MegaH2048, MegaF8192)      \
    X(128, MegaH5120, MegaF13824, false, MegaH5120, MegaF13824)   \
    X(64, MegaSmall, MegaSmall, false, MegaSmall, MegaSmall)      \
    X(128, MegaH4096, MegaF12288, false, MegaH4096, MegaF12288)   \
    X(128, MegaH4096, MegaF14336, true, Q8H4096, Q8F14336)        \
    X(128, MegaH4096, MegaF12288, true, Q8H4096, Q8F12288)        \
    X(64, MegaSmall, MegaSmall, true, Q8Small, Q8Small)

cudaError_t setup_kernels() {
    cudaError_t e;
#define WICI_MEGA_ATTR(DD, SH, SF, Q8, QH, QF) \
    if ((e = mega_smem<DD, SH, SF, Q8, QH, QF, false>()) != cudaSuccess) return e;
    WICI_MEGA_SHAPES(WICI_MEGA_ATTR)
#undef WICI_MEGA_ATTR
    if ((e = setup_mega_any()) != cudaSuccess) return e;
    return set_gemv_attrs<EpiArgmax>();
}

// Ring geometry: slots of gemv_rps(K) rows, as many as fit kGemvRingBytes (2 to 8).
static void ring_geometry(GemvIn &g) {
    const int rps = gemv_rps(g.K);
    g.slot_bytes = ((uint32_t)rps * (uint32_t)g.K * 2u + 127u) & ~127u;
    int st = (int)(kGemvRingBytes / g.slot_bytes);
    g.stages = st < 2 ? 2 : (st > kGemvMaxStages ? kGemvMaxStages : st);
}

static cudaError_t launch_lm_head(GemvIn g, float *logits, int2 *partials, int *hist, int pos_add, int grid,
                                  cudaStream_t st, bool pdl) {
    ring_geometry(g);
    void *fn = gemv_fn<EpiArgmax>(g.K);
    if (!fn) return cudaErrorInvalidValue;
    EpiArgmax e = {};
    e.logits = logits;
    e.partial = partials;
    e.ctrl = g.ctrl;
    e.hist = hist;
    e.pos_add = pos_add;
    e.best = -INFINITY;
    e.bidx = 0x7fffffff;
    return launch_kernel(reinterpret_cast<void (*)(const GemvIn, const EpiArgmax)>(fn), dim3(grid), kGemvThreads,
                         gemv_smem_bytes(g.stages, g.slot_bytes), st, 1, pdl, g, e);
}

static GemvIn lm_head_in(const uint16_t *W, const uint16_t *gain, const float *x, int H, int V, float eps, int *ctrl) {
    GemvIn g = {};
    g.W = W;
    g.K = H;
    g.n_units = V;
    g.in = x;
    g.gain = gain;
    g.ctrl = ctrl;
    g.eps = eps;
    return g;
}

cudaError_t enqueue_lm_head(const Plan &p, const Bufs &b, const float *x, cudaStream_t st, bool pdl, int pos_add,
                            LaunchHook *hook) {
    GemvIn g = lm_head_in(b.W + p.w_lm, b.W + p.w_final_norm, x, p.H, p.V, p.cfg.rms_eps, b.ctrl);
    if (!p.q8) {   // a decode step follows: the first rows of its first matrix
        g.next_W = b.W + p.layer[0].wqkv;
        g.next_K = p.H;
        g.next_n_units = p.nqkv / 2;
        g.next_rpu = 2;
    }
    if (hook) hook->before("lm_head_argmax");
    const cudaError_t e = launch_lm_head(g, b.logits, b.amax, b.hist, pos_add, p.num_sms * kGemvCtasPerSm, st, pdl);
    if (hook) hook->after("lm_head_argmax");
    return e;
}

cudaError_t enqueue_lm_head_argmax_raw(const uint16_t *W, const uint16_t *gain, const float *x, int H, int V,
                                       float eps, float *logits, int *ctrl, int2 *partials, int *hist, int grid,
                                       cudaStream_t st) {
    return launch_lm_head(lm_head_in(W, gain, x, H, V, eps, ctrl), logits, partials, hist, 0, grid, st, false);
}

// ------------------------------------------------------- persistent decode: host
template <class S>
static bool shape_is(int K) {
    return gemv_nch(K) == S::NCH && gemv_rps(K) == S::RPS && ((K / 8) == S::NCH * kGemvConsumers) == S::FULL;
}

// 8-bit block rows: 16-element chunks, and S::RPS rows of the format in a slot
template <class S>
static bool q8_shape_is(int K) {
    const int nch = (K / 16 + kGemvConsumers - 1) / kGemvConsumers;
    return nch == S::NCH && ((K / 16) == nch * kGemvConsumers) == S::FULL &&
           (size_t)S::RPS * q8_row_bytes((size_t)K) <= kMegaSlotBytes;
}

// the instantiation of this plan's widths and format, or nullptr
static MegaLaunch mega_named_launcher(const Plan &p) {
    if (p.qdim != p.H) return nullptr;
#define WICI_MEGA_PICK(DD, SH, SF, Q8, QH, QF)                                                       \
    if (p.q8 == Q8 && p.d == DD && shape_is<SH>(p.H) && shape_is<SF>(p.F) &&                            \
        (!Q8 || (q8_shape_is<QH>(p.H) && q8_shape_is<QF>(p.F))))                                        \
        return launch_mega<DD, SH, SF, Q8, QH, QF, false>;
    WICI_MEGA_SHAPES(WICI_MEGA_PICK)
#undef WICI_MEGA_PICK
    return nullptr;
}

bool decode_has_named_shape(const Plan &p) { return mega_named_launcher(p) != nullptr; }

static cudaError_t enqueue_mega(const Plan &p, const Bufs &b, const CUtensorMap &map_kv, cudaStream_t st,
                                MegaLaunch fn) {
    MegaArgs a = {};
    a.W = b.W;
    a.lstride = p.L > 1 ? p.layer[1].wqkv - p.layer[0].wqkv : 0;
    a.l0 = p.layer[0];
    a.w_embed = p.w_embed;
    a.w_final_norm = p.w_final_norm;
    a.w_lm = p.w_lm;
    a.KV = b.KV;
    a.kv_layer_elems = p.kv_layer_elems;
    a.page_elems = p.kv_page_elems;
    a.ctrl = b.ctrl;
    a.hist = b.hist;
    a.logits = b.logits;
    a.amax = b.amax;
    a.rope = b.rope;
    a.pages = b.pages;
    a.tqkv = b.tqkv; a.tpart = b.tpart; a.to = b.to; a.txo = b.txo; a.txd = b.txd; a.tm = b.tm;
    a.bound = b.mega_bound;
    a.cta_time = b.mega_time;
    a.L = p.L; a.H = p.H; a.F = p.F; a.V = p.V;
    a.nqkv = p.nqkv; a.qdim = p.qdim; a.kvdim = p.kvdim; a.nkv = p.nkv; a.group = p.group;
    a.max_pages = p.max_pages;
    // warps that take pages: as many as the group's states leave room for
    const int fit = (int)(kMegaStateBytes / ((size_t)p.group * (p.d + 4) * sizeof(float)));
    a.nsets = fit < kGemvWarps ? fit : kGemvWarps;
    const int grid = p.num_sms;   // the row-share table has an entry for each
    // one CTA per (KV head, split); more KV heads than CTAs: one split each
    a.splits = grid / p.nkv < 1 ? 1 : grid / p.nkv < kMaxSplits ? grid / p.nkv : kMaxSplits;
    a.bias = p.cfg.qkv_bias;
    a.qk_norm = p.qk_norm;
    a.eps = p.cfg.rms_eps;
    a.qscale = 1.4426950408889634f / sqrtf((float)p.d);
    return fn(map_kv, a, grid, st);
}

cudaError_t enqueue_decode_step(const Plan &p, const Bufs &b, const CUtensorMap &map_kv, cudaStream_t st,
                                LaunchHook *hook) {
    MegaLaunch fn = mega_named_launcher(p);
    if (!fn && (p.q8 || p.qk_norm)) return cudaErrorInvalidValue;   // refused at create
    // also a share of fewer SMs than KV heads: the bf16 shapes give a CTA one head at most
    if (!fn || (!p.q8 && p.num_sms < p.nkv)) fn = mega_any_launcher(p.d);
    if (hook) hook->before("decode_step");
    const cudaError_t e = enqueue_mega(p, b, map_kv, st, fn);
    if (hook) hook->after("decode_step");
    return e;
}

cudaError_t enqueue_bounded_wait_probe(int *err, int64_t limit_ns, cudaStream_t st) {
    bounded_wait_probe_kernel<<<1, 32, 0, st>>>(err, (long long)limit_ns);
    return cudaGetLastError();
}

}  // namespace wici
