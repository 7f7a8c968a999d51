// The persistent decode step: device code and its launch.
#pragma once
#include "gemv.cuh"

namespace wici {

// ======================================================= persistent decode ====
// The whole decode step (Sec. 5.1: one forward pass per generated token) as one
// cooperative kernel, one CTA per SM.  Weight streaming does not depend on the
// data, so the producer warp walks the step's weights (per layer: this CTA's
// rows of Wqkv, its KV pages, its rows of Wo, Wg|Wu and Wd; then the LM head)
// through one TMA ring without ever waiting on a data dependency, only on free
// ring slots.  The eight consumer warps run the phases in order.
//
// Exchange between CTAs: every vector one phase hands to the next (q|k|v, the
// attention split states and output, the residual after O and after down, the
// SwiGLU vector) is an array of 64-bit words, the fp32 value below a 32-bit tag
// that names the layer of the step.  A consumer polls the words it
// needs until they carry the tag; a word is written with one 64-bit store, so a
// value is never seen without its tag and no fence, counter or grid barrier is
// needed.  A grid barrier (store, fence, atomic, poll, then load) cost 1.0 to 2.2
// us and the load after it 0.7 us, five times a layer; polling the data itself
// is one store and one load.
//
// No word is overwritten while someone may still poll its old tag: a CTA that
// has rows of a phase publishes them only after it has read that phase's whole
// input, every phase's input holds words of every CTA that has rows of the phase
// before, and a CTA without rows of a phase does not read its input.  So a CTA
// that writes layer l+1's words of an array has read words that depend on every
// read of layer l's.
//
// Measured (per layer of a decode step, 8B widths at context ~1060, bf16): 79.9
// us with five grid barriers a layer, 70 us now; at 1B widths 35.0 and 27.5 us.
constexpr int kMegaSlots = 6;
constexpr uint32_t kMegaSlotBytes = 32768;
constexpr int kMaxSplits = 32;                  // attention splits of one KV head
// attention scratch: per page set, per query head of the group, an O row, m and l
constexpr size_t kMegaStateBytes = 21504;
// dynamic shared memory: [ring, 1024-byte aligned for the swizzled page boxes][reduction scratch][attention states]
constexpr size_t kMegaSmem = 1024 + (size_t)kMegaSlots * kMegaSlotBytes + kGemvRedBytes + kMegaStateBytes;

enum : int { SITE_MEGA_EMPTY = 51, SITE_MEGA_FULL = 52, SITE_MEGA_DRAIN = 53, SITE_MEGA_DATA = 54 };

template <int NCH_, int RPS_, bool FULL_>
struct GShape {
    static constexpr int NCH = NCH_, RPS = RPS_;
    static constexpr bool FULL = FULL_;
};

struct MegaArgs {
    const uint16_t *W;          // weight arena
    size_t lstride;             // elements between the same tensor of consecutive layers
    LayerOffsets l0;            // layer 0 offsets
    size_t w_embed, w_final_norm, w_lm;
    uint16_t *KV;
    size_t kv_layer_elems, page_elems;
    int *ctrl, *hist;
    float *logits;
    int2 *amax;
    const float2 *rope;
    const int *pages;
    // tagged words: q|k|v [nqkv] (qk_norm: q and k before their norms and RoPE), attention split
    // states [nkv][splits][group][d + 2], attention output [qdim], the residual after O and
    // after down [H], the SwiGLU vector [F]
    uint64_t *tqkv, *tpart, *to, *txo, *txd, *tm;
    uint32_t *bound;            // [grid + 1] share boundaries of the GEMV phases (2^24 = all rows)
    float *cta_time;            // [grid] each CTA's gate/up streaming time in the last step (us)
    int L, H, F, V, nqkv, qdim, kvdim, nkv, group, nsets, splits, max_pages;
    int bias, qk_norm;
    float eps, qscale;
};

struct MegaRing {
    uint32_t full0, empty0, data0;   // shared-memory addresses
    int n;   // slots issued (producer) or consumed (consumer) so far
    int *abort;                      // shared flag: a consumer wait gave up
    uint32_t b0, b1;                 // this CTA's share of every GEMV phase: [b0, b1) / 2^24
};

// units [u0, u1) of an n-unit phase for the share [b0, b1) (fixed point, 2^24 = all)
__device__ __forceinline__ int mega_unit(uint32_t b, int n_units) {
    return (int)(((unsigned long long)b * (unsigned long long)n_units) >> 24);
}

// ------------------------------------------------------------ tagged words --
__device__ __forceinline__ uint64_t tagged(float v, uint32_t tag) {
    return ((uint64_t)tag << 32) | (uint64_t)__float_as_uint(v);
}
__device__ __forceinline__ float tagged_value(uint64_t w) { return __uint_as_float((uint32_t)w); }
__device__ __forceinline__ bool has_tag(uint64_t w, uint32_t tag) { return (uint32_t)(w >> 32) == tag; }

__device__ __forceinline__ void st_tagged(uint64_t *p, float v, uint32_t tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(tagged(v, tag)) : "memory");
}
__device__ __forceinline__ void st_tagged2(uint64_t *p, float v0, float v1, uint32_t tag) {   // 16-byte aligned
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(tagged(v0, tag)), "l"(tagged(v1, tag))
                 : "memory");
}
__device__ __forceinline__ uint64_t ld_tagged(const uint64_t *p) {
    uint64_t w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ void ld_tagged2(const uint64_t *p, uint64_t &a, uint64_t &b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
// four words when `go`, 32-byte aligned; the old contents of w otherwise
__device__ __forceinline__ void ld_tagged4_if(const uint64_t *p, uint64_t (&w)[4], bool go) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
        "@p ld.relaxed.gpu.global.v4.u64 {%0, %1, %2, %3}, [%4];\n\t}"
        : "+l"(w[0]), "+l"(w[1]), "+l"(w[2]), "+l"(w[3])
        : "l"(p), "r"((uint32_t)go)
        : "memory");
}

// Bounds one thread's polling: false once the wait limit has passed or another
// CTA has recorded an error.  No sleep between polls: one of 20 ns cost 1% of a
// 1B-width step and 4% of an 8-bit one, 200 ns 3% and 5%.
struct PollLimit {
    uint64_t t0;
    uint32_t it;
    __device__ __forceinline__ PollLimit() : t0(0), it(0) {}
    __device__ __forceinline__ bool again(int *err) {
        if (it == 0) t0 = globaltimer_ns();
        if ((++it & 31u) == 0u) {
            if (*reinterpret_cast<volatile int *>(err) != 0) return false;
            if (globaltimer_ns() - t0 > kWaitLimitNs) {
                atomicCAS(err, 0, SITE_MEGA_DATA);
                return false;
            }
        }
        return it < 0x7FFFFFFFu;
    }
};

// This thread's chunks c = tid + 256 j of CW elements of a tagged vector, every
// load in flight at once; words that do not carry `tag` yet are loaded again.
template <int NCH, int CW, bool FULL>
__device__ __forceinline__ bool mega_input(float (&h)[NCH][CW], const uint64_t *in, uint32_t tag, int nchunks,
                                           int *err) {
    constexpr int V = CW / 4, NV = NCH * V;
    static_assert(NV <= 32, "pending mask");
    uint64_t w[NV][4];
    uint32_t pend = 0;
#pragma unroll
    for (int j = 0; j < NCH; ++j)
        if (FULL || (int)threadIdx.x + kGemvConsumers * j < nchunks) pend |= ((1u << V) - 1u) << (V * j);
#pragma unroll
    for (int i = 0; i < NV; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) w[i][e] = 0;
    PollLimit lim;
    bool ok = true;
    while (true) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
            ld_tagged4_if(in + ((size_t)threadIdx.x + kGemvConsumers * (i / V)) * CW + 4 * (i % V), w[i],
                          (pend >> i) & 1u);
#pragma unroll
        for (int i = 0; i < NV; ++i)
            if (has_tag(w[i][0], tag) && has_tag(w[i][1], tag) && has_tag(w[i][2], tag) && has_tag(w[i][3], tag))
                pend &= ~(1u << i);
        if (pend == 0) break;
        if (!lim.again(err)) {
            ok = false;
            break;
        }
    }
#pragma unroll
    for (int i = 0; i < NV; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) h[i / V][4 * (i % V) + e] = tagged_value(w[i][e]);
    return ok;
}

// ------------------------------------------------------- decode epilogues --
// unit(u, v): v[0..rpu) are the finished dot products of unit u's rows;
// prefetch(u): this thread finishes unit u in the phase's first batch of rows, so
// what the epilogue needs from memory is loaded while the weights stream.

struct MEpiResidual {  // out[u] = prev[u] + v   (O projection, down projection)
    const uint64_t *prev;    // the residual before this phase (this CTA wrote its own units), or
    const uint16_t *embed;   // layer 0: the token's embedding row
    uint32_t prev_tag;
    uint64_t *out;
    uint32_t tag;
    uint64_t pre;
    __device__ uint64_t base(int u) const {
        return embed ? tagged(bf16_to_f32(embed[u]), prev_tag) : ld_tagged(prev + u);
    }
    __device__ void prefetch(int u) { pre = base(u); }
    __device__ void unit(int u, const float *v, bool first) {
        // written by this CTA before the barriers of this phase: a word loaded too early
        // for it still carries an old tag, one loaded here does not
        uint64_t w = first ? pre : base(u);
        if (!has_tag(w, prev_tag)) w = base(u);
        st_tagged(out + u, tagged_value(w) + v[0], tag);
    }
};

struct MEpiSwiGLU {    // rows (2u, 2u+1) are (gate_u, up_u): m[u] = silu(g) * u
    uint64_t *m;
    uint32_t tag;
    __device__ void prefetch(int) {}
    __device__ void unit(int u, const float *v, bool) {
        const float gt = v[0];
        st_tagged(m + u, gt / (1.0f + expf(-gt)) * v[1], tag);
    }
};

// Packed QKV rows (rows i and i + D/2 of a head are neighbours): q and k after RoPE (before their norms
// with qk_norm) and v, in natural order; the attention phase stores K and V.
template <int D>
struct MEpiQKV {
    uint64_t *t;
    uint32_t tag;
    const float2 *rope;      // (cos, sin) of this position, in shared memory
    const uint16_t *bias;    // packed like the rows, or nullptr
    int qkdim;
    bool raw;
    uint32_t pre;
    __device__ void prefetch(int u) {
        if (bias) pre = *reinterpret_cast<const uint32_t *>(bias + 2 * u);
    }
    __device__ void unit(int u, const float *v, bool first) {
        const int r0 = 2 * u;
        float a = v[0], b = v[1];
        if (bias) {
            const uint32_t w = first ? pre : *reinterpret_cast<const uint32_t *>(bias + r0);
            a += bf16lo(w);
            b += bf16hi(w);
        }
        if (r0 < qkdim) {
            const int i = (r0 % D) >> 1;
            uint64_t *dst = t + (r0 - r0 % D) + i;
            if (!raw) {
                const float2 cs = rope[i];
                const float ra = a * cs.x - b * cs.y;
                b = b * cs.x + a * cs.y;
                a = ra;
            }
            st_tagged(dst, a, tag);
            st_tagged(dst + D / 2, b, tag);
        } else {
            st_tagged2(t + r0, a, b, tag);
        }
    }
};

struct MEpiArgmax : EpiArgmax {
    __device__ void prefetch(int) {}
    __device__ void unit(int u, const float *v, bool) { EpiArgmax::unit(u, v); }
};

// ----------------------------------------------------------- producer side --
// The producer keeps at least kMegaFlightBytes of copies in flight per SM (and two
// slots), and lets landed slots fill the rest of the ring.  That is
// what the HBM needs (152 SMs x 64 KB over ~1.3 us); more only queues in the memory
// system, in front of the words that the phases exchange: with the whole ring in
// flight and 192 KB of gate/up rows per SM moved to L2 during the attention phase,
// a word took up to 4 us to arrive, and a step of the 8B widths 2636 us against
// 2491 (1B: 589 against 555); one slot in flight starves the HBM (3136 us).
constexpr uint32_t kMegaFlightBytes = 65536;
__device__ __forceinline__ int mega_flight(uint32_t slot_bytes) {
    return min(kMegaSlots, max(2, (int)((kMegaFlightBytes + slot_bytes - 1) / slot_bytes)));
}

// wait until ring slot R.n is free and at most `flight` - 1 earlier copies are still landing
__device__ __forceinline__ bool mp_slot(const MegaRing &R, int flight, int *err) {
    if (R.n >= kMegaSlots &&
        !mbar_wait(R.empty0 + 8 * (R.n % kMegaSlots), ((R.n / kMegaSlots) + 1) & 1, err, SITE_MEGA_EMPTY))
        return false;
    const int k = R.n - flight;
    return k < 0 || mbar_wait(R.full0 + 8 * (k % kMegaSlots), (k / kMegaSlots) & 1, err, SITE_MEGA_EMPTY);
}

// this CTA's rows of an n_units-unit matrix whose rows are row_bytes long (bf16:
// 2K; the 8-bit block format: q8_row_bytes(K)), RPS rows per ring slot
__device__ inline bool mp_rows(MegaRing &R, const uint16_t *W, uint32_t row_bytes, int n_units, int rpu, int RPS,
                        int *err, uint64_t pol) {
    const int u0 = mega_unit(R.b0, n_units);
    const int u1 = mega_unit(R.b1, n_units);
    const int total_rows = (u1 - u0) * rpu;
    const int nst = (total_rows + RPS - 1) / RPS;
    const uint8_t *src = reinterpret_cast<const uint8_t *>(W) + (size_t)u0 * rpu * row_bytes;
    const int flight = mega_flight((uint32_t)RPS * row_bytes);
    for (int s = 0; s < nst; ++s) {
        const int slot = R.n % kMegaSlots;
        if (!mp_slot(R, flight, err)) return false;
        const int rows = min(RPS, total_rows - s * RPS);
        const uint32_t bytes = (uint32_t)rows * row_bytes;
        mbar_arrive_expect_tx(R.full0 + 8 * slot, bytes);
        bulk_g2s(R.data0 + slot * kMegaSlotBytes, src + (size_t)s * RPS * row_bytes, bytes, R.full0 + 8 * slot, pol);
        ++R.n;
    }
    return true;
}

// the pages of this CTA's attention split (its K and V blocks)
struct MegaSplit {
    int g, r, p0, n, npages, splits;
    bool active;
};

// unit: a (KV head, split) pair; a CTA has more than one only where KV heads outnumber the
// grid, and then every head is one split
__device__ __forceinline__ MegaSplit mega_split(const MegaArgs &a, int len, int unit) {
    MegaSplit sp;
    sp.npages = (len + kPage - 1) / kPage;
    // as many splits as there are: a page takes its warp longer than a state takes to combine
    // (a page for every warp of a split before the next split: 8B widths 2481 -> 2512 us)
    const int pps = (sp.npages + a.splits - 1) / a.splits;
    sp.splits = (sp.npages + pps - 1) / pps;
    sp.g = unit / a.splits;
    sp.r = unit % a.splits;
    sp.active = unit < a.nkv * a.splits && sp.r < sp.splits;
    sp.p0 = sp.r * pps;
    sp.n = sp.active ? min(sp.npages, sp.p0 + pps) - sp.p0 : 0;
    return sp;
}

// A page in a ring slot: K then V, each as D/64 boxes of 16 keys x 64 d values
// (128-byte rows, 128-byte swizzle: conflict-free ldmatrix), kPagesPerSlot pages
// to a slot.
template <int D>
struct MegaPage {
    static constexpr uint32_t CHUNK = kPage * 128;                 // one box
    static constexpr uint32_t V = (D / 64) * CHUNK;                // V's offset in the page
    static constexpr uint32_t BYTES = 2 * V;
    static constexpr int PER_SLOT = (int)(kMegaSlotBytes / BYTES);
};

__device__ __forceinline__ void mega_tma_page(uint32_t dst, const CUtensorMap *map, int d0, int g, int kv, int page,
                                              uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
        "%6}], [%7];" ::"r"(dst),
        "l"((uint64_t)map), "r"(d0), "r"(0), "r"(g), "r"(kv), "r"(page), "r"(bar)
        : "memory");
}

template <int D>
__device__ bool mp_pages(MegaRing &R, const MegaArgs &a, const CUtensorMap *map_kv, int layer, const MegaSplit &sp,
                         int *err) {
    using PG = MegaPage<D>;
    for (int i0 = 0; i0 < sp.n; i0 += PG::PER_SLOT) {
        const int slot = R.n % kMegaSlots;
        if (!mp_slot(R, 2, err)) return false;
        const int np = min(PG::PER_SLOT, sp.n - i0);
        const uint32_t fb = R.full0 + 8 * slot;
        mbar_arrive_expect_tx(fb, (uint32_t)np * PG::BYTES);
        for (int i = 0; i < np; ++i) {
            const int page = layer * a.max_pages + a.pages[sp.p0 + i0 + i];
            const uint32_t dst = R.data0 + slot * kMegaSlotBytes + (uint32_t)i * PG::BYTES;
#pragma unroll
            for (int c = 0; c < D / 64; ++c) {
                mega_tma_page(dst + c * PG::CHUNK, map_kv, 64 * c, sp.g, 0, page, fb);
                mega_tma_page(dst + PG::V + c * PG::CHUNK, map_kv, 64 * c, sp.g, 1, page, fb);
            }
        }
        ++R.n;
    }
    return true;
}

// ----------------------------------------------------------- consumer side --
// consumers only (8 warps): bar.sync 1, 256 is consumer_sync()

// The rows of a finished batch, summed over the eight warps in fixed order, to the epilogue.
template <class Epi>
__device__ __forceinline__ void mega_flush(const float *red, int buf, int bunits, int rpu, int unit0, bool first,
                                           float scale, Epi &epi) {
    for (int t = threadIdx.x; t < bunits; t += kGemvConsumers) {
        float v[2];
        for (int j = 0; j < rpu; ++j) {
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < kGemvWarps; ++w) sum += red[(size_t)(buf * kGemvWarps + w) * kRedRows + t * rpu + j];
            v[j] = sum * scale;
        }
        epi.unit(unit0 + t, v, first);
    }
}

// One GEMV phase of the consumers: the rows of units [u0, u1) of a K-column matrix
// against the tagged vector `in` (RMSNorm'd with `gain` when given), or against the
// token's embedding row `embed` (layer 0).  *t_data, when given, receives the time
// at which the input was complete.
template <class SH, class Epi>
__device__ bool mc_gemv(MegaRing &R, float *red, int K, int n_units, int rpu, const uint64_t *in, uint32_t tag,
                        const uint16_t *gain, const uint16_t *embed, float eps, int *err, Epi &epi, float *s_part,
                        uint64_t *t_data) {
    constexpr int NCH = SH::NCH, RPS = SH::RPS;
    constexpr bool FULL = SH::FULL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int u0 = mega_unit(R.b0, n_units);
    const int u1 = mega_unit(R.b1, n_units);
    const int total_rows = (u1 - u0) * rpu;
    const int nst = (total_rows + RPS - 1) / RPS;
    if (nst == 0) return true;   // no rows: the input is not read (see the exchange rule above)
    [[maybe_unused]] const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const int nchunks = K >> 3;
    if (tid < u1 - u0) epi.prefetch(u0 + tid);
    uint4 gw[NCH];
    if (gain) {   // the norm's gain comes from HBM: ask for it before waiting for the input
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = tid + kGemvConsumers * j;
            gw[j] = FULL || c < nchunks ? *reinterpret_cast<const uint4 *>(gain + c * 8) : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    float h[NCH][8];
    bool ok = true;
    if (embed) {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = tid + kGemvConsumers * j;
            const uint4 w =
                FULL || c < nchunks ? *reinterpret_cast<const uint4 *>(embed + c * 8) : make_uint4(0u, 0u, 0u, 0u);
            h[j][0] = bf16lo(w.x); h[j][1] = bf16hi(w.x); h[j][2] = bf16lo(w.y); h[j][3] = bf16hi(w.y);
            h[j][4] = bf16lo(w.z); h[j][5] = bf16hi(w.z); h[j][6] = bf16lo(w.w); h[j][7] = bf16hi(w.w);
        }
    } else {
        ok = mega_input<NCH, 8, FULL>(h, in, tag, nchunks, err);
    }
    if (gain) {
        float ss = 0.f;
#pragma unroll
        for (int j = 0; j < NCH; ++j)
#pragma unroll
            for (int e = 0; e < 8; ++e) ss = fmaf(h[j][e], h[j][e], ss);
        ss = warp_sum(ss);
        if (lane == 0) s_part[warp] = ss;
        if (consumer_sync_or(!ok)) return false;
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < kGemvWarps; ++w) tot += s_part[w];
        const float rinv = 1.0f / sqrtf(tot / (float)K + eps);
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const float gg[8] = {bf16lo(gw[j].x), bf16hi(gw[j].x), bf16lo(gw[j].y), bf16hi(gw[j].y),
                                 bf16lo(gw[j].z), bf16hi(gw[j].z), bf16lo(gw[j].w), bf16hi(gw[j].w)};
#pragma unroll
            for (int e = 0; e < 8; ++e) h[j][e] = h[j][e] * rinv * gg[e];
        }
    } else if (consumer_sync_or(!ok)) {   // also: every warp is past the previous phase's last flush
        return false;
    }
    if (t_data) *t_data = globaltimer_ns();

    const uint32_t row_bytes = (uint32_t)K * 2u;
    const bool tail_ok = FULL || tid + kGemvConsumers * (NCH - 1) < nchunks;
    int buf = 0, brow = 0, bunit0 = 0;
    for (int s = 0; s < nst; ++s) {
        const int slot = R.n % kMegaSlots;
        const int rows = min(RPS, total_rows - s * RPS);
        // after a wait gives up every thread still reaches the same barriers; they
        // leave together at the next flush
        ok = ok && !*reinterpret_cast<volatile int *>(R.abort) &&
             mbar_wait(R.full0 + 8 * slot, (R.n / kMegaSlots) & 1, err, SITE_MEGA_FULL);
        if (!ok) *R.abort = 1;
        float acc[RPS];
        const uint32_t sb = R.data0 + (uint32_t)slot * kMegaSlotBytes + (uint32_t)tid * 16u;
        if constexpr (!FULL) {
            // this thread's chunks of all RPS rows into registers (past the last row: old bytes of
            // the ring; no row's sum meets another's, and those are dropped), then the slot is free:
            // its next copy need not wait for the products (steps of hidden 3072 414 -> 367 us,
            // Qwen2.5-14B widths 637 -> 597, the 8-bit format at Qwen3-8B widths 524 -> 470)
            uint4 w[RPS][NCH];
#pragma unroll
            for (int r = 0; r < RPS; ++r)
#pragma unroll
                for (int j = 0; j < NCH; ++j)
                    w[r][j] = j < NCH - 1 || tail_ok ? lds128(sb + r * row_bytes + j * kGemvConsumers * 16) : zero;
            __syncwarp();
            if (lane == 0) mbar_arrive(R.empty0 + 8 * slot);
            ++R.n;
#pragma unroll
            for (int r = 0; r < RPS; ++r) {
                acc[r] = 0.f;
#pragma unroll
                for (int j = 0; j < NCH; ++j) acc[r] = dot8(w[r][j], h[j], acc[r]);
            }
        } else {
            // without tails, loads and products interleaved: measured better at the 1B widths (520 us
            // against 540) and equal at the 8B ones, the two of these shapes that were tried
#pragma unroll
            for (int r = 0; r < RPS; ++r) acc[r] = 0.f;
            if (!ok) {
            } else if (rows == RPS) {
#pragma unroll
                for (int r = 0; r < RPS; ++r)
#pragma unroll
                    for (int j = 0; j < NCH; ++j)
                        acc[r] = dot8(lds128(sb + r * row_bytes + j * kGemvConsumers * 16), h[j], acc[r]);
            } else {
#pragma unroll
                for (int r = 0; r < RPS; ++r)
                    if (r < rows)
#pragma unroll
                        for (int j = 0; j < NCH; ++j)
                            acc[r] = dot8(lds128(sb + r * row_bytes + j * kGemvConsumers * 16), h[j], acc[r]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(R.empty0 + 8 * slot);
            ++R.n;
        }
        warp_rows_store<RPS>(acc, red + (size_t)(buf * kGemvWarps + warp) * kRedRows + brow, rows, lane);
        brow += rows;
        if (s == nst - 1 || brow + RPS > kRedRows) {
            if (consumer_sync_or(!ok)) return false;
            const int bunits = brow / rpu;
            mega_flush(red, buf, bunits, rpu, u0 + bunit0, bunit0 == 0, 1.0f, epi);
            bunit0 += bunits;
            brow = 0;
            buf ^= 1;
        }
    }
    return true;
}

// One GEMV phase over a matrix in the 8-bit block format (rows of
// q8_row_bytes(K) bytes), same role as mc_gemv.  Thread t owns the 16-element
// chunks c = t + 256 j of the input, as byte digits of its fixed-point form.
// ND: byte digits of the fixed-point input (3: 24 bits; 2: 16 bits)
template <class QS, int ND, class Epi>
__device__ bool mc_gemv_q8(MegaRing &R, float *red, int K, int n_units, int rpu, const uint64_t *in, uint32_t tag,
                           const uint16_t *gain, const uint16_t *embed, float eps, int *err, Epi &epi, float *s_part,
                           uint64_t *t_data) {
    static_assert(ND == 2 || ND == 3, "two or three input digits");
    constexpr int NCH = QS::NCH, RPS = QS::RPS;
    constexpr bool FULL = QS::FULL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int u0 = mega_unit(R.b0, n_units);
    const int u1 = mega_unit(R.b1, n_units);
    const int total_rows = (u1 - u0) * rpu;
    const int nst = (total_rows + RPS - 1) / RPS;
    if (nst == 0) return true;   // no rows: the input is not read (see the exchange rule above)
    [[maybe_unused]] const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const int nchunks = K >> 4;
    if (tid < u1 - u0) epi.prefetch(u0 + tid);
    uint4 gw[NCH][2];
    if (gain) {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = tid + kGemvConsumers * j;
#pragma unroll
            for (int hv = 0; hv < 2; ++hv)
                gw[j][hv] = FULL || c < nchunks ? *reinterpret_cast<const uint4 *>(gain + c * 16 + hv * 8)
                                                : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    float h[NCH][16];
    bool ok = true;
    if (embed) {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = tid + kGemvConsumers * j;
#pragma unroll
            for (int hv = 0; hv < 2; ++hv) {
                const uint4 w = FULL || c < nchunks ? *reinterpret_cast<const uint4 *>(embed + c * 16 + hv * 8)
                                                    : make_uint4(0u, 0u, 0u, 0u);
                float *d = h[j] + hv * 8;
                d[0] = bf16lo(w.x); d[1] = bf16hi(w.x); d[2] = bf16lo(w.y); d[3] = bf16hi(w.y);
                d[4] = bf16lo(w.z); d[5] = bf16hi(w.z); d[6] = bf16lo(w.w); d[7] = bf16hi(w.w);
            }
        }
    } else {
        ok = mega_input<NCH, 16, FULL>(h, in, tag, nchunks, err);
    }
    // with the RMSNorm gain applied (before the common factor 1/rms), and the
    // largest magnitude for the fixed point: one reduction of (sum of squares, max)
    float ss = 0.f, mx = 0.f;
    if (gain) {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
#pragma unroll
            for (int e = 0; e < 16; ++e) ss = fmaf(h[j][e], h[j][e], ss);
#pragma unroll
            for (int hv = 0; hv < 2; ++hv) {
                const uint4 g4 = gw[j][hv];
                const float gg[8] = {bf16lo(g4.x), bf16hi(g4.x), bf16lo(g4.y), bf16hi(g4.y),
                                     bf16lo(g4.z), bf16hi(g4.z), bf16lo(g4.w), bf16hi(g4.w)};
#pragma unroll
                for (int e = 0; e < 8; ++e) h[j][hv * 8 + e] *= gg[e];
            }
        }
    }
#pragma unroll
    for (int j = 0; j < NCH; ++j)
#pragma unroll
        for (int e = 0; e < 16; ++e) mx = fmaxf(mx, fabsf(h[j][e]));
    if (gain) ss = warp_sum(ss);
    mx = warp_max(mx);
    if (lane == 0) {
        s_part[warp] = ss;
        s_part[kGemvWarps + warp] = mx;
    }
    if (consumer_sync_or(!ok)) return false;
    float tot = 0.f, M = 0.f;
#pragma unroll
    for (int w = 0; w < kGemvWarps; ++w) {
        tot += s_part[w];
        M = fmaxf(M, s_part[kGemvWarps + w]);
    }
    if (gain) {
        const float rinv = 1.0f / sqrtf(tot / (float)K + eps);
        M *= rinv;
#pragma unroll
        for (int j = 0; j < NCH; ++j)
#pragma unroll
            for (int e = 0; e < 16; ++e) h[j][e] *= rinv;
    }
    // fixed point: M * 2^E just below 2^(8 ND - 1) for the largest magnitude M
    // (values that round past the limit are clamped to it)
    constexpr int XBITS = 8 * ND - 1;
    const int E = M > 0.f ? min(XBITS - 1 - ilogbf(M), 120) : 0;
    const float to_fixed = ldexpf(1.0f, E), from_fixed = ldexpf(1.0f, -E);
    // byte digits, most significant (signed) first: X = sum_i X_i 256^(ND-1-i); four
    // values' bytes are transposed into ND words with byte permutes
    uint32_t dg[NCH][ND][4];   // [chunk][digit][4 words of 4 byte digits]
#pragma unroll
    for (int j = 0; j < NCH; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t X[4];
#pragma unroll
            for (int b = 0; b < 4; ++b)
                X[b] = (uint32_t)max(min(__float2int_rn(h[j][4 * k + b] * to_fixed), (1 << XBITS) - 1),
                                     -(1 << XBITS) + 1);
            // bytes (0, 1) of X0, X1 and of X2, X3 side by side, then byte i of all four
            const uint32_t lo01 = __byte_perm(X[0], X[1], 0x5140), lo23 = __byte_perm(X[2], X[3], 0x5140);
            dg[j][ND - 1][k] = __byte_perm(lo01, lo23, 0x5410);
            dg[j][ND - 2][k] = __byte_perm(lo01, lo23, 0x7632);
            if constexpr (ND == 3) {
                const uint32_t hi01 = __byte_perm(X[0], X[1], 0x0062), hi23 = __byte_perm(X[2], X[3], 0x0062);
                dg[j][0][k] = __byte_perm(hi01, hi23, 0x5410);
            }
        }
    if (t_data) *t_data = globaltimer_ns();

    const uint32_t row_bytes = (uint32_t)q8_row_bytes((size_t)K);
    const bool tail_ok = FULL || tid + kGemvConsumers * (NCH - 1) < nchunks;
    int buf = 0, brow = 0, bunit0 = 0;
    for (int s = 0; s < nst; ++s) {
        const int slot = R.n % kMegaSlots;
        const int rows = min(RPS, total_rows - s * RPS);
        ok = ok && !*reinterpret_cast<volatile int *>(R.abort) &&
             mbar_wait(R.full0 + 8 * slot, (R.n / kMegaSlots) & 1, err, SITE_MEGA_FULL);
        if (!ok) *R.abort = 1;
        // as mc_gemv's shapes with tails; chunk c: codes at byte 16 c of the row, its block's scale at byte K + 2 (c / 2)
        const uint32_t s0 = R.data0 + (uint32_t)slot * kMegaSlotBytes;
        const uint32_t sb = s0 + (uint32_t)tid * 16u, sc = s0 + (uint32_t)K + (uint32_t)(tid >> 1) * 2u;
        uint4 w[RPS][NCH];
        float d[RPS][NCH];
#pragma unroll
        for (int r = 0; r < RPS; ++r)
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const bool in = j < NCH - 1 || tail_ok;
                w[r][j] = in ? lds128(sb + r * row_bytes + j * kGemvConsumers * 16) : zero;
                d[r][j] = in ? lds_f16(sc + r * row_bytes + j * (kGemvConsumers / 2) * 2) : 0.f;
            }
        __syncwarp();
        if (lane == 0) mbar_arrive(R.empty0 + 8 * slot);
        ++R.n;
        float acc[RPS];
#pragma unroll
        for (int r = 0; r < RPS; ++r) {
            acc[r] = 0.f;
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const uint32_t ws[4] = {w[r][j].x, w[r][j].y, w[r][j].z, w[r][j].w};
                int a[ND];
#pragma unroll
                for (int i = 0; i < ND; ++i) a[i] = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int i = 0; i < ND; ++i)
                        a[i] = i == 0 ? dp4a_ss(ws[k], dg[j][i][k], a[i]) : dp4a_su(ws[k], dg[j][i][k], a[i]);
                float cv = small_int_to_f32(a[0]);
#pragma unroll
                for (int i = 1; i < ND; ++i) cv = fmaf(cv, 256.0f, small_int_to_f32(a[i]));
                acc[r] = fmaf(d[r][j], cv, acc[r]);
            }
        }
        warp_rows_store<RPS>(acc, red + (size_t)(buf * kGemvWarps + warp) * kRedRows + brow, rows, lane);
        brow += rows;
        if (s == nst - 1 || brow + RPS > kRedRows) {
            if (consumer_sync_or(!ok)) return false;
            const int bunits = brow / rpu;
            mega_flush(red, buf, bunits, rpu, u0 + bunit0, bunit0 == 0, from_fixed, epi);
            bunit0 += bunits;
            brow = 0;
            buf ^= 1;
        }
    }
    return true;
}

// Input digits of the 8-bit GEMV phases: three (24 bits) for QKV, whose outputs
// become the bf16 K/V and the queries, and kQ8RestDigits for O, gate/up, down.
#ifndef WICI_Q8_REST_DIGITS
#define WICI_Q8_REST_DIGITS 3
#endif
constexpr int kQ8QkvDigits = 3, kQ8RestDigits = WICI_Q8_REST_DIGITS;

// one GEMV phase in its matrix's format; ANY: the bf16 shape of K, of at most MAXN chunks
// a thread, picked here
template <bool ANY, bool Q8, class S, int ND, int MAXN, class Epi>
__device__ __forceinline__ bool mc_phase(MegaRing &R, float *red, int K, int n_units, int rpu, const uint64_t *in,
                                         uint32_t tag, const uint16_t *gain, const uint16_t *embed, float eps, int *err,
                                         Epi &epi, float *s_part, uint64_t *t_data = nullptr) {
    if constexpr (ANY) {
#define WICI_ANY_CASE(N, RPS)                                                                              \
    case N:                                                                                                \
        if constexpr (N <= MAXN)                                                                           \
            return mc_gemv<GShape<N, RPS, false>>(R, red, K, n_units, rpu, in, tag, gain, embed, eps, err, epi, s_part, \
                                                  t_data);                                                 \
        break;
        switch (gemv_nch(K)) {   // with gemv_rps of the K it covers
            WICI_ANY_CASE(1, 8) WICI_ANY_CASE(2, 4) WICI_ANY_CASE(3, 2) WICI_ANY_CASE(4, 2)
            WICI_ANY_CASE(5, 1) WICI_ANY_CASE(6, 1) WICI_ANY_CASE(7, 1) WICI_ANY_CASE(8, 1)
        }
#undef WICI_ANY_CASE
        return false;
    } else if constexpr (Q8) {
        return mc_gemv_q8<S, ND>(R, red, K, n_units, rpu, in, tag, gain, embed, eps, err, epi, s_part, t_data);
    } else {
        return mc_gemv<S>(R, red, K, n_units, rpu, in, tag, gain, embed, eps, err, epi, s_part, t_data);
    }
}

// ------------------------------------------------- attention of one token ----
// CTA (g, r) covers split r of KV head g: pages [p0, p0 + n).  One warp takes a
// whole page for all the group's query heads, on mma.m16n8k16 (a contraction of
// 16 keys with up to 8 heads: the 128-row tcgen05 tile would be nearly empty):
//   S (8 heads x 16 keys)  A = q as bf16 terms (rows 0..7 term 0, rows 8..15 term 1,
//                          then term 2), B = K;
//   O (8 heads x D)        A = P as bf16 terms in the same way, B = V (transposed
//                          ldmatrix).
// q and P are fp32 values split into three bf16 terms (24 bits: their fp32
// precision) and K and V are exact bf16, so every product is exact.  The sums are fp32
// in the accumulators, O's over every page that a warp takes: its error against 64 bits
// grows with them (8B widths, 8000 keys: 3.2e-7 at four pages a warp, 7.0e-7 at 63)
// and stays below that of fp32 FMAs in its place (8.5e-7).  A scalar version (one warp per
// head and page, lane-transposed dot products) took about 1 us per page: 29 us a layer at
// 8K cached tokens.
// The warps' states (O, m, l) are merged in shared memory and published as tagged
// words; each CTA of the head then combines every split's states for its share
// of the group's outputs.
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t addr, uint32_t &r0, uint32_t &r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, "
        "%2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// two fp32 values as three bf16 terms each, packed (first value in the low half)
__device__ __forceinline__ void split_pair(float x, float y, uint32_t (&t)[3]) {
    uint16_t x0, x1, x2, y0, y1, y2;
    split_bf16x3(x, x0, x1, x2);
    split_bf16x3(y, y0, y1, y2);
    t[0] = (uint32_t)x0 | ((uint32_t)y0 << 16);
    t[1] = (uint32_t)x1 | ((uint32_t)y1 << 16);
    t[2] = (uint32_t)x2 | ((uint32_t)y2 << 16);
}

// Qwen3 block, for one head held by a warp (lane l has elements l*EPL ..): RMS
// norm over the head with the gain, then rotate-half RoPE (the partner of element
// i < D/2 is i + D/2, EPL elements further in lane l + 16; rope: this position's row).
template <int D>
__device__ __forceinline__ void head_norm_rope(float *v, const uint16_t *gain, float eps, const float2 *rope,
                                               int lane) {
    constexpr int EPL = D / 32, HALF = D / 2;
    float ss = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) ss = fmaf(v[e], v[e], ss);
    const float rinv = 1.0f / sqrtf(warp_sum(ss) / (float)D + eps);
#pragma unroll
    for (int e = 0; e < EPL; ++e) v[e] = v[e] * rinv * bf16_to_f32(gain[lane * EPL + e]);
    const bool lower = lane < 16;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        const float other = __shfl_xor_sync(0xffffffffu, v[e], 16);
        const float2 cs = rope[(lane * EPL + e) % HALF];
        v[e] = lower ? v[e] * cs.x - other * cs.y : v[e] * cs.x + other * cs.y;
    }
}

// EPL consecutive tagged words of lane `lane` (a head's row spread over a warp), polled
template <int EPL>
__device__ __forceinline__ bool mega_row(const uint64_t *p, uint32_t tag, int lane, float (&v)[EPL], int *err) {
    PollLimit lim;
    uint64_t w[EPL];
    bool ok = true;
    while (true) {
        bool all = true;
#pragma unroll
        for (int e = 0; e < EPL; e += 2) ld_tagged2(p + lane * EPL + e, w[e], w[e + 1]);
#pragma unroll
        for (int e = 0; e < EPL; ++e) all = all && has_tag(w[e], tag);
        if (all) break;
        if (!lim.again(err)) {
            ok = false;
            break;
        }
    }
#pragma unroll
    for (int e = 0; e < EPL; ++e) v[e] = tagged_value(w[e]);
    __syncwarp();
    return ok;
}

template <int D>
struct MegaAttnSmem {
    static constexpr uint32_t Q_ROW = D * 2 + 16;              // padded: conflict-free ldmatrix
    static constexpr uint32_t Q_TERM = 8 * Q_ROW;              // 8 heads of one term
    static constexpr uint32_t KV_OFF = 3 * Q_TERM;             // this step's k and v rows, bf16
    static constexpr int STATE = D + 4;                        // floats per state: O[D], m, l, pad
    static_assert(KV_OFF + 2 * D * 2 <= kGemvRedBytes, "q terms fit the reduction scratch");
};

template <int D>
__device__ bool mc_attn(MegaRing &R, const MegaArgs &a, uint16_t *kvl, const MegaSplit &sp, int len, uint32_t tag,
                        uint8_t *qs, float *state, const float2 *rope, const uint16_t *qn, const uint16_t *kn) {
    using SM = MegaAttnSmem<D>;
    using PG = MegaPage<D>;
    constexpr int EPL = D / 32;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    int *err = a.ctrl + CTRL_ERR;
    if (!sp.active) return true;
    const bool last_split = sp.p0 + sp.n == sp.npages;
    const uint32_t qs0 = smem_u32(qs);
    bool ok = true;
    consumer_sync();   // the reduction scratch is free: every warp is past the last flush
    // q rows: warp w holds head w (zeros past the group); this step's k and v rows
    for (int row = w; row < 10; row += kGemvWarps) {
        float v[EPL];
        if (row < 8) {
            uint8_t *dst = qs + row * SM::Q_ROW + lane * EPL * 2;
            uint32_t t[EPL / 2][3] = {};
            if (row < a.group) {
                ok = mega_row<EPL>(a.tqkv + (size_t)(sp.g * a.group + row) * D, tag, lane, v, err) && ok;
                if (qn) head_norm_rope<D>(v, qn, a.eps, rope, lane);
#pragma unroll
                for (int e = 0; e < EPL; e += 2) split_pair(v[e] * a.qscale, v[e + 1] * a.qscale, t[e >> 1]);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int e = 0; e < EPL / 2; ++e)
                    *reinterpret_cast<uint32_t *>(dst + k * SM::Q_TERM + 4 * e) = t[e][k];
        } else if (last_split) {
            const bool is_v = row == 9;
            ok = mega_row<EPL>(a.tqkv + a.qdim + (is_v ? a.kvdim : 0) + (size_t)sp.g * D, tag, lane, v, err) && ok;
            if (!is_v && kn) head_norm_rope<D>(v, kn, a.eps, rope, lane);
            const int slot = (len - 1) % kPage, page = a.pages[sp.npages - 1];
            uint16_t *g = kvl + (size_t)page * a.page_elems + (is_v ? (size_t)a.nkv * kPage * D : 0) +
                          ((size_t)sp.g * kPage + slot) * D + lane * EPL;
            uint8_t *dst = qs + SM::KV_OFF + (is_v ? D * 2 : 0) + lane * EPL * 2;
#pragma unroll
            for (int e = 0; e < EPL; e += 2) {
                const uint32_t b = (uint32_t)f32_to_bf16(v[e]) | ((uint32_t)f32_to_bf16(v[e + 1]) << 16);
                *reinterpret_cast<uint32_t *>(g + e) = b;
                *reinterpret_cast<uint32_t *>(dst + 2 * e) = b;
            }
        }
    }
    if (consumer_sync_or(!ok)) return false;

    float o[D / 8][4];
#pragma unroll
    for (int i = 0; i < D / 8; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
    float m = -INFINITY, l = 0.f;    // of head lane / 4
    const int j2 = 2 * (lane & 3), mi = lane >> 3, mr = lane & 7;
    for (int i0 = 0; i0 < sp.n; i0 += PG::PER_SLOT) {
        const int slot = R.n % kMegaSlots;
        ok = ok && !*reinterpret_cast<volatile int *>(R.abort) &&
             mbar_wait(R.full0 + 8 * slot, (R.n / kMegaSlots) & 1, err, SITE_MEGA_FULL);
        ok = __all_sync(0xffffffffu, ok);   // the warp's matrix instructions run with all its lanes or not at all
        if (!ok) *R.abort = 1;
        const int np = min(PG::PER_SLOT, sp.n - i0);
        for (int i = 0; i < np && ok; ++i) {
            if ((i0 + i) % a.nsets != w) continue;
            const uint32_t kb = R.data0 + (uint32_t)slot * kMegaSlotBytes + (uint32_t)i * PG::BYTES, vb = kb + PG::V;
            const int ntok = min(kPage, len - (sp.p0 + i0 + i) * kPage);
            if (sp.p0 + i0 + i == sp.npages - 1) {
                // the copy may predate this step's row, and holds anything past it: the row from
                // shared memory, zeros for the V rows behind it (their weights are zero)
                for (int u = lane; u < 2 * (D / 8) + (kPage - ntok) * (D / 8); u += 32) {
                    const bool cur = u < 2 * (D / 8);
                    const int du = u % (D / 8), isv = cur ? u / (D / 8) : 1;
                    const int r = cur ? ntok - 1 : ntok + (u - 2 * (D / 8)) / (D / 8);
                    const uint32_t dst = (isv ? vb : kb) + (du >> 3) * PG::CHUNK + r * 128 + (((du & 7) ^ (r & 7)) << 4);
                    uint4 x = make_uint4(0u, 0u, 0u, 0u);
                    if (cur) x = lds128(qs0 + SM::KV_OFF + isv * D * 2 + du * 16);
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(x.x), "r"(x.y), "r"(x.z),
                                 "r"(x.w)
                                 : "memory");
                }
                __syncwarp();
                // these stores come before the next copy into this slot
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            // S: s01 rows 0..7 term 0, rows 8..15 term 1; s2 rows 0..7 term 2.  Fragments are
            // loaded one step ahead of the matrix instructions that take them.
            float s01[2][4] = {}, s2[2][4] = {};
            uint32_t qa[2][4], q2[2][2], kf[2][4];
            auto load_s = [&](int kk) {
                const int key = (mi >> 1) * 8 + mr, u = (kk & 3) * 2 + (mi & 1);
                ldsm4(kb + (kk >> 2) * PG::CHUNK + key * 128 + ((u ^ (key & 7)) << 4), kf[kk & 1]);
                ldsm4(qs0 + (mi & 1) * SM::Q_TERM + mr * SM::Q_ROW + (16 * kk + (mi >> 1) * 8) * 2, qa[kk & 1]);
                ldsm2(qs0 + 2 * SM::Q_TERM + mr * SM::Q_ROW + (16 * kk + (mi & 1) * 8) * 2, q2[kk & 1][0], q2[kk & 1][1]);
            };
            uint32_t vf[2][4];
            auto load_v = [&](int n) {
                const int key = (mi & 1) * 8 + mr, u = 2 * n + (mi >> 1);
                ldsm4t(vb + (u >> 3) * PG::CHUNK + key * 128 + (((u & 7) ^ (key & 7)) << 4), vf[n & 1]);
            };
            load_s(0);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                if (kk + 1 < D / 16) load_s(kk + 1);
                const uint32_t(&q)[4] = qa[kk & 1], (&k)[4] = kf[kk & 1];
#pragma unroll
                for (int t = 0; t < 2; ++t) mma_bf16(s01[t], q[0], q[1], q[2], q[3], k[2 * t], k[2 * t + 1]);
#pragma unroll
                for (int t = 0; t < 2; ++t) mma_bf16(s2[t], q2[kk & 1][0], 0u, q2[kk & 1][1], 0u, k[2 * t], k[2 * t + 1]);
            }
            load_v(0);
            float s[2][2];
            float mx = m;
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    s[t][e] = (s2[t][e] + s01[t][2 + e]) + s01[t][e];
                    if (8 * t + j2 + e >= ntok) s[t][e] = -INFINITY;
                    mx = fmaxf(mx, s[t][e]);
                }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float corr = exp2f(m - mx);
            uint32_t p[2][3];
            float ps = 0.f;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const float p0 = exp2f(s[t][0] - mx), p1 = exp2f(s[t][1] - mx);   // 0 for masked keys
                ps += p0 + p1;
                split_pair(p0, p1, p[t]);
            }
            l = l * corr + ps;
            if (__any_sync(0xffffffffu, mx != m)) {
#pragma unroll
                for (int n = 0; n < D / 8; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[n][e] *= corr;
            }
            m = mx;
#pragma unroll
            for (int n = 0; n < D / 16; ++n) {
                if (n + 1 < D / 16) load_v(n + 1);
                const uint32_t(&v)[4] = vf[n & 1];
#pragma unroll
                for (int t = 0; t < 2; ++t) mma_bf16(o[2 * n + t], p[0][2], 0u, p[1][2], 0u, v[2 * t], v[2 * t + 1]);
#pragma unroll
                for (int t = 0; t < 2; ++t)
                    mma_bf16(o[2 * n + t], p[0][0], p[0][1], p[1][0], p[1][1], v[2 * t], v[2 * t + 1]);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(R.empty0 + 8 * slot);
        ++R.n;
    }
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    const int sets = min(a.nsets, sp.n);    // warps that held pages
    if (w < sets && (lane >> 2) < a.group) {
        float *st = state + (size_t)(w * a.group + (lane >> 2)) * SM::STATE;
#pragma unroll
        for (int n = 0; n < D / 8; ++n)
            *reinterpret_cast<float2 *>(st + 8 * n + j2) = make_float2(o[n][0] + o[n][2], o[n][1] + o[n][3]);
        if ((lane & 3) == 0) *reinterpret_cast<float2 *>(st + D) = make_float2(m, l);
    }
    if (consumer_sync_or(!ok)) return false;

    // merge the page sets in set order; publish this split's state
    const int E = a.group * D;
    uint64_t *part = a.tpart + (size_t)sp.g * a.splits * a.group * (D + 2);
    for (int e = tid; e < E; e += kGemvConsumers) {
        const int hd = e / D, c = e % D;
        const float *st = state + (size_t)hd * SM::STATE;
        const int stride = a.group * SM::STATE;
        float M = st[D];
        for (int t = 1; t < sets; ++t) M = fmaxf(M, st[t * stride + D]);
        float acc = 0.f, L = 0.f;
        for (int t = 0; t < sets; ++t) {
            const float f = exp2f(st[t * stride + D] - M);
            acc = fmaf(st[t * stride + c], f, acc);
            L = fmaf(st[t * stride + D + 1], f, L);
        }
        if (sp.splits == 1) {
            st_tagged(a.to + (size_t)sp.g * E + e, acc * (1.0f / L), tag);
        } else {
            uint64_t *mine = part + (size_t)(sp.r * a.group + hd) * (D + 2);
            st_tagged(mine + c, acc, tag);
            if (c == 0) st_tagged2(mine + D, M, L, tag);
        }
    }
    if (sp.splits == 1) return true;

    // combine: this CTA's share [e0, e1) of the group's outputs over every split; warps
    // (ws, we): splits ws, ws + nws, ... of the 32-output blocks we, we + 8 / nws, ...
    const int e0 = sp.r * E / sp.splits, ne = (sp.r + 1) * E / sp.splits - e0;
    const int nws = sp.splits >= 8 ? 8 : sp.splits >= 4 ? 4 : 2;
    const int ws = w % nws, we = w / nws;
    constexpr int MAXQ = kMaxSplits / 8;    // splits of one warp
    float *scr = state;                       // [nws][ne] x (acc, m, l)
    consumer_sync();                          // the states have been merged
    for (int x = we * 32 + lane; x < ne; x += 32 * (kGemvWarps / nws)) {
        const int hd = (e0 + x) / D, c = (e0 + x) % D;
        uint64_t wv[MAXQ], wm[MAXQ], wl[MAXQ];
        PollLimit lim;
        while (true) {
            bool all = true;
#pragma unroll
            for (int q = 0; q < MAXQ; ++q)
                if (ws + q * nws < sp.splits) {
                    const uint64_t *src = part + (size_t)((ws + q * nws) * a.group + hd) * (D + 2);
                    wv[q] = ld_tagged(src + c);
                    ld_tagged2(src + D, wm[q], wl[q]);
                }
#pragma unroll
            for (int q = 0; q < MAXQ; ++q)
                if (ws + q * nws < sp.splits)
                    all = all && has_tag(wv[q], tag) && has_tag(wm[q], tag) && has_tag(wl[q], tag);
            if (all) break;
            if (!lim.again(err)) {
                ok = false;
                break;
            }
        }
        float M = -INFINITY, acc = 0.f, L = 0.f;
#pragma unroll
        for (int q = 0; q < MAXQ; ++q)
            if (ws + q * nws < sp.splits) M = fmaxf(M, tagged_value(wm[q]));
#pragma unroll
        for (int q = 0; q < MAXQ; ++q)
            if (ws + q * nws < sp.splits) {
                const float f = exp2f(tagged_value(wm[q]) - M);
                acc = fmaf(tagged_value(wv[q]), f, acc);
                L = fmaf(tagged_value(wl[q]), f, L);
            }
        float *d = scr + (size_t)(ws * ne + x) * 3;
        d[0] = acc;
        d[1] = M;
        d[2] = L;
    }
    if (consumer_sync_or(!ok)) return false;
    for (int x = tid; x < ne; x += kGemvConsumers) {
        float M = scr[x * 3 + 1];
        for (int t = 1; t < nws; ++t) M = fmaxf(M, scr[(t * ne + x) * 3 + 1]);
        float acc = 0.f, L = 0.f;
        for (int t = 0; t < nws; ++t) {
            const float *d = scr + (size_t)(t * ne + x) * 3;
            const float f = exp2f(d[1] - M);
            acc = fmaf(d[0], f, acc);
            L = fmaf(d[2], f, L);
        }
        st_tagged(a.to + (size_t)sp.g * E + e0 + x, acc * (1.0f / L), tag);
    }
    return true;
}

// The SMs do not draw equal HBM bandwidth, and which SMs are slow stays the same
// from step to step, so the GEMV rows are split in proportion to each CTA's
// measured speed instead of evenly.  Run by the consumers of the last CTA of a
// step: the new share of CTA b blends its old share with old share / time of
// its gate/up phases (normalised), half and half, with a floor of a quarter of
// an even share.  Which CTA streams which rows changes no result.
__device__ inline void mega_rebalance(const MegaArgs &a, float *scr) {
    const int G = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    static_assert(kMaxCtas <= kGemvConsumers, "one thread per CTA");
    // sum of v over the consumers, with the inclusive prefix sums in *pre
    auto block_sum = [&](float v, float *pre) {
        float p = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float q = __shfl_up_sync(0xffffffffu, p, o);
            if (lane >= o) p += q;
        }
        consumer_sync();   // the scratch of the sum before is read
        if (lane == 31) scr[warp] = p;
        consumer_sync();
        float tot = 0.f;
        for (int w = 0; w < kGemvWarps; ++w) {
            if (w == warp) *pre = tot + p;
            tot += scr[w];
        }
        return tot;
    };
    float share = 0.f, rate = 0.f, pre;
    if (tid < G) {
        share = (float)(__ldcg(a.bound + tid + 1) - __ldcg(a.bound + tid)) * (1.0f / 16777216.0f);
        const float t = __ldcg(a.cta_time + tid);
        rate = t > 0.f ? share / t : 0.f;
    }
    const float tot = block_sum(rate, &pre);
    if (!(tot > 0.f)) return;
    const float ns = tid < G ? fmaxf(0.5f * share + 0.5f * rate / tot, 0.25f / (float)G) : 0.f;
    const float sum = block_sum(ns, &pre);
    // every thread has read the old table before the first barrier above
    if (tid < G - 1) a.bound[tid + 1] = (uint32_t)fminf(pre / sum * 16777216.0f, 16777216.0f);
    if (tid == G - 1) {
        a.bound[0] = 0;
        a.bound[G] = 1u << 24;
    }
}

// Registers: nine warps get 168 each, the register file's share of three warps on one SM
// partition.  Where a thread holds two or more chunks of every hidden-wide row (bf16 rows of
// more than 2048 elements in a named shape), the step is launched with twelve warps of 168
// and the producer's warpgroup hands its own on: 384 x 168 = 128 x 104 + 256 x 200.  The
// compiler then keeps more loads of a phase in flight.  The line lies between the measured
// shapes: Llama-3-8B widths, 2 layers and 6360 tokens of context, 180 us a step -> 176; 14B
// widths, 6 layers, 599 -> 580 (hidden 4096 and 5120 are all that takes it).  The other
// shapes lose with it (1B 518 -> 536 us, 8-bit Qwen3-8B 9 layers 471 -> 482, widths picked
// at run time 366 -> 370) and keep nine warps.  A producer of 24 and consumers of 240
// measured the same (174 to 176, 579).
template <class SH, bool Q8, bool ANY>
struct MegaRegs {
    static constexpr bool kSplit = !Q8 && !ANY && SH::NCH >= 2;
    static constexpr int kThreads = kSplit ? 384 : kGemvThreads;
    static constexpr int kProducer = 104, kConsumer = 200;
    // above the launch's own registers the consumers would wait for ever: launch_mega checks
    static constexpr int kNeeded = 128 * kProducer + 256 * kConsumer;
};

// SH, SF: GEMV shapes of K = hidden and K = ffn for bf16 rows; with Q8 the seven
// per-layer matrices are in the 8-bit block format and stream with the shapes
// QH, QF (16-element chunks, rows per slot sized for the shorter rows), while
// the LM head stays bf16 (SH).  ANY: bf16 matrices of any widths the configuration
// allows, the shape of each phase picked at run time (SH .. QF are ignored).
template <int D, class SH, class SF, bool Q8, class QH, class QF, bool ANY>
__global__ void __launch_bounds__((MegaRegs<SH, Q8, ANY>::kThreads), 1)
    decode_step_kernel(const __grid_constant__ CUtensorMap map_kv, const MegaArgs a) {
    using LH = std::conditional_t<Q8, QH, SH>;   // layer matrices with K = hidden (and K = n_q * d)
    using LF = std::conditional_t<Q8, QF, SF>;   // the down projection, K = ffn
    constexpr bool LOOP = ANY || Q8;             // a CTA may have several KV heads
    const uint32_t rb_h = Q8 ? (uint32_t)q8_row_bytes((size_t)a.H) : (uint32_t)a.H * 2u;
    const uint32_t rb_q = Q8 ? (uint32_t)q8_row_bytes((size_t)a.qdim) : (uint32_t)a.qdim * 2u;
    const uint32_t rb_f = Q8 ? (uint32_t)q8_row_bytes((size_t)a.F) : (uint32_t)a.F * 2u;
    // rows per ring slot of the matrices with K = hidden, K = n_q * d and K = ffn
    const int rps_h = ANY ? gemv_rps(a.H) : LH::RPS, rps_q = ANY ? gemv_rps(a.qdim) : LH::RPS;
    const int rps_f = ANY ? gemv_rps(a.F) : LF::RPS;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t bars[2 * kMegaSlots];
    __shared__ float2 s_rope[D / 2];          // this position's (cos, sin)
    __shared__ float s_part[2 * kGemvWarps];  // per-warp partials: sums, then maxima (8-bit phases)
    __shared__ float s_bv[kGemvWarps];
    __shared__ int s_bi[kGemvWarps];
    __shared__ int s_last, s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int *err = a.ctrl + CTRL_ERR;
    uint8_t *ring = smem + ((1024u - (smem_u32(smem) & 1023u)) & 1023u);
    float *red = reinterpret_cast<float *>(ring + (size_t)kMegaSlots * kMegaSlotBytes);
    float *state = red + kGemvRedBytes / 4;

    MegaRing R;
    R.full0 = smem_u32(bars);
    R.empty0 = smem_u32(bars + kMegaSlots);
    R.data0 = smem_u32(ring);
    R.n = 0;
    R.abort = &s_abort;
    // the table changes only at the very end of a step, after every CTA read it here
    R.b0 = a.bound[blockIdx.x];
    R.b1 = a.bound[blockIdx.x + 1];
    // so do the position, the input token and the step count (last LM-head CTA)
    const int len = *reinterpret_cast<volatile int *>(a.ctrl + CTRL_POS) + 1;
    if (tid == 0) {
        s_abort = 0;
        for (int s = 0; s < kMegaSlots; ++s) {
            mbar_init(R.full0 + 8 * s, 1);
            mbar_init(R.empty0 + 8 * s, kGemvWarps);
        }
        fence_barrier_init();
    }
    if (tid < D / 2) s_rope[tid] = a.rope[(size_t)(len - 1) * (D / 2) + tid];
    __syncthreads();
    const MegaSplit sp0 = mega_split(a, len, blockIdx.x);
    const int units = a.nkv * a.splits;

    using Regs = MegaRegs<SH, Q8, ANY>;
    if (warp >= kGemvWarps) {  // ------------------------------------ producer
        if constexpr (Regs::kSplit) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Regs::kProducer));
        if (warp == kGemvWarps && lane == 0) {
            const uint64_t pol = l2_evict_first();
            bool ok = true;
            for (int l = 0; l < a.L && ok; ++l) {
                const size_t lo = (size_t)l * a.lstride;
                ok = mp_rows(R, a.W + a.l0.wqkv + lo, rb_h, a.nqkv / 2, 2, rps_h, err, pol) &&
                     mp_pages<D>(R, a, &map_kv, l, sp0, err);
                if constexpr (LOOP)
                    for (int u = blockIdx.x + gridDim.x; ok && u < units; u += gridDim.x)
                        ok = mp_pages<D>(R, a, &map_kv, l, mega_split(a, len, u), err);
                ok = ok && mp_rows(R, a.W + a.l0.wo + lo, rb_q, a.H, 1, rps_q, err, pol) &&
                     mp_rows(R, a.W + a.l0.wgu + lo, rb_h, a.F, 2, rps_h, err, pol) &&
                     mp_rows(R, a.W + a.l0.wd + lo, rb_f, a.H, 1, rps_f, err, pol);
            }
            if (ok) mp_rows(R, a.W + a.w_lm, (uint32_t)a.H * 2u, a.V, 1, ANY ? rps_h : SH::RPS, err, pol);
            // no copy may still be landing in shared memory when the CTA exits
            for (int s = max(0, R.n - kMegaSlots); s < R.n; ++s)
                mbar_wait(R.full0 + 8 * (s % kMegaSlots), (s / kMegaSlots) & 1, err, SITE_MEGA_DRAIN);
        }
        return;
    }

    // ---------------------------------------------------------------- consumers
    if constexpr (Regs::kSplit) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Regs::kConsumer));
    const uint16_t *embed = a.W + a.w_embed + (size_t)a.ctrl[CTRL_TOKEN] * a.H;
    // tag of layer l: unique over the last 2^32 / L steps
    const uint32_t tag0 = (uint32_t)a.ctrl[CTRL_EPOCH] * (uint32_t)a.L;
    bool ok = true;
    uint64_t gu_ns = 0;   // this CTA's streaming time in the gate/up phases (thread 0's clock)
    for (int l = 0; l < a.L; ++l) {
        const size_t lo = (size_t)l * a.lstride;
        const uint32_t tag = tag0 + (uint32_t)l + 1u;
        const uint16_t *e0 = l == 0 ? embed : nullptr;
        MEpiQKV<D> eq;
        eq.t = a.tqkv; eq.tag = tag; eq.rope = s_rope;
        eq.bias = a.bias ? a.W + a.l0.bqkv + lo : nullptr;
        eq.qkdim = a.qdim + a.kvdim;
        eq.raw = a.qk_norm != 0;
        ok = mc_phase<ANY, Q8, LH, kQ8QkvDigits, 4>(R, red, a.H, a.nqkv / 2, 2, a.txd, tag - 1u,
                                                 a.W + a.l0.attn_norm + lo, e0, a.eps, err, eq, s_part);
        if (!ok) break;
        MegaSplit sp = sp0;
        for (int u = blockIdx.x;;) {
            ok = mc_attn<D>(R, a, a.KV + (size_t)l * a.kv_layer_elems, sp, len, tag, reinterpret_cast<uint8_t *>(red),
                            state, s_rope, a.qk_norm ? a.W + a.l0.qn + lo : nullptr,
                            a.qk_norm ? a.W + a.l0.kn + lo : nullptr);
            if constexpr (!LOOP) break;
            u += gridDim.x;
            if (!ok || u >= units) break;
            sp = mega_split(a, len, u);
        }
        if (!ok) break;
        MEpiResidual er;
        er.prev = a.txd; er.embed = e0; er.prev_tag = tag - 1u; er.out = a.txo; er.tag = tag;
        ok = mc_phase<ANY, Q8, LH, kQ8RestDigits, 8>(R, red, a.qdim, a.H, 1, a.to, tag, nullptr, nullptr, a.eps, err, er, s_part);
        if (!ok) break;
        MEpiSwiGLU es{a.tm, tag};
        uint64_t t_gu = 0;
        ok = mc_phase<ANY, Q8, LH, kQ8RestDigits, 4>(R, red, a.H, a.F, 2, a.txo, tag, a.W + a.l0.ffn_norm + lo, nullptr, a.eps, err, es,
                                   s_part, &t_gu);
        if (!ok) break;
        if (t_gu) gu_ns += globaltimer_ns() - t_gu;
        er.prev = a.txo; er.embed = nullptr; er.prev_tag = tag; er.out = a.txd;
        ok = mc_phase<ANY, Q8, LF, kQ8RestDigits, 8>(R, red, a.F, a.H, 1, a.tm, tag, nullptr, nullptr, a.eps, err, er, s_part);
        if (!ok) break;
    }
    if (tid == 0) a.cta_time[blockIdx.x] = (float)gu_ns * 1e-3f;
    if (!ok) return;
    MEpiArgmax ea;
    ea.logits = a.logits; ea.partial = a.amax; ea.ctrl = a.ctrl; ea.hist = a.hist; ea.pos_add = 1;
    ea.best = -INFINITY; ea.bidx = 0x7fffffff;
    if (!mc_phase<ANY, false, SH, kQ8RestDigits, 4>(R, red, a.H, a.V, 1, a.txd, tag0 + (uint32_t)a.L, a.W + a.w_final_norm, nullptr, a.eps, err, ea,
                     s_part, nullptr))
        return;
    if (!lm_argmax(ea, s_bv, s_bi, &s_last)) return;
    if (tid == 0) a.ctrl[CTRL_EPOCH] += 1;   // the next step's words carry other tags
    mega_rebalance(a, state);
}

// ------------------------------------------------------------------ launch ----
typedef cudaError_t (*MegaLaunch)(const CUtensorMap &, const MegaArgs &, int grid, cudaStream_t);

template <int D, class SH, class SF, bool Q8, class QH, class QF, bool ANY>
cudaError_t launch_mega(const CUtensorMap &map_kv, const MegaArgs &a, int grid, cudaStream_t st) {
    using Regs = MegaRegs<SH, Q8, ANY>;
    if constexpr (Regs::kSplit) {   // a property of the compiled kernel, asked once
        static const int regs = [] {
            cudaFuncAttributes fa = {};
            return cudaFuncGetAttributes(&fa, decode_step_kernel<D, SH, SF, Q8, QH, QF, ANY>) == cudaSuccess ? fa.numRegs : 0;
        }();
        if (regs * Regs::kThreads < Regs::kNeeded) return cudaErrorLaunchOutOfResources;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(Regs::kThreads);
    cfg.dynamicSmemBytes = kMegaSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // every CTA resident: they wait for one another's words
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, decode_step_kernel<D, SH, SF, Q8, QH, QF, ANY>, map_kv, a);
}

template <int D, class SH, class SF, bool Q8, class QH, class QF, bool ANY>
cudaError_t mega_smem() {
    return cudaFuncSetAttribute(decode_step_kernel<D, SH, SF, Q8, QH, QF, ANY>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMegaSmem);
}

// the step for bf16 matrices of any widths (kernels_decode_any.cu)
MegaLaunch mega_any_launcher(int head_dim);
cudaError_t setup_mega_any();

}  // namespace wici
