// Decode-step kernels (batch 1): weight-streaming GEMVs with fused prologues
// and epilogues, and split-K flash-decode over the paged KV cache.
//
// A decode step is HBM-bound: every weight byte is read once per token
// (arithmetic intensity ~1 FLOP/byte).  The GEMV streams each CTA's rows through
// a 3-stage ring in shared memory with 1-D TMA bulk copies (cp.async.bulk,
// completion on mbarriers); one producer warp issues the copies, eight consumer
// warps do the dot products with the input vector held in registers.  The
// producer starts before griddepcontrol.wait, so under programmatic dependent
// launch a GEMV's first weight tiles stream in while its predecessor finishes.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace wici {

// wait-site ids recorded in ctrl[CTRL_ERR]
enum : int { SITE_GEMV_EMPTY = 11, SITE_GEMV_FULL = 12, SITE_GEMV_DRAIN = 13, SITE_PROBE = 99 };

struct GemvIn {
    const uint16_t *W;      // rows of this matrix, [n_units * rpu][K]
    int K, n_units, rpu, ups;
    int stages;             // ring slots (<= kGemvMaxStages)
    uint32_t slot_bytes;    // bytes per ring slot (>= ups * rpu * K * 2, multiple of 128)
    const float *in;        // input vector (x when gain != nullptr)
    const uint16_t *gain;   // RMSNorm gain (bf16) or nullptr for a plain input
    const uint16_t *embed;  // non-null: the input is embed[ctrl[CTRL_TOKEN]] (layer 0)
    float *x_out;           // embed variant: CTA 0 stores the embedded row here
    int *ctrl;
    float eps;
    // the GEMV launched after this one: the producer moves the first rows of
    // this CTA's share of it into L2 once its own rows are issued
    const uint16_t *next_W;  // nullptr: none
    int next_K, next_n_units, next_rpu;
};

// ---------------------------------------------------------------- epilogues --
// unit(u, v): v[0..rpu) are the finished dot products of unit u's rows.

struct EpiResidual {  // x[u] += W x_in   (O projection, down projection)
    float *x;
    static constexpr bool kArgmax = false;
    __device__ void unit(int u, const float *v) { x[u] += v[0]; }
};

struct EpiSwiGLU {    // rows (2u, 2u+1) are (gate_u, up_u): m[u] = silu(g) * u
    float *m;
    static constexpr bool kArgmax = false;
    __device__ void unit(int u, const float *v) {
        const float gt = v[0];
        m[u] = gt / (1.0f + expf(-gt)) * v[1];
    }
};

// Packed QKV rows: for every q and k head the rows are paired (i, i + d/2) as
// adjacent rows (2i, 2i + 1), so one unit holds one RoPE pair; v rows are in
// natural order, two per unit.
struct EpiQKV {
    float *q;
    uint16_t *kv;          // this layer's pages
    const int *pages;
    const float2 *rope;
    const int *ctrl;
    const uint16_t *bias;  // packed like the rows, or nullptr
    int qdim, kvdim, d, nkv;
    size_t page_elems;
    static constexpr bool kArgmax = false;
    __device__ void unit(int u, const float *v) {
        const int r0 = 2 * u;
        float a = v[0], b = v[1];
        if (bias) {
            a += bf16_to_f32(bias[r0]);
            b += bf16_to_f32(bias[r0 + 1]);
        }
        const int pos = ctrl[CTRL_POS];
        uint16_t *page = kv + (size_t)pages[pos / kPage] * page_elems;
        const int slot = pos % kPage;
        if (r0 < qdim + kvdim) {
            const int hd = r0 / d, i = (r0 % d) >> 1, half = d >> 1;
            const float2 cs = rope[(size_t)pos * half + i];
            const float ra = a * cs.x - b * cs.y;
            const float rb = b * cs.x + a * cs.y;
            if (r0 < qdim) {
                q[hd * d + i] = ra;
                q[hd * d + i + half] = rb;
            } else {
                const int kh = hd - qdim / d;
                uint16_t *kr = page + ((size_t)kh * kPage + slot) * d;
                kr[i] = f32_to_bf16(ra);
                kr[i + half] = f32_to_bf16(rb);
            }
        } else {
            const int j = r0 - qdim - kvdim, vh = j / d, e = j % d;
            uint16_t *vr = page + (size_t)nkv * kPage * d + ((size_t)vh * kPage + slot) * d;
            vr[e] = f32_to_bf16(a);
            vr[e + 1] = f32_to_bf16(b);
        }
    }
};

struct EpiArgmax {    // logits[u] = v; greedy argmax (lowest index on ties) across the grid
    float *logits;
    int2 *partial;
    int *ctrl;
    int *hist;
    int pos_add;
    float best;
    int bidx;
    static constexpr bool kArgmax = true;
    __device__ void unit(int u, const float *v) {
        logits[u] = v[0];
        if (v[0] > best || (v[0] == best && u < bidx)) {
            best = v[0];
            bidx = u;
        }
    }
};

__device__ __forceinline__ bool better(float av, int ai, float bv, int bi) {
    return av > bv || (av == bv && ai < bi);
}


constexpr int kRedRows = 128;  // rows of partial sums per reduction batch

constexpr int kGemvMaxStages = 8;
// dynamic shared memory: [reduction scratch 2 x 8 warps x kRedRows fp32][ring]
constexpr size_t kGemvRedBytes = 2 * 8 * kRedRows * 4;
static inline size_t gemv_smem_bytes(int stages, uint32_t slot_bytes) {
    return kGemvRedBytes + (size_t)stages * slot_bytes;
}

// ------------------------------------------------------------------- GEMV ----
// Grid: num_sms CTAs, each owning a contiguous, balanced range of units.  Each
// consumer thread holds NCH 8-element chunks of the input vector in registers
// (chunk c = tid + 256 j) and, for every row of a stage, contributes the dot
// product over its chunks; warp sums go to shared memory and are reduced over
// the 8 warps (fixed order) once per batch of up to kRedRows rows.
// Shapes: every slot holds RPS rows (RPS a power of two, at most 8, RPS x K x 2
// <= 32 KB, a multiple of the unit); consumer thread t covers the 8-element
// chunks c = t + 256 j, j < NCH; FULL when the chunks cover K exactly (no tail
// check in the inner loop).
__host__ __device__ constexpr int gemv_rps(int K) {
    return 2 * K * 8 <= 32768 ? 8 : 2 * K * 4 <= 32768 ? 4 : 2 * K * 2 <= 32768 ? 2 : 1;
}
__host__ __device__ constexpr int gemv_nch(int K) { return (K / 8 + 255) / 256; }

constexpr int kGemvConsumers = 256;
constexpr int kGemvWarps = 8;

__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// consumer barrier that also returns the OR of every consumer thread's flag, so
// all of them take the same branch afterwards
__device__ __forceinline__ bool consumer_sync_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, 1, 256, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 r;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "r"(addr));
    return r;
}

// a + (8 bf16 weights) . (8 fp32 inputs)
__device__ __forceinline__ float dot8(const uint4 w, const float *h, float a) {
    a = fmaf(bf16lo(w.x), h[0], a);
    a = fmaf(bf16hi(w.x), h[1], a);
    a = fmaf(bf16lo(w.y), h[2], a);
    a = fmaf(bf16hi(w.y), h[3], a);
    a = fmaf(bf16lo(w.z), h[4], a);
    a = fmaf(bf16hi(w.z), h[5], a);
    a = fmaf(bf16lo(w.w), h[6], a);
    a = fmaf(bf16hi(w.w), h[7], a);
    return a;
}

// Warp sums of a slot's RPS rows (each lane holds its partial of every row),
// stored to rb[0, rows): a transposed butterfly.  R = RPS rounded up to a power
// of two; at each of the first log2(R) levels a lane keeps one half of its rows
// and trades the other half with its partner, so one shuffle moves one row (R - 1
// shuffles in all instead of 5 R); plain butterflies finish the sum.  Lane l then
// holds the row whose index is spelled by lane bits 4, 3, ... (most significant
// first), and the lanes whose remaining low bits are zero store it.
template <int RPS>
__device__ __forceinline__ void warp_rows_store(const float (&acc)[RPS], float *rb, int rows, int lane) {
    constexpr int R = RPS <= 1 ? 1 : RPS <= 2 ? 2 : RPS <= 4 ? 4 : 8;
    static_assert(RPS <= 8, "at most 8 rows per slot");
    float v[R];
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = i < RPS ? acc[i] : 0.f;
    int row = 0;
#pragma unroll
    for (int o = 16, cnt = R; o > 0; o >>= 1) {
        if (cnt > 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int t = 0; t < cnt / 2; ++t) {
                const float send = up ? v[t] : v[t + cnt / 2];
                const float keep = up ? v[t + cnt / 2] : v[t];
                v[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
            if (up) row += cnt / 2;
            cnt >>= 1;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
    if ((lane & (32 / R - 1)) == 0 && row < rows) rb[row] = v[0];
}

// ------------------------------------------------- 8-bit block rows (decode) --
// A row of the 8-bit block format in shared memory: K int8 codes (two's
// complement), then the row's K/32 fp16 block scales.
//
// The input vector of a phase is put once into fixed point, X[c] = rint(h[c] *
// 2^E) with |X| < 2^23 (three byte digits) or 2^15 (two), E from the vector's
// largest magnitude (one rounding of at most 2^-24, or 2^-16, of it), and X is
// cut into byte digits, e.g. X = 65536 X2 + 256 X1 + X0 (X2 signed, the others
// unsigned).  The
// integer dot products of 16 codes with each digit (dp4a, exact in int32) make
// the chunk's exact sum q . X, which one fp32 rounding carries into the row's
// fp32 accumulator with the block scale; 2^-E is applied once per row.  That is
// 12 dp4a and a handful of fp32 operations per 16 codes, where converting every
// code to fp32 costs three operations per code.
__device__ __forceinline__ int dp4a_ss(uint32_t a, uint32_t b, int c) {
    int d;
    asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ int dp4a_su(uint32_t a, uint32_t b, int c) {
    int d;
    asm("dp4a.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// exact int -> fp32 for |v| < 2^22: the integer added under the exponent of 1.5 * 2^23
__device__ __forceinline__ float small_int_to_f32(int v) {
    return __int_as_float(0x4B400000 + v) - 12582912.0f;
}

__device__ __forceinline__ float lds_f16(uint32_t addr) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return __half2float(__ushort_as_half(v));
}

// The eight consumer warps' best (value, lowest index) of thread candidates; valid in thread 0.
__device__ __forceinline__ void block_argmax(float &bv, int &bi, float *s_bv, int *s_bi) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
    }
    if (lane == 0) { s_bv[warp] = bv; s_bi[warp] = bi; }
    consumer_sync();
    if (threadIdx.x == 0)
        for (int w = 1; w < kGemvWarps; ++w)
            if (better(s_bv[w], s_bi[w], bv, bi)) { bv = s_bv[w]; bi = s_bi[w]; }
}

// End of an LM head: this CTA's argmax to its partial and a ticket; the last CTA
// reduces every partial (value, lowest index: any order gives the same), writes the
// token and advances the position.  True in that CTA.  The partials are read by all
// consumer threads at once: one thread walking the 152 of them (and the row shares
// after them) took about 25 us of every decode step.
__device__ bool lm_argmax(const EpiArgmax &e, float *s_bv, int *s_bi, int *s_last) {
    const int tid = threadIdx.x, G = gridDim.x;
    float bv = e.best;
    int bi = e.bidx;
    block_argmax(bv, bi, s_bv, s_bi);
    if (tid == 0) {
        e.partial[blockIdx.x] = make_int2(__float_as_int(bv), bi);
        __threadfence();
        const int t = atomicAdd(e.ctrl + CTRL_LM_TICKET, 1);
        *s_last = t == G - 1;
        if (t == G - 1) __threadfence();
    }
    consumer_sync();
    if (!*s_last) return false;
    bv = -INFINITY;
    bi = 0x7fffffff;
    for (int c = tid; c < G; c += kGemvConsumers) {
        const int2 pr = __ldcg(e.partial + c);
        if (better(__int_as_float(pr.x), pr.y, bv, bi)) { bv = __int_as_float(pr.x); bi = pr.y; }
    }
    block_argmax(bv, bi, s_bv, s_bi);
    if (tid == 0) {
        if (bi == 0x7fffffff) bi = 0;
        const int np = e.ctrl[CTRL_POS] + e.pos_add;
        e.ctrl[CTRL_TOKEN] = bi;
        e.ctrl[CTRL_POS] = np;
        e.hist[np] = bi;
        e.ctrl[CTRL_LM_TICKET] = 0;
    }
    return true;
}

// ------------------------------------------------------------------- GEMV ----
// Grid: num_sms CTAs, each owning a contiguous, balanced range of units.  The
// producer warp streams the CTA's rows, RPS per slot, through the ring; each of
// the 8 consumer warps adds its chunks of every row and reduces the slot's RPS
// rows with interleaved butterflies; warp sums go to shared memory and are
// reduced over the warps (fixed order) once per kRedRows rows, then passed to
// the epilogue.
template <int NCH, int RPS, bool FULL, class Epi>
__global__ void __launch_bounds__(kGemvThreads, 1) gemv_kernel(const GemvIn g, const Epi epi_in) {
    extern __shared__ __align__(128) uint8_t smem[];
    float *red = reinterpret_cast<float *>(smem);  // [2][kGemvWarps][kRedRows]
    uint8_t *ring = smem + kGemvRedBytes;
    __shared__ __align__(8) uint64_t bars[2 * kGemvMaxStages];  // full[S], empty[S]
    __shared__ float s_part[kGemvWarps];
    __shared__ int s_abort;
    __shared__ float s_bv[kGemvWarps];
    __shared__ int s_bi[kGemvWarps];
    __shared__ int s_last;
    const int S = g.stages;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x;
    const int u0 = (int)(((long long)blockIdx.x * g.n_units) / G);
    const int u1 = (int)(((long long)(blockIdx.x + 1) * g.n_units) / G);
    const int nunits = u1 - u0;
    const int total_rows = nunits * g.rpu;
    const int nst = (total_rows + RPS - 1) / RPS;
    int *err = g.ctrl + CTRL_ERR;

    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kGemvMaxStages);
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, kGemvWarps);
        }
        fence_barrier_init();
        s_abort = 0;
    }
    __syncthreads();
    griddep_launch_dependents();

    if (warp == kGemvWarps) {  // ------------------------------------ producer
        if (lane == 0) {
            const uint64_t pol = l2_evict_first();
            const uint32_t ring0 = smem_u32(ring);
            const uint16_t *src = g.W + (size_t)u0 * g.rpu * g.K;
            int issued = 0;
            for (int s = 0; s < nst; ++s) {
                const int slot = s % S;
                if (s >= S && !mbar_wait(empty0 + 8 * slot, ((s / S) + 1) & 1, err, SITE_GEMV_EMPTY)) break;
                const int rows = min(RPS, total_rows - s * RPS);
                const uint32_t bytes = (uint32_t)rows * (uint32_t)g.K * 2u;
                mbar_arrive_expect_tx(full0 + 8 * slot, bytes);
                bulk_g2s(ring0 + slot * g.slot_bytes, src + (size_t)s * RPS * g.K, bytes, full0 + 8 * slot, pol);
                issued = s + 1;
            }
            if (g.next_W) {
                // the next kernel's CTA of the same index streams units [nu0, nu1); its
                // first ring-full is fetched while this CTA drains, so the HBM stays busy
                // across the kernel boundary
                const int nu0 = (int)(((long long)blockIdx.x * g.next_n_units) / G);
                const int nu1 = (int)(((long long)(blockIdx.x + 1) * g.next_n_units) / G);
                const size_t total = (size_t)(nu1 - nu0) * g.next_rpu * g.next_K * 2;
                const size_t want = total < (size_t)kGemvRingBytes ? total : (size_t)kGemvRingBytes;
                const uint8_t *src = reinterpret_cast<const uint8_t *>(g.next_W + (size_t)nu0 * g.next_rpu * g.next_K);
                for (size_t off = 0; off < want; off += 32768)
                    bulk_prefetch_l2(src + off, (uint32_t)(want - off < 32768 ? want - off : 32768));
            }
            // no copy may still be landing in this CTA's shared memory when it exits
            for (int s = max(0, issued - S); s < issued; ++s)
                mbar_wait(full0 + 8 * (s % S), (s / S) & 1, err, SITE_GEMV_DRAIN);
        }
        return;
    }

    // --------------------------------------------------------------- consumers
    Epi epi = epi_in;
    griddep_wait();
    const int nchunks = g.K >> 3;
    float h[NCH][8];
    float ss = 0.f;
    const int tok = g.embed ? g.ctrl[CTRL_TOKEN] : 0;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int c = tid + kGemvConsumers * j;
        if (FULL || c < nchunks) {
            if (g.embed) {
                const uint4 w = *reinterpret_cast<const uint4 *>(g.embed + (size_t)tok * g.K + c * 8);
                h[j][0] = bf16lo(w.x); h[j][1] = bf16hi(w.x); h[j][2] = bf16lo(w.y); h[j][3] = bf16hi(w.y);
                h[j][4] = bf16lo(w.z); h[j][5] = bf16hi(w.z); h[j][6] = bf16lo(w.w); h[j][7] = bf16hi(w.w);
                if (blockIdx.x == 0) {
                    float4 *dst = reinterpret_cast<float4 *>(g.x_out + c * 8);
                    dst[0] = make_float4(h[j][0], h[j][1], h[j][2], h[j][3]);
                    dst[1] = make_float4(h[j][4], h[j][5], h[j][6], h[j][7]);
                }
            } else {
                const float4 a = *reinterpret_cast<const float4 *>(g.in + c * 8);
                const float4 b = *reinterpret_cast<const float4 *>(g.in + c * 8 + 4);
                h[j][0] = a.x; h[j][1] = a.y; h[j][2] = a.z; h[j][3] = a.w;
                h[j][4] = b.x; h[j][5] = b.y; h[j][6] = b.z; h[j][7] = b.w;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) ss = fmaf(h[j][e], h[j][e], ss);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) h[j][e] = 0.f;
        }
    }
    if (g.gain) {  // RMSNorm prologue: every CTA reduces the whole vector in the same order
        ss = warp_sum(ss);
        if (lane == 0) s_part[warp] = ss;
        consumer_sync();
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < kGemvWarps; ++w) tot += s_part[w];
        const float rinv = 1.0f / sqrtf(tot / (float)g.K + g.eps);
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = tid + kGemvConsumers * j;
            if (FULL || c < nchunks) {
                const uint4 gw = *reinterpret_cast<const uint4 *>(g.gain + c * 8);
                const float gg[8] = {bf16lo(gw.x), bf16hi(gw.x), bf16lo(gw.y), bf16hi(gw.y),
                                     bf16lo(gw.z), bf16hi(gw.z), bf16lo(gw.w), bf16hi(gw.w)};
#pragma unroll
                for (int e = 0; e < 8; ++e) h[j][e] = h[j][e] * rinv * gg[e];
            }
        }
    }

    const uint32_t row_bytes = (uint32_t)g.K * 2u;
    const uint32_t my0 = smem_u32(ring) + (uint32_t)tid * 16u;   // this thread's chunk 0 in slot 0
    const bool tail_ok = FULL || tid + kGemvConsumers * (NCH - 1) < nchunks;
    int buf = 0, brow = 0, bunit0 = 0, slot = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int s = 0; s < nst; ++s) {
        const int rows = min(RPS, total_rows - s * RPS);
        ok = ok && !*reinterpret_cast<volatile int *>(&s_abort) &&
             mbar_wait(full0 + 8 * slot, phase, err, SITE_GEMV_FULL);
        if (!ok) s_abort = 1;
        float acc[RPS];
#pragma unroll
        for (int r = 0; r < RPS; ++r) acc[r] = 0.f;
        if (ok) {
            const uint32_t sb = my0 + (uint32_t)slot * g.slot_bytes;
            if (rows == RPS) {
#pragma unroll
                for (int r = 0; r < RPS; ++r)
#pragma unroll
                    for (int j = 0; j < NCH; ++j)
                        if (j < NCH - 1 || tail_ok)
                            acc[r] = dot8(lds128(sb + r * row_bytes + j * kGemvConsumers * 16), h[j], acc[r]);
            } else {   // the CTA's last slot may hold fewer rows
#pragma unroll
                for (int r = 0; r < RPS; ++r)
                    if (r < rows)
#pragma unroll
                        for (int j = 0; j < NCH; ++j)
                            if (j < NCH - 1 || tail_ok)
                                acc[r] = dot8(lds128(sb + r * row_bytes + j * kGemvConsumers * 16), h[j], acc[r]);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8 * slot);
        if (++slot == S) {
            slot = 0;
            phase ^= 1u;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < RPS; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
        if (lane == 0) {
            float *rb = red + (size_t)(buf * kGemvWarps + warp) * kRedRows + brow;
#pragma unroll
            for (int r = 0; r < RPS; ++r)
                if (r < rows) rb[r] = acc[r];
        }
        brow += rows;
        if (s == nst - 1 || brow + RPS > kRedRows) {
            consumer_sync();
            if (s_abort) break;
            const int bunits = brow / g.rpu;
            for (int t = tid; t < bunits; t += kGemvConsumers) {
                float v[2];
                for (int j = 0; j < g.rpu; ++j) {
                    float sum = 0.f;
#pragma unroll
                    for (int w = 0; w < kGemvWarps; ++w)
                        sum += red[(size_t)(buf * kGemvWarps + w) * kRedRows + t * g.rpu + j];
                    v[j] = sum;
                }
                epi.unit(u0 + bunit0 + t, v);
            }
            bunit0 += bunits;
            brow = 0;
            buf ^= 1;
        }
    }

    if constexpr (Epi::kArgmax) lm_argmax(epi, s_bv, s_bi, &s_last);
}

// ------------------------------------------------------------ flash-decode ----
// Split-K attention of one query token over the paged cache (Sec. 5.1 decode
// step).  Grid (S, nkv): CTA (r, g) covers split r of KV head g, a contiguous
// range of the cached pages; block = group x wph query warps + 1 producer warp.
// The producer streams the range's pages (the K and V blocks of head g, 16 x d
// bf16 each, contiguous in a page) through a small TMA ring; query warp
// (j, set) runs an online softmax for query head g*group + j over the pages
// i = set (mod wph) of the range, and the wph states of a head are merged in
// shared memory.  Each CTA writes its per-head state (acc, m, l) to global
// memory and takes a ticket; the last CTA of head g combines the splits in
// split order, so the result does not depend on which CTA finishes last.
//
// No cluster and a small footprint (<= 288 threads, 32 KB ring): the CTAs fit
// beside a GEMV CTA on the same SM, so under programmatic dependent launch the
// kernel starts streaming pages while the QKV GEMV still runs, and the O
// projection's weight ring fills while the attention finishes.  The length comes
// from the device position, so one captured graph serves every step; the split
// count adapts to it at run time (at most gridDim.x splits).
constexpr uint32_t kFdRingBytes = 32768;
constexpr int kFdMaxQueryWarps = 8;
constexpr int kFdMaxSplits = 32;

struct FDArgs {
    const float *q;
    const uint16_t *kv;  // this layer's pages
    const int *pages;
    int *ctrl;
    float *o;
    float *part;         // [nkv][splits][group][d + 4]: acc[d], m, l of each split
    int nkv, group, wph;
    size_t page_elems;
    float qscale;        // log2(e) / sqrt(d)
};

enum : int { SITE_FD_EMPTY = 31, SITE_FD_FULL = 32, SITE_FD_DRAIN = 33 };

// (m, l, acc) online-softmax merge of b into a (log2 domain)
// An empty state (no keys seen) has m = -inf, l = 0, acc = 0 and is skipped:
// exp2(m - M) with both maxima -inf would be NaN.
template <int EPL>
__device__ __forceinline__ void fd_merge(float &m, float &l, float *acc, float mb, float lb, const float *accb) {
    if (mb == -INFINITY) return;
    if (m == -INFINITY) {
        m = mb;
        l = lb;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] = accb[e];
        return;
    }
    const float M = fmaxf(m, mb);
    const float fa = exp2f(m - M), fb = exp2f(mb - M);
    l = l * fa + lb * fb;
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = acc[e] * fa + accb[e] * fb;
    m = M;
}

template <int D>
__global__ void __launch_bounds__(32 * (kFdMaxQueryWarps + 1)) flash_decode_kernel(const FDArgs a) {
    constexpr int EPL = D / 32;
    constexpr uint32_t BLK = kPage * D * 2;              // bytes of one K (or V) block of a page
    constexpr int STAGES = (int)(kFdRingBytes / (2 * BLK));
    constexpr int STRIDE = D + 4;                        // floats per state: acc[D], m, l, pad
    extern __shared__ __align__(128) uint8_t fsm[];      // [STAGES][K block | V block]
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES];
    __shared__ __align__(16) float s_state[kFdMaxQueryWarps][STRIDE];
    __shared__ int s_last;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nq = a.group * a.wph;   // query warps
    const int g = blockIdx.y;
    const int r = blockIdx.x;
    int *err = a.ctrl + CTRL_ERR;

    // the position is only advanced at the end of a step, so it is stable here
    const int len = *reinterpret_cast<volatile int *>(a.ctrl + CTRL_POS) + 1;
    const int npages = (len + kPage - 1) / kPage;
    const int pps = (npages + (int)gridDim.x - 1) / (int)gridDim.x;
    const int splits = (npages + pps - 1) / pps;          // every split below this has pages
    if (r >= splits) return;                              // idle CTA: no state, no ticket
    const int p0 = r * pps;
    const int n = min(npages, p0 + pps) - p0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), a.group);
        }
        fence_barrier_init();
    }
    __syncthreads();
    griddep_launch_dependents();

    if (w == nq) {  // ---------------------------------------------- producer
        // the whole warp walks the pages so that 32 page-table entries are read at
        // once (one coalesced load) and handed out by shuffle; lane 0 issues
        const uint32_t ring0 = smem_u32(fsm);
        int issued = 0, my_page = 0;
        bool waited = false;
        for (int i = 0; i < n; ++i) {
            if ((i & 31) == 0 && i + lane < n) my_page = a.pages[p0 + i + lane];
            const int page = __shfl_sync(0xffffffffu, my_page, i & 31);
            const int s = i % STAGES;
            bool ok = true;
            if (lane == 0 && i >= STAGES)
                ok = mbar_wait(smem_u32(&empty_bar[s]), ((i / STAGES) + 1) & 1, err, SITE_FD_EMPTY);
            if (!__shfl_sync(0xffffffffu, (int)ok, 0)) break;
            // the page holding the current position is written by the preceding kernel
            if (!waited && p0 + i == npages - 1) {
                griddep_wait();
                waited = true;
            }
            if (lane == 0) {
                const uint16_t *Kb = a.kv + (size_t)page * a.page_elems + (size_t)g * kPage * D;
                const uint16_t *Vb = Kb + (size_t)a.nkv * kPage * D;
                const uint32_t fb = smem_u32(&full_bar[s]);
                mbar_arrive_expect_tx(fb, 2 * BLK);
                bulk_g2s(ring0 + s * 2 * BLK, Kb, BLK, fb);
                bulk_g2s(ring0 + s * 2 * BLK + BLK, Vb, BLK, fb);
            }
            issued = i + 1;
        }
        if (lane == 0)
            for (int i = max(0, issued - STAGES); i < issued; ++i)
                mbar_wait(smem_u32(&full_bar[i % STAGES]), (i / STAGES) & 1, err, SITE_FD_DRAIN);
        __syncwarp();
        return;   // the producer takes no part in the named barriers below
    }

    // ------------------------------------------------------------ query warps
    griddep_wait();
    const int j = w % a.group, set = w / a.group;
    const int head = g * a.group + j;
    float qv[EPL], acc[EPL];
    if constexpr (EPL == 4) {
        const float4 q4 = *reinterpret_cast<const float4 *>(a.q + head * D + lane * 4);
        qv[0] = q4.x * a.qscale; qv[1] = q4.y * a.qscale; qv[2] = q4.z * a.qscale; qv[3] = q4.w * a.qscale;
    } else {
        const float2 q2 = *reinterpret_cast<const float2 *>(a.q + head * D + lane * 2);
        qv[0] = q2.x * a.qscale; qv[1] = q2.y * a.qscale;
    }
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
    float m = -INFINITY, l = 0.f;
    const int key = lane >> 1;   // the key whose score this lane ends with
    bool ok = true;
    for (int i = set; i < n && ok; i += a.wph) {
        const int s = i % STAGES;
        ok = mbar_wait(smem_u32(&full_bar[s]), (i / STAGES) & 1, err, SITE_FD_FULL);
        if (!ok) break;
        const uint8_t *Ks = fsm + (size_t)s * 2 * BLK;
        const uint8_t *Vs = Ks + BLK;
        const int ntok = min(kPage, len - (p0 + i) * kPage);
        // partial dot products of this lane's d-slice with the 16 keys
        float sc[kPage];
#pragma unroll
        for (int t = 0; t < kPage; ++t) {
            const uint8_t *kr = Ks + (t * D + lane * EPL) * 2;
            if constexpr (EPL == 4) {
                const uint2 kw = *reinterpret_cast<const uint2 *>(kr);
                sc[t] = qv[0] * bf16lo(kw.x) + qv[1] * bf16hi(kw.x) + qv[2] * bf16lo(kw.y) + qv[3] * bf16hi(kw.y);
            } else {
                const uint32_t kw = *reinterpret_cast<const uint32_t *>(kr);
                sc[t] = qv[0] * bf16lo(kw) + qv[1] * bf16hi(kw);
            }
        }
        // transposed butterfly: lanes 2k and 2k+1 end with the full score of key k
#pragma unroll
        for (int o = 16, cnt = kPage; o > 0; o >>= 1) {
            if (cnt > 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int t = 0; t < cnt / 2; ++t) {
                    const float send = up ? sc[t] : sc[t + cnt / 2];
                    const float keep = up ? sc[t + cnt / 2] : sc[t];
                    sc[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
                cnt >>= 1;
            } else {
                sc[0] += __shfl_xor_sync(0xffffffffu, sc[0], o);
            }
        }
        const float my = key < ntok ? sc[0] : -INFINITY;   // slots past the length are masked
        const float mx = fmaxf(m, warp_max(my));
        const float corr = exp2f(m - mx);
        const float pme = exp2f(my - mx);                  // 0 for masked keys
        l = l * corr + pme;   // per-lane share of the denominator (every key is held by two lanes)
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] *= corr;
#pragma unroll
        for (int t = 0; t < kPage; ++t) {
            // slots past the length are never used: they may hold stale values
            const bool valid = t < ntok;
            const float pt = __shfl_sync(0xffffffffu, pme, 2 * t);
            const uint8_t *vr = Vs + (t * D + lane * EPL) * 2;
            if constexpr (EPL == 4) {
                uint2 vw = *reinterpret_cast<const uint2 *>(vr);
                if (!valid) vw = make_uint2(0u, 0u);
                acc[0] = fmaf(pt, bf16lo(vw.x), acc[0]);
                acc[1] = fmaf(pt, bf16hi(vw.x), acc[1]);
                acc[2] = fmaf(pt, bf16lo(vw.y), acc[2]);
                acc[3] = fmaf(pt, bf16hi(vw.y), acc[3]);
            } else {
                uint32_t vw = *reinterpret_cast<const uint32_t *>(vr);
                if (!valid) vw = 0u;
                acc[0] = fmaf(pt, bf16lo(vw), acc[0]);
                acc[1] = fmaf(pt, bf16hi(vw), acc[1]);
            }
        }
        m = mx;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
    }
    l = warp_sum(l) * 0.5f;
    if (a.wph > 1) {
#pragma unroll
        for (int e = 0; e < EPL; ++e) s_state[w][lane * EPL + e] = acc[e];
        if (lane == 0) {
            s_state[w][D] = m;
            s_state[w][D + 1] = l;
        }
        // merge the wph page sets of each head into set 0 (fixed set order)
        asm volatile("bar.sync 1, %0;" ::"r"(32 * nq) : "memory");
        if (set == 0)
            for (int t = 1; t < a.wph; ++t) {
                const float *o = s_state[t * a.group + j];
                float ob[EPL];
#pragma unroll
                for (int e = 0; e < EPL; ++e) ob[e] = o[lane * EPL + e];
                fd_merge<EPL>(m, l, acc, o[D], o[D + 1], ob);
            }
    }
    // this split's state of head j -> global; then the ticket
    float *mine = a.part + ((size_t)(g * gridDim.x + r) * a.group + j) * STRIDE;
    if (set == 0) {
        if constexpr (EPL == 4)
            *reinterpret_cast<float4 *>(mine + lane * 4) = make_float4(acc[0], acc[1], acc[2], acc[3]);
        else
            *reinterpret_cast<float2 *>(mine + lane * 2) = make_float2(acc[0], acc[1]);
        if (lane == 0) *reinterpret_cast<float2 *>(mine + D) = make_float2(m, l);
    }
    // the CTA barrier orders every warp's stores before thread 0's fence, which
    // publishes them at GPU scope ahead of the ticket (and, for the last CTA, orders
    // the other splits' stores before the loads below)
    asm volatile("bar.sync 1, %0;" ::"r"(32 * nq) : "memory");
    if (threadIdx.x == 0) {
        __threadfence();
        const int t = atomicAdd(a.ctrl + CTRL_ATTN_TICKET0 + g, 1);
        s_last = (t == splits - 1);
        if (s_last) __threadfence();
    }
    asm volatile("bar.sync 1, %0;" ::"r"(32 * nq) : "memory");
    if (!s_last || set != 0) return;

    // ------------------------------------------- last CTA of head g: combine
    const float *base = a.part + ((size_t)g * gridDim.x * a.group + j) * STRIDE;
    const size_t sstride = (size_t)a.group * STRIDE;     // floats between splits of one head
    float2 ml = make_float2(-INFINITY, 0.f);
    if (lane < splits) ml = __ldcg(reinterpret_cast<const float2 *>(base + lane * sstride + D));
    const float M = warp_max(ml.x);
    const float f = lane < splits ? exp2f(ml.x - M) : 0.f;
    const float L = warp_sum(ml.y * f);
    float out[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) out[e] = 0.f;
    for (int s0 = 0; s0 < splits; s0 += 8) {
        float v[8][EPL];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int sp = min(s0 + u, splits - 1);
            const float *src = base + sp * sstride + lane * EPL;
            if constexpr (EPL == 4) {
                const float4 t4 = __ldcg(reinterpret_cast<const float4 *>(src));
                v[u][0] = t4.x; v[u][1] = t4.y; v[u][2] = t4.z; v[u][3] = t4.w;
            } else {
                const float2 t2 = __ldcg(reinterpret_cast<const float2 *>(src));
                v[u][0] = t2.x; v[u][1] = t2.y;
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float fs = __shfl_sync(0xffffffffu, f, (s0 + u) & 31);
            if (s0 + u < splits)
#pragma unroll
                for (int e = 0; e < EPL; ++e) out[e] = fmaf(v[u][e], fs, out[e]);
        }
    }
    const float inv = 1.0f / L;
    if constexpr (EPL == 4)
        *reinterpret_cast<float4 *>(a.o + head * D + lane * 4) =
            make_float4(out[0] * inv, out[1] * inv, out[2] * inv, out[3] * inv);
    else
        *reinterpret_cast<float2 *>(a.o + head * D + lane * 2) = make_float2(out[0] * inv, out[1] * inv);
    if (j == 0 && lane == 0) a.ctrl[CTRL_ATTN_TICKET0 + g] = 0;   // ready for the next layer
}

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
// that names the layer of the step (mega_tag).  A consumer polls the words it
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
// us with five grid barriers a layer, 72 us now; at 1B widths 35.0 and 27.5 us.
constexpr int kMegaSlots = 6;
constexpr uint32_t kMegaSlotBytes = 32768;
constexpr int kMegaMaxCtas = 256;               // grid size limit (one CTA per SM)
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

// one word, polled
__device__ __forceinline__ bool mega_word(const uint64_t *p, uint32_t tag, float *v, int *err) {
    PollLimit lim;
    uint64_t w = ld_tagged(p);
    while (!has_tag(w, tag)) {
        if (!lim.again(err)) return false;
        w = ld_tagged(p);
    }
    *v = tagged_value(w);
    return true;
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
    static constexpr bool kArgmax = false;
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
    static constexpr bool kArgmax = false;
    __device__ void prefetch(int) {}
    __device__ void unit(int u, const float *v, bool) {
        const float gt = v[0];
        st_tagged(m + u, gt / (1.0f + expf(-gt)) * v[1], tag);
    }
};

// Packed QKV rows (pairs as in EpiQKV): q and k after RoPE (before their norms
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
    static constexpr bool kArgmax = false;
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
// The producer keeps about kMegaFlightBytes of copies in flight per SM (never
// fewer than two slots), and lets landed slots fill the rest of the ring.  That is
// what the HBM needs (152 SMs x 64 KB over ~1.3 us); more only queues in the memory
// system, in front of the words that the phases exchange: with the whole ring in
// flight and 192 KB of gate/up rows per SM moved to L2 during the attention phase,
// a word took up to 4 us to arrive, and a step of the 8B widths 2636 us against
// 2491 (1B: 589 against 555); one slot in flight starves the HBM (3136 us).
constexpr uint32_t kMegaFlightBytes = 65536;
__device__ __forceinline__ int mega_flight(uint32_t slot_bytes) {
    return min(kMegaSlots, max(2, (int)(kMegaFlightBytes / slot_bytes)));
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
__device__ bool mp_rows(MegaRing &R, const uint16_t *W, uint32_t row_bytes, int n_units, int rpu, int RPS,
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

__device__ __forceinline__ MegaSplit mega_split(const MegaArgs &a, int len) {
    MegaSplit sp;
    const int unit = blockIdx.x;
    sp.npages = (len + kPage - 1) / kPage;
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
#pragma unroll
        for (int r = 0; r < RPS; ++r) acc[r] = 0.f;
        const uint32_t sb = R.data0 + (uint32_t)slot * kMegaSlotBytes + (uint32_t)tid * 16u;
        if (!ok) {
        } else if (rows == RPS) {
#pragma unroll
            for (int r = 0; r < RPS; ++r)
#pragma unroll
                for (int j = 0; j < NCH; ++j)
                    if (j < NCH - 1 || tail_ok)
                        acc[r] = dot8(lds128(sb + r * row_bytes + j * kGemvConsumers * 16), h[j], acc[r]);
        } else {
#pragma unroll
            for (int r = 0; r < RPS; ++r)
                if (r < rows)
#pragma unroll
                    for (int j = 0; j < NCH; ++j)
                        if (j < NCH - 1 || tail_ok)
                            acc[r] = dot8(lds128(sb + r * row_bytes + j * kGemvConsumers * 16), h[j], acc[r]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(R.empty0 + 8 * slot);
        ++R.n;
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
        float acc[RPS];
#pragma unroll
        for (int r = 0; r < RPS; ++r) acc[r] = 0.f;
        // chunk c: codes at byte 16 c of the row, its block's scale at byte K + 2 (c / 2)
        const uint32_t s0 = R.data0 + (uint32_t)slot * kMegaSlotBytes;
        const uint32_t sb = s0 + (uint32_t)tid * 16u;
        const uint32_t sc = s0 + (uint32_t)K + (uint32_t)(tid >> 1) * 2u;
        if (ok) {
#pragma unroll
            for (int r = 0; r < RPS; ++r)
                if (rows == RPS || r < rows)
#pragma unroll
                    for (int j = 0; j < NCH; ++j)
                        if (j < NCH - 1 || tail_ok) {
                            const uint4 w = lds128(sb + r * row_bytes + j * kGemvConsumers * 16);
                            const float d = lds_f16(sc + r * row_bytes + j * (kGemvConsumers / 2) * 2);
                            const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
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
                            acc[r] = fmaf(d, cv, acc[r]);
                        }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(R.empty0 + 8 * slot);
        ++R.n;
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

// a per-layer GEMV phase in the layer matrices' format
template <bool Q8, class S, int ND = kQ8RestDigits, class Epi>
__device__ __forceinline__ bool mc_layer_gemv(MegaRing &R, float *red, int K, int n_units, int rpu,
                                              const uint64_t *in, uint32_t tag, const uint16_t *gain,
                                              const uint16_t *embed, float eps, int *err, Epi &epi, float *s_part,
                                              uint64_t *t_data = nullptr) {
    if constexpr (Q8)
        return mc_gemv_q8<S, ND>(R, red, K, n_units, rpu, in, tag, gain, embed, eps, err, epi, s_part, t_data);
    else
        return mc_gemv<S>(R, red, K, n_units, rpu, in, tag, gain, embed, eps, err, epi, s_part, t_data);
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
// precision) and K and V are exact bf16, so every product is exact and the sums
// are fp32.  A scalar version (one warp per head and page, lane-transposed dot
// products) took about 1 us per page: 29 us a layer at 8K cached tokens.
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
    asm volatile(
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
            // S: acc01 rows 0..7 term 0, rows 8..15 term 1; acc2 rows 0..7 term 2
            float s01[2][4] = {}, s2[2][4] = {};
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                uint32_t qa[4], q2a, q2b, kf[4];
                ldsm4(qs0 + (mi & 1) * SM::Q_TERM + mr * SM::Q_ROW + (16 * kk + (mi >> 1) * 8) * 2, qa);
                ldsm2(qs0 + 2 * SM::Q_TERM + mr * SM::Q_ROW + (16 * kk + (mi & 1) * 8) * 2, q2a, q2b);
                const int key = (mi >> 1) * 8 + mr, u = (kk & 3) * 2 + (mi & 1);
                ldsm4(kb + (kk >> 2) * PG::CHUNK + key * 128 + ((u ^ (key & 7)) << 4), kf);
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    mma_bf16(s01[t], qa[0], qa[1], qa[2], qa[3], kf[2 * t], kf[2 * t + 1]);
                    mma_bf16(s2[t], q2a, 0u, q2b, 0u, kf[2 * t], kf[2 * t + 1]);
                }
            }
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
                uint32_t vf[4];
                const int key = (mi & 1) * 8 + mr, u = 2 * n + (mi >> 1);
                ldsm4t(vb + (u >> 3) * PG::CHUNK + key * 128 + (((u & 7) ^ (key & 7)) << 4), vf);
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    mma_bf16(o[2 * n + t], p[0][2], 0u, p[1][2], 0u, vf[2 * t], vf[2 * t + 1]);
                    mma_bf16(o[2 * n + t], p[0][0], p[0][1], p[1][0], p[1][1], vf[2 * t], vf[2 * t + 1]);
                }
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
    constexpr int MAXQ = kFdMaxSplits / 8;    // splits of one warp
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
__device__ void mega_rebalance(const MegaArgs &a, float *scr) {
    const int G = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    static_assert(kMegaMaxCtas <= kGemvConsumers, "one thread per CTA");
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

// SH, SF: GEMV shapes of K = hidden and K = ffn for bf16 rows; with Q8 the seven
// per-layer matrices are in the 8-bit block format and stream with the shapes
// QH, QF (16-element chunks, rows per slot sized for the shorter rows), while
// the LM head stays bf16 (SH).
template <int D, class SH, class SF, bool Q8, class QH, class QF>
__global__ void __launch_bounds__(kGemvThreads, 1)
    decode_step_kernel(const __grid_constant__ CUtensorMap map_kv, const MegaArgs a) {
    using LH = std::conditional_t<Q8, QH, SH>;   // layer matrices with K = hidden (and K = n_q * d)
    using LF = std::conditional_t<Q8, QF, SF>;   // the down projection, K = ffn
    const uint32_t rb_h = Q8 ? (uint32_t)q8_row_bytes((size_t)a.H) : (uint32_t)a.H * 2u;
    const uint32_t rb_q = Q8 ? (uint32_t)q8_row_bytes((size_t)a.qdim) : (uint32_t)a.qdim * 2u;
    const uint32_t rb_f = Q8 ? (uint32_t)q8_row_bytes((size_t)a.F) : (uint32_t)a.F * 2u;
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
    const MegaSplit sp = mega_split(a, len);

    if (warp == kGemvWarps) {  // ------------------------------------ producer
        if (lane == 0) {
            const uint64_t pol = l2_evict_first();
            bool ok = true;
            for (int l = 0; l < a.L && ok; ++l) {
                const size_t lo = (size_t)l * a.lstride;
                ok = mp_rows(R, a.W + a.l0.wqkv + lo, rb_h, a.nqkv / 2, 2, LH::RPS, err, pol) &&
                     mp_pages<D>(R, a, &map_kv, l, sp, err) &&
                     mp_rows(R, a.W + a.l0.wo + lo, rb_q, a.H, 1, LH::RPS, err, pol) &&
                     mp_rows(R, a.W + a.l0.wgu + lo, rb_h, a.F, 2, LH::RPS, err, pol) &&
                     mp_rows(R, a.W + a.l0.wd + lo, rb_f, a.H, 1, LF::RPS, err, pol);
            }
            if (ok) mp_rows(R, a.W + a.w_lm, (uint32_t)a.H * 2u, a.V, 1, SH::RPS, err, pol);
            // no copy may still be landing in shared memory when the CTA exits
            for (int s = max(0, R.n - kMegaSlots); s < R.n; ++s)
                mbar_wait(R.full0 + 8 * (s % kMegaSlots), (s / kMegaSlots) & 1, err, SITE_MEGA_DRAIN);
        }
        return;
    }

    // ---------------------------------------------------------------- consumers
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
        ok = mc_layer_gemv<Q8, LH, kQ8QkvDigits>(R, red, a.H, a.nqkv / 2, 2, a.txd, tag - 1u,
                                                 a.W + a.l0.attn_norm + lo, e0, a.eps, err, eq, s_part);
        if (!ok) break;
        ok = mc_attn<D>(R, a, a.KV + (size_t)l * a.kv_layer_elems, sp, len, tag, reinterpret_cast<uint8_t *>(red),
                        state, s_rope, a.qk_norm ? a.W + a.l0.qn + lo : nullptr,
                        a.qk_norm ? a.W + a.l0.kn + lo : nullptr);
        if (!ok) break;
        MEpiResidual er;
        er.prev = a.txd; er.embed = e0; er.prev_tag = tag - 1u; er.out = a.txo; er.tag = tag;
        ok = mc_layer_gemv<Q8, LH>(R, red, a.qdim, a.H, 1, a.to, tag, nullptr, nullptr, a.eps, err, er, s_part);
        if (!ok) break;
        MEpiSwiGLU es{a.tm, tag};
        uint64_t t_gu = 0;
        ok = mc_layer_gemv<Q8, LH>(R, red, a.H, a.F, 2, a.txo, tag, a.W + a.l0.ffn_norm + lo, nullptr, a.eps, err, es,
                                   s_part, &t_gu);
        if (!ok) break;
        if (t_gu) gu_ns += globaltimer_ns() - t_gu;
        er.prev = a.txo; er.embed = nullptr; er.prev_tag = tag; er.out = a.txd;
        ok = mc_layer_gemv<Q8, LF>(R, red, a.F, a.H, 1, a.tm, tag, nullptr, nullptr, a.eps, err, er, s_part);
        if (!ok) break;
    }
    if (tid == 0) a.cta_time[blockIdx.x] = (float)gu_ns * 1e-3f;
    if (!ok) return;
    MEpiArgmax ea;
    ea.logits = a.logits; ea.partial = a.amax; ea.ctrl = a.ctrl; ea.hist = a.hist; ea.pos_add = 1;
    ea.best = -INFINITY; ea.bidx = 0x7fffffff;
    if (!mc_gemv<SH>(R, red, a.H, a.V, 1, a.txd, tag0 + (uint32_t)a.L, a.W + a.w_final_norm, nullptr, a.eps, err, ea,
                     s_part, nullptr))
        return;
    if (!lm_argmax(ea, s_bv, s_bi, &s_last)) return;
    if (tid == 0) a.ctrl[CTRL_EPOCH] += 1;   // the next step's words carry other tags
    mega_rebalance(a, state);
}

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

template <typename Kern, typename... Args>
static cudaError_t launch(Kern kern, dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                          Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// query warps per head: at most kFdMaxQueryWarps query warps per CTA
static int fd_wph(int group) { return group >= kFdMaxQueryWarps ? 1 : kFdMaxQueryWarps / group; }

int fd_splits(int max_pages) {
    const int s = (max_pages + 3) / 4;   // about four pages per split at the largest length
    return s < 1 ? 1 : (s > kFdMaxSplits ? kFdMaxSplits : s);
}

size_t fd_part_floats(int nkv, int group, int d, int max_pages) {
    (void)max_pages;   // room for the largest split count of either decode path
    return (size_t)nkv * kFdMaxSplits * group * (d + 4);
}

size_t mega_part_words(int nkv, int group, int d) { return (size_t)nkv * kFdMaxSplits * group * (d + 2); }

template <int D>
static cudaError_t launch_fd(const Plan &p, const FDArgs &fa, cudaStream_t st, bool pdl) {
    constexpr uint32_t BLK = kPage * D * 2;
    return launch(flash_decode_kernel<D>, dim3(fd_splits(p.max_pages), p.nkv), dim3(32 * (fa.group * fa.wph + 1)),
                  (size_t)(kFdRingBytes / (2 * BLK)) * 2 * BLK, st, pdl, fa);
}

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
#define WICI_MEGA_ATTR(DD, SH, SF, Q8, QH, QF)                                                        \
    if ((e = cudaFuncSetAttribute(decode_step_kernel<DD, SH, SF, Q8, QH, QF>,                          \
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMegaSmem)) != cudaSuccess) \
        return e;
    WICI_MEGA_SHAPES(WICI_MEGA_ATTR)
#undef WICI_MEGA_ATTR
    if ((e = set_gemv_attrs<EpiResidual>()) != cudaSuccess) return e;
    if ((e = set_gemv_attrs<EpiSwiGLU>()) != cudaSuccess) return e;
    if ((e = set_gemv_attrs<EpiQKV>()) != cudaSuccess) return e;
    if ((e = set_gemv_attrs<EpiArgmax>()) != cudaSuccess) return e;
    return cudaSuccess;
}

// Ring geometry: slots of gemv_rps(K) rows, as many as fit kGemvRingBytes (2 to 8).
static void ring_geometry(GemvIn &g) {
    const int rps = gemv_rps(g.K);
    g.ups = rps / g.rpu;
    g.slot_bytes = ((uint32_t)rps * (uint32_t)g.K * 2u + 127u) & ~127u;
    int st = (int)(kGemvRingBytes / g.slot_bytes);
    g.stages = st < 2 ? 2 : (st > kGemvMaxStages ? kGemvMaxStages : st);
}

template <class Epi>
static cudaError_t launch_gemv(const Plan &p, GemvIn g, Epi epi, cudaStream_t st, bool pdl,
                               LaunchHook *hook, const char *name) {
    ring_geometry(g);
    void *fn = gemv_fn<Epi>(g.K);
    if (!fn || g.ups < 1) return cudaErrorInvalidValue;
    const int grid = p.num_sms * kGemvCtasPerSm;
    if (hook) hook->before(name);
    cudaError_t e = launch(reinterpret_cast<void (*)(const GemvIn, const Epi)>(fn),
                           dim3(grid), dim3(kGemvThreads), gemv_smem_bytes(g.stages, g.slot_bytes), st, pdl,
                           g, epi);
    if (hook) hook->after(name);
    return e;
}

static GemvIn gemv_in(const Plan &p, const Bufs &b, const uint16_t *W, int K, int n_units, int rpu,
                      const float *in, const uint16_t *gain) {
    GemvIn g = {};
    g.W = W;
    g.K = K;
    g.n_units = n_units;
    g.rpu = rpu;
    g.in = in;
    g.gain = gain;
    g.ctrl = b.ctrl;
    g.eps = p.cfg.rms_eps;
    return g;
}

// Decode-step GEMVs in launch order: per layer QKV, O, gate/up, down; then the LM head.
enum GemvId : int { G_QKV = 0, G_O = 1, G_GU = 2, G_DOWN = 3, G_LM = 4 };

static void set_next(const Plan &p, const Bufs &b, GemvIn &g, int layer, int id) {
    if (id == G_LM) {
        layer = 0;
        id = G_QKV;        // the next step starts with layer 0
    } else if (id == G_DOWN) {
        if (++layer == p.L) id = G_LM;
        else id = G_QKV;
    } else {
        ++id;
    }
    if (id == G_LM) {
        g.next_W = b.W + p.w_lm; g.next_K = p.H; g.next_n_units = p.V; g.next_rpu = 1;
        return;
    }
    const LayerOffsets &lo = p.layer[layer];
    switch (id) {
        case G_QKV: g.next_W = b.W + lo.wqkv; g.next_K = p.H; g.next_n_units = p.nqkv / 2; g.next_rpu = 2; break;
        case G_O: g.next_W = b.W + lo.wo; g.next_K = p.qdim; g.next_n_units = p.H; g.next_rpu = 1; break;
        case G_GU: g.next_W = b.W + lo.wgu; g.next_K = p.H; g.next_n_units = p.F; g.next_rpu = 2; break;
        default: g.next_W = b.W + lo.wd; g.next_K = p.F; g.next_n_units = p.H; g.next_rpu = 1; break;
    }
}

cudaError_t enqueue_lm_head(const Plan &p, const Bufs &b, const float *x, cudaStream_t st, bool pdl, int pos_add,
                            LaunchHook *hook) {
    GemvIn g = gemv_in(p, b, b.W + p.w_lm, p.H, p.V, 1, x, b.W + p.w_final_norm);
    set_next(p, b, g, p.L - 1, G_LM);   // a decode step (layer 0) follows
    EpiArgmax e = {};
    e.logits = b.logits;
    e.partial = b.amax;
    e.ctrl = b.ctrl;
    e.hist = b.hist;
    e.pos_add = pos_add;
    e.best = -INFINITY;
    e.bidx = 0x7fffffff;
    return launch_gemv(p, g, e, st, pdl, hook, "lm_head_argmax");
}

cudaError_t enqueue_lm_head_argmax_raw(const uint16_t *W, const uint16_t *gain, const float *x, int H, int V,
                                       float eps, float *logits, int *ctrl, int2 *partials, int *hist, int grid,
                                       cudaStream_t st) {
    GemvIn g = {};
    g.W = W;
    g.K = H;
    g.n_units = V;
    g.rpu = 1;
    g.in = x;
    g.gain = gain;
    g.ctrl = ctrl;
    g.eps = eps;
    ring_geometry(g);
    void *fn = gemv_fn<EpiArgmax>(g.K);
    if (!fn || g.ups < 1) return cudaErrorInvalidValue;
    EpiArgmax e = {};
    e.logits = logits;
    e.partial = partials;
    e.ctrl = ctrl;
    e.hist = hist;
    e.pos_add = 0;
    e.best = -INFINITY;
    e.bidx = 0x7fffffff;
    return launch(reinterpret_cast<void (*)(const GemvIn, const EpiArgmax)>(fn), dim3(grid), dim3(kGemvThreads),
                  gemv_smem_bytes(g.stages, g.slot_bytes), st, false, g, e);
}


// ------------------------------------------------------- persistent decode: host
typedef cudaError_t (*MegaLaunch)(const CUtensorMap &, const MegaArgs &, int grid, cudaStream_t);

template <int D, class SH, class SF, bool Q8, class QH, class QF>
static cudaError_t launch_mega(const CUtensorMap &map_kv, const MegaArgs &a, int grid, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kGemvThreads);
    cfg.dynamicSmemBytes = kMegaSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // every CTA resident: they wait for one another's words
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, decode_step_kernel<D, SH, SF, Q8, QH, QF>, map_kv, a);
}

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

static MegaLaunch mega_launcher(const Plan &p) {
    if (p.qdim != p.H || p.nkv > 64 || p.num_sms > kMegaMaxCtas) return nullptr;
    // every layer's tensors must sit at one fixed stride
    if (p.L > 1) {
        const size_t st = p.layer[1].wqkv - p.layer[0].wqkv;
        for (int l = 0; l < p.L; ++l) {
            const LayerOffsets &a = p.layer[l], &b = p.layer[0];
            const size_t o = st * (size_t)l;
            if (a.attn_norm != b.attn_norm + o || a.wqkv != b.wqkv + o || a.wo != b.wo + o ||
                a.ffn_norm != b.ffn_norm + o || a.wgu != b.wgu + o || a.wd != b.wd + o ||
                (p.cfg.qkv_bias && a.bqkv != b.bqkv + o) || (p.qk_norm && (a.qn != b.qn + o || a.kn != b.kn + o)))
                return nullptr;
        }
    }
#define WICI_MEGA_PICK(DD, SH, SF, Q8, QH, QF)                                                       \
    if (p.q8 == Q8 && p.d == DD && shape_is<SH>(p.H) && shape_is<SF>(p.F) &&                            \
        (!Q8 || (q8_shape_is<QH>(p.H) && q8_shape_is<QF>(p.F))))                                        \
        return launch_mega<DD, SH, SF, Q8, QH, QF>;
    WICI_MEGA_SHAPES(WICI_MEGA_PICK)
#undef WICI_MEGA_PICK
    return nullptr;
}

bool decode_is_persistent(const Plan &p) { return mega_launcher(p) != nullptr; }

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
    const int grid = p.num_sms;
    a.splits = grid / p.nkv < kFdMaxSplits ? grid / p.nkv : kFdMaxSplits;
    a.bias = p.cfg.qkv_bias;
    a.qk_norm = p.qk_norm;
    a.eps = p.cfg.rms_eps;
    a.qscale = 1.4426950408889634f / sqrtf((float)p.d);
    return fn(map_kv, a, grid, st);
}

cudaError_t enqueue_decode_step(const Plan &p, const Bufs &b, const CUtensorMap &map_kv, cudaStream_t st, bool pdl,
                                LaunchHook *hook) {
    if (MegaLaunch fn = mega_launcher(p)) {
        if (hook) hook->before("decode_step");
        cudaError_t e = enqueue_mega(p, b, map_kv, st, fn);
        if (hook) hook->after("decode_step");
        return e;
    }
    cudaError_t e;
    const float qscale = 1.4426950408889634f / sqrtf((float)p.d);
    for (int l = 0; l < p.L; ++l) {
        const LayerOffsets &lo = p.layer[l];
        uint16_t *kvl = b.KV + (size_t)l * p.kv_layer_elems;
        // A3 + A4: RMSNorm, QKV, RoPE, KV append (layer 0 also gathers the embedding, A2)
        GemvIn g = gemv_in(p, b, b.W + lo.wqkv, p.H, p.nqkv / 2, 2, b.x, b.W + lo.attn_norm);
        if (l == 0) {
            g.embed = b.W + p.w_embed;
            g.x_out = b.x;
        }
        set_next(p, b, g, l, G_QKV);
        EpiQKV eq = {};
        eq.q = b.q;
        eq.kv = kvl;
        eq.pages = b.pages;
        eq.rope = b.rope;
        eq.ctrl = b.ctrl;
        eq.bias = p.cfg.qkv_bias ? b.W + lo.bqkv : nullptr;
        eq.qdim = p.qdim;
        eq.kvdim = p.kvdim;
        eq.d = p.d;
        eq.nkv = p.nkv;
        eq.page_elems = p.kv_page_elems;
        if ((e = launch_gemv(p, g, eq, st, pdl && l > 0, hook, "qkv_rope_kvappend")) != cudaSuccess) return e;
        // A5: attention
        FDArgs fa = {b.q, kvl, b.pages, b.ctrl, b.o, b.fd_part, p.nkv, p.group, fd_wph(p.group), p.kv_page_elems,
                     qscale};
        if (hook) hook->before("flash_decode");
        if (p.d == 128)
            e = launch_fd<128>(p, fa, st, pdl);
        else
            e = launch_fd<64>(p, fa, st, pdl);
        if (hook) hook->after("flash_decode");
        if (e != cudaSuccess) return e;
        // A6: O projection + residual
        g = gemv_in(p, b, b.W + lo.wo, p.qdim, p.H, 1, b.o, nullptr);
        set_next(p, b, g, l, G_O);
        if ((e = launch_gemv(p, g, EpiResidual{b.x}, st, pdl, hook, "o_proj_residual")) != cudaSuccess)
            return e;
        // A7: RMSNorm + gate/up + SwiGLU
        g = gemv_in(p, b, b.W + lo.wgu, p.H, p.F, 2, b.x, b.W + lo.ffn_norm);
        set_next(p, b, g, l, G_GU);
        if ((e = launch_gemv(p, g, EpiSwiGLU{b.m}, st, pdl, hook, "gate_up_swiglu")) != cudaSuccess)
            return e;
        // A8: down projection + residual
        g = gemv_in(p, b, b.W + lo.wd, p.F, p.H, 1, b.m, nullptr);
        set_next(p, b, g, l, G_DOWN);
        if ((e = launch_gemv(p, g, EpiResidual{b.x}, st, pdl, hook, "down_residual")) != cudaSuccess)
            return e;
    }
    // A9: final norm + LM head + greedy argmax; advances the position by one
    return enqueue_lm_head(p, b, b.x, st, pdl, 1, hook);
}

cudaError_t enqueue_bounded_wait_probe(int *err, int64_t limit_ns, cudaStream_t st) {
    bounded_wait_probe_kernel<<<1, 32, 0, st>>>(err, (long long)limit_ns);
    return cudaGetLastError();
}

}  // namespace wici
