// Weight-streaming GEMV: one launch over a matrix, with a fused RMSNorm prologue and
// the argmax epilogue of the LM head (after a prefill, and for callers that cannot
// allocate), and the helpers it shares with the persistent decode step.
//
// HBM-bound: every weight byte is read once (arithmetic intensity ~1 FLOP/byte).  A
// producer warp streams each CTA's rows through a ring in shared memory with 1-D TMA
// bulk copies (completion on mbarriers); eight consumer warps do the dot products with
// the input vector held in registers.  The producer starts before griddepcontrol.wait,
// so under programmatic dependent launch the first weights stream in while the
// predecessor finishes.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace wici {

// wait-site ids recorded in ctrl[CTRL_ERR]
enum : int { SITE_GEMV_EMPTY = 11, SITE_GEMV_FULL = 12, SITE_GEMV_DRAIN = 13 };

struct GemvIn {
    const uint16_t *W;      // rows of this matrix, [n_units][K]
    int K, n_units;
    int stages;             // ring slots (<= kGemvMaxStages)
    uint32_t slot_bytes;    // bytes per ring slot (>= gemv_rps(K) * K * 2, multiple of 128)
    const float *in;        // input vector (x when gain != nullptr)
    const uint16_t *gain;   // RMSNorm gain (bf16) or nullptr for a plain input
    int *ctrl;
    float eps;
    // the GEMV launched after this one: the producer moves the first rows of
    // this CTA's share of it into L2 once its own rows are issued
    const uint16_t *next_W;  // nullptr: none
    int next_K, next_n_units, next_rpu;
};

// ---------------------------------------------------------------- epilogues --
struct EpiArgmax {    // logits[u] = v; greedy argmax (lowest index on ties) across the grid
    float *logits;
    int2 *partial;
    int *ctrl;
    int *hist;
    int pos_add;
    float best;
    int bidx;
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

// ------------------------------------------------------------ GEMV shapes ----
// (NCH, RPS, FULL): every slot holds RPS rows (a power of two, at most 8, RPS x K x 2 <=
// 32 KB); consumer thread t covers the 8-element chunks c = t + 256 j, j < NCH; FULL when
// the chunks cover K exactly (no tail check in the inner loop).
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
__device__ inline bool lm_argmax(const EpiArgmax &e, float *s_bv, int *s_bi, int *s_last) {
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
// Grid: num_sms CTAs, each owning a contiguous, balanced range of rows.  The producer warp
// streams them, RPS per slot, through the ring; each consumer thread adds its chunks of
// every row of a slot, each warp sums the slot's RPS rows with interleaved butterflies, and
// the warp sums go to shared memory, where they are reduced over the 8 warps (fixed order)
// once per batch of up to kRedRows rows and passed to the epilogue.
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
    const int total_rows = u1 - u0;
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
            const uint16_t *src = g.W + (size_t)u0 * g.K;
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
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int c = tid + kGemvConsumers * j;
        if (FULL || c < nchunks) {
            const float4 a = *reinterpret_cast<const float4 *>(g.in + c * 8);
            const float4 b = *reinterpret_cast<const float4 *>(g.in + c * 8 + 4);
            h[j][0] = a.x; h[j][1] = a.y; h[j][2] = a.z; h[j][3] = a.w;
            h[j][4] = b.x; h[j][5] = b.y; h[j][6] = b.z; h[j][7] = b.w;
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
            for (int t = tid; t < brow; t += kGemvConsumers) {
                float v = 0.f;
#pragma unroll
                for (int w = 0; w < kGemvWarps; ++w) v += red[(size_t)(buf * kGemvWarps + w) * kRedRows + t];
                epi.unit(u0 + bunit0 + t, &v);
            }
            bunit0 += brow;
            brow = 0;
            buf ^= 1;
        }
    }

    lm_argmax(epi, s_bv, s_bi, &s_last);
}

}  // namespace wici
