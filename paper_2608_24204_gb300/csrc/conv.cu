// C ABI of the CNN-training sample's convolution layer (include/wici.h):
// tensor maps, tile counts and launches of conv_tc_kernel.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdarg.h>
#include <stdio.h>

#include "../../include/wici.h"
#include "conv2_tc.cuh"
#include "conv_plan.h"
#include "conv_tc.cuh"
#include "device_table.h"
#include "kernels.h"

using namespace wici;

namespace {

constexpr size_t kConvErrBytes = 256;   // the error word, then the transposed filter

int fail(int code, const char *fmt, ...) {
    char buf[256];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    set_thread_error(buf);
    return code;
}

const char *check_shape(const wici_conv_shape *s) {
    if (!s) return "null shape";
    if (s->n < 1 || s->c < 1 || s->k < 1 || s->h < 2 || s->w < 2) return "non-positive dimension";
    if (s->c % CV_BN || s->k % CV_BN) return "c and k must be multiples of 256";
    if (s->h % 2 || s->w % 2) return "h and w must be even";
    return nullptr;
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

DeviceTable<ConvDevice> g_devices;

template <int MODE>
cudaError_t setup_mode() {
    cudaError_t e = cudaSuccess;
    for (const void *f : {(const void *)conv_tc_kernel<MODE, 1>, (const void *)conv_tc_kernel<MODE, 2>,
                          (const void *)conv_tc_kernel<MODE, 4>, (const void *)conv_tc_kernel<MODE, 8>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CV_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(conv2_tc_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CV2_SMEM);
    return e;
}

template <int SPLIT>
cudaError_t count_clusters(int nsm, int *n) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SPLIT * nsm);
    cfg.blockDim = dim3(CV_THREADS);
    cfg.dynamicSmemBytes = CV_SMEM;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = SPLIT;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(n, conv_tc_kernel<CONV_FWD, SPLIT>, &cfg);
}

// the current device's counts, with the kernels' shared-memory limits set there
cudaError_t setup(ConvDevice *out) {
    int dev = 0;
    if (const cudaError_t e = cudaGetDevice(&dev)) return e;
    return g_devices.get(dev, out, [dev](ConvDevice *d) {
        cudaError_t e;
        if ((e = cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = setup_mode<CONV_FWD>()) != cudaSuccess || (e = setup_mode<CONV_DGRAD>()) != cudaSuccess ||
            (e = setup_mode<CONV_WGRAD>()) != cudaSuccess)
            return e;
        d->clusters[0] = d->sms;
        if ((e = count_clusters<2>(d->sms, &d->clusters[1])) != cudaSuccess ||
            (e = count_clusters<4>(d->sms, &d->clusters[2])) != cudaSuccess ||
            (e = count_clusters<8>(d->sms, &d->clusters[3])) != cudaSuccess)
            return e;
        return cudaSuccess;
    });
}

ConvArgs make_args(const wici_conv_shape *s, float *out, void *ws) {
    ConvArgs a = {};
    a.n = s->n; a.c = s->c; a.h = s->h; a.w = s->w; a.k = s->k;
    a.p = s->h / 2; a.q = s->w / 2;
    a.pt = (a.p + 7) / 8;
    a.qt = (a.q + 15) / 16;
    a.out = out;
    a.wide = ((uintptr_t)out & 31u) == 0;
    a.err = (int *)ws;
    return a;
}

// x [n][h][w][c] with element strides 2 in w and h: boxes of 64 c x `wbox` w x `hbox` h
bool map_x_strided(CUtensorMap *m, const void *x, const wici_conv_shape *s, int wbox, int hbox) {
    const uint64_t dims[4] = {(uint64_t)s->c, (uint64_t)s->w, (uint64_t)s->h, (uint64_t)s->n};
    const uint64_t st[3] = {(uint64_t)s->c * 2, (uint64_t)s->w * s->c * 2, (uint64_t)s->h * s->w * s->c * 2};
    const uint32_t box[4] = {64, (uint32_t)wbox, (uint32_t)hbox, 1};
    const uint32_t es[4] = {1, 2, 2, 1};
    return encode_tiled(m, 4, x, dims, st, box, es);
}

// dy [n][p][q][k]: boxes of 64 k x 16 q x `pbox` p
bool map_dy(CUtensorMap *m, const void *dy, const wici_conv_shape *s, int pbox) {
    const int p = s->h / 2, q = s->w / 2;
    const uint64_t dims[4] = {(uint64_t)s->k, (uint64_t)q, (uint64_t)p, (uint64_t)s->n};
    const uint64_t st[3] = {(uint64_t)s->k * 2, (uint64_t)q * s->k * 2, (uint64_t)p * q * s->k * 2};
    const uint32_t box[4] = {64, 16, (uint32_t)pbox, 1};
    const uint32_t es[4] = {1, 1, 1, 1};
    return encode_tiled(m, 4, dy, dims, st, box, es);
}

// a row-major bf16 matrix [rows][cols]: boxes of 64 columns x `box_rows` rows
bool map_rows(CUtensorMap *m, const void *ptr, uint64_t rows, uint64_t cols, int box_rows) {
    const uint64_t dims[2] = {cols, rows};
    const uint64_t st[1] = {cols * 2};
    const uint32_t box[2] = {64, (uint32_t)box_rows};
    const uint32_t es[2] = {1, 1};
    return encode_tiled(m, 2, ptr, dims, st, box, es);
}

template <int MODE, int SPLIT>
cudaError_t launch_split(const ConvDevice &d, const CUtensorMap &ma, const CUtensorMap &mb, const ConvArgs &a,
                         cudaStream_t st) {
    // one tile per cluster where tiles are shared, otherwise persistent
    const int grid = SPLIT > 1 ? a.ntiles * SPLIT : a.ntiles < d.sms ? a.ntiles : d.sms;
    return launch_kernel(conv_tc_kernel<MODE, SPLIT>, dim3(grid), CV_THREADS, CV_SMEM, st, SPLIT, true, ma, mb, a);
}

// ctas: pick_ctas; mb: boxes of 128 rows for pairs, of 256 otherwise (the same for the filter gradient)
template <int MODE>
cudaError_t launch(const ConvDevice &d, int ctas, const CUtensorMap &ma, const CUtensorMap &mb, ConvArgs a, int tiles,
                   cudaStream_t st) {
    a.ntiles = ctas == 0 ? cv_pair_tiles<MODE>(a) : tiles;
    switch (ctas) {
        case 0: {
            const int grid = 2 * (a.ntiles < d.clusters[1] ? a.ntiles : d.clusters[1]);
            // __cluster_dims__ gives the pairs
            return launch_kernel(conv2_tc_kernel<MODE>, dim3(grid), CV_THREADS, CV2_SMEM, st, 1, true, ma, mb, a);
        }
        case 1: return launch_split<MODE, 1>(d, ma, mb, a, st);
        case 2: return launch_split<MODE, 2>(d, ma, mb, a, st);
        case 4: return launch_split<MODE, 4>(d, ma, mb, a, st);
        default: return launch_split<MODE, 8>(d, ma, mb, a, st);
    }
}

constexpr int kPick = -1;   // CTAs per tile: pick_ctas of the call's shape

// the CTAs per tile of a call, or a negative number when the device has none resident that way
int ctas_of(const ConvDevice &d, int ctas, int tiles, int pair_tiles, int nkb) {
    if (ctas == kPick) return pick_ctas(d, tiles, pair_tiles, nkb);
    switch (ctas) {
        case 0: case 2: return d.clusters[1] > 0 ? ctas : kPick;
        case 1: return ctas;
        case 4: return d.clusters[2] > 0 ? ctas : kPick;
        case 8: return d.clusters[3] > 0 ? ctas : kPick;
        default: return kPick;
    }
}

int forward(cudaStream_t st, const wici_conv_shape *s, const void *x, const void *w, float *y, void *workspace,
            int ctas) {
    if (const char *m = check_shape(s)) return fail(WICI_E_ARG, "conv: %s", m);
    if (!aligned16(x) || !aligned16(w) || !aligned16(y) || !aligned16(workspace) || !workspace)
        return fail(WICI_E_ARG, "conv: null or unaligned buffer");
    ConvDevice dev;
    cudaError_t e = setup(&dev);
    if (e != cudaSuccess) return fail(WICI_E_CUDA, "conv: %s", cudaGetErrorString(e));
    CUtensorMap ma, mb;
    const ConvArgs a = make_args(s, y, workspace);
    const int tiles = a.n * a.pt * a.qt * (a.k / CV_BN);
    ctas = ctas_of(dev, ctas, tiles, cv_pair_tiles<CONV_FWD>(a), 9 * (a.c / CV_BK));
    if (ctas < 0) return fail(WICI_E_ARG, "conv: CTAs per tile");
    if (!map_x_strided(&ma, x, s, 32, 16) ||
        !map_rows(&mb, w, (uint64_t)s->k, (uint64_t)9 * s->c, ctas == 0 ? CV_BN / 2 : CV_BN))
        return fail(WICI_E_CUDA, "conv: cuTensorMapEncodeTiled failed");
    if ((e = launch<CONV_FWD>(dev, ctas, ma, mb, a, tiles, st)) != cudaSuccess)
        return fail(WICI_E_CUDA, "conv forward: %s", cudaGetErrorString(e));
    return WICI_OK;
}

int backward_data(cudaStream_t st, const wici_conv_shape *s, const void *dy, const void *w, float *dx, void *workspace,
                  int ctas) {
    if (const char *m = check_shape(s)) return fail(WICI_E_ARG, "conv: %s", m);
    if (!aligned16(dy) || !aligned16(w) || !aligned16(dx) || !aligned16(workspace) || !workspace)
        return fail(WICI_E_ARG, "conv: null or unaligned buffer");
    ConvDevice dev;
    cudaError_t e = setup(&dev);
    if (e != cudaSuccess) return fail(WICI_E_CUDA, "conv: %s", cudaGetErrorString(e));
    const ConvArgs a = make_args(s, dx, workspace);
    const int tiles = 4 * a.n * a.pt * a.qt * (a.c / CV_BN);
    ctas = ctas_of(dev, ctas, tiles, cv_pair_tiles<CONV_DGRAD>(a), 4 * (a.k / CV_BK));
    if (ctas < 0) return fail(WICI_E_ARG, "conv: CTAs per tile");
    uint16_t *wt = (uint16_t *)((uint8_t *)workspace + kConvErrBytes);
    if ((e = launch_kernel(conv_transpose_filter_kernel, dim3((s->c + 31) / 32, (s->k + 31) / 32, 9), 256, 0, st, 1,
                           true, (const uint16_t *)w, wt, s->k, s->c)) != cudaSuccess)
        return fail(WICI_E_CUDA, "conv transpose: %s", cudaGetErrorString(e));
    CUtensorMap ma, mb;
    if (!map_dy(&ma, dy, s, 8) ||
        !map_rows(&mb, wt, (uint64_t)9 * s->c, (uint64_t)s->k, ctas == 0 ? CV_BN / 2 : CV_BN))
        return fail(WICI_E_CUDA, "conv: cuTensorMapEncodeTiled failed");
    if ((e = launch<CONV_DGRAD>(dev, ctas, ma, mb, a, tiles, st)) != cudaSuccess)
        return fail(WICI_E_CUDA, "conv data gradient: %s", cudaGetErrorString(e));
    return WICI_OK;
}

int backward_filter(cudaStream_t st, const wici_conv_shape *s, const void *x, const void *dy, float *dw,
                    void *workspace, int ctas) {
    if (const char *m = check_shape(s)) return fail(WICI_E_ARG, "conv: %s", m);
    if (!aligned16(x) || !aligned16(dy) || !aligned16(dw) || !aligned16(workspace) || !workspace)
        return fail(WICI_E_ARG, "conv: null or unaligned buffer");
    ConvDevice dev;
    cudaError_t e = setup(&dev);
    if (e != cudaSuccess) return fail(WICI_E_CUDA, "conv: %s", cudaGetErrorString(e));
    CUtensorMap ma, mb;
    if (!map_dy(&ma, dy, s, 4) || !map_x_strided(&mb, x, s, 32, 8))
        return fail(WICI_E_CUDA, "conv: cuTensorMapEncodeTiled failed");
    const ConvArgs a = make_args(s, dw, workspace);
    const int tiles = 9 * (a.k / CV_BM) * (a.c / CV_BN);
    ctas = ctas_of(dev, ctas, tiles, cv_pair_tiles<CONV_WGRAD>(a), a.n * ((a.p + 3) / 4) * a.qt);
    if (ctas < 0) return fail(WICI_E_ARG, "conv: CTAs per tile");
    if ((e = launch<CONV_WGRAD>(dev, ctas, ma, mb, a, tiles, st)) != cudaSuccess)
        return fail(WICI_E_CUDA, "conv filter gradient: %s", cudaGetErrorString(e));
    return WICI_OK;
}

}  // namespace

extern "C" {

int wici_conv_workspace_bytes(const wici_conv_shape *s, size_t *bytes) {
    if (const char *m = check_shape(s)) return fail(WICI_E_ARG, "conv: %s", m);
    if (!bytes) return fail(WICI_E_ARG, "conv: null output");
    *bytes = kConvErrBytes + (size_t)9 * s->c * s->k * 2;
    return WICI_OK;
}

int wici_conv_forward(void *cuda_stream, const wici_conv_shape *s, const void *x, const void *w, float *y,
                      void *workspace) {
    return forward((cudaStream_t)cuda_stream, s, x, w, y, workspace, kPick);
}

int wici_conv_backward_data(void *cuda_stream, const wici_conv_shape *s, const void *dy, const void *w, float *dx,
                            void *workspace) {
    return backward_data((cudaStream_t)cuda_stream, s, dy, w, dx, workspace, kPick);
}

int wici_conv_backward_filter(void *cuda_stream, const wici_conv_shape *s, const void *x, const void *dy, float *dw,
                              void *workspace) {
    return backward_filter((cudaStream_t)cuda_stream, s, x, dy, dw, workspace, kPick);
}

int wici_internal_conv(int mode, int ctas, void *cuda_stream, const wici_conv_shape *s, const void *a, const void *b,
                       float *out, void *workspace) {
    if (ctas == kPick) return fail(WICI_E_ARG, "conv: CTAs per tile");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    switch (mode) {
        case CONV_FWD: return forward(st, s, a, b, out, workspace, ctas);
        case CONV_DGRAD: return backward_data(st, s, a, b, out, workspace, ctas);
        case CONV_WGRAD: return backward_filter(st, s, a, b, out, workspace, ctas);
        default: return fail(WICI_E_ARG, "conv: mode");
    }
}

int wici_conv_status(void *cuda_stream, void *workspace) {
    if (!workspace) return fail(WICI_E_ARG, "conv: null workspace");
    int h = 0;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    cudaError_t e = cudaMemcpyAsync(&h, workspace, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(WICI_E_CUDA, "conv status: %s", cudaGetErrorString(e));
    if (h != 0) {
        cudaMemsetAsync(workspace, 0, sizeof(int), st);
        cudaStreamSynchronize(st);
        return fail(WICI_E_TIMEOUT, "conv: a device-side wait gave up (site %d)", h);
    }
    return WICI_OK;
}

}  // extern "C"
