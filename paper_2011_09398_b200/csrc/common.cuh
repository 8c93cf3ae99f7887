// Shared host-side helpers of the library: geometry of an LceBConv2d call and launch checks.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "lce.h"

namespace lce {

// TensorFlow VALID / SAME extents (paper Section 3.2: LCE extends TFLite, "same" padding).
struct Axis {
    int32_t out;         // output extent
    int32_t pad_before;  // padding in front of element 0
};

inline Axis axis_geometry(int32_t in, int32_t k, int32_t stride, int32_t padding)
{
    Axis a{0, 0};
    if (padding == LCE_PAD_VALID) {
        a.out = in >= k ? (in - k) / stride + 1 : 0;
        return a;
    }
    a.out = (in + stride - 1) / stride;
    int32_t total = (a.out - 1) * stride + k - in;
    if (total < 0) total = 0;
    a.pad_before = total / 2;
    return a;
}

struct ConvGeom {
    int32_t N, H, W, Cin, Cw, Cout, Cow, KH, KW, sh, sw, OH, OW, pt, pl;
    int32_t padding, out_type, activation;
    int64_t M;  // N*OH*OW output pixels
};

// Output extents under a padding mode.  The index arithmetic of the kernels is 32-bit on words: every tensor stays below
// 2^31 words.
inline lce_status set_padding(ConvGeom *g, int32_t padding)
{
    const Axis ah = axis_geometry(g->H, g->KH, g->sh, padding), aw = axis_geometry(g->W, g->KW, g->sw, padding);
    if (ah.out <= 0 || aw.out <= 0) return LCE_ERR_INVALID_ARG;
    g->padding = padding;
    g->OH = ah.out; g->OW = aw.out; g->pt = ah.pad_before; g->pl = aw.pad_before;
    g->M = (int64_t)g->N * g->OH * g->OW;
    const int64_t in_words = (int64_t)g->N * g->H * g->W * g->Cw;
    const int64_t out_elems = g->M * g->Cout;
    const int64_t w_words = (int64_t)g->Cout * g->KH * g->KW * g->Cw;
    return in_words >= (1ll << 31) || out_elems >= (1ll << 31) || w_words >= (1ll << 31) ? LCE_ERR_UNSUPPORTED : LCE_OK;
}

// Whether `covers` holds for the geometry under one padding mode at least.  Packed weights serve every padding mode, so
// which parts their buffer has must not depend on the mode they are packed under: a part is there for all modes if its
// kernel covers any of them (the kernels' limits on shared memory and taps differ between the modes).
template <typename Covers>
bool covers_some_padding(const ConvGeom &g, Covers covers)
{
    for (const int32_t padding : {LCE_PAD_VALID, LCE_PAD_SAME_ONE, LCE_PAD_SAME_ZERO}) {
        ConvGeom t = g;
        if (set_padding(&t, padding) == LCE_OK && covers(t)) return true;
    }
    return false;
}

inline lce_status make_geom(const lce_bconv2d_desc *d, ConvGeom *g)
{
    if (!d) return LCE_ERR_INVALID_ARG;
    if (d->batch <= 0 || d->in_h <= 0 || d->in_w <= 0 || d->in_c <= 0 || d->out_c <= 0 ||
        d->kernel_h <= 0 || d->kernel_w <= 0 || d->stride_h <= 0 || d->stride_w <= 0)
        return LCE_ERR_INVALID_ARG;
    if (d->padding < LCE_PAD_VALID || d->padding > LCE_PAD_SAME_ZERO) return LCE_ERR_INVALID_ARG;
    if (d->out_type < LCE_OUT_FLOAT32 || d->out_type > LCE_OUT_INT32) return LCE_ERR_INVALID_ARG;
    if (d->activation < LCE_ACT_NONE || d->activation > LCE_ACT_RELU) return LCE_ERR_INVALID_ARG;
    if (d->kernel < LCE_KERNEL_AUTO || d->kernel > LCE_KERNEL_TENSOR) return LCE_ERR_INVALID_ARG;
    if (d->weights_packed != 0 && d->weights_packed != 1) return LCE_ERR_INVALID_ARG;
    g->N = d->batch; g->H = d->in_h; g->W = d->in_w; g->Cin = d->in_c; g->Cw = (d->in_c + 31) / 32;
    g->Cout = d->out_c; g->Cow = (d->out_c + 31) / 32;
    g->KH = d->kernel_h; g->KW = d->kernel_w; g->sh = d->stride_h; g->sw = d->stride_w;
    g->out_type = d->out_type; g->activation = d->activation;
    return set_padding(g, d->padding);
}

inline bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

// floor(n / d) = (n * mul) >> sh for every 0 <= n < 2^31: sh = 31 + ceil(log2 d), mul = floor(2^sh / d) + 1
// (the excess mul * d - 2^sh is at most d <= 2^(sh - 31), so n * excess < 2^sh)
inline void fast_div_constants(uint32_t d, uint32_t *mul, uint32_t *sh)
{
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    *sh = 31 + l;
    *mul = (uint32_t)(((1ull << (31 + l)) / d) + 1);
}

inline lce_status launch_status()
{
    return cudaGetLastError() == cudaSuccess ? LCE_OK : LCE_ERR_CUDA;
}

// The opt-in to more than 48 KB of dynamic shared memory is a driver call; it is made once per kernel,
// device and size (a larger request later raises it), not on every launch.  One instance per kernel.
struct SmemOptIn {
    static constexpr int kDevices = 64;
    std::atomic<size_t> granted[kDevices];
    SmemOptIn() { for (auto &g : granted) g.store(0, std::memory_order_relaxed); }
    template <typename Kernel>
    bool ensure(Kernel kernel, size_t smem_bytes)
    {
        if (smem_bytes <= 48 * 1024) return true;
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess) return false;
        const bool tracked = dev >= 0 && dev < kDevices;
        if (tracked && granted[dev].load(std::memory_order_acquire) >= smem_bytes) return true;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes) != cudaSuccess) return false;
        if (tracked) {  // concurrent callers may both set the attribute; the recorded size only grows
            size_t seen = granted[dev].load(std::memory_order_relaxed);
            while (seen < smem_bytes && !granted[dev].compare_exchange_weak(seen, smem_bytes, std::memory_order_release)) {}
        }
        return true;
    }
};

// Launches a kernel with programmatic stream serialization: its CTAs may be scheduled while the previous kernel
// of the stream drains (if that kernel lets its dependents start early), and wait for its completion themselves
// (griddepcontrol.wait) before they touch anything it may have written or may still read.  Also the cheaper launch
// for the host (2.4 us against 2.9 us measured).
template <typename... Params, typename... Args>
lce_status launch_dependent(void (*kernel)(Params...), dim3 grid, int threads, size_t smem_bytes, cudaStream_t s, const Args &...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...) != cudaSuccess) {
        cudaGetLastError();
        return LCE_ERR_CUDA;
    }
    return LCE_OK;
}

// A launch worked out ahead of time for a geometry: everything but the buffers (filled in by the prepare functions,
// read by the launch functions of the same kernel).
struct PreparedLaunch {
    alignas(16) unsigned char bytes[1536];
};

// Kernel entry points implemented in the other translation units.
lce_status launch_bconv_direct(const ConvGeom &g, const uint32_t *in, const uint32_t *w, const float *mult,
                               const float *bias, const int32_t *thr, void *out, cudaStream_t s);
// Returns LCE_ERR_UNSUPPORTED without launching when the tiled kernel does not cover the shape.
// w_image: the tiled part of a packed-weights buffer, or nullptr to derive operands from `w`.
// residual / out_packed: fused shortcut add and fused LceQuantize of a float output (both optional;
// with out_packed given, `out` may be null).
lce_status launch_bconv_tiled(const ConvGeom &g, const uint32_t *in, const uint32_t *w, const uint32_t *w_image,
                              const float *mult, const float *bias, const int32_t *thr, void *out, cudaStream_t s,
                              const float *residual = nullptr, uint32_t *out_packed = nullptr,
                              const float *in_f32 = nullptr);
// One-word-patch kernel for tiny channel counts (KH*KW*Cin <= 32); plain words, `packed` when they are the first part
// of a packed-weights buffer.
bool patch_covers(const ConvGeom &g);
lce_status launch_bconv_patch(const ConvGeom &g, const uint32_t *in, const uint32_t *w, bool packed, const float *mult,
                              const float *bias, const int32_t *thr, void *out, cudaStream_t s);
// Latency kernel for small layers (any filter, stride and channel count whose tile fits in shared memory).
// w_image: the part of a packed-weights buffer launch_pack_weights_small wrote, or null to use the plain words.
// residual / out_packed as for the tiled kernel.
struct TiledPlanInfo;
bool small_covers(const ConvGeom &g);
int64_t small_ctas(const ConvGeom &g);
void small_plan_info(const ConvGeom &g, TiledPlanInfo *info);
size_t small_weight_image_bytes(const ConvGeom &g);
lce_status launch_pack_weights_small(const ConvGeom &g, const uint32_t *w, uint32_t *plain, uint32_t *image, cudaStream_t s);  // plain: a copy of w
lce_status prepare_bconv_small(const ConvGeom &g, PreparedLaunch *prepared);
lce_status launch_bconv_small(const PreparedLaunch &prepared, const uint32_t *in, const uint32_t *w, const uint32_t *w_image, const float *mult,
                              const float *bias, const int32_t *thr, void *out, cudaStream_t s,
                              const float *residual = nullptr, uint32_t *out_packed = nullptr);
// Tensor-core kernel (tcgen05 kind::mxf4 on e2m1 operands): any filter of up to 64 taps, equal strides
// of 1 or 2, every padding mode; needs the weight image that launch_pack_weights_tensor writes at load
// time (w_image; null -> LCE_ERR_UNSUPPORTED).  residual / out_packed as for the tiled kernel (float
// output, out_c a multiple of 32).
bool tensor_covers(const ConvGeom &g);
size_t tensor_weight_image_bytes(const ConvGeom &g);
lce_status launch_pack_weights_tensor(const ConvGeom &g, const uint32_t *w, void *image, cudaStream_t s);
lce_status prepare_bconv_tensor(const ConvGeom &g, bool fused, PreparedLaunch *prepared);
lce_status launch_bconv_tensor(const PreparedLaunch &prepared, const uint32_t *in, const void *w_image, const float *mult,
                               const float *bias, const int32_t *thr, void *out, cudaStream_t s,
                               const float *residual = nullptr, uint32_t *out_packed = nullptr);
struct TensorPlanInfo {
    int32_t tile_positions, ctas, weight_stages, weights_resident, phases;
    int64_t shared_bytes;
    double clocks;  // of a CTA's share, by the cost model of the plan
};
lce_status tensor_plan_info(const ConvGeom &g, TensorPlanInfo *info);
// Bounded device-side waits: status word, its reset, the host-visible flag (no synchronisation), and a
// tiny kernel whose wait is meant to run out (nobody arrives at its barrier).
lce_status tensor_device_status(int *status);
lce_status tensor_device_status_reset();
bool tensor_timeout_flagged();
lce_status tensor_wait_probe(uint64_t limit_ns, cudaStream_t s);
// Copies between pinned host memory and the device in one kernel; arrays on 4 bytes, sizes multiples of 4 below 2^31 in
// all, empty ones allowed.  pinned_host_view: where a kernel may access a host array (`write`: store to it), null
// where the array is the copy engine's (host_view.cuh).
constexpr int kHostCopies = 5;
struct HostCopy {
    const void *src;
    void *dst;
    size_t bytes;
};
void *pinned_host_view(const void *host, size_t bytes, bool write);
lce_status launch_host_copies(const HostCopy (&copies)[kHostCopies], cudaStream_t s);
// Bytes of the tiled kernel's weight image for this geometry (0 if the kernel does not cover it).
// Launch plan of the tiled kernels for a geometry (no buffers involved), for lce_bconv2d_plan.
struct TiledPlanInfo {
    int32_t pointwise, warps_per_cta, pixels_per_thread, tile_pixels, ctas, ctas_half_block, pixels_per_cta,
        pixels_per_cta_half_block;
    int64_t shared_bytes;
};
lce_status tiled_plan_info(const ConvGeom &g, TiledPlanInfo *info);
size_t tiled_weight_image_bytes(const ConvGeom &g);
lce_status launch_pack_weights_tiled(const ConvGeom &g, const uint32_t *w, uint32_t *image, cudaStream_t s);

}  // namespace lce
