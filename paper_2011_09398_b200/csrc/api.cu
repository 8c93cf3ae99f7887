// C ABI front: version/status strings, shape query and the LceBConv2d dispatch (device- and
// host-buffer forms).  All argument checks happen here, before anything is launched.
#include "common.cuh"

#include <string.h>

#include <atomic>
#include <memory>
#include <new>

namespace lce {
namespace {

lce_status check_conv_buffers(const ConvGeom &g, const void *input, const void *weights, const void *multiplier, const void *bias,
                              const void *thresholds, const void *output)
{
    if (!input || !weights || !output) return LCE_ERR_INVALID_ARG;
    if (g.out_type == LCE_OUT_FLOAT32 && (!multiplier || !bias)) return LCE_ERR_INVALID_ARG;
    if (g.out_type == LCE_OUT_BITPACKED) {
        if (!thresholds) return LCE_ERR_INVALID_ARG;
        if (g.activation != LCE_ACT_NONE) return LCE_ERR_INVALID_ARG;
    }
    return LCE_OK;
}

bool conv_buffers_aligned(const void *input, const void *weights, const void *multiplier, const void *bias, const void *thresholds, const void *output)
{
    return aligned(input, 4) && aligned(weights, 4) && aligned(output, 4) && aligned(multiplier, 4) && aligned(bias, 4) && aligned(thresholds, 4);
}

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

size_t plain_weight_bytes(const ConvGeom &g) { return round_up((size_t)g.Cout * g.KH * g.KW * g.Cw * 4, 256); }

// A packed-weights buffer = [plain words][operand image of the tiled XOR/POPC kernel][operand image of
// the tensor-core kernel][tile image of the latency kernel], each part rounded up to 256 bytes; a part is
// empty if its kernel covers the geometry under no padding mode (the buffer is the same under all of them).
struct WeightParts {
    size_t tiled, tensor, small, total;  // byte offsets; 0: no such part
};

WeightParts weight_parts(const ConvGeom &g)
{
    WeightParts w{};
    size_t off = plain_weight_bytes(g);
    const size_t tiled = tiled_weight_image_bytes(g), tensor = tensor_weight_image_bytes(g), small = small_weight_image_bytes(g);
    if (tiled > 0) w.tiled = off;
    off += round_up(tiled, 256);
    if (tensor > 0) w.tensor = off;
    off += round_up(tensor, 256);
    if (small > 0) w.small = off;
    w.total = off + round_up(small, 256);
    return w;
}

enum KernelPick { PICK_NONE = 0, PICK_DIRECT, PICK_PATCH, PICK_TILED, PICK_TENSOR, PICK_SMALL };

// Which kernel weights packed at load time go to: the one whose estimated time is the shorter.  The estimates (us) were
// fitted to 180 layers of 2^26 - 2^31 binary MACs, 1x1 - 5x5, 32 - 512 channels, strides 1 and 2, as the kernels were then (10%
// rms each; on 180 others of that range, as they are now, 14% and 11%): the
// latency kernel pays per output and per 128-deep step of an output, the tensor-core kernel a start-up and the clocks its
// plan predicts; staging the four phase grids of a stride-2 layer word by word grows with the square of the depth (fewer
// positions fit a tile).  Of those 180 others the slower of the two is picked in 10, by 10% on average and 26% at most.  One
// image of 14x14x64 is 1.8 on the latency kernel and 3.6 on the tensor cores; 21 images of 14x14x256, 1x1 (2^28.0), 5.7 and
// 4.0; one of 56x56x512, stride 2 (2^30.8), 9.9 and 12.5.  The XOR/POPC kernel is ahead of both in one of the 180.
// Where one of the two does not cover the layer the other competes with the integer kernels: from 2^28 (weights
// resident) or 2^29 MACs (streamed) the tensor cores are ahead, up to 2^29 and 600 CTAs the latency kernel is.
// `extra`: what the tensor-core kernel costs besides.  PICK_NONE: neither.
KernelPick pick_packed(const ConvGeom &g, bool tensor_ok, double extra = 0.0)
{
    TensorPlanInfo t{};
    tensor_ok = tensor_ok && !patch_covers(g) && tensor_plan_info(g, &t) == LCE_OK;
    const bool small_ok = small_covers(g);
    const double macs = (double)g.M * g.Cout * g.KH * g.KW * g.Cin, outs = (double)g.M * g.Cow * 32;
    if (!tensor_ok) return small_ok && macs < 536870912.0 && small_ctas(g) <= 600 ? PICK_SMALL : PICK_NONE;
    if (!small_ok) return macs >= (t.weights_resident ? 268435456.0 : 536870912.0) ? PICK_TENSOR : PICK_NONE;
    const double small_us = 2.2 + outs * (2.3e-6 + 5.6e-7 * ((g.KH * g.KW * g.Cw + 3) / 4));
    const double tensor_us = 4.0 + 3.85e-4 * t.clocks + (t.phases > 1 ? 0.017 * g.Cw * g.Cw : 0.0) + extra;
    return small_us <= tensor_us ? PICK_SMALL : PICK_TENSOR;
}

// One place decides which kernel a call gets; lce_bconv2d_plan shows the same decision.
// tiled_buffers_ok: the tiled kernels write float / int32 rows with 128-bit accesses when the channel count allows it,
// and then need 16-byte aligned buffers.
KernelPick pick_kernel(const lce_bconv2d_desc *desc, const ConvGeom &g, bool have_tensor_image, bool tiled_buffers_ok)
{
    TiledPlanInfo info{};
    switch (desc->kernel) {
        case LCE_KERNEL_DIRECT: return PICK_DIRECT;
        case LCE_KERNEL_TENSOR: return have_tensor_image && tensor_covers(g) ? PICK_TENSOR : PICK_NONE;
        case LCE_KERNEL_TILED:
            if (patch_covers(g)) return PICK_PATCH;
            return tiled_buffers_ok && tiled_plan_info(g, &info) == LCE_OK ? PICK_TILED : PICK_NONE;
        default: break;
    }
    // a stem's patch kernel beats the latency kernel at every batch (one 224x224x3 image 2.0 against 4.1 us)
    const bool stem = patch_covers(g) && g.out_type == LCE_OUT_BITPACKED && g.padding != LCE_PAD_SAME_ZERO;
    const KernelPick packed = desc->weights_packed && !stem ? pick_packed(g, have_tensor_image) : PICK_NONE;
    if (packed != PICK_NONE) return packed;
    if (patch_covers(g)) return PICK_PATCH;
    if (tiled_buffers_ok && tiled_plan_info(g, &info) == LCE_OK) return PICK_TILED;
    return PICK_DIRECT;
}

// The fused form (shortcut, re-quantised copy): the shapes the tiled kernels cover; the tensor-core kernel wants whole
// 32-channel words and 16-byte rows.
KernelPick pick_fused(const lce_bconv2d_desc *desc, const ConvGeom &g, const WeightParts &parts, bool rows_aligned)
{
    if (desc->kernel == LCE_KERNEL_DIRECT || patch_covers(g)) return PICK_NONE;
    const bool tensor_ok = desc->weights_packed && parts.tensor && tensor_covers(g) && (g.Cout & 31) == 0 && rows_aligned;
    if (desc->kernel == LCE_KERNEL_TENSOR) return tensor_ok ? PICK_TENSOR : PICK_NONE;
    if (desc->kernel != LCE_KERNEL_AUTO || !desc->weights_packed) return PICK_TILED;
    const KernelPick packed = pick_packed(g, tensor_ok);
    if (packed == PICK_SMALL && tiled_weight_image_bytes(g) == 0) return tensor_ok ? PICK_TENSOR : PICK_TILED;
    return packed == PICK_NONE ? PICK_TILED : packed;
}

// The host-buffer form brings plain weights along: the kernels that want packed ones are open to it, too, if there is
// room in the workspace to pack them (`image_fits`; the latency kernel reads plain words).  28x28x128 at batch 64: the
// XOR/POPC kernel 38 us, packing and the tensor-core kernel 10 us.
constexpr double kPackImage = 2.5;  // us: packing, behind the copies
KernelPick pick_host(const lce_bconv2d_desc *desc, const ConvGeom &g, bool image_fits)
{
    if (desc->kernel != LCE_KERNEL_AUTO) return pick_kernel(desc, g, false, true);
    const KernelPick packed = patch_covers(g) ? PICK_NONE : pick_packed(g, image_fits, kPackImage);
    return packed == PICK_NONE ? pick_kernel(desc, g, false, true) : packed;
}

// Everything about a call that follows from its descriptor: geometry, parts of the packed weights, which kernel and
// the launch worked out for it.
struct Prepared {
    lce_bconv2d_desc desc;
    int device;
    uint32_t form;      // FORM_*: what else the choice depends on
    lce_status status;
    ConvGeom g;
    WeightParts parts;
    KernelPick pick;
    PreparedLaunch launch;
};
enum { FORM_FUSED = 1, FORM_ROWS_UNALIGNED = 2, FORM_HOST = 4, FORM_NO_IMAGE = 8 };  // float / int32 rows that are not on 16 bytes (relevant for out_c % 4 == 0)

void prepare(const lce_bconv2d_desc *desc, int device, uint32_t form, Prepared *p)
{
    p->desc = *desc;
    p->device = device;
    p->form = form;
    p->status = make_geom(desc, &p->g);
    if (p->status != LCE_OK) return;
    p->parts = weight_parts(p->g);
    const bool rows_aligned = !(form & FORM_ROWS_UNALIGNED);
    p->pick = form & FORM_HOST ? pick_host(desc, p->g, !(form & FORM_NO_IMAGE)) : form & FORM_FUSED ? pick_fused(desc, p->g, p->parts, rows_aligned) : pick_kernel(desc, p->g, desc->weights_packed && p->parts.tensor, rows_aligned);
    if (p->pick == PICK_SMALL) p->status = prepare_bconv_small(p->g, &p->launch);
    if (p->pick == PICK_TENSOR) p->status = prepare_bconv_tensor(p->g, form & FORM_FUSED, &p->launch);
}

// A network repeats few descriptors: the last ones of each host thread are kept.  Working a call out costs 1 - 2 us of
// host time, against 2.4 us for the launch itself.
const Prepared &prepared_for(const lce_bconv2d_desc *desc, uint32_t form)
{
    constexpr int kSlots = 64, kWays = 4;
    struct Cache {
        Prepared slots[kSlots] = {};
        bool used[kSlots] = {};
        uint32_t turn = 0;
    };
    static thread_local std::unique_ptr<Cache> cache;
    static thread_local Prepared uncached;  // where there is no memory for the cache
    if (!cache) cache.reset(new (std::nothrow) Cache);
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) device = -1;
    if (!cache) {
        prepare(desc, device, form, &uncached);
        return uncached;
    }
    uint32_t hash = form * 2654435761u;
    int32_t fields[sizeof(lce_bconv2d_desc) / 4];
    memcpy(fields, desc, sizeof(fields));
    for (int32_t f : fields) hash = (hash ^ (uint32_t)f) * 16777619u;
    const uint32_t base = (hash >> 16) % (kSlots / kWays) * kWays;
    for (uint32_t i = base; i < base + kWays; ++i) {
        const Prepared &p = cache->slots[i];
        if (cache->used[i] && p.device == device && p.form == form && memcmp(&p.desc, desc, sizeof(*desc)) == 0) return p;
    }
    const uint32_t i = base + cache->turn++ % kWays;
    prepare(desc, device, form, &cache->slots[i]);
    cache->used[i] = true;
    return cache->slots[i];
}

uint32_t rows_form(const lce_bconv2d_desc *desc, const void *out, const void *residual)
{
    const bool wide_rows = (desc->out_c & 3) == 0 && desc->out_type != LCE_OUT_BITPACKED;
    return wide_rows && (!aligned(out, 16) || !aligned(residual, 16)) ? FORM_ROWS_UNALIGNED : 0;
}

lce_status dispatch(const Prepared &p, const uint32_t *input, const uint32_t *weights, const float *multiplier, const float *bias,
                    const int32_t *thresholds, void *output, cudaStream_t s, const float *residual = nullptr, uint32_t *out_packed = nullptr)
{
    if (tensor_timeout_flagged()) return LCE_ERR_DEVICE_TIMEOUT;  // an earlier kernel on this device gave up a wait
    const bool packed = p.desc.weights_packed != 0;
    if (packed && !aligned(weights, 256)) return LCE_ERR_ALIGNMENT;
    const auto part = [&](size_t off) { return packed && off ? reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(weights) + off) : nullptr; };
    switch (p.pick) {
        case PICK_DIRECT: return launch_bconv_direct(p.g, input, weights, multiplier, bias, thresholds, output, s);
        case PICK_PATCH: return launch_bconv_patch(p.g, input, weights, packed, multiplier, bias, thresholds, output, s);
        case PICK_TILED: return launch_bconv_tiled(p.g, input, weights, part(p.parts.tiled), multiplier, bias, thresholds, output, s, residual, out_packed);
        case PICK_TENSOR: return launch_bconv_tensor(p.launch, input, part(p.parts.tensor), multiplier, bias, thresholds, output, s, residual, out_packed);
        case PICK_SMALL: return launch_bconv_small(p.launch, input, weights, part(p.parts.small), multiplier, bias, thresholds, output, s, residual, out_packed);
        default: return LCE_ERR_UNSUPPORTED;
    }
}

struct HostLayout {
    size_t in, w, mult, bias, thr, out, total;  // total: what a call needs at least
    size_t image;                               // beyond that, room for packed weights (0: of no use to this layer)
    size_t in_bytes, w_bytes, ch_bytes, out_bytes;
};

HostLayout host_layout(const ConvGeom &g)
{
    HostLayout L{};
    L.in_bytes = (size_t)g.N * g.H * g.W * g.Cw * 4;
    L.w_bytes = (size_t)g.Cout * g.KH * g.KW * g.Cw * 4;
    L.ch_bytes = (size_t)g.Cout * 4;
    L.out_bytes = (size_t)g.M * (g.out_type == LCE_OUT_BITPACKED ? g.Cow : g.Cout) * 4;
    size_t off = 0;
    L.in = off;   off += round_up(L.in_bytes, 256);
    L.w = off;    off += round_up(L.w_bytes, 256);
    L.mult = off; off += round_up(L.ch_bytes, 256);
    L.bias = off; off += round_up(L.ch_bytes, 256);
    L.thr = off;  off += round_up(L.ch_bytes, 256);
    L.out = off;  off += round_up(L.out_bytes, 256);
    L.total = off;
    if (!patch_covers(g) && pick_packed(g, true, kPackImage) == PICK_TENSOR) L.image = round_up(tensor_weight_image_bytes(g), 256);
    return L;
}

}  // namespace
}  // namespace lce

extern "C" const char *lce_version(void) { return "lce-b200 0.1 (sm_100a)"; }

extern "C" const char *lce_status_string(lce_status status)
{
    switch (status) {
        case LCE_OK: return "ok";
        case LCE_ERR_INVALID_ARG: return "invalid argument";
        case LCE_ERR_UNSUPPORTED: return "unsupported";
        case LCE_ERR_ALIGNMENT: return "misaligned pointer";
        case LCE_ERR_CUDA: return "CUDA error";
        case LCE_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
        case LCE_ERR_WORKSPACE: return "workspace too small";
    }
    return "unknown status";
}

extern "C" lce_status lce_device_status(int32_t *status)
{
    if (!status) return LCE_ERR_INVALID_ARG;
    int v = 0;
    lce_status st = lce::tensor_device_status(&v);
    if (st != LCE_OK) return st;
    *status = v;
    return LCE_OK;
}

extern "C" lce_status lce_device_status_reset(void) { return lce::tensor_device_status_reset(); }

extern "C" lce_status lce_device_wait_probe(uint64_t limit_ns, void *stream)
{
    if (limit_ns == 0 || limit_ns > 1000000000ull) return LCE_ERR_INVALID_ARG;  // at most a second
    return lce::tensor_wait_probe(limit_ns, static_cast<cudaStream_t>(stream));
}

extern "C" lce_status lce_bconv2d_out_shape(const lce_bconv2d_desc *desc, int32_t *out_h, int32_t *out_w)
{
    lce::ConvGeom g;
    lce_status st = lce::make_geom(desc, &g);
    if (st != LCE_OK) return st;
    if (!out_h || !out_w) return LCE_ERR_INVALID_ARG;
    *out_h = g.OH;
    *out_w = g.OW;
    return LCE_OK;
}

extern "C" lce_status lce_bconv2d_plan(const lce_bconv2d_desc *desc, lce_bconv2d_plan_info *plan)
{
    using namespace lce;
    ConvGeom g;
    lce_status st = make_geom(desc, &g);
    if (st != LCE_OK) return st;
    if (!plan) return LCE_ERR_INVALID_ARG;
    *plan = lce_bconv2d_plan_info{};
    // the decision dispatch() makes, for 16-byte aligned buffers
    const bool have_tensor_image = desc->weights_packed && tensor_weight_image_bytes(g) > 0;
    TiledPlanInfo info{};
    switch (pick_kernel(desc, g, have_tensor_image, true)) {
        case PICK_DIRECT: plan->kernel = LCE_KERNEL_DIRECT; return LCE_OK;
        case PICK_PATCH: plan->kernel = LCE_KERNEL_TILED; plan->patch = 1; return LCE_OK;
        case PICK_TENSOR: {
            TensorPlanInfo t{};
            st = tensor_plan_info(g, &t);
            if (st != LCE_OK) return st;
            plan->kernel = LCE_KERNEL_TENSOR;
            plan->tile_pixels = t.tile_positions;
            plan->ctas = t.ctas;
            plan->weight_stages = t.weight_stages;
            plan->weights_resident = t.weights_resident;
            plan->shared_bytes = t.shared_bytes;
            return LCE_OK;
        }
        case PICK_TILED:
            st = tiled_plan_info(g, &info);
            if (st != LCE_OK) return st;
            break;
        case PICK_SMALL: small_plan_info(g, &info); break;
        default: return LCE_ERR_UNSUPPORTED;
    }
    plan->kernel = LCE_KERNEL_TILED;
    plan->pointwise = info.pointwise;
    plan->warps_per_cta = info.warps_per_cta;
    plan->pixels_per_thread = info.pixels_per_thread;
    plan->tile_pixels = info.tile_pixels;
    plan->ctas = info.ctas;
    plan->ctas_half_block = info.ctas_half_block;
    plan->pixels_per_cta = info.pixels_per_cta;
    plan->pixels_per_cta_half_block = info.pixels_per_cta_half_block;
    plan->shared_bytes = info.shared_bytes;
    return LCE_OK;
}

extern "C" lce_status lce_bconv2d(const lce_bconv2d_desc *desc, const uint32_t *input, const uint32_t *weights,
                                  const float *multiplier, const float *bias, const int32_t *thresholds,
                                  void *output, void *stream)
{
    using namespace lce;
    if (!desc) return LCE_ERR_INVALID_ARG;
    const Prepared &p = prepared_for(desc, rows_form(desc, output, nullptr));
    if (p.status != LCE_OK) return p.status;
    const lce_status st = check_conv_buffers(p.g, input, weights, multiplier, bias, thresholds, output);
    if (st != LCE_OK) return st;
    if (!conv_buffers_aligned(input, weights, multiplier, bias, thresholds, output)) return LCE_ERR_ALIGNMENT;
    return dispatch(p, input, weights, multiplier, bias, thresholds, output, static_cast<cudaStream_t>(stream));
}

// ---- plan objects: the checks of lce_bconv2d once, the launch many times ---------------------------
struct lce_plan {
    lce::Prepared prepared;
    const uint32_t *input, *weights;
    const float *multiplier, *bias;
    const int32_t *thresholds;
    void *output;
};

extern "C" lce_status lce_bconv2d_plan_create(const lce_bconv2d_desc *desc, const uint32_t *input, const uint32_t *weights,
                                              const float *multiplier, const float *bias, const int32_t *thresholds,
                                              void *output, lce_plan **plan)
{
    using namespace lce;
    if (!plan) return LCE_ERR_INVALID_ARG;
    *plan = nullptr;
    if (!desc) return LCE_ERR_INVALID_ARG;
    const Prepared &p = prepared_for(desc, rows_form(desc, output, nullptr));
    if (p.status != LCE_OK) return p.status;
    const lce_status st = check_conv_buffers(p.g, input, weights, multiplier, bias, thresholds, output);
    if (st != LCE_OK) return st;
    if (!conv_buffers_aligned(input, weights, multiplier, bias, thresholds, output)) return LCE_ERR_ALIGNMENT;
    // is there a kernel for this shape, these buffers and a forced kernel choice?  (A float / int32 output
    // that is only 4-byte aligned rules the tiled kernel out: AUTO then records another kernel, a
    // forced LCE_KERNEL_TILED fails here rather than at every run.)
    if (desc->weights_packed && !aligned(weights, 256)) return LCE_ERR_ALIGNMENT;
    if (p.pick == PICK_NONE) return LCE_ERR_UNSUPPORTED;
    lce_plan *h = new (std::nothrow) lce_plan;
    if (!h) return LCE_ERR_CUDA;
    h->prepared = p;
    h->input = input; h->weights = weights; h->multiplier = multiplier; h->bias = bias; h->thresholds = thresholds;
    h->output = output;
    *plan = h;
    return LCE_OK;
}

extern "C" lce_status lce_plan_run(const lce_plan *plan, void *stream)
{
    using namespace lce;
    if (!plan) return LCE_ERR_INVALID_ARG;
    int device = -1;
    // on another device than the plan was made on: its launch is worked out for that one
    const bool same = cudaGetDevice(&device) == cudaSuccess && device == plan->prepared.device;
    const Prepared &p = same ? plan->prepared : prepared_for(&plan->prepared.desc, plan->prepared.form);
    return dispatch(p, plan->input, plan->weights, plan->multiplier, plan->bias, plan->thresholds, plan->output, static_cast<cudaStream_t>(stream));
}

extern "C" void lce_plan_destroy(lce_plan *plan) { delete plan; }

extern "C" lce_status lce_bconv2d_fused(const lce_bconv2d_desc *desc, const uint32_t *input, const uint32_t *weights,
                                        const float *multiplier, const float *bias, const float *residual,
                                        float *out_float, uint32_t *out_packed, void *stream)
{
    using namespace lce;
    if (!desc) return LCE_ERR_INVALID_ARG;
    const Prepared &p = prepared_for(desc, FORM_FUSED | (aligned(out_float, 16) && aligned(residual, 16) ? 0 : FORM_ROWS_UNALIGNED));
    if (p.status != LCE_OK) return p.status;
    if (p.g.out_type != LCE_OUT_FLOAT32) return LCE_ERR_INVALID_ARG;
    if (!input || !weights || !multiplier || !bias || (!out_float && !out_packed)) return LCE_ERR_INVALID_ARG;
    if (!conv_buffers_aligned(input, weights, multiplier, bias, out_packed, out_float) || !aligned(residual, 4)) return LCE_ERR_ALIGNMENT;
    return dispatch(p, input, weights, multiplier, bias, nullptr, out_float, static_cast<cudaStream_t>(stream), residual, out_packed);
}

extern "C" lce_status lce_bconv2d_f32(const lce_bconv2d_desc *desc, const float *input, const uint32_t *weights,
                                      const float *multiplier, const float *bias, const int32_t *thresholds,
                                      void *output, void *stream)
{
    using namespace lce;
    ConvGeom g;
    lce_status st = make_geom(desc, &g);
    if (st != LCE_OK) return st;
    st = check_conv_buffers(g, input, weights, multiplier, bias, thresholds, output);
    if (st != LCE_OK) return st;
    if (!conv_buffers_aligned(input, weights, multiplier, bias, thresholds, output)) return LCE_ERR_ALIGNMENT;
    const uint32_t *image = nullptr;
    if (desc->weights_packed) {
        if (!aligned(weights, 256)) return LCE_ERR_ALIGNMENT;
        const size_t off = weight_parts(g).tiled;
        if (off) image = reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(weights) + off);
    }
    if (desc->kernel == LCE_KERNEL_DIRECT || desc->kernel == LCE_KERNEL_TENSOR) return LCE_ERR_UNSUPPORTED;
    return launch_bconv_tiled(g, nullptr, weights, image, multiplier, bias, thresholds, output,
                              static_cast<cudaStream_t>(stream), nullptr, nullptr, input);
}

extern "C" size_t lce_bconv2d_packed_weights_bytes(const lce_bconv2d_desc *desc)
{
    using namespace lce;
    if (!desc) return 0;
    const Prepared &p = prepared_for(desc, 0);
    return p.status == LCE_OK ? p.parts.total : 0;
}

extern "C" lce_status lce_bconv2d_pack_weights(const lce_bconv2d_desc *desc, const uint32_t *weights, void *packed,
                                               void *stream)
{
    using namespace lce;
    ConvGeom g;
    lce_status st = make_geom(desc, &g);
    if (st != LCE_OK) return st;
    if (!weights || !packed) return LCE_ERR_INVALID_ARG;
    if (!aligned(weights, 4) || !aligned(packed, 256)) return LCE_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t plain = (size_t)g.Cout * g.KH * g.KW * g.Cw * 4;
    const WeightParts parts = weight_parts(g);
    char *base = static_cast<char *>(packed);
    if (!parts.small && cudaMemcpyAsync(packed, weights, plain, cudaMemcpyDeviceToDevice, s) != cudaSuccess) return LCE_ERR_CUDA;
    if (parts.tiled && (st = launch_pack_weights_tiled(g, weights, reinterpret_cast<uint32_t *>(base + parts.tiled), s)) != LCE_OK) return st;
    if (parts.tensor && (st = launch_pack_weights_tensor(g, weights, base + parts.tensor, s)) != LCE_OK) return st;
    if (parts.small) return launch_pack_weights_small(g, weights, static_cast<uint32_t *>(packed), reinterpret_cast<uint32_t *>(base + parts.small), s);
    return LCE_OK;
}

extern "C" size_t lce_bconv2d_host_workspace_bytes(const lce_bconv2d_desc *desc)
{
    lce::ConvGeom g;
    if (lce::make_geom(desc, &g) != LCE_OK) return 0;
    const lce::HostLayout L = lce::host_layout(g);
    return L.total + L.image;
}

namespace lce {
namespace {
// An engine copy costs about 4 us however short, and where a kernel follows or goes before it some 8 us more; one kernel
// over pinned memory moves all the arrays of a call in about 3 us and the PCIe time (0.8 MB: 20.6 us, the engine 18.0),
// so the two draw level at some 2.5 MB.  28x28x128, 64 images, 0.8 MB in and out: 64 -> 61 us a call; 56x56x128, 8 images:
// 55 -> 43.  An output written by the convolution itself saves the copy's launch as well: one 20x20x32 image 33 -> 21 us,
// 51 KB of floats 28.4 -> 21.6, 86 KB 31.0 -> 27.6.
constexpr size_t kKernelCopy = 2048 * 1024;
// float / int32 rows leave as 128-byte lines, bit-packed words four bytes at a time (0.8 MB of them straight to the host:
// 203 us a call)
constexpr size_t kSmallRows = 256 * 1024, kSmallWords = 32 * 1024;

lce_status host_conv(const lce_bconv2d_desc *desc, const uint32_t *input, const uint32_t *weights, const float *multiplier,
                     const float *bias, const int32_t *thresholds, void *output, void *workspace, size_t workspace_bytes,
                     void *stream, bool synchronise)
{
    ConvGeom g;
    lce_status st = make_geom(desc, &g);
    if (st == LCE_OK) st = check_conv_buffers(g, input, weights, multiplier, bias, thresholds, output);
    if (st != LCE_OK) return st;
    if (!workspace || desc->weights_packed) return LCE_ERR_INVALID_ARG;
    if (!aligned(workspace, 256)) return LCE_ERR_ALIGNMENT;
    const HostLayout L = host_layout(g);
    if (workspace_bytes < L.total) return LCE_ERR_WORKSPACE;
    const Prepared &p = prepared_for(desc, FORM_HOST | (workspace_bytes < L.total + L.image ? FORM_NO_IMAGE : 0));
    if (p.status != LCE_OK) return p.status;
    if (p.pick == PICK_NONE) return LCE_ERR_UNSUPPORTED;
    if (tensor_timeout_flagged()) return LCE_ERR_DEVICE_TIMEOUT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char *ws = static_cast<char *>(workspace);
    // arrays of up to kKernelCopy bytes in pinned memory travel together in one kernel, the others (first: the rest is
    // prepared while they run) by the copy engine
    HostCopy copies[kHostCopies] = {{input, ws + L.in, L.in_bytes}, {weights, ws + L.w, L.w_bytes}, {multiplier, ws + L.mult, L.ch_bytes},
                                    {bias, ws + L.bias, L.ch_bytes}, {thresholds, ws + L.thr, L.ch_bytes}};
    for (HostCopy &c : copies) {
        if (!c.src) c.bytes = 0;
        const void *view = c.bytes > 0 && c.bytes <= kKernelCopy ? pinned_host_view(c.src, c.bytes, false) : nullptr;
        if (view) {
            c.src = view;
            continue;
        }
        if (c.bytes > 0 && cudaMemcpyAsync(c.dst, c.src, c.bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return LCE_ERR_CUDA;
        c.bytes = 0;
    }
    st = launch_host_copies(copies, s);
    if (st != LCE_OK) return st;
    // a small output in pinned memory is written there directly
    void *out_view = L.out_bytes <= (g.out_type == LCE_OUT_BITPACKED ? kSmallWords : kSmallRows) && aligned(output, 16) ? pinned_host_view(output, L.out_bytes, true) : nullptr;
    void *d_out = out_view ? out_view : ws + L.out;
    const auto at = [&](size_t off) { return reinterpret_cast<uint32_t *>(ws + off); };
    const uint32_t *d_in = at(L.in), *d_w = at(L.w);
    const float *d_mult = multiplier ? reinterpret_cast<const float *>(ws + L.mult) : nullptr, *d_bias = bias ? reinterpret_cast<const float *>(ws + L.bias) : nullptr;
    const int32_t *d_thr = thresholds ? reinterpret_cast<const int32_t *>(ws + L.thr) : nullptr;
    if (p.pick == PICK_TENSOR) {
        st = launch_pack_weights_tensor(g, d_w, ws + L.total, s);
        if (st == LCE_OK) st = launch_bconv_tensor(p.launch, d_in, ws + L.total, d_mult, d_bias, d_thr, d_out, s);
    } else {
        st = dispatch(p, d_in, d_w, d_mult, d_bias, d_thr, d_out, s);
    }
    if (st != LCE_OK) return st;
    void *back_view = !out_view && L.out_bytes <= kKernelCopy ? pinned_host_view(output, L.out_bytes, true) : nullptr;
    if (back_view) {
        const HostCopy back[kHostCopies] = {{ws + L.out, back_view, L.out_bytes}};
        st = launch_host_copies(back, s);
        if (st != LCE_OK) return st;
    } else if (!out_view && cudaMemcpyAsync(output, ws + L.out, L.out_bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) {
        return LCE_ERR_CUDA;
    }
    if (synchronise && cudaStreamSynchronize(s) != cudaSuccess) return LCE_ERR_CUDA;
    return LCE_OK;
}
}  // namespace
}  // namespace lce

extern "C" lce_status lce_bconv2d_host(const lce_bconv2d_desc *desc, const uint32_t *input, const uint32_t *weights,
                                       const float *multiplier, const float *bias, const int32_t *thresholds,
                                       void *output, void *workspace, size_t workspace_bytes, void *stream)
{
    return lce::host_conv(desc, input, weights, multiplier, bias, thresholds, output, workspace, workspace_bytes, stream, true);
}

extern "C" lce_status lce_bconv2d_host_async(const lce_bconv2d_desc *desc, const uint32_t *input, const uint32_t *weights,
                                             const float *multiplier, const float *bias, const int32_t *thresholds,
                                             void *output, void *workspace, size_t workspace_bytes, void *stream)
{
    return lce::host_conv(desc, input, weights, multiplier, bias, thresholds, output, workspace, workspace_bytes, stream, false);
}

// ---- host-buffer convolution that allocates nothing ---------------------------------------------
// Some callers cannot give lce_bconv2d_host the device workspace it asks for, because they are not
// in a position to call cudaMalloc at all: code running inside a memory-capped or allocator-less
// host process, a real-time loop that must not take the allocator's locks, a plug-in that is only
// handed host tensors.  For them the staging area lives inside the library itself, as a
// file-scope device array that every GPU loading the library carries until the process exits.

#define LCE_STATIC_WORKSPACE_BYTES (8u << 20)

static __device__ __align__(256) unsigned char g_static_workspace[LCE_STATIC_WORKSPACE_BYTES];

namespace lce {
namespace {

constexpr int kMaxDevices = 64;
std::atomic<void *> g_static_workspace_addr[kMaxDevices];  // device address of g_static_workspace, per device; null = not looked up yet

}  // namespace
}  // namespace lce

extern "C" size_t lce_bconv2d_host_noalloc_max_bytes(void) { return LCE_STATIC_WORKSPACE_BYTES; }

extern "C" lce_status lce_bconv2d_host_noalloc(const lce_bconv2d_desc *desc, const uint32_t *input,
                                               const uint32_t *weights, const float *multiplier, const float *bias,
                                               const int32_t *thresholds, void *output, void *stream)
{
    using namespace lce;
    ConvGeom g;
    lce_status st = make_geom(desc, &g);
    if (st == LCE_OK) st = check_conv_buffers(g, input, weights, multiplier, bias, thresholds, output);
    if (st != LCE_OK) return st;
    if (desc->weights_packed) return LCE_ERR_INVALID_ARG;
    if (host_layout(g).total > LCE_STATIC_WORKSPACE_BYTES) return LCE_ERR_WORKSPACE;  // this call does not fit the built-in array

    // In host code the array's name is only a stand-in for the symbol, not a device address: ask the
    // runtime for the address once per device, with that device current.  (Two threads making the
    // first call together both look it up and store the same value.)
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return LCE_ERR_CUDA;
    void *addr = g_static_workspace_addr[dev].load(std::memory_order_acquire);
    if (addr == nullptr) {
        if (cudaGetSymbolAddress(&addr, g_static_workspace) != cudaSuccess || addr == nullptr) return LCE_ERR_CUDA;
        g_static_workspace_addr[dev].store(addr, std::memory_order_release);
    }
    // Nothing in the array has to start at zero: every region is written in full (by the copies in,
    // or by the kernel) before anything reads it.  From here on this is lce_bconv2d_host on that array.
    return host_conv(desc, input, weights, multiplier, bias, thresholds, output, addr, LCE_STATIC_WORKSPACE_BYTES, stream, true);
}
