// LceBConv2d, tiled XOR/POPC kernels for 3x3 and 5x5 filters (and, further down, 1x1) (paper
// Section 3.2: im2col -> BGEMM -> output transform, here as one implicit-GEMM kernel: the im2col
// matrix is never materialised and the accumulators never leave registers before the output
// transform).
//
// Stride 1 or 2, any channel counts and image sizes:
//   * a CTA of 8 (or 4) warps owns one contiguous range of output pixels (flat (n, oh, ow) order)
//     times 64 output channels; a warp works on 4 pixels x 8 channel groups at a time (8 x 4 in a
//     channel block that has at most 32 channels), a thread on TP pixels x 8 channels, i.e. TP x 8
//     accumulators in registers.  All ranges are equal to within two pixels per thread: the last step
//     of a range runs the two-pixel form of the same code;
//   * the CTA copies the packed input rows its pixels need into shared memory, a tile of up to
//     8 x 32 x TP pixels at a time (the next tile while the current one is computed), one plane per
//     channel word, in "padded image" coordinates: rows/columns outside the image hold zero words,
//     which is exactly the paper's one-padding (a zero bit is +1.0);
//   * the weights of its 64 channels arrive as carry-save operands (csa.cuh): either copied in
//     16-byte pieces from a buffer prepared once by lce_bconv2d_pack_weights (the paper's
//     load-time "weight packing"), or derived on the fly from the plain packed weights;
//   * for every channel word nine taps of a (pixel, channel) pair form one nine-word carry-save
//     group (a 5x5 filter is three groups, the last two words zero): 16 LOP3 + 4 POPC + 4 IMAD
//     instead of 9 XOR + 9 POPC + 9 adds.  The activation-side operands of the thread's TP pixels
//     sit in registers for the whole group; the weight-side operands of one channel are read from
//     shared memory once and used for all TP pixels (shared-memory bandwidth, not issue slots, is
//     what this ordering saves);
//   * epilogue: acc = K - 2*count, then float multiply-add, threshold + bit-pack, or raw int32.
#include "common.cuh"

#include "csa.cuh"
#include "tiled_common.cuh"
#include "bconv_kxk.cuh"
#include "bconv_1x1.cuh"

namespace lce {
namespace {

// ---- host side: launchers, the tile / range chooser, weight packing, plan and launch ----------------

template <int TP>
lce_status launch1x1(const TiledParams &p, size_t smem_bytes, dim3 grid, cudaStream_t s)
{
    auto kernel = bconv1x1_kernel<TP>;
    static SmemOptIn opted;
    if (!opted.ensure(kernel, smem_bytes)) return LCE_ERR_CUDA;
    return launch_dependent(kernel, grid, kThreads, smem_bytes, s, p);
}

template <int KS, int STRIDE, int TP, int NW, bool F32 = false>
lce_status launch_kxk(const TiledParams &p, size_t smem_bytes, dim3 grid, cudaStream_t s)
{
    auto kernel = bconv3x3_kernel<KS, STRIDE, TP, NW, F32>;
    static SmemOptIn opted;
    if (!opted.ensure(kernel, smem_bytes)) return LCE_ERR_CUDA;
    return launch_dependent(kernel, grid, 32 * NW, smem_bytes, s, p);
}

// CTAs of 128 threads that the register file lets share an SM, per pixels-per-thread variant
// (must match the __launch_bounds__ of the kernel).
int reg_limited_ctas(int tp, int nw) { return (tp <= 2 ? 24 : 16) / nw; }

size_t smem_bytes_for(const ConvGeom &g, const TiledParams &p)
{
    return ((size_t)g.Cw * groups_per_word(g.KH) * kChanGroups * kWGroupStride + kWsumWords + 2 * (size_t)g.Cw * p.plane) * 4;
}

void set_tile(const ConvGeom &g, TiledParams *p, int tile_pixels)
{
    p->tile_pixels = tile_pixels;
    int rows_max = (tile_pixels - 1) / g.OW + 2;  // output rows a run of tile_pixels flat pixels can touch
    if (rows_max > tile_pixels) rows_max = tile_pixels;
    const int nv_max = (rows_max - 1) * g.KH + g.KH;  // consecutive output rows are at most KH virtual rows apart
    p->plane = nv_max * p->pitch;
}

// the KxK kernel keeps two pixels' counts in one 32-bit accumulator: a count can reach K, so K < 65536
bool covers3x3(const ConvGeom &g)
{
    return g.KH == g.KW && (g.KH == 3 || g.KH == 5) && g.sh == g.sw && g.sh <= 2 && (int64_t)g.KH * g.KW * g.Cin < 65536;
}
bool covers1x1(const ConvGeom &g) { return g.KH == 1 && g.KW == 1 && g.sh == g.sw; }

bool tiled_covers(const ConvGeom &g)
{
    return (covers3x3(g) || covers1x1(g)) && g.M < (1ll << 31) - 256 &&
           (g.Cout + kChanPerCta - 1) / kChanPerCta <= 65535;
}

void pointwise_split(int Cw, int *n9, int *rem3)
{
    *n9 = Cw / 9;
    const int rem = Cw % 9;
    if (rem > 6) { ++*n9; *rem3 = 0; }
    else *rem3 = (rem + 2) / 3;
}

int image_groups(const ConvGeom &g)
{
    if (covers3x3(g)) return g.Cw * groups_per_word(g.KH);
    int n9, rem3;
    pointwise_split(g.Cw, &n9, &rem3);
    return pointwise_groups(n9, rem3);
}

#ifndef LCE_MAX_ROUNDS
#define LCE_MAX_ROUNDS 8
#endif
constexpr int kMaxRounds = LCE_MAX_ROUNDS;

struct TileChoice {
    int tp, tile, ctas_x, ctas_half, range_full, range_half;
    double cost;
};

// Pixels per thread (TP) and tile size: a tile covers 16*TP*rounds flat pixels and the grid is
// persistent (each CTA walks tiles x, x + gridDim.x, ...).  Pick the pair that balances the SMs
// best: cost = (CTAs on the busiest SM) x (tiles of the busiest CTA) x (tile work), with a
// penalty when too few warps share an SM to keep the logic pipe busy.
template <typename SmemFn>
bool choose_tile(const ConvGeom &g, int chan_blocks, SmemFn smem_for_tile, TileChoice *best, int nw = kWarps,
                 size_t smem_limit = 110 * 1024, bool has_half_block = false, bool ranged = false, bool allow_tp1 = false)
{
    int sms = 148;
    {
        int dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    double best_cost = 0;
    best->tile = 0;
    // one pixel per thread exists for the KxK kernel with 4-warp CTAs only: the finest split of a
    // single image over the SMs (latency, not throughput)
    for (int tp = (ranged && nw == 4 && allow_tp1) ? 1 : 2; tp <= 4; ++tp) {
        const int unit = 4 * nw * tp;
        for (int rounds = 1; rounds <= kMaxRounds; ++rounds) {
            // a half channel block takes two units of pixels per step
            if (has_half_block && (rounds & 1)) continue;
            const int tile = unit * rounds;
            const size_t smem = smem_for_tile(tile);
            if (smem > smem_limit) continue;
            int per_sm = (int)((220 * 1024) / (smem + 1024));
            if (per_sm < 1) per_sm = 1;
            if (per_sm > reg_limited_ctas(tp, nw)) per_sm = reg_limited_ctas(tp, nw);
            const double smem_penalty[5] = {0, 1.2, 1.06, 1.02, 1.0};  // fewer pixels per thread re-read the weight operands more often
            const int full_blocks = has_half_block ? chan_blocks - 1 : chan_blocks;
            const int64_t slots = (int64_t)sms * per_sm;
            int64_t ctas_x, ctas_half = 0, range_full = 0, range_half = 0;
            double t_cta;  // time of the busiest CTA, in pixel-steps of a full block
            if (ranged) {
                // KxK kernel: a CTA owns a contiguous range of pixels, a whole number of granules; a
                // granule is the smallest step the kernel has (2 pixels per thread when TP > 2)
                const bool tail = kTailStep && tp > 2;
                const int64_t pps = 4 * nw;                     // pixels per step and pixel-per-thread, full block
                const int64_t granule = tail ? pps : unit;      // ranges are whole numbers of granules
                // per tile: barrier bubbles and the halo rows that are staged again (measured at
                // 56x56x64: about a fifth of the time of computing those rows)
                const double tile_overhead = 4.0 + 0.2 * (g.KH - 1) * g.OW;
                auto range_for = [&](int64_t ctas, int64_t gran) { return ((g.M + ctas - 1) / ctas + gran - 1) / gran * gran; };
                auto time_of = [&](int64_t range, int pixel_scale) {  // pixel_scale 2: a half block's step covers twice the pixels
                    double t = (double)((range + tile - 1) / tile) * tile_overhead;
                    for (int64_t r = range / pixel_scale; r > 0;) {  // the kernel's own decomposition into steps
                        if (tail && r <= 2 * pps) { t += 2 * pps * smem_penalty[2]; r = 0; }
                        else { t += unit * smem_penalty[tp]; r -= unit; }
                    }
                    return t;
                };
                ctas_x = has_half_block ? (2 * slots) / (2 * full_blocks + 1) : slots / chan_blocks;
                if (ctas_x < 1) ctas_x = 1;
                t_cta = 0;
                if (full_blocks > 0) {
                    range_full = range_for(ctas_x, granule);
                    ctas_x = (g.M + range_full - 1) / range_full;
                    t_cta = time_of(range_full, 1);
                }
                if (has_half_block) {
                    ctas_half = full_blocks > 0 ? (ctas_x + 1) / 2 : (slots < 1 ? 1 : slots);
                    range_half = range_for(ctas_half, 2 * granule);
                    ctas_half = (g.M + range_half - 1) / range_half;
                    const double t_half = time_of(range_half, 2);
                    if (t_half > t_cta) t_cta = t_half;
                }
            } else {
                const int64_t n_tiles = (g.M + tile - 1) / tile;
                ctas_x = slots / chan_blocks;
                if (ctas_x < 1) ctas_x = 1;
                if (ctas_x > n_tiles) ctas_x = n_tiles;
                t_cta = (double)((n_tiles + ctas_x - 1) / ctas_x) * (tile * smem_penalty[tp] + 4.0);
            }
            const int64_t total_ctas = ctas_x * full_blocks + ctas_half;
            const int64_t ctas_on_sm = (total_ctas + sms - 1) / sms;
            const double warps = (double)total_ctas / sms * nw;
            const double eff = warps >= 16 ? 1.0 : (warps >= 8 ? 0.8 + 0.2 * (warps - 8) / 8 : 0.4 + 0.4 * warps / 8);
            const double cost = (double)ctas_on_sm * t_cta / eff;
            if (best->tile == 0 || cost < best_cost) {
                best->tile = tile; best->tp = tp; best->ctas_x = (int)ctas_x; best->ctas_half = (int)ctas_half;
                best->range_full = (int)range_full; best->range_half = (int)range_half;
                best_cost = best->cost = cost;
            }
        }
    }
    return best->tile != 0;
}

}  // namespace

size_t tiled_weight_image_bytes(const ConvGeom &g)
{
    if (!covers_some_padding(g, tiled_covers)) return 0;
    const int chan_blocks = (g.Cout + kChanPerCta - 1) / kChanPerCta;
    return (size_t)chan_blocks * image_block_words(image_groups(g)) * 4;
}

lce_status launch_pack_weights_tiled(const ConvGeom &g, const uint32_t *w, uint32_t *image, cudaStream_t s)
{
    const int chan_blocks = (g.Cout + kChanPerCta - 1) / kChanPerCta;
    const int groups = image_groups(g);
    const int64_t entries = (int64_t)chan_blocks * kChanPerCta * groups;
    int blocks = (int)((entries + 127) / 128);
    if (blocks > 148 * 8) blocks = 148 * 8;
    if (covers3x3(g))
        pack_weights_kernel<<<blocks, 128, 0, s>>>(w, image, g.Cout, g.Cw, g.Cin, chan_blocks, g.KH);
    else
        pack_weights_pointwise_kernel<<<blocks, 128, 0, s>>>(w, image, g.Cout, g.Cw, groups, chan_blocks);
    return launch_status();
}

// Everything the launch needs that does not depend on the buffers: geometry fields of the kernel
// parameters, the chosen variant and the launch dimensions.
inline bool geom_equal(const ConvGeom &a, const ConvGeom &b)
{
    return a.N == b.N && a.H == b.H && a.W == b.W && a.Cin == b.Cin && a.Cout == b.Cout && a.KH == b.KH && a.KW == b.KW &&
           a.sh == b.sh && a.sw == b.sw && a.padding == b.padding && a.out_type == b.out_type && a.activation == b.activation;
}

struct TiledPlan {
    bool pointwise;
    int nw, tp;
    size_t smem_bytes;
    dim3 grid;
};

static lce_status plan_tiled_uncached(const ConvGeom &g, bool f32_input, TiledParams *pp, TiledPlan *plan)
{
    TiledParams &p = *pp;
    if (!tiled_covers(g)) return LCE_ERR_UNSUPPORTED;
    if (f32_input && !covers3x3(g)) return LCE_ERR_UNSUPPORTED;
    p.N = g.N; p.H = g.H; p.W = g.W; p.Cin = g.Cin; p.Cw = g.Cw; p.Cout = g.Cout; p.Cow = g.Cow;
    p.OH = g.OH; p.OW = g.OW; p.pt = g.pt; p.pl = g.pl;
    p.padding = g.padding; p.out_type = g.out_type; p.activation = g.activation;
    p.M = (int32_t)g.M;
    p.stride = g.sh;
    p.cw_shift = -1;
    p.half_block = -1;
    for (int b = 0; b < 16; ++b)
        if ((1 << b) == g.Cw) p.cw_shift = b;
    const int chan_blocks = (g.Cout + kChanPerCta - 1) / kChanPerCta;
    TileChoice c;

    if (covers1x1(g)) {
        pointwise_split(g.Cw, &p.n9, &p.rem3);
        p.cwp = 9 * p.n9 + 3 * p.rem3;
        const int groups = pointwise_groups(p.n9, p.rem3);
        auto smem_for = [&](int tile) {
            return ((size_t)groups * kChanGroups * kWGroupStride + kWsumWords + 2 * (size_t)tile * p.cwp) * 4;
        };
        if (!choose_tile(g, chan_blocks, smem_for, &c)) return LCE_ERR_UNSUPPORTED;
        p.tile_pixels = c.tile;
        p.n_tiles = (int32_t)((g.M + c.tile - 1) / c.tile);
        plan->pointwise = true;
        plan->nw = kWarps;
        plan->tp = c.tp;
        plan->grid = dim3((unsigned)c.ctas_x, (unsigned)chan_blocks, 1);
        plan->smem_bytes = smem_for(c.tile);
        return LCE_OK;
    }

    p.Hp = (g.OH - 1) * g.sh + g.KH;
    p.Wp = (g.OW - 1) * g.sh + g.KW;
    if (p.Wp < g.W + g.pl) p.Wp = g.W + g.pl;  // staging writes the whole image row; columns past the taps are unused
    p.pitch = p.Wp | 1;  // odd pitch: the 4 pixels of a warp in 4 different rows hit 4 different banks
    auto smem_for = [&](int tile) {
        set_tile(g, &p, tile);
        return smem_bytes_for(g, p);
    };
    // Candidates: CTAs of 8 or 4 warps (eight warps share one copy of the weight operands and one
    // staging buffer, which measures faster wherever whole tiles of 32*TP pixels are useful work;
    // four-warp CTAs remain for problems too small for that), with or without the half-block lane
    // mapping (which needs tiles of two units: not worth it on very small problems).
    const int tail_channels = g.Cout % kChanPerCta;
    const bool can_half = tail_channels >= 1 && tail_channels <= kChanPerCta / 2;
    int nw = 0;
    bool half = false;
    c.cost = 0;
    for (int use_half = can_half ? 1 : 0; use_half >= 0; --use_half) {
        for (int w = 8; w >= 4; w -= 4) {
            if (w == 8 && f32_input) continue;  // the float-input loader exists for four-warp CTAs only
            TileChoice t;
            bool ok = choose_tile(g, chan_blocks, smem_for, &t, w, w == 8 ? 226 * 1024 : 110 * 1024, use_half != 0, true, !f32_input);
            if (!ok && w == 4 && f32_input)
                ok = choose_tile(g, chan_blocks, smem_for, &t, 4, 226 * 1024, use_half != 0, true);
            if (ok && (nw == 0 || t.cost < c.cost)) { c = t; nw = w; half = use_half != 0; }
        }
    }
    if (nw == 0) return LCE_ERR_UNSUPPORTED;
    set_tile(g, &p, c.tile);
    p.n_tiles = (int32_t)((g.M + c.tile - 1) / c.tile);
    p.half_block = half ? chan_blocks - 1 : -1;
    p.full_blocks = half ? chan_blocks - 1 : chan_blocks;
    p.ctas_full = c.ctas_x;
    p.ctas_half = half ? c.ctas_half : 0;
    p.range_full = c.range_full;
    p.range_half = c.range_half;
    plan->pointwise = false;
    plan->nw = nw;
    plan->tp = c.tp;
    plan->smem_bytes = smem_bytes_for(g, p);
    plan->grid = dim3((unsigned)(p.full_blocks * p.ctas_full + p.ctas_half), 1, 1);
    return LCE_OK;
}

// The plan depends on the geometry alone, and a network repeats few geometries: the last few plans
// of each host thread are kept (the cost model walks a few hundred candidates per call otherwise).
static lce_status plan_tiled(const ConvGeom &g, bool f32_input, TiledParams *pp, TiledPlan *plan)
{
    struct Entry {
        ConvGeom g;
        bool f32_input, valid;
        int device;  // the plan depends on the SM count of the current device
        lce_status status;
        TiledParams p;
        TiledPlan plan;
    };
    constexpr int kEntries = 16;
    static thread_local Entry cache[kEntries];
    static thread_local int next = 0;
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) device = -1;
    for (int i = 0; i < kEntries; ++i) {
        const Entry &e = cache[i];
        if (e.valid && e.f32_input == f32_input && e.device == device && geom_equal(e.g, g)) {
            *pp = e.p;
            *plan = e.plan;
            return e.status;
        }
    }
    Entry &e = cache[next];
    next = (next + 1) % kEntries;
    e.valid = false;
    e.p = TiledParams{};
    e.plan = TiledPlan{};
    e.status = plan_tiled_uncached(g, f32_input, &e.p, &e.plan);
    e.g = g;
    e.f32_input = f32_input;
    e.device = device;
    e.valid = true;
    *pp = e.p;
    *plan = e.plan;
    return e.status;
}

lce_status tiled_plan_info(const ConvGeom &g, TiledPlanInfo *info)
{
    TiledParams p{};
    TiledPlan plan{};
    const lce_status st = plan_tiled(g, false, &p, &plan);
    if (st != LCE_OK) return st;
    info->pointwise = plan.pointwise ? 1 : 0;
    info->warps_per_cta = plan.nw;
    info->pixels_per_thread = plan.tp;
    info->tile_pixels = p.tile_pixels;
    info->ctas = (int32_t)(plan.grid.x * plan.grid.y);
    info->ctas_half_block = plan.pointwise ? 0 : p.ctas_half;
    info->pixels_per_cta = plan.pointwise ? 0 : p.range_full;
    info->pixels_per_cta_half_block = plan.pointwise ? 0 : p.range_half;
    info->shared_bytes = (int64_t)plan.smem_bytes;
    return LCE_OK;
}

lce_status launch_bconv_tiled(const ConvGeom &g, const uint32_t *in, const uint32_t *w, const uint32_t *w_image,
                              const float *mult, const float *bias, const int32_t *thr, void *out, cudaStream_t s,
                              const float *residual, uint32_t *out_packed, const float *in_f32)
{
    // 128-bit epilogue accesses need 16-byte aligned buffers when the channel count allows them
    if ((g.Cout & 3) == 0 && g.out_type != LCE_OUT_BITPACKED && (!aligned(out, 16) || !aligned(residual, 16)))
        return LCE_ERR_UNSUPPORTED;
    if (w_image && !aligned(w_image, 16)) return LCE_ERR_ALIGNMENT;
    TiledParams p{};
    TiledPlan plan{};
    const lce_status st = plan_tiled(g, in_f32 != nullptr, &p, &plan);
    if (st != LCE_OK) return st;
    p.in = in; p.w = w; p.w_image = w_image; p.mult = mult; p.bias = bias; p.thr = thr; p.out = out;
    p.residual = residual; p.out_packed = out_packed; p.in_f32 = in_f32;
    const size_t smem_bytes = plan.smem_bytes;
    const dim3 grid = plan.grid;
    const int nw = plan.nw;
    struct { int tp; } c{plan.tp};
    if (plan.pointwise) {
        if (c.tp == 2) return launch1x1<2>(p, smem_bytes, grid, s);
        if (c.tp == 3) return launch1x1<3>(p, smem_bytes, grid, s);
        return launch1x1<4>(p, smem_bytes, grid, s);
    }
#define LCE_LAUNCH_TP(KS, ST, NW)                                                   \
    do {                                                                            \
        if (c.tp == 1) return launch_kxk<KS, ST, 1, 4>(p, smem_bytes, grid, s);     \
        if (c.tp == 2) return launch_kxk<KS, ST, 2, NW>(p, smem_bytes, grid, s);    \
        if (c.tp == 3) return launch_kxk<KS, ST, 3, NW>(p, smem_bytes, grid, s);    \
        return launch_kxk<KS, ST, 4, NW>(p, smem_bytes, grid, s);                   \
    } while (0)
    if (in_f32) {
#define LCE_LAUNCH_F32(KS, ST)                                                         \
    do {                                                                               \
        if (c.tp == 2) return launch_kxk<KS, ST, 2, 4, true>(p, smem_bytes, grid, s);  \
        if (c.tp == 3) return launch_kxk<KS, ST, 3, 4, true>(p, smem_bytes, grid, s);  \
        return launch_kxk<KS, ST, 4, 4, true>(p, smem_bytes, grid, s);                 \
    } while (0)
        if (g.KH == 3 && g.sh == 1) LCE_LAUNCH_F32(3, 1);
        if (g.KH == 3) LCE_LAUNCH_F32(3, 2);
        if (g.sh == 1) LCE_LAUNCH_F32(5, 1);
        LCE_LAUNCH_F32(5, 2);
#undef LCE_LAUNCH_F32
    }
    if (g.KH == 3 && g.sh == 1) { if (nw == 8) LCE_LAUNCH_TP(3, 1, 8); else LCE_LAUNCH_TP(3, 1, 4); }
    if (g.KH == 3) { if (nw == 8) LCE_LAUNCH_TP(3, 2, 8); else LCE_LAUNCH_TP(3, 2, 4); }
    if (g.sh == 1) { if (nw == 8) LCE_LAUNCH_TP(5, 1, 8); else LCE_LAUNCH_TP(5, 1, 4); }
    if (nw == 8) LCE_LAUNCH_TP(5, 2, 8); else LCE_LAUNCH_TP(5, 2, 4);
#undef LCE_LAUNCH_TP
}

}  // namespace lce

