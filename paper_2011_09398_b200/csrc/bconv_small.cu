// LceBConv2d for small layers (single images, late stages of a network), built for latency.
//
// What bounds these calls: a layer of one image is 2^22 - 2^28 binary MACs, well under a microsecond of work if
// every SM gets its share of it and no SM waits long for its operands.  The tiled kernels give a CTA 64
// channels, the whole depth K and carry-save weight operands of 12 words per nine, so a 7x7x512 layer fills 32
// SMs, each of which copies 77 KB of weights before it starts (9.3 us); the tensor-core kernel sets up TMEM
// and a ring of barriers for one or two tiles (4 - 5 us at least).  Here:
//   * the output is cut into tiles of 8 .. 64 pixels x 32 channels (one bit-packed word per pixel), so that the
//     CTAs spread over all SMs, and inside a CTA the depth K is cut into slices: a warp computes 8 or 16 pixels
//     x 32 channels over its slice, the slices meet in shared memory;
//   * the product is the warp-level integer matrix instruction m16n8k32 (u8 x u8 -> s32, 8 clocks per SM
//     sub-partition, measured: 64 words per clock and SM, against 28 for the best popcount loop).  Of a step of
//     four words of K, lane q of a quad holds word q of its row; in four instructions t = 0..3 it feeds the bits t
//     and t + 4 of every byte, one AND each, so its activation bytes are bit << t.  The weights are laid out with
//     the bits of every byte reversed, so theirs are bit << (7 - t), and every product of two set bits is 2^7.  The
//     sum is 128 popcount(a AND w), and with the popcounts of the two rows the accumulator of Section 2 is
//     K - 2 popcount(a XOR w) = K - 2 popcount(a) - 2 popcount(w) + 4 popcount(a AND w), exactly;
//   * a tile's weights are 32 rows of K words, laid out at load time as the shared-memory image
//     (lce_bconv2d_pack_weights).  The input rows a tile touches are fetched once into shared memory, with zero
//     words (= +1.0, one-padding) around the image, and im2col (Section 3.2) is a table: the offset of each of the
//     K words from the corner of a pixel's window.  Fetching im2col rows from memory asks for every word once per
//     tap, and the whole input of a 7x7x512 layer is 24 cache lines that all SMs want at once: the L2 served
//     those in 2000 clocks, against 600 for one fetch; making im2col rows in shared memory cost another 500 - 900;
//   * pitches in shared memory keep a warp's reads of 8 rows x 4 words in 32 different banks (stride 1);
//   * with so little work per CTA every dependent step shows (a dynamic loop over the slices' partial sums took
//     350 - 560 clocks; now they are added up by shared-memory atomics): address divisions are done before the
//     dependency wait, and the transform's form is a template argument;
//   * programmatic dependent launch: weights and per-channel constants are on their way while the previous
//     kernel of the stream drains.
#include "common.cuh"
#include "mx_common.cuh"
#include "u8_mma.cuh"

namespace lce {
namespace {

constexpr int kChannels = 32;      // channels per CTA
constexpr int kGroupPixels = 8;    // pixels of a warp's tile
constexpr int kRedPitch = 36;      // words per pixel of the sums (32 channels + 4: conflict-free updates)
constexpr int kMaxWarps = 16;

// n / d for 0 <= n < 2^31 in a multiply-high, an add and a shift (Granlund and Montgomery, PLDI 1994, Figure 4.1)
struct FastDiv {
    uint32_t mul, sh;
    __device__ __forceinline__ int operator()(int n) const { return (int)((__umulhi((uint32_t)n, mul) + (uint32_t)n) >> sh); }
};

FastDiv fast_div(uint32_t d)
{
    FastDiv f{0, 0};
    while ((1ull << f.sh) < d) ++f.sh;
    f.mul = (uint32_t)((((1ull << f.sh) - d) << 32) / d + 1);
    return f;
}

struct SmallParams {
    const uint32_t *in;
    const uint32_t *w;            // plain words, or the tile images (image != 0)
    const float *mult;
    const float *bias;
    const int32_t *thr;
    const float *residual;
    void *out;
    uint32_t *out_packed;
    int32_t image, N, H, W, Cw, Cin, Cout, Cow, KH, KW, taps, sh, sw, OH, OW, pt, pl;
    int32_t M, K, KD;             // output pixels; packed words per row; true depth taps * Cin
    int32_t Hp, Wp, PW;           // padded rows per image, padded columns per row, words between columns in shared memory
    int32_t steps, per_slice;     // 4-word steps of a row, and of a slice
    int32_t pitch;                // words between weight rows in shared memory
    int32_t tile, slices, slices_sh;   // pixels per CTA (a multiple of 8); slices of K, a power of two
    int32_t raw_words, padded;    // room for the input rows of a tile (a multiple of 4); they have padding
    int32_t vec, pieces;          // words per asynchronous copy of activations: 4, 2 or 1; copies per row
    int32_t zero_pad, out_type, relu;
    FastDiv by_pieces, by_px_pieces, by_cw, by_kw, by_ow, by_oh, by_hp;
};

// Holds a kernel parameter in a register from here on.  Left to itself the compiler reads parameters from the
// constant bank where they are used, 40 and more clocks each, which in code that runs once per CTA adds up to
// more than the work (the transform of two pixels per warp took 1150 clocks).
template <typename T>
__device__ __forceinline__ T keep(T v)
{
    if (sizeof(T) == 8) asm volatile("" : "+l"(reinterpret_cast<uint64_t &>(v)));
    else asm volatile("" : "+r"(reinterpret_cast<uint32_t &>(v)));
    return v;
}

// A load that is issued here and waited for at its first use (an ordinary load of a constant may be moved down to
// its use, behind the dependency wait, and then its latency is paid in full).
__device__ __forceinline__ int load_early(const void *p)
{
    int v;
    asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

enum { SMALL_BITS = 0, SMALL_FLOAT = 1, SMALL_GENERAL = 2 };  // GENERAL: int32 output, shortcut add, re-quantised copy

template <int MODE, int NT>  // NT: groups of 8 pixels per warp job
__global__ void __launch_bounds__(32 * kMaxWarps, 1) bconv_small_kernel(const __grid_constant__ SmallParams p)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int pitch = keep(p.pitch), tile = keep(p.tile), steps = keep(p.steps);
    const bool zero_pad = keep(p.zero_pad) != 0;
    uint32_t *sW = smem;                                                   // [32][pitch]
    int32_t *sOnes = reinterpret_cast<int32_t *>(sW + kChannels * pitch);  // [32] popcounts of the weight rows
    int32_t *sTap = sOnes + kChannels;                                     // zero-padding: [32][taps] sums of a tap's weights
    int32_t *sK = sTap + (zero_pad ? kChannels * p.taps : 0);              // [4 steps] offset of word k from a window's corner
    int32_t *sPx = sK + 4 * steps;                                         // [tile] window corner of a pixel in sRaw
    int32_t *sRed = sPx + tile;                                            // [tile][kRedPitch] sums
    int32_t *sPop = sRed + tile * kRedPitch;                               // [tile] popcounts of the activation rows
    uint32_t *sOutside = reinterpret_cast<uint32_t *>(sPop + tile);        // zero-padding: [tile] taps of a pixel outside the image
    uint32_t *sRaw = sOutside + (zero_pad ? tile : 0);                     // padded input rows

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_threads = blockDim.x, n_warps = n_threads >> 5;
    const int m0 = blockIdx.x * tile, ch0 = blockIdx.y * kChannels;

    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- constants of the model: weights on their way, per-channel values in registers -------------------
    if (p.image) {  // rows, row tails, popcounts and tap sums as they lie in shared memory
        const int image_words = kChannels * (pitch + 1 + p.taps), n = (zero_pad ? image_words : kChannels * (pitch + 1)) >> 2;
        const uint32_t *src = p.w + (int64_t)blockIdx.y * image_words;
        for (int e = tid; e < n; e += n_threads) cp_async_zfill<16>(sW + 4 * e, src + 4 * e, true);
    } else {
        // plain words may come from the kernel before (LceQuantize of the weights), which may still be running
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int r = warp; r < kChannels; r += n_warps) {
            const bool valid = ch0 + r < p.Cout;
            const uint32_t *src = p.w + (valid ? (int64_t)(ch0 + r) * p.K : 0);
            int ones = 0;
            for (int k = lane; k < 4 * steps; k += 32) {
                const uint32_t v = valid && k < p.K ? __ldg(src + k) : 0u;
                sW[r * pitch + k] = reverse_in_bytes(v);
                ones += __popc(v);
            }
            ones = __reduce_add_sync(0xffffffffu, ones);
            if (lane == 0) sOnes[r] = ones;
        }
    }
    const int channel = ch0 + lane;
    const bool ch_ok = channel < p.Cout;
    const int KD = keep(p.KD);
    float mult = 0.f, bias = 0.f;
    int32_t limit = INT32_MIN;  // bit-packed output: the threshold; pad channels are never below it
    if (MODE != SMALL_BITS && p.out_type == LCE_OUT_FLOAT32 && ch_ok) {
        mult = __int_as_float(load_early(p.mult + channel));
        bias = __int_as_float(load_early(p.bias + channel));
    }
    if (MODE == SMALL_BITS && ch_ok) limit = load_early(p.thr + channel);

    // ---- geometry: padded rows v = n * Hp + y of the tile, pixel corners, im2col offsets ---------------------
    const int W = keep(p.W), H = keep(p.H), Cw = keep(p.Cw), PW = keep(p.PW), Wp = keep(p.Wp), M = keep(p.M), K = keep(p.K);
    const auto corner = [&](int m, int *ow) {  // padded row of a pixel's window, and its output column
        const int r = p.by_ow(m), n = p.by_oh(r);
        *ow = r * -p.OW + m;
        return n * p.Hp + (r - n * p.OH) * p.sh;
    };
    int ow_unused;
    const int v_first = corner(m0, &ow_unused), v_end = corner(min(m0 + tile, M) - 1, &ow_unused) + p.KH;
    for (int e = tid; e < tile; e += n_threads) {
        int ow;
        const int v = corner(min(m0 + e, M - 1), &ow);
        sPx[e] = ((v - v_first) * Wp + ow * p.sw) * PW;
        sPop[e] = 0;
        if (zero_pad) {
            const int y0 = v - p.by_hp(v) * p.Hp - p.pt, x0 = ow * p.sw - p.pl;
            uint32_t columns = 0u, outside = 0u;
            for (int kx = 0; kx < p.KW; ++kx) columns |= ((unsigned)(x0 + kx) >= (unsigned)W ? 1u : 0u) << kx;
            for (int ky = 0; ky < p.KH; ++ky) outside |= ((unsigned)(y0 + ky) >= (unsigned)H ? (1u << p.KW) - 1u : columns) << (ky * p.KW);
            sOutside[e] = outside;
        }
    }
    for (int k = tid; k < 4 * steps; k += n_threads) {
        const int tap = p.by_cw(min(k, K - 1)), ky = p.by_kw(tap);
        sK[k] = (ky * Wp + tap - ky * p.KW) * PW + min(k, K - 1) - tap * Cw;
    }
    for (int e = tid; e < tile * kRedPitch; e += n_threads) sRed[e] = 0;
    if (p.padded)
        for (int e = tid; 4 * e < p.raw_words; e += n_threads) reinterpret_cast<uint4 *>(sRaw)[e] = make_uint4(0u, 0u, 0u, 0u);
    // this thread's first copy of activations: (row, column, piece of the column's words)
    const int vec = keep(p.vec), pieces = keep(p.pieces), copies = (v_end - v_first) * pieces, n_images = p.N;
    const uint32_t *const in = keep(p.in);
    const auto activation_copy = [&](int e, const uint32_t **src, uint32_t **dst) {
        const int rr = p.by_pieces(e), j = e - rr * pieces, v = v_first + rr;
        const int n = p.by_hp(v), y = v - n * p.Hp - p.pt;
        const int x = p.by_px_pieces(j), w = j * vec - x * Cw;
        *src = in + ((int64_t)n * H + y) * W * Cw + j * vec;
        *dst = sRaw + (rr * Wp + x + p.pl) * PW + w;
        return e < copies && (unsigned)y < (unsigned)H && n < n_images;
    };
    const uint32_t *src;
    uint32_t *dst;
    bool copy_ok = activation_copy(tid, &src, &dst);
    // what the rest of the kernel needs of the parameters, and this warp's first job
    void *const out = keep(p.out);
    const int slices = keep(p.slices), slices_sh = keep(p.slices_sh), per_slice = keep(p.per_slice);
    const int Cout = keep(p.Cout), Cow = keep(p.Cow), floor_acc = keep(p.relu ? 0 : INT32_MIN);
    const int jobs = tile / (kGroupPixels * NT) * slices;
    __syncthreads();
    if (zero_pad && !p.image) {
        for (int e = tid; e < kChannels * p.taps; e += n_threads) {
            const int r = e / p.taps, tap = e - r * p.taps;
            int ones = 0;
            for (int k = 0; k < Cw; ++k) ones += __popc(sW[r * pitch + tap * Cw + k]);  // reversing bits keeps their number
            sTap[e] = p.Cin - 2 * ones;
        }
    }

    // ---- activations, once the previous kernel is done ---------------------------------------------------
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int e = tid;;) {
        if (copy_ok) {
            if (vec == 4) cp_async_zfill<16>(dst, src, true);
            else if (vec == 2) cp_async_zfill<8>(dst, src, true);
            else cp_async_zfill<4>(dst, src, true);
        }
        e += n_threads;
        if (e >= copies) break;
        copy_ok = activation_copy(e, &src, &dst);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // ---- 128 popcount(a AND w): a warp per (8 NT pixels, slice of K) -------------------------------------------
    const int g = lane >> 2, q = lane & 3;
    const int base = KD - 2 * sOnes[lane];
    for (int job = warp; job < jobs; job += n_warps) {
        const int group = job >> slices_sh, slice = job & (slices - 1);
        int k = 4 * slice * per_slice + q;
        const int k_end = 4 * min(steps, (slice + 1) * per_slice);
        const int px = group * (kGroupPixels * NT) + g;
        const uint32_t *w = sW + g * pitch;
        const uint32_t *a[NT];
        constexpr int kSets = NT == 1 ? 2 : 1;  // sets of sums: an instruction waits 23 clocks for the one before it on the same set
        int acc[kSets][2][NT][4] = {}, ones[NT] = {};
#pragma unroll
        for (int i = 0; i < NT; ++i) a[i] = sRaw + sPx[px + 8 * i];
        // the words of the next step are on their way while the matrix instructions of this one run
        uint32_t wv[4], av[NT];
        const auto fetch = [&](int kk, uint32_t (&wn)[4], uint32_t (&an)[NT]) {
            const int offset = sK[kk];
#pragma unroll
            for (int i = 0; i < 4; ++i) wn[i] = w[8 * i * pitch + kk];
#pragma unroll
            for (int i = 0; i < NT; ++i) an[i] = kk < K ? a[i][offset] : 0u;
        };
        if (k < k_end) fetch(k, wv, av);
        while (k < k_end) {
            uint32_t wn[4], an[NT];
            k += 4;
            fetch(min(k, 4 * steps - 4 + q), wn, an);
#pragma unroll
            for (int i = 0; i < NT; ++i) ones[i] += __popc(av[i]);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const uint32_t w_lo = 0x80808080u >> t, w_hi = 0x08080808u >> t;  // reversed bits t and t + 4 of every byte
                const uint32_t a_lo = 0x01010101u << t, a_hi = 0x10101010u << t;
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        mma_u8(acc[t & (kSets - 1)][j][i], wv[2 * j] & w_lo, wv[2 * j + 1] & w_lo, wv[2 * j] & w_hi, wv[2 * j + 1] & w_hi, av[i] & a_lo, av[i] & a_hi);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) wv[i] = wn[i];
#pragma unroll
            for (int i = 0; i < NT; ++i) av[i] = an[i];
        }
        // rows of the result are channels (g, g + 8), columns pixels (2 q, 2 q + 1)
        int32_t *red = sRed + (group * (kGroupPixels * NT) + 2 * q) * kRedPitch + g;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                int32_t *r = red + 8 * i * kRedPitch + 16 * j;
                atomicAdd(r, acc[0][j][i][0] + (kSets == 2 ? acc[kSets - 1][j][i][0] : 0));
                atomicAdd(r + kRedPitch, acc[0][j][i][1] + (kSets == 2 ? acc[kSets - 1][j][i][1] : 0));
                atomicAdd(r + 8, acc[0][j][i][2] + (kSets == 2 ? acc[kSets - 1][j][i][2] : 0));
                atomicAdd(r + kRedPitch + 8, acc[0][j][i][3] + (kSets == 2 ? acc[kSets - 1][j][i][3] : 0));
            }
            ones[i] += __shfl_xor_sync(0xffffffffu, ones[i], 1);
            ones[i] += __shfl_xor_sync(0xffffffffu, ones[i], 2);
            if (q == 0) atomicAdd(&sPop[px + 8 * i], ones[i]);
        }
    }
    __syncthreads();

    // ---- output transform (Section 3.2): lane = channel, a warp per pixel ----------------------------------
    const int pixels = min(tile, M - m0);
    for (int t = warp; t < pixels; t += n_warps) {
        const int m = m0 + t;
        int acc = base - 2 * sPop[t] + (sRed[t * kRedPitch + lane] >> 5);
        if (zero_pad)  // taps outside the image counted as +1 * w; take them out again
            for (uint32_t outside = sOutside[t]; outside; outside &= outside - 1) acc -= sTap[lane * p.taps + __ffs(outside) - 1];
        if (MODE == SMALL_BITS) {
            const uint32_t word = __ballot_sync(0xffffffffu, acc < limit);
            if (lane == 0) static_cast<uint32_t *>(out)[(int64_t)m * Cow + blockIdx.y] = word;
        } else if (MODE == SMALL_FLOAT) {
            const float y = __fmaf_rn((float)max(acc, floor_acc), mult, bias);
            if (ch_ok) static_cast<float *>(out)[(int64_t)m * Cout + channel] = y;
        } else if (p.out_type == LCE_OUT_INT32) {
            if (ch_ok) static_cast<int32_t *>(out)[(int64_t)m * Cout + channel] = acc;
        } else {
            float y = __fmaf_rn((float)max(acc, floor_acc), mult, bias);
            const int64_t o = (int64_t)m * Cout + channel;
            if (p.residual && ch_ok) y = __fadd_rn(y, p.residual[o]);
            if (out && ch_ok) static_cast<float *>(out)[o] = y;
            if (p.out_packed) {
                const uint32_t word = __ballot_sync(0xffffffffu, ch_ok && y < 0.f);
                if (lane == 0) p.out_packed[(int64_t)m * Cow + blockIdx.y] = word;
            }
        }
    }
}

// ---- load-time weight image ----------------------------------------------------------------------------------
// plain packed words [Cout][K] -> per block of 32 channels: [32][pitch] words with the bits of every byte reversed
// (zero past K and past Cout), [32] popcounts of the rows, [32][taps] per-tap weight sums (for zero-padding); and the
// plain words themselves to the front of the packed buffer, which as a copy of its own was one more operation on the
// stream for each layer of a model.  A sum is a warp's: a thread that adds up a whole row waits for one load after
// another (512 channels 3x3: 9.2 us, now 4.8 with the copy).  Packing seventeen 3x3 layers of 32 - 512 channels through
// the binding, all images: 312 -> 243 us (253 without this image, but with the copy apart).
__global__ void small_pack_weights_kernel(const uint32_t *w, uint32_t *plain, uint32_t *image, int Cout, int Cow, int Cin, int Cw, int taps, int pitch)
{
    const int K = taps * Cw, rows_words = kChannels * pitch, block_words = kChannels * (pitch + 1 + taps);
    const int64_t thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = thread; e < (int64_t)Cout * K; e += threads) plain[e] = w[e];
    for (int64_t e = thread; e < (int64_t)Cow * rows_words; e += threads) {
        const int64_t o = e / pitch;   // channel: rows of all blocks one after the other
        const int k = (int)(e - o * pitch), block = (int)(o / kChannels);
        image[(int64_t)block * block_words + (e - (int64_t)block * rows_words)] = o < Cout && k < K ? reverse_in_bytes(w[o * K + k]) : 0u;
    }
    const int lane = threadIdx.x & 31;
    for (int64_t e = thread >> 5; e < (int64_t)Cow * kChannels * (1 + taps); e += threads >> 5) {  // in the order they lie in the image
        const int block = (int)(e / (kChannels * (1 + taps))), i = (int)(e - (int64_t)block * kChannels * (1 + taps));
        const bool whole = i < kChannels;
        const int t = whole ? i : i - kChannels, r = whole ? t : t / taps, first = whole ? 0 : (t - r * taps) * Cw, n = whole ? K : Cw;
        const int64_t o = (int64_t)block * kChannels + r;
        int ones = 0;
        if (o < Cout)
            for (int k = lane; k < n; k += 32) ones += __popc(w[o * K + first + k]);
        ones = __reduce_add_sync(0xffffffffu, ones);
        if (lane == 0) image[(int64_t)block * block_words + rows_words + i] = (uint32_t)(whole ? ones : o < Cout ? Cin - 2 * ones : 0);
    }
}

struct SmallShape {
    int tile, slices, warps, groups;  // pixels per CTA, slices of K, warps, groups of 8 pixels per warp job
    size_t smem;
};

int small_steps(const ConvGeom &g) { return (g.KH * g.KW * g.Cw + 3) / 4; }
// an odd multiple of 4 words: 8 rows x 4 words in 32 banks
int small_pitch(const ConvGeom &g) { return 4 * (small_steps(g) | 1); }
int small_column_words(const ConvGeom &g) { return g.Cw % 8 == 0 ? g.Cw + 4 : g.Cw; }
int small_columns(const ConvGeom &g) { return max((g.OW - 1) * g.sw + g.KW, g.pl + g.W); }

// the padded input rows a tile can touch
int64_t small_raw_words(const ConvGeom &g, int tile)
{
    const int64_t out_rows = (tile + g.OW - 2) / g.OW + 1;   // output rows of a run of `tile` pixels, at most
    const int64_t crossings = (out_rows + g.OH - 2) / g.OH;   // image boundaries among them: windows of two images share no row
    const int64_t rows = (out_rows - 1) * g.sh + crossings * max(0, g.KH - g.sh) + g.KH;
    return (rows * small_columns(g) * small_column_words(g) + 3) / 4 * 4;
}

size_t small_smem(const ConvGeom &g, int tile)
{
    const size_t tap_sums = g.padding == LCE_PAD_SAME_ZERO ? (size_t)kChannels * g.KH * g.KW + tile : 0;
    return 4 * ((size_t)kChannels * (small_pitch(g) + 1) + tap_sums + 4 * (size_t)small_steps(g) + (size_t)tile * (kRedPitch + 2) + (size_t)small_raw_words(g, tile));
}

template <int MODE, int NT>
lce_status launch_small_mode(const SmallParams &p, const SmallShape &shape, cudaStream_t s)
{
    static SmemOptIn opted;
    if (!opted.ensure(bconv_small_kernel<MODE, NT>, shape.smem)) return LCE_ERR_CUDA;
    return launch_dependent(bconv_small_kernel<MODE, NT>, dim3((unsigned)((p.M + shape.tile - 1) / shape.tile), (unsigned)p.Cow), 32 * shape.warps, shape.smem, s, p);
}

struct SmallLaunch {
    SmallParams params;
    SmallShape shape;
};
static_assert(sizeof(SmallLaunch) <= sizeof(PreparedLaunch), "PreparedLaunch too small");

// the activations are copied in pieces of `vec` words
void small_set_vec(SmallParams *p, int vec)
{
    p->vec = vec;
    p->pieces = p->W * p->Cw / vec;
    p->by_pieces = fast_div((uint32_t)p->pieces);
    p->by_px_pieces = fast_div((uint32_t)(p->Cw / vec));
}

void prepare_small_as(const ConvGeom &g, const SmallShape &shape, SmallLaunch *l)
{
    l->shape = shape;
    l->params = SmallParams{};
    SmallParams &p = l->params;
    p.N = g.N; p.H = g.H; p.W = g.W; p.Cw = g.Cw; p.Cin = g.Cin; p.Cout = g.Cout; p.Cow = g.Cow; p.KH = g.KH; p.KW = g.KW; p.taps = g.KH * g.KW;
    p.sh = g.sh; p.sw = g.sw; p.OH = g.OH; p.OW = g.OW; p.pt = g.pt; p.pl = g.pl;
    p.M = (int32_t)g.M; p.K = p.taps * g.Cw; p.KD = p.taps * g.Cin;
    p.Hp = (g.OH - 1) * g.sh + g.KH; p.Wp = small_columns(g); p.PW = small_column_words(g);
    p.steps = small_steps(g); p.pitch = small_pitch(g);
    p.tile = shape.tile; p.slices = shape.slices; p.per_slice = (p.steps + shape.slices - 1) / shape.slices;
    while ((1 << p.slices_sh) < shape.slices) ++p.slices_sh;
    p.raw_words = (int32_t)small_raw_words(g, shape.tile);
    p.padded = g.padding != LCE_PAD_VALID && (g.KH > 1 || g.KW > 1);
    small_set_vec(&p, g.Cw % 4 == 0 ? 4 : g.Cw % 2 == 0 ? 2 : 1);
    p.by_cw = fast_div((uint32_t)g.Cw);
    p.by_kw = fast_div((uint32_t)g.KW); p.by_ow = fast_div((uint32_t)g.OW); p.by_oh = fast_div((uint32_t)g.OH); p.by_hp = fast_div((uint32_t)p.Hp);
    p.zero_pad = g.padding == LCE_PAD_SAME_ZERO; p.out_type = g.out_type; p.relu = g.activation == LCE_ACT_RELU;
}

lce_status launch_small_as(const SmallLaunch &l, const uint32_t *in, const uint32_t *w, const uint32_t *w_image, const float *mult,
                           const float *bias, const int32_t *thr, void *out, cudaStream_t s, const float *residual, uint32_t *out_packed)
{
    SmallParams p = l.params;
    p.in = in; p.w = w_image ? w_image : w; p.image = w_image != nullptr;
    p.mult = mult; p.bias = bias; p.thr = thr; p.residual = residual; p.out = out; p.out_packed = out_packed;
    while (!aligned(in, 4 * (size_t)p.vec)) small_set_vec(&p, p.vec / 2);
    const bool wide = l.shape.groups == 2;
    if (p.out_type == LCE_OUT_BITPACKED) return wide ? launch_small_mode<SMALL_BITS, 2>(p, l.shape, s) : launch_small_mode<SMALL_BITS, 1>(p, l.shape, s);
    if (p.out_type == LCE_OUT_FLOAT32 && !residual && !out_packed)
        return wide ? launch_small_mode<SMALL_FLOAT, 2>(p, l.shape, s) : launch_small_mode<SMALL_FLOAT, 1>(p, l.shape, s);
    return wide ? launch_small_mode<SMALL_GENERAL, 2>(p, l.shape, s) : launch_small_mode<SMALL_GENERAL, 1>(p, l.shape, s);
}

constexpr size_t kSmallSmem = 100 * 1024;  // two CTAs per SM, so that a CTA of the next kernel finds room to prepare itself

// The shape of a launch, by the best of sweeps over tiles, slices and warps on 40 layers (M = 49 .. 50176 pixels,
// 1 .. 16 channel blocks, 1 .. 36 steps): the smallest tile that leaves few enough CTAs (more than two or three
// per SM only repeat the set-up), 8 warps, and as many slices as give every warp a job.  Jobs of 16 pixels use a
// weight operand twice and win in tiles of 32 pixels and more, and where the depth gives enough steps to share out (8 and
// more).  With few steps (below 8, in tiles of 32 below 20) a second slice is enough in tiles of 16 and 32 pixels, even if half
// of the warps then have no job: every job ends in 8 updates of shared sums.  The line at 20 is a compromise, not an edge.  Two
// slices against four in tiles of 32, us at 14, 16, 18, 21, 23, 25, 27 and 30 steps: 10x10 -> 192, 16 images (300 CTAs) 4.9 /
// 5.2, 5.6 / 5.6, 5.6 / 6.0, 6.6 / 7.0, 6.7 / 6.8, 7.5 / 7.8, 7.3 / 7.3, 8.6 / 8.7, and much the same with 265 CTAs;
// 10x10 -> 109, 17 images (216 CTAs) 4.2 / 4.1, 4.7 / 4.4, 4.9 / 4.6, 5.0 / 5.4, 5.1 / 5.2, 5.6 / 5.9, 6.5 / 5.5, 7.3 / 6.6.  One image of 56x56x64 (tiles of 32) 3.3 -> 2.8 us, of 56x56x64 -> 128 at
// stride 2 (16) 2.8 -> 2.5, three of 33x33x100 (32) 4.5 -> 4.2, 53 of 8x8x160, 1x1 (64) 4.1 -> 3.8.
// Tiles of 64 pixels in more CTAs than fit at once do better with four warps each; of 16 pixels they do not (14x14x256,
// three images 3.8 us, 4.9 with four).
SmallShape small_shape(const ConvGeom &g)
{
    const int steps = small_steps(g);
    SmallShape s{8, 1, 8, 1, 0};
    const auto ctas = [&](int tile) { return (g.M + tile - 1) / tile * g.Cow; };
    const auto most_ctas = [&](int tile) { return tile == 8 ? 220 : tile == 16 && steps < 8 ? 300 : 420; };
    while (s.tile < 64 && ctas(s.tile) > most_ctas(s.tile) && small_smem(g, 2 * s.tile) <= kSmallSmem) s.tile *= 2;
    s.groups = s.tile >= 32 || (s.tile == 16 && steps >= 8) ? 2 : 1;
    const int jobs = s.tile / (8 * s.groups);           // of one slice
    const int most = (s.tile == 32 && steps < 20) || (s.tile == 16 && s.groups == 1) || (s.tile == 8 && steps < 32) ? 4 : 8;
    while (s.slices * jobs < most && 2 * s.slices <= steps) s.slices *= 2;
    if (s.tile == 64 && ctas(64) > 400) s.warps = 4;
    s.smem = small_smem(g, s.tile);
    return s;
}

}  // namespace

bool small_covers(const ConvGeom &g)
{
    if (g.padding == LCE_PAD_SAME_ZERO && g.KH * g.KW > 31) return false;  // a pixel's taps outside the image are one word of bits
    return small_smem(g, 8) <= kSmallSmem && g.M < (1ll << 31) - 64 && g.Cow <= 65535 &&
           (int64_t)g.N * ((int64_t)(g.OH - 1) * g.sh + g.KH) < (1ll << 31) && (int64_t)g.KH * g.KW * g.Cin < (1 << 23);
}

// CTAs of a launch
int64_t small_ctas(const ConvGeom &g)
{
    const SmallShape s = small_shape(g);
    return (g.M + s.tile - 1) / s.tile * g.Cow;
}

void small_plan_info(const ConvGeom &g, TiledPlanInfo *info)
{
    const SmallShape s = small_shape(g);
    *info = TiledPlanInfo{};
    info->pointwise = g.KH == 1 && g.KW == 1;
    info->warps_per_cta = s.warps;
    info->tile_pixels = s.tile;
    info->ctas = (int32_t)((g.M + s.tile - 1) / s.tile * g.Cow);
    info->shared_bytes = (int64_t)s.smem;
}

size_t small_weight_image_bytes(const ConvGeom &g)
{
    return covers_some_padding(g, small_covers) ? (size_t)g.Cow * kChannels * (small_pitch(g) + 1 + g.KH * g.KW) * 4 : 0;
}

lce_status launch_pack_weights_small(const ConvGeom &g, const uint32_t *w, uint32_t *plain, uint32_t *image, cudaStream_t s)
{
    const int taps = g.KH * g.KW, pitch = small_pitch(g);
    const int64_t words = (int64_t)g.Cow * kChannels * pitch, sums = (int64_t)g.Cow * kChannels * (1 + taps);
    const int64_t blocks = max((words + 255) / 256, (sums + 7) / 8);  // a word per thread, a sum per warp
    small_pack_weights_kernel<<<(unsigned)min(blocks, (int64_t)148 * 8), 256, 0, s>>>(w, plain, image, g.Cout, g.Cow, g.Cin, g.Cw, taps, pitch);
    return launch_status();
}

lce_status prepare_bconv_small(const ConvGeom &g, PreparedLaunch *prepared)
{
    if (!small_covers(g)) return LCE_ERR_UNSUPPORTED;
    prepare_small_as(g, small_shape(g), reinterpret_cast<SmallLaunch *>(prepared->bytes));
    return LCE_OK;
}

lce_status launch_bconv_small(const PreparedLaunch &prepared, const uint32_t *in, const uint32_t *w, const uint32_t *w_image, const float *mult,
                              const float *bias, const int32_t *thr, void *out, cudaStream_t s, const float *residual, uint32_t *out_packed)
{
    return launch_small_as(*reinterpret_cast<const SmallLaunch *>(prepared.bytes), in, w, w_image, mult, bias, thr, out, s, residual, out_packed);
}

}  // namespace lce
