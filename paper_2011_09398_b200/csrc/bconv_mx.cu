// LceBConv2d on the 5th-generation tensor cores with 4-bit operands (tcgen05 kind::mxf4, accumulators
// in TMEM).  The +-1 multiply-accumulate of the paper's binary GEMM (Section 2: dot = K - 2 popcount(a
// XOR w); Section 3.2, LceBConv2d) is an exact contraction in any number format that holds +1, -1 and
// 0: e2m1 holds all three in four bits, block scales of 1.0 change nothing, and the fp32 accumulator
// is exact for |sum| < 2^24.  One instruction multiplies 128 x N x 64 values, twice the depth of an
// 8-bit instruction for the same operand bytes, and a zero operand gives the paper's zero-padding
// variant and the channel padding without any correction term.
//
// The packed bits stay the storage and transfer format (32x smaller, Section 3.2).  A 32-bit word
// of activations or weights becomes one 16-byte row chunk of 32 e2m1 values in shared memory:
// nibble = 0x2 (+1.0) | bit << 3 (sign), four shift-and-mask operations per word; pad channels of
// the weights and, for zero-padding, pad pixels are the nibble 0 (0.0).
//
// Implicit GEMM, D[channel][position] = W[channel][k] * X[position][k]^T, M = 128 output channels (TMEM
// lanes), N = a tile of up to 224 grid positions (TMEM columns), K = 64 per instruction:
//   * positions: the images are stacked into one grid of row pitch Wg and Hg rows per image.  For
//     stride 1 the pixel (y, x) sits at (y + pad_top, x + pad_left) and rows / images share their pad
//     positions (the right pad of a row is the left pad of the next); output (oh, ow) is the
//     position of its window's top-left corner and tap (ky, kx) reads position + ky * Wg + kx.  For
//     stride 2 the padded image is split into four phase grids (row parity x column parity), in
//     which tap (ky, kx) of output (oh, ow) is position + (ky / 2) * Wg + kx / 2 of phase
//     (ky % 2, kx % 2).  Positions that are no output (pad columns, pad rows) are computed and dropped.
//   * shared memory holds, per phase, [channel word][position][16 bytes]: the B operand of a tap is
//     the same buffer shifted by the tap's position offset (K-major, no swizzle, rows 16 bytes
//     apart), so every staged position is expanded once for all taps.  T consecutive tiles share one
//     buffer of T * Nt + halo rows, so the halo a tile reads beyond its own positions is staged once
//     per T tiles; there are two to four such buffers (as many as shared memory has room for, up to what
//     lets the loaders run four tiles ahead), one where a CTA has no second super-tile.
//   * K is the taps' channel words, 32 values each, two to an instruction (mx_word): the two chunks of its B operand are
//     rows of one buffer any distance apart, so the last words of an odd count pair up across taps.  A word of zeros
//     per tap instead cost 9 MMAs for 9 words (32 channels, 3x3; now 5) and 75 for 125 (160 channels, 5x5; now 63:
//     32x32x160, 64 images, float 36.4 -> 33.3 us).
//   * the weights were expanded when the model was loaded (lce_bconv2d_pack_weights) into the exact
//     operand image [channel block][pair of words][2][128 channels][16 bytes] (for out_c <= 64 the
//     channel block is repeated down the 128 rows, so that every TMEM lane quarter holds values a
//     finisher warp can work on); the bulk-copy engine brings pairs into a ring of shared-memory stages
//     (cp.async.bulk + mbarrier transaction count).  If every pair fits they are fetched once per CTA,
//     all counted on one barrier; otherwise they stream past once per tile, in groups of pairs that
//     alternate between two stages (one copy, one wait and one commit per group).
//   * roles: 8 loader warps (prefetch the packed words of the next chunk with cp.async, expand the
//     current one), one warp that issues the MMAs (all lanes run the same code, the elected lane
//     issues), one warp that feeds the weight ring and, once the weights are resident, issues the MMAs
//     of every other tile, 16 finisher warps (tcgen05.ld, output transform, stores).  Two accumulator
//     buffers: the MMAs of tile t and the output transform of tile t-1 overlap, and the loaders run up
//     to four tiles ahead of the finished MMAs (rings of four barriers).  The roles meet only through
//     mbarriers; every wait is bounded by time, after which the kernel records a status, waits (bounded)
//     for what it has in flight, frees its TMEM and returns.
//   * output transform (Section 3.2): a TMEM lane is a channel and a column a position.  Bit-packed
//     output: the sign of (accumulator - threshold) of 32 positions per lane, then a 32 x 32 bit
//     transpose across the warp gives each lane the finished word of one pixel.  Float / int32 output
//     is written straight from the registers: per position a warp stores its 32 consecutive channels as
//     one 128-byte line.
//   * few output channels on grids that fill the SMs go with the operands exchanged, positions on the TMEM lanes: a kernel of its own
//     (bconv_mx_positions.cuh) on the same loaders, weight image and grid, four issuers, no weight ring; mx_positions_pay draws the line.
//   * launched with programmatic stream serialization, dependents released at kernel entry: set-up and
//     the weight copies may overlap the tail of the previous kernel of the stream; activations, shortcut
//     and outputs are touched only after griddepcontrol.wait.
#include <atomic>
#include <math.h>
#include <mutex>
#include <stdlib.h>
#include <string.h>

#include "common.cuh"
#include "mx_columns.cuh"
#include "mx_common.cuh"
#include "mx_rings.cuh"

namespace lce {
namespace {

constexpr int kFinishers = 512;                              // warps 0-15 (warp % 4 = TMEM lane quarter, four column groups)
constexpr int kLoaders = 256;                                // warps 16-23
constexpr int kMxThreads = kFinishers + kLoaders + 64;       // + MMA issuer warp + weight producer warp
constexpr int kIssuerWarp = (kFinishers + kLoaders) / 32;
constexpr int kProducerTid = (kIssuerWarp + 1) * 32;
static_assert(kColGroups == kFinishers / 128, "finisher warps per TMEM lane quarter");
constexpr int kMaxNt = 224;                                  // tile width (positions); two accumulators + scales fit 512 columns
constexpr uint32_t kD1Col = 240;                             // TMEM column of the second accumulator buffer
constexpr uint32_t kSfaCol = 480, kSfbCol = 496;             // block scales (all 1.0) of the A / B operand
constexpr int kMaxTaps = 64;
constexpr int kPairBytes = 4096;                             // weights of an MMA: two words of K, 128 rows, 16 bytes each
constexpr int kMaxStages = 32;
// shared-memory map (bytes)
constexpr int kOffBars = 0;          // full_x[4] tile_done[4] full_d[2] empty_d[2] done[2] scales full_w[32] empty_w[32]
constexpr int kOffSlot = 1000;       // TMEM base address; 1004 fills issued, 1008 fills consumed
constexpr int kOffPix = 1024;        // int32[16][2][32]: for every finisher warp the output pixels (or offsets) of the positions it works on, two chunks of a tile at most; int32[32]: -1
constexpr int kOffDyn = 5248;       // raw words, uint2[MMAs of a tile]: operand offsets (A, B; 16-byte units), weight ring, position buffers

enum { BAR_FULL_X0 = 0, BAR_FULL_X3 = 3, BAR_TILE_DONE0, BAR_TILE_DONE3 = BAR_TILE_DONE0 + 3, BAR_FULL_D0, BAR_FULL_D1, BAR_EMPTY_D0, BAR_EMPTY_D1, BAR_DONE, BAR_DONE_B,
       BAR_SCALES, BAR_FULL_W0,
       BAR_EMPTY_W0 = BAR_FULL_W0 + kMaxStages, BAR_COUNT = BAR_EMPTY_W0 + kMaxStages };
static_assert((kMaxNt + 31) / 32 <= 2 * kColGroups, "a finisher warp has two chunks of a tile at most");
static_assert(BAR_COUNT * 8 <= kOffSlot, "barriers overlap the TMEM slot");


// ---- what a wait that gave up leaves behind --------------------------------------------------------------
// A device word (read by lce_device_status) and, once it has been set up, a word in mapped host memory
// that the host reads without synchronising: the next call on that device reports LCE_ERR_DEVICE_TIMEOUT.
__device__ int g_mx_status = 0;

__device__ __forceinline__ void mx_report_timeout(int *host_flag)
{
    g_mx_status = 1;
    if (host_flag) {
        *reinterpret_cast<volatile int *>(host_flag) = 1;
        __threadfence_system();
    }
}

constexpr int kFlagDevices = 64;
std::mutex g_flag_mutex;
std::atomic<int *> g_flag_host{nullptr};   // int[kFlagDevices] in mapped, portable host memory
std::atomic<int *> g_flag_dev{nullptr};    // the same array as the devices see it

// Sets the flag array up on first use.  Not a stream operation: must not run while a stream is capturing.
int *mx_flag_array(bool device_view)
{
    int *h = g_flag_host.load(std::memory_order_acquire);
    if (!h) {
        std::lock_guard<std::mutex> lock(g_flag_mutex);
        h = g_flag_host.load(std::memory_order_acquire);
        if (!h) {
            void *mem = nullptr, *dev = nullptr;
            if (cudaHostAlloc(&mem, kFlagDevices * sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
                cudaGetLastError();
                return nullptr;
            }
            memset(mem, 0, kFlagDevices * sizeof(int));
            if (cudaHostGetDevicePointer(&dev, mem, 0) != cudaSuccess) {
                cudaGetLastError();
                cudaFreeHost(mem);
                return nullptr;
            }
            g_flag_dev.store(static_cast<int *>(dev), std::memory_order_release);
            g_flag_host.store(static_cast<int *>(mem), std::memory_order_release);
            h = static_cast<int *>(mem);
        }
    }
    return device_view ? g_flag_dev.load(std::memory_order_acquire) : h;
}

int current_device_index()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kFlagDevices) return -1;
    return dev;
}

// the current device's flag as a kernel argument; null while it cannot be set up (a capturing stream)
int *mx_flag_for_launch(cudaStream_t s)
{
    const int dev = current_device_index();
    if (dev < 0) return nullptr;
    if (!g_flag_host.load(std::memory_order_acquire)) {
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) {
            cudaGetLastError();
            return nullptr;
        }
    }
    int *arr = mx_flag_array(true);
    return arr ? arr + dev : nullptr;
}

// an advance by a fixed number of grid positions
struct MxStep {
    int n, r, c;
};

struct MxParams {
    const uint32_t *in;
    const uint8_t *wimg;
    const float *mult;
    const float *bias;
    const int32_t *thr;
    void *out;
    const float *residual;   // fused shortcut (float output), or null
    uint32_t *out_packed;    // fused LceQuantize of the float result, or null
    int *host_flag;          // host-mapped word set when a wait gives up, or null
    int32_t N, H, W, Cw, Cout, Cow;
    int32_t OH, OW, KH, KW, stride, pt, pl, K;
    int32_t Wg, Hg, n_phase;
    uint32_t Wg_mul, Wg_sh, Hg_mul, Hg_sh;                // divisions by Wg, Hg as multiply + shift
    MxStep step_across, step_tile;                        // kLoaders positions; to the next tile of a super-tile
    MxStep step_chunk_first, step_chunk_super;            // from a super-tile's first chunk to its second; from its last one to the next super-tile's first
    int32_t Nt, P;           // tile width; rows of a position buffer per phase and channel word = T * Nt + halo
    int32_t T, halo;         // tiles that share a position buffer; positions a tile reads beyond its own
    int32_t n_tiles, n_super, total_q;
    int32_t pairs, stages, resident;
    int32_t group_pairs, groups;  // streamed weights: pairs per ring stage, stages' worth of pairs per tile = ceil(pairs / group_pairs)
    int32_t x_bytes;
    int32_t n_xbuf, ahead;   // position buffers (1..4); tiles the loaders may be ahead of the finished MMAs (2..4)
    int32_t off_tbl, off_w, off_x;    // byte offsets in shared memory
    int32_t cp_words;        // words per cp.async: 4, 2 or 1
    int32_t pad_zero, out_type, activation, write_float;
    uint32_t even_mul, even_sh;            // divisions by the even number of channel words, as multiply + shift
    uint16_t tap_rows[kMaxTaps];           // first row of a tap's words in a position buffer, taps in the order of mx_word
    int32_t dup_log2;        // log2 of the copies of the channel block in the 128 rows: 1 for out_c <= 64, 2 for out_c <= 32, else 0
};

// ---- loaders --------------------------------------------------------------------------------------------
// A grid position as image, grid row inside the image and grid column; a thread's positions advance by a few
// fixed numbers of positions (to the next chunk, the next super-tile, its next position of a chunk), so the
// coordinates are carried along with two compares instead of being divided out of the position every time (two
// 64-bit multiply-shift divisions per position and one more pair per output column were most of a loader's
// instructions: a tile of a 64-channel layer took 2550 clocks, its matrix instructions 1320).
struct MxPos {
    int n, r, c;
};

__device__ __forceinline__ void mx_advance(MxPos &a, const MxStep &d, int Wg, int Hg)
{
    a.c += d.c;
    a.r += d.r;
    a.n += d.n;
    if (a.c >= Wg) { a.c -= Wg; ++a.r; }
    if (a.r >= Hg) { a.r -= Hg; ++a.n; }
}

__device__ __forceinline__ MxPos mx_position(int f, const MxParams &p)
{
    MxPos a;
    const int row = fast_div(f, p.Wg_mul, p.Wg_sh);
    a.c = f - row * p.Wg;
    a.n = fast_div(row, p.Hg_mul, p.Hg_sh);
    a.r = row - a.n * p.Hg;
    return a;
}

// What the loader threads keep in registers for the whole kernel (kernel parameters read inside their loops
// cost more than the arithmetic).
struct MxLoad {
    int N, H, W, Cw, Wg, Hg, P, pt, pl, origin;  // origin: the words from pixel (-pt, -pl) to pixel (0, 0)
    int col_words, row_words, image_words;       // words between positions of a grid column, row and image
    const uint32_t *in;
    MxStep across;                               // kLoaders positions
};

// How a position's words are brought in and expanded.  CW: channel words, 0 = any number, read in pieces of
// cp_words.  FORM: stride 1; stride 2 with its four phases one by one; stride 2 where image width and left pad
// are even, so that the pixels of the two column phases are neighbours in memory (one copy of 2 CW words).
enum { MX_S1 = 0, MX_S2 = 1, MX_S2_PAIR = 2 };

template <int CW>
__device__ __forceinline__ void mx_copy_words(uint32_t *dst, const uint32_t *src, int words, int cp_words, bool ok)
{
    if (CW == 1) {
        cp_async_zfill<4>(dst, src, ok);
    } else if (CW == 2) {
        cp_async_zfill<8>(dst, src, ok);
    } else if (CW > 2) {
#pragma unroll
        for (int w = 0; w < CW; w += 4) cp_async_zfill<16>(dst + w, src + w, ok);
    } else if (cp_words == 4) {
        for (int w = 0; w < words; w += 4) cp_async_zfill<16>(dst + w, src + w, ok);
    } else if (cp_words == 2) {
        for (int w = 0; w < words; w += 2) cp_async_zfill<8>(dst + w, src + w, ok);
    } else {
        for (int w = 0; w < words; ++w) cp_async_zfill<4>(dst + w, src + w, ok);
    }
}

// packed words of the chunk's `count` positions, of which this thread's first is `a` -> raw (pad positions:
// zero words), asynchronously; raw holds the phases of a position one after the other.  One buffer is enough: every
// thread fetches only into places whose words it has itself just expanded.
template <int CW, int FORM>
__device__ __forceinline__ void mx_prefetch(const MxLoad &l, MxPos a, int count, uint32_t *raw, int ltid, int cp_words)
{
    const int cw = CW ? CW : l.Cw;
    for (int j = ltid; j < count; j += kLoaders) {
        const bool image = a.n < l.N;
        if (FORM == MX_S1) {
            const bool ok = image && (unsigned)(a.r - l.pt) < (unsigned)l.H && (unsigned)(a.c - l.pl) < (unsigned)l.W;
            const int off = a.n * l.image_words + a.r * l.row_words + a.c * l.col_words - l.origin;
            mx_copy_words<CW>(raw + j * cw, l.in + (ok ? off : 0), cw, cp_words, ok);
        } else {
            const int y = 2 * a.r - l.pt, x = 2 * a.c - l.pl;
            const int off = a.n * l.image_words + 2 * (a.r * l.row_words + a.c * cw) - l.origin;
#pragma unroll
            for (int py = 0; py < 2; ++py) {
                const bool row_ok = image && (unsigned)(y + py) < (unsigned)l.H;
                uint32_t *dst = raw + (j * 4 + 2 * py) * cw;
                if (FORM == MX_S2_PAIR) {
                    const bool ok = row_ok && (unsigned)x < (unsigned)l.W;  // column phase 0; phase 1 is the next pixel, inside with it
                    mx_copy_words<2 * CW>(dst, l.in + (ok ? off + py * l.row_words : 0), 2 * cw, cp_words, ok);
                } else {
#pragma unroll
                    for (int px = 0; px < 2; ++px) {
                        const bool ok = row_ok && (unsigned)(x + px) < (unsigned)l.W;
                        mx_copy_words<CW>(dst + px * cw, l.in + (ok ? off + py * l.row_words + px * cw : 0), cw, cp_words, ok);
                    }
                }
            }
        }
        mx_advance(a, l.across, l.Wg, l.Hg);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// one phase of a position: cw words from src -> cw chunks of 16 bytes, P positions apart
template <int CW>
__device__ __forceinline__ void mx_expand_phase(uint4 *dst, int P, const uint32_t *src, int words, bool zero)
{
    if (CW == 0) {
        for (int k = 0; k < words; ++k) {
            uint4 v = mx_expand_word(src[k]);
            if (zero) v = make_uint4(0u, 0u, 0u, 0u);
            dst[k * P] = v;
        }
        return;
    }
    uint32_t w[CW ? CW : 1];
    if (CW == 1) {
        w[0] = *src;
    } else if (CW == 2) {
        const uint2 q = *reinterpret_cast<const uint2 *>(src);
        w[0] = q.x; w[1] = q.y;
    } else {
#pragma unroll
        for (int k = 0; k < CW; k += 4) {
            const uint4 q = *reinterpret_cast<const uint4 *>(src + k);
            w[k] = q.x; w[k + 1] = q.y; w[k + 2] = q.z; w[k + 3] = q.w;
        }
    }
#pragma unroll
    for (int k = 0; k < CW; ++k) {
        uint4 v = mx_expand_word(w[k]);
        if (zero) v = make_uint4(0u, 0u, 0u, 0u);
        dst[k * P] = v;
    }
}

// The chunk's words -> e2m1 in the position buffer, from row `lo` on.  Every thread expands the words it
// prefetched itself (same item mapping): waiting for its own copies is enough.  With zero-padding the positions
// outside the image become 0.0; `a` is the thread's first position again.
template <int CW, int FORM>
__device__ __forceinline__ void mx_expand(const MxLoad &l, MxPos a, int count, const uint32_t *raw, uint4 *X, int plane, int ltid, bool pad_zero)
{
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int cw = CW ? CW : l.Cw;
    for (int j = ltid; j < count; j += kLoaders) {
        bool zero_y[2] = {false, false}, zero_x[2] = {false, false};
        if (pad_zero) {
            const int y = FORM == MX_S1 ? a.r - l.pt : 2 * a.r - l.pt, x = FORM == MX_S1 ? a.c - l.pl : 2 * a.c - l.pl;
#pragma unroll
            for (int k = 0; k < (FORM == MX_S1 ? 1 : 2); ++k) {
                zero_y[k] = a.n >= l.N || (unsigned)(y + k) >= (unsigned)l.H;
                zero_x[k] = (unsigned)(x + k) >= (unsigned)l.W;
            }
            mx_advance(a, l.across, l.Wg, l.Hg);
        }
        if (FORM == MX_S1) {
            mx_expand_phase<CW>(X + j, l.P, raw + j * cw, cw, zero_y[0] || zero_x[0]);
        } else {
#pragma unroll
            for (int ph = 0; ph < 4; ++ph)
                mx_expand_phase<CW>(X + ph * plane + j, l.P, raw + (j * 4 + ph) * cw, cw, zero_y[ph >> 1] || zero_x[ph & 1]);
        }
    }
}

// which form the loaders use: channel words (0 = any) + 32 * FORM
__device__ __forceinline__ int mx_form(const MxParams &p)
{
    const bool words_ok = (p.Cw == 1) || (p.Cw == 2 && p.cp_words >= 2) || ((p.Cw == 4 || p.Cw == 8 || p.Cw == 16) && p.cp_words == 4);
    if (p.n_phase == 1) return words_ok && p.Cw >= 2 ? p.Cw : 0;
    const bool pairs = (p.W & 1) == 0 && (p.pl & 1) == 0 && (reinterpret_cast<uintptr_t>(p.in) & 15) == 0 && words_ok && p.Cw <= 4;
    return pairs ? 32 * MX_S2_PAIR + p.Cw : words_ok && p.Cw == 8 ? 32 * MX_S2 + 8 : 32 * MX_S2;
}

// a loader's registers; the form
__device__ __forceinline__ int mx_load_setup(const MxParams &p, MxLoad &ld)
{
    ld.N = p.N; ld.H = p.H; ld.W = p.W; ld.Cw = p.Cw; ld.Wg = p.Wg; ld.Hg = p.Hg; ld.P = p.P; ld.pt = p.pt; ld.pl = p.pl;
    ld.in = p.in;
    ld.col_words = p.Cw;
    ld.row_words = p.W * p.Cw;
    ld.image_words = p.H * ld.row_words;
    ld.origin = p.pt * ld.row_words + p.pl * p.Cw;
    if (p.stride == 2 && p.n_phase == 1) {  // 1x1: every second pixel of every second row, none of them padding
        ld.H = p.OH; ld.W = p.OW;
        ld.col_words *= 2;
        ld.row_words *= 2;
    }
    ld.across = p.step_across;
    return mx_form(p);
}

#define LCE_MX_FORMS(CALL)                                                                                                       \
    switch (form) {                                                                                                             \
        case 2: CALL(2, MX_S1); break;                                                                                          \
        case 4: CALL(4, MX_S1); break;                                                                                          \
        case 8: CALL(8, MX_S1); break;                                                                                          \
        case 16: CALL(16, MX_S1); break;                                                                                        \
        case 32 * MX_S2 + 8: CALL(8, MX_S2); break;                                                                             \
        case 32 * MX_S2: CALL(0, MX_S2); break;                                                                                 \
        case 32 * MX_S2_PAIR + 1: CALL(1, MX_S2_PAIR); break;                                                                   \
        case 32 * MX_S2_PAIR + 2: CALL(2, MX_S2_PAIR); break;                                                                   \
        case 32 * MX_S2_PAIR + 4: CALL(4, MX_S2_PAIR); break;                                                                   \
        default: CALL(0, MX_S1); break;                                                                                         \
    }

// The loaders' loop over the CTA's tiles: expand the chunk whose words have arrived, hand the tile to the issuer, and only then ask for the words of the next chunk
// (the tile's MMAs must not wait for loads they do not need).  False when a wait gave up.
template <int CW, int FORM>
__device__ __forceinline__ bool mx_load_tiles(const MxParams &p, const MxLoad &l, MxPos stage, uint64_t *bars, uint32_t *raw0, uint8_t *sX0,
                                              int tid, int first_tile, int tile_step)
{
    const int Nt = p.Nt, T = p.T, halo = p.halo, n_tiles = p.n_tiles, n_super = p.n_super, n_xbuf = p.n_xbuf, ahead = p.ahead;
    const int plane = p.Cw * p.P, cp_words = p.cp_words;
    const uint32_t x_bytes = (uint32_t)p.x_bytes;
    const bool pad_zero = p.pad_zero != 0;
    const MxStep tile_d = p.step_tile, chunk_first = p.step_chunk_first, chunk_super = p.step_chunk_super;
    int it = 0, xbuf = 0;
    for (int st = first_tile; st < n_super; st += tile_step, xbuf = xbuf + 1 == n_xbuf ? 0 : xbuf + 1) {
        uint4 *X = reinterpret_cast<uint4 *>(sX0 + xbuf * x_bytes);
        for (int k = 0; k < T && st * T + k < n_tiles; ++k, ++it) {
            if (it >= ahead) {
                // At most `ahead` tiles in front of the finished MMAs: those of tile it - ahead are done (a
                // ring of four barriers, one commit per tile).  That keeps the arrivals on the four full_x
                // barriers within one phase of what the issuer has seen, and (the MMAs finish in order; with more than one
                // super-tile ahead <= (n_xbuf - 1) * T + 1) it means that the super-tile whose position buffer this chunk
                // overwrites has been read completely.
                const int done = it - ahead;
                if (!mbar_wait_bounded(&bars[BAR_TILE_DONE0 + (done & 3)], (uint32_t)(done >> 2) & 1u)) return false;
            }
            mx_expand<CW, FORM>(l, stage, k ? Nt : Nt + halo, raw0, X + (k ? k * Nt + halo : 0), plane, tid, pad_zero);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&bars[BAR_FULL_X0 + (it & 3)]);
            const bool more_here = k + 1 < T && st * T + k + 1 < n_tiles;
            if (more_here || st + tile_step < n_super) {
                mx_advance(stage, !more_here ? chunk_super : k ? tile_d : chunk_first, l.Wg, l.Hg);
                mx_prefetch<CW, FORM>(l, stage, more_here ? Nt : Nt + halo, raw0, tid, cp_words);
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    return true;
}

// The order of K: word i of an output's taps x Cw words, as a tap (row, column) and a channel word.  Taps by their place
// in a position buffer, which for stride 2 is phase by phase; every tap's channel words two by two; where their number
// is odd, the taps' last ones at the end.  Two words of a pair are then one behind the other in the buffer (the distance
// in the operand descriptor has no sign), and pairs are as few as the words allow.
struct MxWord {
    int ky, kx, cw;
};

__host__ __device__ __forceinline__ MxWord mx_word(int i, int KH, int KW, int Cw, int stride)
{
    const int even = Cw & ~1, paired = KH * KW * even;
    MxWord w;
    int tap = i < paired ? i / even : i - paired;
    w.cw = i < paired ? i - tap * even : Cw - 1;
    if (stride == 1) {
        w.ky = tap / KW;
        w.kx = tap - w.ky * KW;
        return w;
    }
    w.ky = w.kx = 0;
    for (int phase = 0; phase < 4; ++phase) {
        const int py = phase >> 1, px = phase & 1, rows = (KH - py + 1) / 2, cols = (KW - px + 1) / 2;
        if (tap < rows * cols) {
            w.ky = py + 2 * (tap / cols);
            w.kx = px + 2 * (tap % cols);
            break;
        }
        tap -= rows * cols;
    }
    return w;
}

// its first row in a position buffer, in 16-byte units: the tap's (worked out on the host: dividing it out here, from cold
// code, took 0.2 us of every launch) in the plane of its channel word
__device__ __forceinline__ uint32_t word_b_offset(const MxParams &p, int i, int even, int paired)
{
    const int tap = i < paired ? fast_div(i, p.even_mul, p.even_sh) : i - paired;
    return p.tap_rows[tap] + (uint32_t)((i < paired ? i - tap * even : even) * p.P);
}

// One lane of the converged warp, the same one every time
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(pred));
    return pred != 0;
}

// One MMA, by one lane.  Descriptors: low words a and b, the same high word
__device__ __forceinline__ void mx_mma(uint32_t tmem_d, uint32_t a, uint32_t b, uint32_t desc_hi, uint32_t idesc, uint32_t sfa, uint32_t sfb, bool accumulate)
{
    asm volatile(
        "{\n\t.reg .pred pa;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 pa, %7, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\t mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], da, db, %4, [%5], [%6], pa;\n\t}"
        :
        : "r"(tmem_d), "r"(a), "r"(b), "r"(desc_hi), "r"(idesc), "r"(sfa), "r"(sfb), "r"((uint32_t)accumulate)
        : "memory");
}

// The MMAs of a table of operand offsets, in one loop of the elected lane.  The issuer's code comes by once per tile, while 24
// other warps of the SM run loops of their own, so it is fetched anew every time: what bounds it is its length (blocks of 8, 4, 2
// and 1 MMAs written out, all lanes of the warp with them, took 100 clocks an MMA where the tensor pipe needs 50 - 105).
// Eight a turn: 64 images of 7x7x512 float 9.2 -> 8.4 us, 256 of 14x14x256 -> 512 at stride 2 18.3 -> 17.3, 64 of 32x32x160
// 5x5 bits 28.0 -> 26.5; with one a turn these take 9.2, 19.3 and 27.1, and 28x28x128 7.6 instead of 7.1; with two it is 7.8, 17.8
// and 26.2, but 28x28x128 float 9.2 instead of 9.05.  What is left of a turn goes four at once, then one by one: 14x14x256, 1x1, one image
// (four instructions) float 3.51 -> 3.37 us, 64 images 5.66 -> 5.50, 64 of 32x32x160 5x5 bits 25.87 -> 25.74.
__device__ __forceinline__ void mx_issue_table(uint32_t tmem_d, const uint2 *tbl, int count, uint32_t a_base, uint32_t b_base, uint32_t desc_hi,
                                               uint32_t idesc, uint32_t sfa, uint32_t sfb, uint32_t &accumulate)
{
    if (elect_one()) {
        const auto mma = [&](int i) {
            const uint2 o = tbl[i];
            mx_mma(tmem_d, a_base + o.x, b_base + o.y, desc_hi, idesc, sfa, sfb, accumulate || i > 0);
        };
        int i = 0;
#pragma unroll 1
        for (; i + 8 <= count; i += 8) {
#pragma unroll
            for (int k = 0; k < 8; ++k) mma(i + k);
        }
        if (count & 4) {
#pragma unroll
            for (int k = 0; k < 4; ++k) mma(i + k);
            i += 4;
        }
#pragma unroll 1
        for (; i < count; ++i) mma(i);
    }
    accumulate = 1;
}

// Two additions in one instruction
__device__ __forceinline__ void add_pair(float &x, float &y, float c)
{
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %2};\n\tadd.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}" : "+f"(x), "+f"(y) : "f"(c));
}

// 32 x 32 bit transpose across the warp: in: lane = row, bit j = column j; out: lane j holds column j.
// Five butterfly steps; in step k a lane keeps the bits under its mask and takes the others from its
// partner's word rotated by k towards them (the bits that wrap around fall under the kept mask).  The
// per-lane masks and rotation counts are worked out once per warp: a step is one shuffle, one funnel shift
// and one three-input logic operation, the first two (whole bytes) one shuffle and one byte permutation.
struct Transpose32 {
    uint32_t bytes[2];  // byte selectors of the steps k = 16, 8
    uint32_t keep[3];   // bits this lane keeps in the steps k = 4, 2, 1
    uint32_t rot[3];    // left-rotation of the partner's word
};

__device__ __forceinline__ Transpose32 transpose32_setup(int lane)
{
    // a lane without bit k keeps its low halves and takes the partner's low halves moved up by k;
    // a lane with bit k keeps its high halves and takes the partner's high halves moved down by k
    Transpose32 t;
    t.bytes[0] = (lane & 16) ? 0x3276u : 0x5410u;
    t.bytes[1] = (lane & 8) ? 0x3715u : 0x6240u;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int k = 4 >> i;
        const uint32_t low = k == 4 ? 0x0F0F0F0Fu : k == 2 ? 0x33333333u : 0x55555555u;
        t.keep[i] = (lane & k) ? ~low : low;
        t.rot[i] = (lane & k) ? 32u - (uint32_t)k : (uint32_t)k;
    }
    return t;
}

__device__ __forceinline__ uint32_t warp_transpose32(uint32_t m, const Transpose32 &t)
{
    m = __byte_perm(m, __shfl_xor_sync(0xffffffffu, m, 16), t.bytes[0]);
    m = __byte_perm(m, __shfl_xor_sync(0xffffffffu, m, 8), t.bytes[1]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, m, 4 >> i);
        const uint32_t moved = __funnelshift_l(y, y, t.rot[i]);
        m = (m & t.keep[i]) | (moved & ~t.keep[i]);
    }
    return m;
}

// The finishers.  All transforms take the accumulator 16 columns at a time (32 left no register free: the bit-packed one
// spilled), know their positions' output pixels before the accumulator is there, and do one compare a position.  Instructions
// bound the thin layers (5900 a tile of 208 positions on 56x56x64): 64 channels, 56x56, 64 images, float 14.0 -> 13.8 us; 256 images,
// bits, 28.4 -> 26.5 (a layer that has gone to bconv_mx_positions.cuh since: 21.8).  Setting the accumulators to minus the threshold beforehand (tcgen05.st) instead of
// adding it to every value was slower (28.4 -> 36 us): the store waits for the other tile's matrix instructions.
//
// What a finisher warp needs for every tile, worked out once before its tile loop (divisions and
// kernel-parameter reads per tile cost a third of the warp's instructions when they sat in the epilogue).
struct MxFin : MxColumns, MxGrid {
    uint32_t lane_off;       // TMEM lane offset of its quarter
    float minus_thr, mult, bias;  // this lane's channel: minus its threshold (inf if it does not exist), multiplier, bias
    int cout, cow;
    uint32_t *out_words;     // bit-packed output, at this warp's channel word
    float *outp;             // float / int32 output, at this lane's channel
    const float *resp;       // shortcut tensor at this lane's channel, or null
    uint32_t *packp;         // re-quantised copy at this warp's channel word, or null
    bool relu, write_float;
    int lane_step;           // from lane_positions of the first chunk to that of the second
    int32_t *positions;      // shared memory: output pixels or offsets of the two chunks' positions (one array per warp)
    const int32_t *lane_positions;  // the same for this lane; a row of -1 if its channel does not exist
};

__device__ __forceinline__ MxFin mx_fin_context(const MxParams &p, int32_t *sPix, int fw, int lane, int ch0)
{
    MxFin f;
    mx_columns(f, p.Nt, p.Cout, ch0, p.dup_log2, fw);
    const int cq = f.word, channel = ch0 + cq * 32 + lane;
    f.lane_off = (uint32_t)((fw & 3) * 32) << 16;
    const bool ch_ok = channel < p.Cout;
    // this lane's constants straight from global memory (constants of the model, never the previous kernel's
    // output): their latency passes while the first tile is being staged
    f.minus_thr = INFINITY;
    if (ch_ok && p.out_type == LCE_OUT_BITPACKED) {
        // acc < thr is unchanged by clamping thr to [-K-1, K+1] (|acc| <= K), and then thr is exact in fp32
        f.minus_thr = -(float)max(-p.K - 1, min(p.K + 1, __ldg(p.thr + channel)));
    }
    f.mult = (ch_ok && p.out_type == LCE_OUT_FLOAT32) ? __ldg(p.mult + channel) : 0.f;
    f.bias = (ch_ok && p.out_type == LCE_OUT_FLOAT32) ? __ldg(p.bias + channel) : 0.f;
    f.cout = p.Cout;
    f.cow = p.Cow;
    f.out_words = static_cast<uint32_t *>(p.out) + (ch0 >> 5) + cq;
    f.outp = static_cast<float *>(p.out) + channel;
    f.resp = p.residual ? p.residual + channel : nullptr;
    f.packp = p.out_packed ? p.out_packed + (ch0 >> 5) + cq : nullptr;
    f.relu = p.activation == LCE_ACT_RELU;
    f.write_float = p.write_float != 0;
    f.N = p.N; f.OH = p.OH; f.OW = p.OW; f.Wg = p.Wg; f.Hg = p.Hg;
    f.Wg_mul = p.Wg_mul; f.Wg_sh = p.Wg_sh; f.Hg_mul = p.Hg_mul; f.Hg_sh = p.Hg_sh;
    f.positions = sPix + fw * 64;
    f.lane_step = ch_ok ? 32 : 0;
    f.lane_positions = ch_ok ? f.positions : sPix + 2 * kFinishers;
    return f;
}

// The warp has read its last columns of the accumulator
__device__ __forceinline__ void mx_hand_back(uint64_t *empty_d, int lane)
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(empty_d);
}

// Bit-packed output of one tile (Section 3.2: accumulator compared with the per-channel threshold).
// Lane = channel; per 32-column chunk the sign of (accumulator - threshold) of 32 positions, then a 32 x 32 bit transpose across the warp gives every
// lane the finished word of one pixel.
__device__ __forceinline__ void mx_epilogue_bits(const MxFin &f, const Transpose32 &tr, uint32_t tmem_d, int pix, int pix2, int lane, uint64_t *empty_d)
{
    for (int ck = f.group; ck <= f.last_chunk; ck += f.n_groups) {
        const int c0 = ck * 32;
        const bool full = c0 + 32 <= f.Nt;
        uint32_t m = 0u;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (half == 0 || full) {
                float v[16];
                tmem_ld16(tmem_d + f.lane_off + (uint32_t)(c0 + half * 16), v);
                if (ck == f.last_chunk && (half == 1 || !full)) mx_hand_back(empty_d, lane);  // before the arithmetic
                // bit j = (acc_j < thr): the sign of acc - thr (both are small integers held exactly), two columns to an
                // addition; two short chains of shifts instead of one long one
#pragma unroll
                for (int j = 0; j < 16; j += 2) add_pair(v[j], v[j + 1], f.minus_thr);
                uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
                for (int j = 7; j >= 0; --j) {
                    m0 = __funnelshift_l(__float_as_uint(v[j]), m0, 1);
                    m1 = __funnelshift_l(__float_as_uint(v[8 + j]), m1, 1);
                }
                m |= (m0 | m1 << 8) << (half * 16);
            }
        }
        const uint32_t word = warp_transpose32(m, tr);
        if (pix >= 0) f.out_words[(int64_t)pix * f.cow] = word;
        pix = pix2;
    }
    if (f.last_chunk < 0) mx_hand_back(empty_d, lane);  // nothing to read for this warp
}

// Float / int32 output of one tile (Section 3.2: int -> float, fused activation, one multiply-add;
// Section 5.3: optional shortcut add and re-quantisation).  A lane holds one channel of 32 positions:
// for every position the warp writes its 32 consecutive channels as one 128-byte store, so a value
// costs one multiply-add and one store instruction and nothing is staged.  The pixels of the positions come from
// shared memory, -1 where nothing is to be written: one compare a position.
enum { EPI_FLOAT = 0, EPI_FLOAT_FUSED = 1, EPI_INT32 = 2, EPI_BITS = 3, EPI_PLAIN = 4 };

// the chunks' positions, for the whole warp to see: output pixels, -1 where nothing is to be written, or (the fused form) the
// offsets of their elements from a channel's first one, which are below 2^31
__device__ __forceinline__ void mx_share_positions(const MxFin &f, int first, int second, int lane)
{
    __syncwarp();  // the tile before is through with the array
    f.positions[lane] = first;
    f.positions[32 + lane] = second;
    __syncwarp();
}

template <int MODE>
__device__ __forceinline__ void mx_epilogue_values(const MxFin &f, uint32_t tmem_d, int lane, uint64_t *empty_d)
{
    const int32_t *lane_positions = f.lane_positions;
    for (int ck = f.group; ck <= f.last_chunk; ck += f.n_groups) {
        const int c0 = ck * 32;
        const bool full = c0 + 32 <= f.Nt;
        // straight-line code: every store is predicated, nothing branches, so the positions' address
        // arithmetic, multiply-adds and stores overlap instead of running one position after the other
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (half == 0 || full) {
                float v[16];
                tmem_ld16(tmem_d + f.lane_off + (uint32_t)(c0 + half * 16), v);
                if (ck == f.last_chunk && (half == 1 || !full)) mx_hand_back(empty_d, lane);
#pragma unroll
                for (int j4 = 0; j4 < 16; j4 += 4) {
                    const int4 o4 = *reinterpret_cast<const int4 *>(lane_positions + half * 16 + j4);
                    const int o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        float *at = f.outp + (int64_t)o[u] * f.cout;  // outside the condition: nothing branches
                        if (MODE != EPI_INT32) {
                            const float y = __fmaf_rn(v[j4 + u], f.mult, f.bias);
                            if (o[u] >= 0) *at = y;
                        } else {
                            const int32_t y = __float2int_rn(v[j4 + u]);
                            if (o[u] >= 0) *reinterpret_cast<int32_t *>(at) = y;
                        }
                    }
                }
            }
        }
        lane_positions += f.lane_step;
    }
    if (f.last_chunk < 0) mx_hand_back(empty_d, lane);  // nothing to read for this warp
}

// Float output with activation, shortcut add and re-quantised copy fused in (Section 5.3); the latter two only where every
// channel of the block exists.
// The shortcut values of a warp's first chunk of a tile are asked for before it waits for the accumulator
// (mx_shortcut: 32 independent 128-byte loads a warp), those of its next one when it is through with the first.  The
// re-quantised copy is the sign bits and the bit transpose of the bit-packed form; y + 0 makes -0.0 and NaN, which
// quantize to 0 bits, positive (PTX: a NaN result has no sign).
// Positions come as offsets of elements: multiplying pixels by the channels at each use took 36.9 us on the 56x56x64 block at 128
// images, 34.5 then (40.6 with ballots and loads behind the wait; with positions on the lanes, as that block goes now, 25.0); the plain float form, which has registers to spare, is
// faster with pixels (13.9 us against 14.4 on 56x56x64, 64 images).
// With all three parts there are registers for 16 values ahead only, those of the next half chunk: 32 spilled into the loop, 78.5 us
// on that block with everything, 57.5 with 16 (58.0 with no value before the wait; 40.6 with positions on the lanes); shortcut and float
// output 51.3 and 49.3.  What is left here of that form are 96 channels, 3x3, blocks of 128 and more, and grids that do not fill the SMs.
template <bool RES, int AHEAD>
__device__ __forceinline__ void mx_shortcut(const MxFin &f, const int32_t *offsets, float (&r)[AHEAD])
{
    if (!RES) return;
#pragma unroll
    for (int j4 = 0; j4 < AHEAD; j4 += 4) {
        const int4 o4 = *reinterpret_cast<const int4 *>(offsets + j4);  // the same for every lane
        const int o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            r[j4 + u] = o[u] >= 0 ? __ldg(f.resp + (o[u] >= 0 ? o[u] : 0)) : 0.f;
        }
    }
}

template <bool RES, bool PACK, bool WRITE_FLOAT, int AHEAD>
__device__ __forceinline__ void mx_epilogue_fused(const MxFin &f, const Transpose32 &tr, uint32_t tmem_d, float (&r)[AHEAD], int lane, uint64_t *empty_d)
{
    // which of the three parts (shortcut add, re-quantised copy, float output) a launch has is a template
    // argument: a test of a pointer per position turns the unrolled block below into branchy code that
    // runs at a third of the speed (measured on the plain float transform, and again here)
    const float floor_v = f.relu ? 0.f : -INFINITY;
    const int32_t *lane_positions = f.lane_positions;
    for (int ck = f.group; ck <= f.last_chunk; ck += f.n_groups) {
        const int c0 = ck * 32;
        const bool full = c0 + 32 <= f.Nt;  // otherwise 16 columns, the tile's last
        if (AHEAD == 32 && ck != f.group) mx_shortcut<RES>(f, f.positions + 32, r);
        uint32_t m = 0u;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (half == 0 || full) {
                float v[16];
                tmem_ld16(tmem_d + f.lane_off + (uint32_t)(c0 + half * 16), v);
                if (ck == f.last_chunk && (half == 1 || !full)) mx_hand_back(empty_d, lane);
#pragma unroll
                for (int j4 = 0; j4 < 16; j4 += 4) {
                    int o[4];
                    if (WRITE_FLOAT) {
                        const int4 o4 = *reinterpret_cast<const int4 *>(lane_positions + half * 16 + j4);
                        o[0] = o4.x; o[1] = o4.y; o[2] = o4.z; o[3] = o4.w;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        float y = __fmaf_rn(fmaxf(v[j4 + u], floor_v), f.mult, f.bias);
                        if (RES) y = __fadd_rn(y, r[(half * 16 + j4 + u) & (AHEAD - 1)]);
                        if (WRITE_FLOAT) {
                            if (o[u] >= 0) f.outp[o[u]] = y;
                        }
                        if (PACK) v[j4 + u] = y;
                    }
                }
                if (AHEAD == 16) {  // the next 16 columns, while the signs of these are collected
                    if (half == 0 && full) mx_shortcut<RES>(f, f.positions + (ck == f.group ? 16 : 48), r);
                    else if (ck != f.last_chunk) mx_shortcut<RES>(f, f.positions + 32, r);
                }
                if (PACK) {
                    uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
                    for (int j = 0; j < 16; j += 2) add_pair(v[j], v[j + 1], 0.f);
#pragma unroll
                    for (int j = 7; j >= 0; --j) {
                        m0 = __funnelshift_l(__float_as_uint(v[j]), m0, 1);
                        m1 = __funnelshift_l(__float_as_uint(v[8 + j]), m1, 1);
                    }
                    m |= (m0 | m1 << 8) << (half * 16);
                }
            }
        }
        if (PACK) {
            const uint32_t word = warp_transpose32(m, tr);
            const int o = lane_positions[lane];
            if (o >= 0) f.packp[o >> 5] = word;  // whole words of channels: 32 values to a word
        }
        lane_positions += f.lane_step;
    }
    if (f.last_chunk < 0) mx_hand_back(empty_d, lane);  // nothing to read for this warp
}

// The finishers' loop over the CTA's tiles.  FORM: which transform; the fused one by its three parts.
template <int MODE, bool RES, bool PACK, bool WRITE_FLOAT>
__device__ __forceinline__ bool mx_finish_tiles(const MxParams &p, const MxFin &f, uint64_t *bars, uint32_t tmem_base, int lane, int first_tile, int tile_step)
{
    const int T = p.T, n_tiles = p.n_tiles, n_super = p.n_super;
    Transpose32 tr;
    if (MODE == EPI_BITS || PACK) tr = transpose32_setup(lane);
    int it = 0;
    for (int st = first_tile; st < n_super; st += tile_step) {
        for (int tile = st * T; tile < st * T + T && tile < n_tiles; ++tile, ++it) {
            const int buf = it & 1;
            // what does not depend on the accumulator, before it is there (the pixels are worked out here: as a table written by
            // the loaders they were on those warps' critical chain)
            const int pix = mx_chunk_pixel(f, f, tile, 0, lane), pix2 = mx_chunk_pixel(f, f, tile, 1, lane);
            float r[RES && PACK && WRITE_FLOAT ? 16 : 32];
            if (MODE != EPI_BITS) mx_share_positions(f, MODE == EPI_FLOAT_FUSED && pix >= 0 ? pix * f.cout : pix, MODE == EPI_FLOAT_FUSED && pix2 >= 0 ? pix2 * f.cout : pix2, lane);
            if (MODE == EPI_FLOAT_FUSED) mx_shortcut<RES>(f, f.positions, r);
            // the warp goes on together (its transform uses warp-wide shuffles)
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&bars[BAR_FULL_D0 + buf], (uint32_t)(it >> 1) & 1u))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t tmem_d = tmem_base + (buf ? kD1Col : 0u);
            uint64_t *empty_d = &bars[BAR_EMPTY_D0 + buf];
            if (MODE == EPI_FLOAT_FUSED) mx_epilogue_fused<RES, PACK, WRITE_FLOAT>(f, tr, tmem_d, r, lane, empty_d);
            else if (MODE == EPI_BITS) mx_epilogue_bits(f, tr, tmem_d, pix, pix2, lane, empty_d);
            else mx_epilogue_values<MODE>(f, tmem_d, lane, empty_d);
        }
    }
    return true;
}

// EPI: EPI_PLAIN carries the three plain output transforms (bit-packed, float, int32; chosen per launch by the
// output type), EPI_FLOAT_FUSED the float transform with the shortcut add, the activation and the re-quantised
// copy.  One instantiation for the plain forms matters more than their few KB of code: a network alternates
// bit-packed and float layers, and two kernels of 160 KB alternating evict each other from the SMs' instruction
// caches at every launch (config 2 as one flushed step: 103 us with a kernel per form, 87 us with one for all
// three); the fused form stays apart because its register needs spoil the float form's code when they share one.
template <int EPI>
__global__ void __launch_bounds__(kMxThreads, 1) bconv_mx_kernel(const __grid_constant__ MxParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBars);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kOffSlot);
    int32_t *fills = reinterpret_cast<int32_t *>(smem + kOffSlot + 4);  // [0] issued by the producer, [1] consumed by the issuer
    int32_t *sPix = reinterpret_cast<int32_t *>(smem + kOffPix);
    uint32_t *raw0 = reinterpret_cast<uint32_t *>(smem + kOffDyn);
    uint8_t *sW = smem + p.off_w;
    uint8_t *sX0 = smem + p.off_x;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ch0 = blockIdx.y * 128;
    const int first_tile = blockIdx.x, tile_step = gridDim.x;

    // the next kernel of the stream may start setting itself up as soon as every CTA of this one has got here
    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- set-up, its parts side by side: the issuer warp allocates TMEM, the producer warp initialises the
    // barriers and starts the weight copies, the finisher warps fill the table of operand offsets, the
    // loaders fetch the first chunk of activations ---------------------------------------------------------
    const int n_mma = p.pairs;
    // the weight producer's progress (one thread): fills issued, ring stage and (tile-local) group of pairs of the next one
    int prod_g = 0, prod_total = 0, prod_stage = 0, prod_group = 0;
    uint32_t prod_parity = 1;  // the first pass over the ring waits for nothing
    if (warp == kIssuerWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp == kIssuerWarp + 1) {
        for (int b = lane; b < BAR_COUNT; b += 32) {
            const uint32_t count = b <= BAR_FULL_X3 ? kLoaders : (b == BAR_EMPTY_D0 || b == BAR_EMPTY_D1) ? kFinishers / 32 : b == BAR_SCALES ? 4 : 1;
            mbar_init(&bars[b], count);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncwarp();
        // The weights are constants of the model: their copies start at once, whatever the previous kernel of
        // the stream is still doing, one lane per copy.  Resident: all pairs, every copy counted on the same
        // barrier; streamed: the first pass over the ring (stage = fill number; at most 32 stages).
        const uint8_t *src = p.wimg + (size_t)blockIdx.y * p.pairs * kPairBytes;
        if (p.resident) {
            if (lane == 0) mbar_expect_tx(&bars[BAR_FULL_W0], (uint32_t)(p.pairs * kPairBytes));
            __syncwarp();
            const int share = (p.pairs + 31) >> 5, first = lane * share, n = min(share, p.pairs - first);
            if (n > 0) bulk_copy_g2s(sW + (size_t)first * kPairBytes, src + (size_t)first * kPairBytes, (uint32_t)(n * kPairBytes), &bars[BAR_FULL_W0]);
            prod_g = 1;
        } else {
            int my_tiles = 0;
            for (int st = first_tile; st < p.n_super; st += tile_step) my_tiles += min(p.T, p.n_tiles - st * p.T);
            // a fill = one group of up to group_pairs consecutive pairs (one copy: they are contiguous in the image)
            prod_total = my_tiles * p.groups;
            prod_g = min(p.stages, prod_total);
            if (lane < prod_g) {
                const int first = (lane % p.groups) * p.group_pairs;
                const uint32_t bytes = (uint32_t)(min(p.group_pairs, p.pairs - first) * kPairBytes);
                mbar_expect_tx(&bars[BAR_FULL_W0 + lane], bytes);
                bulk_copy_g2s(sW + (size_t)lane * p.group_pairs * kPairBytes, src + (size_t)first * kPairBytes, bytes, &bars[BAR_FULL_W0 + lane]);
            }
            prod_group = prod_g % p.groups;   // the next fill's group within its tile
            if (prod_g == p.stages) prod_parity ^= 1u; else prod_stage = prod_g;
        }
        __syncwarp();
        if (lane == 0) {
            fills[0] = prod_g;
            fills[1] = 0;
        }
    } else if (tid < kFinishers) {
        uint2 *tbl = reinterpret_cast<uint2 *>(smem + p.off_tbl);
        if (warp == 0) sPix[2 * kFinishers + lane] = -1;  // the pixels of channels that do not exist
        const int even = p.Cw & ~1, paired = p.KH * p.KW * even, words = p.KH * p.KW * p.Cw;
        for (int e = tid; e < n_mma; e += kFinishers) {
            // A: the pair's place among the resident ones or in its group of streamed ones.  B: the first word's rows, and in
            // the upper half the distance from there to the second word's; an odd last word has a second one of zero
            // weights, whose rows may be any (the next ones: a position buffer has one row to spare)
            const uint32_t first = word_b_offset(p, 2 * e, even, paired);
            const uint32_t apart = 2 * e < paired ? (uint32_t)p.P : 2 * e + 1 < words ? word_b_offset(p, 2 * e + 1, even, paired) - first : 1u;
            tbl[e] = make_uint2((uint32_t)(p.resident ? e : e % p.group_pairs) * (kPairBytes >> 4), first | apart << 16);
        }
    }
    // The loaders' first prefetch goes out before the CTA-wide barrier of the set-up: it needs the previous
    // kernel's output (hence the dependency wait) and plain shared memory, nothing that is set up above.
    MxLoad ld;
    MxPos stage{0, 0, 0};
    int form = 0;
    const int ltid = tid - kFinishers;  // a loader's number
    const bool loader = ltid >= 0 && ltid < kLoaders;
    if (loader) {
        form = mx_load_setup(p, ld);
        stage = mx_position(first_tile * p.T * p.Nt + ltid, p);
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the activations may come from the previous kernel
        if (first_tile < p.n_super) {
            // through the general forms, whose staging layout is everybody's: one more copy of every special form
            // costs more in code size than it saves here
            if (p.n_phase == 1) mx_prefetch<0, MX_S1>(ld, stage, p.Nt + p.halo, raw0, ltid, p.cp_words);
            else mx_prefetch<0, MX_S2>(ld, stage, p.Nt + p.halo, raw0, ltid, p.cp_words);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    if (warp < 4) {
        // block scales: every byte 0x7F = 2^0 (ue8m0), for all 128 lanes of the 32 scale columns, written by the
        // first four finisher warps (one per lane quarter; they have nothing else to do yet); the issuer
        // waits for the four arrivals before its first MMA
        const uint32_t one = 0x7F7F7F7Fu;
        const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + kSfaCol;
#pragma unroll
        for (int c = 0; c < 32; c += 8)
            asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr + c), "r"(one) : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[BAR_SCALES]);
    }

    bool ok = true;
    if (loader) {
        // ======================= loaders ==============================================================
#define LCE_MX_LOAD(CW, FORM) ok = mx_load_tiles<CW, FORM>(p, ld, stage, bars, raw0, sX0, ltid, first_tile, tile_step)
        LCE_MX_FORMS(LCE_MX_LOAD)
    } else if (tid < kFinishers) {
        // ======================= finishers ============================================================
        const MxFin fin = mx_fin_context(p, sPix, warp, lane, ch0);  // lane quarter warp & 3, column group warp >> 2
        asm volatile("griddepcontrol.wait;" ::: "memory");  // outputs and the shortcut tensor: only after the previous kernel
#define LCE_MX_FINISH(...) mx_finish_tiles<__VA_ARGS__>(p, fin, bars, tmem_base, lane, first_tile, tile_step)
        if (EPI == EPI_FLOAT_FUSED) {
            switch ((fin.resp != nullptr ? 4 : 0) | (fin.packp != nullptr ? 2 : 0) | (fin.write_float ? 1 : 0)) {
                case 1: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, false, false, true); break;
                case 2: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, false, true, false); break;
                case 3: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, false, true, true); break;
                case 5: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, true, false, true); break;
                case 6: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, true, true, false); break;
                case 7: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, true, true, true); break;
                default: ok = LCE_MX_FINISH(EPI_FLOAT_FUSED, false, false, false); break;  // nothing to write: only hands the accumulator back
            }
        } else if (p.out_type == LCE_OUT_BITPACKED) {
            ok = LCE_MX_FINISH(EPI_BITS, false, false, false);
        } else if (p.out_type == LCE_OUT_INT32) {
            ok = LCE_MX_FINISH(EPI_INT32, false, false, false);
        } else {
            ok = LCE_MX_FINISH(EPI_FLOAT, false, false, false);
        }
    } else if (warp == kIssuerWarp || (warp == kIssuerWarp + 1 && p.resident != 0)) {
        // ======================= MMA issuer: a warp, every lane with the same values ==================
        // With the weights resident the producer warp has nothing left to do and becomes a second issuer: the
        // two take alternate tiles (one accumulator buffer each), so that one warp's per-tile bookkeeping and
        // waits run while the other's MMAs are in the pipe.
        const int my_parity = warp - kIssuerWarp;
        const uint2 *tbl = reinterpret_cast<const uint2 *>(smem + p.off_tbl);
        // instruction descriptor (block-scaled kinds): A, B = e2m1 (1), both K-major, N >> 3 at bit 17,
        // scales ue8m0 (bit 23), M >> 4 at bit 24, scale-factor ids 0
        const uint32_t idesc = (1u << 7) | (1u << 10) | ((uint32_t)(p.Nt >> 3) << 17) | (1u << 23) | ((uint32_t)(128 >> 4) << 24);
        // shared-memory descriptors (units of 16 bytes): low = start | K-chunk stride << 16 (B: from the table); high = 8-row
        // group stride (128 bytes) | version 1 at bit 46; no swizzle
        const uint32_t desc_hi = 8u | (1u << 14);
        // everything the loops use, read from the kernel parameters once
        const int T = p.T, n_tiles = p.n_tiles, n_super = p.n_super, Nt = p.Nt, stages = p.stages, group_pairs = p.group_pairs;
        const bool resident = p.resident != 0;
        const uint32_t w_lo0 = ((uint32_t)p.off_w >> 4) + (smem_u32(smem) >> 4) + (128u << 16);
        const uint32_t x_lo_buf0 = ((uint32_t)p.off_x >> 4) + (smem_u32(smem) >> 4);
        const uint32_t x_units = (uint32_t)p.x_bytes >> 4, group_units = (uint32_t)(kPairBytes >> 4) * (uint32_t)p.group_pairs;
        const uint32_t sfa = tmem_base + kSfaCol, sfb = tmem_base + kSfbCol;
        const int n_xbuf = p.n_xbuf;
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bars[BAR_SCALES], 0));  // the block scales are in TMEM
        int g = 0, stage_i = 0;
        uint32_t w_parity = 0;
        int it = 0;
        int xbuf = 0;
        for (int st = first_tile; st < n_super && ok; st += tile_step, xbuf = xbuf + 1 == n_xbuf ? 0 : xbuf + 1)
        for (int k = 0; k < T && st * T + k < n_tiles && ok; ++k, ++it) {
            const int buf = it & 1;
            if (resident && buf != my_parity) continue;
            ok = mbar_wait_bounded(&bars[BAR_FULL_X0 + (it & 3)], (uint32_t)(it >> 2) & 1u);
            if (ok && it >= 2) {  // the accumulator buffer must have been read out
                ok = mbar_wait_bounded(&bars[BAR_EMPTY_D0 + buf], (uint32_t)((it >> 1) - 1) & 1u);
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t tmem_d = tmem_base + (buf ? kD1Col : 0u);
            // B operand: the super-tile's position buffer from this tile's first row on
            const uint32_t x_lo0 = x_lo_buf0 + (uint32_t)xbuf * x_units + (uint32_t)(k * Nt);
            uint32_t accumulate = 0;
            if (resident) {
                // every pair stays in shared memory: one wait for all of them (a single barrier counts the bytes
                // of all the copies) before the CTA's first tile, then nothing between the MMAs of a tile
                if (it < 2) {  // this warp's first tile
                    ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bars[BAR_FULL_W0], 0));
                    if (!ok) break;
                    if (lane == 0) fills[1] = 1;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                mx_issue_table(tmem_d, tbl, n_mma, w_lo0, x_lo0, desc_hi, idesc, sfa, sfb, accumulate);
            } else {
                // the pairs stream through the ring a group at a time: wait for the group, issue its MMAs in one run, hand
                // its stage back (the wait, the commit and the bookkeeping cost this warp as much as some MMAs: issued tap
                // by tap, a group of five taps cost 600 clocks more than its MMAs)
                int pair = 0;
                while (pair < n_mma) {
                    ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bars[BAR_FULL_W0 + stage_i], w_parity));
                    if (!ok) break;
                    ++g;
                    if (lane == 0) fills[1] = g;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const int n = min(group_pairs, n_mma - pair);
                    mx_issue_table(tmem_d, tbl + pair, n, w_lo0 + (uint32_t)stage_i * group_units, x_lo0, desc_hi, idesc, sfa, sfb, accumulate);
                    pair += n;
                    if (elect_one()) mma_commit(&bars[BAR_EMPTY_W0 + stage_i]);
                    if (++stage_i == stages) { stage_i = 0; w_parity ^= 1u; }
                }
            }
            if (!ok) break;
            if (elect_one()) {
                mma_commit(&bars[BAR_FULL_D0 + buf]);         // to the finishers: the accumulator is complete
                mma_commit(&bars[BAR_TILE_DONE0 + (it & 3)]);  // to the loaders: the tile's operands have been read
            }
        }
    } else if (tid == kProducerTid) {
        // ======================= weight producer: one thread, the rest of the streamed pairs ==========
        const uint8_t *src = p.wimg + (size_t)blockIdx.y * p.pairs * kPairBytes;
        for (; !p.resident && prod_g < prod_total; ++prod_g) {
            ok = mbar_wait_bounded(&bars[BAR_EMPTY_W0 + prod_stage], prod_parity);
            if (!ok) break;
            const int first = prod_group * p.group_pairs;
            const uint32_t bytes = (uint32_t)(min(p.group_pairs, p.pairs - first) * kPairBytes);
            mbar_expect_tx(&bars[BAR_FULL_W0 + prod_stage], bytes);
            bulk_copy_g2s(sW + (size_t)prod_stage * p.group_pairs * kPairBytes, src + (size_t)first * kPairBytes, bytes, &bars[BAR_FULL_W0 + prod_stage]);
            fills[0] = prod_g + 1;
            if (++prod_group == p.groups) prod_group = 0;
            if (++prod_stage == p.stages) { prod_stage = 0; prod_parity ^= 1u; }
        }
    }
    if (!ok) mx_report_timeout(p.host_flag);

    // ---- tear-down: nothing of this CTA may still be in flight when its TMEM and shared memory go ----
    // When no wait gave up, the finishers have waited for the MMAs of every tile and the issuer for every
    // weight copy; otherwise the lane that issued the MMAs waits for what is still under way.
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    const bool all_ok = __syncthreads_and(ok) != 0;
    if (!all_ok || fills[0] != fills[1]) {
        if ((warp == kIssuerWarp || (warp == kIssuerWarp + 1 && p.resident != 0)) && elect_one()) {
            uint64_t *done = &bars[warp == kIssuerWarp ? BAR_DONE : BAR_DONE_B];
            mma_commit(done);                                  // arrives when every MMA this lane issued has finished
            bool drained = mbar_wait_bounded(done, 0);
            // weight copies that were started but never consumed
            const int issued = fills[0], consumed = fills[1];
            for (int g = consumed; warp == kIssuerWarp && g < issued && drained; ++g)
                drained = mbar_wait_bounded(&bars[BAR_FULL_W0 + g % p.stages], (uint32_t)(g / p.stages) & 1u);
            if (!drained) mx_report_timeout(p.host_flag);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == kIssuerWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
}

}  // namespace
}  // namespace lce

#include "bconv_mx_positions.cuh"

namespace lce {
namespace {

// ---- load-time weight image -----------------------------------------------------------------------------
// plain packed words [Cout][KH][KW][Cw] -> e2m1 operand image [channel block][pair of words of K][2][128 channels][16 bytes]
// in the order of mx_word; channels past Cout, the second word of an odd last one and channels past Cin inside a word are
// 0.0; with out_c <= 64 (<= 32) the rows hold two (four) copies of the channels, so that every TMEM lane quarter has work
// for a finisher warp
__global__ void mx_pack_weights_kernel(const uint32_t *w, uint4 *image, int Cout, int Cin, int Cw, int KH, int KW, int stride, int n_blocks, int dup)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int words = KH * KW * Cw, padded = words + (words & 1);
    const int64_t total = (int64_t)n_blocks * padded * 128;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int row = (int)(e & 127);
        const int64_t t = e >> 7;
        const int blk = (int)(t / padded), i = (int)(t - (int64_t)blk * padded);
        const int o = blk * 128 + (row & (128 / dup - 1));  // few output channels: the block is repeated down the 128 rows
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (o < Cout && i < words) {
            const MxWord at = mx_word(i, KH, KW, Cw, stride);
            v = mx_expand_word(w[((int64_t)o * KH * KW + at.ky * KW + at.kx) * Cw + at.cw]);
            const int valid = Cin - at.cw * 32;  // channels of this word that exist
            if (valid < 32) {
                // value (register j, nibble i) is channel 4 i + j of the word
                uint32_t m[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    m[j] = 0u;
                    for (int n = 0; n < 8; ++n)
                        if (4 * n + j < valid) m[j] |= 0xFu << (4 * n);
                }
                v.x &= m[0]; v.y &= m[1]; v.z &= m[2]; v.w &= m[3];
            }
        }
        image[e] = v;
    }
}

struct MxPlan {
    int Nt, P, T, stages, resident, group_pairs, groups, n_blocks, ctas_x, n_tiles, n_super, total_q, Wg, Hg, n_phase, Cw, pairs, taps, halo, cover_halo, n_xbuf, ahead;
    bool positions;  // positions on the TMEM lanes (bconv_mx_positions.cuh)
    size_t raw_words, x_bytes, off_tbl, off_w, off_x, smem;
    double clocks;  // of a CTA's tiles by the cost model
};

constexpr size_t kSmemLimit = 227 * 1024;
constexpr int kMaxPositions = 16383;  // of a position buffer: descriptor strides are 14-bit counts of 16 bytes

bool mx_plan_uncached(const ConvGeom &g, int sms, MxPlan *pl);

// The plan depends on the geometry alone, and a network repeats few geometries: the last few plans of
// each host thread are kept (the search below walks about a hundred candidates otherwise).
bool mx_plan(const ConvGeom &g, int sms, MxPlan *pl)
{
    struct Entry {
        ConvGeom g;
        int sms;
        bool valid, found;
        MxPlan plan;
    };
    constexpr int kEntries = 16;
    static thread_local Entry cache[kEntries];
    static thread_local int next = 0;
    for (int i = 0; i < kEntries; ++i) {
        const Entry &e = cache[i];
        if (e.valid && e.sms == sms && memcmp(&e.g, &g, sizeof(ConvGeom)) == 0) {
            *pl = e.plan;
            return e.found;
        }
    }
    Entry &e = cache[next];
    next = (next + 1) % kEntries;
    memset(&e.g, 0, sizeof(ConvGeom));
    e.g = g;
    e.sms = sms;
    e.found = mx_plan_uncached(g, sms, &e.plan);
    e.valid = true;
    *pl = e.plan;
    return e.found;
}

int mx_pairs(const ConvGeom &g) { return (g.KH * g.KW * g.Cw + 1) / 2; }
int mx_channel_blocks(const ConvGeom &g) { return (g.Cout + 127) / 128; }

// The grid of positions and everything else of a plan that does not depend on the tile; false where the kernel does not
// cover the layer.
bool mx_frame(const ConvGeom &g, MxPlan *pl)
{
    if (g.sh != g.sw || (g.sh != 1 && g.sh != 2)) return false;
    if (g.Cw > 32) return false;
    const int taps = g.KH * g.KW;
    if (taps > kMaxTaps) return false;
    const int s = g.sh;
    int Wg, Hg;
    int64_t halo, cover_halo = -1;
    if (s == 1) {
        const int pr = max(0, (g.OW - 1) + g.KW - g.W - g.pl), pb = max(0, (g.OH - 1) + g.KH - g.H - g.pt);
        Wg = g.W + max(g.pl, pr);
        cover_halo = (int64_t)(g.KH - 1) * Wg + (g.KW - 1);
        if (g.Cw & 1) Wg = max(Wg, g.KW);  // a tap's place in the buffer grows with its number (mx_word) as long as a row holds the window
        Hg = g.H + max(g.pt, pb);
        halo = (int64_t)(g.KH - 1) * Wg + (g.KW - 1);
    } else {
        Wg = g.OW + (g.KW - 1) / 2;
        Hg = g.OH + (g.KH - 1) / 2;
        halo = (int64_t)((g.KH - 1) / 2) * Wg + (g.KW - 1) / 2;
    }
    const int64_t total_q = (int64_t)g.N * Hg * Wg;
    if (total_q >= (1ll << 31) - 4096 || g.M >= (1ll << 31) || halo > kMaxPositions) return false;
    pl->Wg = Wg; pl->Hg = Hg; pl->halo = (int)halo; pl->cover_halo = (int)(cover_halo < 0 ? halo : cover_halo); pl->total_q = (int)total_q;
    // a 1x1 filter at stride 2 reads one phase of the four: staging that one alone took 64 images of 28x28x512 -> 512 from
    // 19.5 to 7.3 us, of 56x56x256 -> 256 from 13.7 to 9.0
    pl->n_phase = taps == 1 ? 1 : s * s;
    pl->Cw = g.Cw;
    pl->taps = taps;
    pl->pairs = mx_pairs(g);
    pl->n_blocks = mx_channel_blocks(g);
    return true;
}

// Shared memory of a tile of nt positions, T of them to a position buffer; false if it does not fit beside two pairs of
// weight words (or the only one).
struct MxRoom {
    int P;
    size_t raw_words, x_bytes, off_tbl, off_w, rest;
};

bool mx_room(const MxPlan &pl, int nt, int T, int n_xbuf, size_t limit, MxRoom *r)
{
    // T tiles share one position buffer of T * nt + halo rows: the halo is staged once per T tiles
    r->P = T * nt + pl.halo;
    if (r->P > kMaxPositions) return false;
    r->raw_words = (((size_t)pl.n_phase * (nt + pl.halo) * pl.Cw + 3) / 4) * 4;
    r->x_bytes = ((size_t)pl.n_phase * pl.Cw * r->P * 16 + 16 + 127) / 128 * 128;  // one row to spare: see the table of operand offsets
    r->off_tbl = kOffDyn + r->raw_words * 4;
    const size_t fixed = r->off_tbl + (size_t)pl.pairs * 8;  // the table no longer than it is: at 512 channels 3x3 the 8 KB saved are a wider tile
    r->off_w = (fixed + 127) / 128 * 128;
    r->rest = n_xbuf * r->x_bytes + 256;
    return r->off_w + r->rest + (size_t)min(2, pl.pairs) * kPairBytes <= limit;
}

// Which layers the kernel takes: those whose smallest tile (16 positions) fits beside two whole taps (one of a 1x1 filter)
// of an even number of words each.  Pairs take less room than that, and a larger tile never less than a smaller one, so
// such a layer has a plan.
bool mx_covers(const ConvGeom &g)
{
    MxPlan pl;
    if (!mx_frame(g, &pl)) return false;
    const size_t Cw2 = g.Cw + (g.Cw & 1), P = 16 + pl.cover_halo;
    const size_t raw = (pl.n_phase * P * g.Cw + 3) / 4 * 16, table = pl.taps * (Cw2 / 2) * 8;
    constexpr size_t kBefore = 8192;  // what lay before these parts when the line was drawn
    return (kBefore + raw + table + 127) / 128 * 128 + 2 * pl.n_phase * Cw2 * P * 16 + 256 + (pl.taps > 1 ? 2 : 1) * Cw2 * 2048 <= kSmemLimit;
}

bool mx_plan_as(const ConvGeom &g, int sms, bool positions, size_t reserved, MxPlan *pl)
{
    const size_t limit = kSmemLimit - reserved;
    if (!mx_frame(g, pl)) return false;
    if (!mx_covers(g)) return false;
    const int pairs = pl->pairs, halo = pl->halo;
    const int64_t total_q = pl->total_q;
    const int ctas_max = max(1, sms / pl->n_blocks);
    double best = 1e30;
    bool found = false;
    pl->positions = positions;
    for (int nt = positions ? kPositionsTile : 16; nt <= (positions ? kPositionsTile : kMaxNt); nt += 16) {
        const int n_tiles = (int)((total_q + nt - 1) / nt);
        for (int T = 1; T <= 8; ++T) {
            if (T > 1 && (T - 1) * ctas_max >= n_tiles) break;   // no CTA would have that many tiles
            MxRoom room;
            // A CTA that has one super-tile needs one position buffer.  28x28x256 at stride 2, 64 images: one tile of 208
            // positions a CTA instead of two of 112 beside two buffers of four phases, 11.2 -> 9.5 us; 7x7x512, 128 images
            // 10.7 -> 10.3; 56x56x64, 64 images, float (seven tiles in one super-tile) 13.8 -> 13.5.
            const int n_super = (n_tiles + T - 1) / T;
            const int ctas_x = min(ctas_max, n_super);
            const bool single = n_super <= ctas_x;
            if (!mx_room(*pl, nt, T, single ? 1 : 2, limit, &room)) break;
            // pairs that fit beside the position buffers: all of them -> resident (one barrier); otherwise a ring of two
            // stages of half the fitting pairs each (a group costs the issuer one wait and one commit, whatever its
            // size: two large groups measured better than three or four smaller ones)
            const int slots = (int)((limit - room.off_w - room.rest) / kPairBytes);
            const bool resident = slots >= pairs;
            if (positions && !resident) break;
            int stages, group_pairs, groups;
            if (resident) {
                stages = groups = 1; group_pairs = pairs;
            } else {
                group_pairs = max(1, slots / 2);
                groups = (pairs + group_pairs - 1) / group_pairs;
                group_pairs = (pairs + groups - 1) / groups;  // even groups
                stages = min(kMaxStages, slots / group_pairs);
            }
            const int per_cta = ((n_super + ctas_x - 1) / ctas_x) * T;
            // clocks per MMA: 43 + N/2, at least 100 (measured); the loaders need about 400 + 8 clocks per staged
            // position and tile
            const double mma1 = fmax(100.0, 43.0 + nt / 2.0);
            const double mma = (double)pairs * mma1;
            // a streamed group: its bytes from L2 (with all SMs streaming at least 38 bytes per clock each), or its share of a copy's latency, or what the single issuer needs
            // per group (wait for the stage, issue, hand the stage back: about 250 clocks on top of the MMAs)
            const double stream = resident ? 0.0 : (double)groups * fmax(fmax(group_pairs * kPairBytes / 38.0, 1300.0 / stages), 250.0 + group_pairs * mma1);
            // stride 2: four phases per position, staged two at a time where the geometry allows (MX_S2_PAIR)
            const double per_position = pl->n_phase == 1 ? 1.0 : ((g.W & 1) == 0 && (g.pl & 1) == 0 && g.Cw <= 4) ? 2.0 : 3.0;
            const double load = 400.0 + 8.0 * per_position * (nt + (double)halo / T);
            // with streamed weights the hand-overs of the ring and of the loaders do not hide each other (112x112x32 stride 2
            // at batch 256: 71 us streamed, 36 us resident, where the three terms alone call it a tie)
            const double cost = per_cta * (fmax(fmax(mma, stream), load) + 0.5 * fmin(stream, load) + 150.0);
            if (cost < best) {
                best = pl->clocks = cost;
                found = true;
                pl->Nt = nt; pl->P = room.P; pl->T = T; pl->stages = stages; pl->resident = resident ? 1 : 0; pl->group_pairs = group_pairs; pl->groups = groups;
                pl->n_tiles = n_tiles; pl->n_super = n_super; pl->ctas_x = ctas_x;
                pl->raw_words = room.raw_words; pl->x_bytes = room.x_bytes;
                pl->off_tbl = room.off_tbl;
                pl->off_w = room.off_w;
                pl->off_x = (room.off_w + (size_t)stages * group_pairs * kPairBytes + 127) / 128 * 128;
                // More position buffers where shared memory is left over (thin layers): the loaders may then be
                // up to four tiles ahead, ahead <= (n_xbuf - 1) * T + 1, and the hand-overs between the roles
                // (a few hundred clocks each) drop out of the per-tile cycle.
                int n_xbuf = single ? 1 : 2;
                while (!single && n_xbuf < 4 && (n_xbuf - 1) * T + 1 < 4 && pl->off_x + (size_t)(n_xbuf + 1) * room.x_bytes <= limit) ++n_xbuf;
                pl->n_xbuf = n_xbuf;
                pl->ahead = single ? 4 : min(4, (n_xbuf - 1) * T + 1);
                pl->smem = pl->off_x + (size_t)n_xbuf * room.x_bytes + reserved;
            }
        }
    }
    return found;
}

// Where positions on the lanes pay, given that all weights fit.  A tile is 256 positions whatever the grid, where the other form cuts
// narrower ones so that every SM has its share: with fewer tiles than SMs, or few in the last wave, SMs have nothing to do.  What the form
// gains per tile must make up for that, and it gains more the fewer words it stores and the fewer matrix instructions there are.  Both
// forms as graphs of 20 launches, 1 - 128 images of 7x7 - 112x112, 32 - 512 -> 32 - 96 channels, 1x1 - 5x5, strides 1 and 2 (711 layers
// with bits, 532 with each fused output); time with positions on the lanes / with channels:
//   bits: 0.60 - 1.02 where taken.  Left to the other form: 0.94 - 1.22 (14x14x256 -> 64 at 32 images 1.10, 14x14x512 -> 96, 1x1, at
//     64 images 1.03).
//   re-quantised copy alone: 0.68 - 1.04; left 0.92 - 1.40 (14x14x96 at 32 images 1.20).
//   floats or a shortcut: 0.55 - 1.03; left 0.88 - 1.79 (one image of 28x28x96 with all three 1.79).
enum MxOutput { MX_BITS, MX_COPY, MX_COPY_FLOATS, MX_SHORTCUT_COPY, MX_SHORTCUT_FLOATS, MX_OUTPUTS };  // the last with or without the copy

bool mx_positions_pay(const ConvGeom &g, const MxPlan &pl, int sms, MxOutput output)
{
    const int words = (g.Cout + 31) / 32, instructions = pl.pairs * words;  // of 32 channels each
    const bool one_phase = pl.n_phase == 1;
    const double waves = (double)pl.n_tiles / sms, full = waves / ceil(waves);
    if (output == MX_BITS)
        return one_phase && waves >= 0.5 || full >= 0.6 || one_phase && instructions <= 10 || words == 1 && waves >= 0.35;
    if (full >= 0.86 || words == 1 && waves >= (one_phase ? 0.5 : 1.0)) return true;
    if (output == MX_COPY) return pl.pairs <= 8 && full >= 0.6 || one_phase && words <= 2 && instructions <= 8;
    if (words == 1 && one_phase && instructions <= 10 && waves >= 0.08) return true;
    return output == MX_SHORTCUT_COPY && waves >= 2.0 || output == MX_SHORTCUT_FLOATS && waves >= 4.0;  // the last wave counts for less
}

// Bit-packed output of up to 96 channels.  With 128 channels an accumulator has 128 columns, three fill TMEM, and it depends: 28x28x128 at
// 64 images 7.2 -> 8.2 us, 56x56x64 -> 128 at stride 2, 256 images, 14.7 -> 14.0.  `clocks` stays that of channels on the lanes: it is what
// the choice between this file and the latency kernel is fitted to, and positions on the lanes are taken where they need no more.
bool mx_plan_uncached(const ConvGeom &g, int sms, MxPlan *pl)
{
    if (!mx_plan_as(g, sms, false, 0, pl)) return false;
    MxPlan positions;
    if (g.out_type == LCE_OUT_BITPACKED && g.Cout <= kPositionsChannels && mx_plan_as(g, sms, true, 0, &positions) &&
        mx_positions_pay(g, positions, sms, MX_BITS)) {
        positions.clocks = pl->clocks;
        *pl = positions;
    }
    return true;
}

template <int EPI>
lce_status launch_mx(const MxParams &p, dim3 grid, size_t smem, cudaStream_t s)
{
    static SmemOptIn opted;
    if (!opted.ensure(bconv_mx_kernel<EPI>, smem)) return LCE_ERR_CUDA;
    return launch_dependent(bconv_mx_kernel<EPI>, grid, kMxThreads, smem, s, p);
}

template <int FORM>
lce_status launch_positions(const MxPositionsParams &p, dim3 grid, size_t smem, cudaStream_t s)
{
    static SmemOptIn opted;
    if (!opted.ensure(bconv_mx_positions_kernel<FORM>, smem)) return LCE_ERR_CUDA;
    return launch_dependent(bconv_mx_positions_kernel<FORM>, grid, kPositionsThreads, smem, s, p);
}

int mx_dup(const ConvGeom &g) { return g.Cout <= 32 ? 4 : g.Cout <= 64 ? 2 : 1; }

int device_sms()
{
    int sms = 148, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 148;
}

}  // namespace

bool tensor_covers(const ConvGeom &g) { return mx_covers(g); }

size_t tensor_weight_image_bytes(const ConvGeom &g)
{
    return covers_some_padding(g, mx_covers) ? (size_t)mx_channel_blocks(g) * mx_pairs(g) * kPairBytes : 0;
}

lce_status launch_pack_weights_tensor(const ConvGeom &g, const uint32_t *w, void *image, cudaStream_t s)
{
    const int n_blocks = mx_channel_blocks(g);
    const int64_t total = (int64_t)n_blocks * mx_pairs(g) * 256;
    const int64_t want = (total + 255) / 256;
    const int blocks = (int)(want < 4096 ? want : 4096);
    const lce_status st = launch_dependent(mx_pack_weights_kernel, dim3((unsigned)blocks), 256, 0, s, w, static_cast<uint4 *>(image), g.Cout, g.Cin, g.Cw, g.KH, g.KW, g.sh, n_blocks, mx_dup(g));
    mx_flag_array(false);  // load time is the moment to set up the host-visible status word (it cannot be done under stream capture)
    return st;
}

lce_status tensor_plan_info(const ConvGeom &g, TensorPlanInfo *info)
{
    MxPlan pl;
    if (!mx_plan(g, device_sms(), &pl)) return LCE_ERR_UNSUPPORTED;
    info->tile_positions = pl.positions ? kUnit : pl.Nt;  // of an accumulator
    info->ctas = pl.ctas_x * pl.n_blocks;
    info->weight_stages = pl.resident ? pl.taps : pl.stages;
    info->weights_resident = pl.resident;
    info->shared_bytes = (int64_t)pl.smem;
    info->clocks = pl.clocks;
    info->phases = pl.n_phase;
    return LCE_OK;
}

namespace {
struct MxLaunch {
    MxParams params;
    dim3 grid;
    size_t smem;
    bool positions;
};

// float output has launches of its own for a re-quantised copy and for a shortcut, taken where they pay
struct MxLaunches {
    MxLaunch plain, copy, shortcut;
    bool pays[MX_OUTPUTS];
};
static_assert(sizeof(MxLaunches) <= sizeof(PreparedLaunch), "PreparedLaunch too small");

MxLaunch mx_launch(const ConvGeom &g, const MxPlan &pl)
{
    MxLaunch l;
    l.params = MxParams{};
    l.grid = dim3((unsigned)pl.ctas_x, (unsigned)pl.n_blocks);
    l.smem = pl.smem;
    l.positions = pl.positions;
    MxParams &p = l.params;
    p.N = g.N; p.H = g.H; p.W = g.W; p.Cw = g.Cw; p.Cout = g.Cout; p.Cow = g.Cow;
    p.OH = g.OH; p.OW = g.OW; p.KH = g.KH; p.KW = g.KW; p.stride = g.sh; p.pt = g.pt; p.pl = g.pl;
    p.K = g.KH * g.KW * g.Cin;
    p.Wg = pl.Wg; p.Hg = pl.Hg; p.n_phase = pl.n_phase;
    fast_div_constants((uint32_t)pl.Wg, &p.Wg_mul, &p.Wg_sh);
    fast_div_constants((uint32_t)pl.Hg, &p.Hg_mul, &p.Hg_sh);
    const auto step = [&](int64_t positions) {
        const int64_t rows = positions / pl.Wg;
        return MxStep{(int)(rows / pl.Hg), (int)(rows % pl.Hg), (int)(positions % pl.Wg)};
    };
    const int64_t last_chunk = pl.T > 1 ? (int64_t)(pl.T - 1) * pl.Nt + pl.halo : 0, super_step = (int64_t)pl.ctas_x * pl.T * pl.Nt;
    p.step_across = step(kLoaders);
    p.step_tile = step(pl.Nt);
    p.step_chunk_first = step(pl.Nt + pl.halo);
    p.step_chunk_super = step(super_step - last_chunk);
    p.Nt = pl.Nt; p.P = pl.P; p.T = pl.T; p.halo = pl.halo; p.n_tiles = pl.n_tiles; p.n_super = pl.n_super; p.total_q = pl.total_q;
    const uint32_t even = (uint32_t)max(2, g.Cw & ~1);
    fast_div_constants(even, &p.even_mul, &p.even_sh);
    for (int tap = 0; tap < pl.taps; ++tap) {  // word 0 of a tap of one word a tap: the tap itself
        const MxWord w = mx_word(tap, g.KH, g.KW, 1, g.sh);
        p.tap_rows[tap] = (uint16_t)(g.sh == 2 ? ((w.ky & 1) * 2 + (w.kx & 1)) * g.Cw * pl.P + (w.ky >> 1) * pl.Wg + (w.kx >> 1) : w.ky * pl.Wg + w.kx);
    }
    p.pairs = pl.pairs; p.stages = pl.stages; p.resident = pl.resident; p.group_pairs = pl.group_pairs; p.groups = pl.groups;
    p.x_bytes = (int32_t)pl.x_bytes;
    p.n_xbuf = pl.n_xbuf; p.ahead = pl.ahead;
    p.off_tbl = (int32_t)pl.off_tbl; p.off_w = (int32_t)pl.off_w; p.off_x = (int32_t)pl.off_x;
    p.pad_zero = g.padding == LCE_PAD_SAME_ZERO;
    p.out_type = g.out_type; p.activation = g.activation;
    p.dup_log2 = mx_dup(g) == 4 ? 2 : mx_dup(g) == 2 ? 1 : 0;
    return l;
}
}  // namespace

// Float output of whole words of up to 96 channels, with a shortcut added or a re-quantised copy written, can go with positions on the
// lanes (us: 56x56x64 at 128 images, copy alone 17.9 -> 15.4, shortcut and copy 34.1 -> 25.0, with the floats 57.7 -> 40.6); a
// shortcut from 96 to 96 channels, 3x3, has no room beside the weights, as a rule.  Floats alone are bound by their stores and have one
// form: 56x56x64 at 64 images 14.1, with positions on the lanes 15.1 (32 bytes of a pixel a store instead of 128).
lce_status prepare_bconv_tensor(const ConvGeom &g, bool fused, PreparedLaunch *prepared)
{
    MxPlan pl;
    const int sms = device_sms();
    if (!mx_plan(g, sms, &pl)) return LCE_ERR_UNSUPPORTED;
    MxLaunches &l = *reinterpret_cast<MxLaunches *>(prepared->bytes);
    l.plain = mx_launch(g, pl);
    memset(l.pays, 0, sizeof(l.pays));
    if (fused && g.out_type == LCE_OUT_FLOAT32 && g.Cout % 32 == 0 && g.Cout <= kPositionsChannels) {
        if (mx_plan_as(g, sms, true, 0, &pl)) {
            l.copy = mx_launch(g, pl);
            for (MxOutput o : {MX_COPY, MX_COPY_FLOATS}) l.pays[o] = mx_positions_pay(g, pl, sms, o);
        }
        if (mx_plan_as(g, sms, true, kShortcutBytes, &pl)) {
            l.shortcut = mx_launch(g, pl);
            for (MxOutput o : {MX_SHORTCUT_COPY, MX_SHORTCUT_FLOATS}) l.pays[o] = mx_positions_pay(g, pl, sms, o);
        }
    }
    return LCE_OK;
}

lce_status launch_bconv_tensor(const PreparedLaunch &prepared, const uint32_t *in, const void *w_image, const float *mult, const float *bias,
                               const int32_t *thr, void *out, cudaStream_t s, const float *residual, uint32_t *out_packed)
{
    if (!w_image) return LCE_ERR_UNSUPPORTED;
    if (!aligned(w_image, 16)) return LCE_ERR_ALIGNMENT;
    const MxLaunches &forms = *reinterpret_cast<const MxLaunches *>(prepared.bytes);
    const MxOutput output = residual ? (out ? MX_SHORTCUT_FLOATS : MX_SHORTCUT_COPY) : out ? MX_COPY_FLOATS : MX_COPY;
    const MxLaunch &l = !(residual || out_packed) || !forms.pays[output] ? forms.plain : residual ? forms.shortcut : forms.copy;
    MxParams p = l.params;
    p.in = in; p.wimg = static_cast<const uint8_t *>(w_image); p.mult = mult; p.bias = bias; p.thr = thr; p.out = out;
    p.residual = residual; p.out_packed = out_packed;
    p.host_flag = mx_flag_for_launch(s);
    p.cp_words = (p.Cw % 4 == 0 && aligned(in, 16)) ? 4 : (p.Cw % 2 == 0 && aligned(in, 8)) ? 2 : 1;
    p.write_float = out != nullptr;
    if (l.positions) {
        MxPositionsParams q;
        q.m = p;
        q.n_dim = (p.Cout + 31) / 32 * 32;
        q.slots = min(4, kPositionsColumns / (2 * q.n_dim));
        q.wide = p.Cow == 2 && aligned(out, 8) ? 2 : 1;
        q.off_shortcut = (int32_t)l.smem - kShortcutBytes;
        if (p.out_type == LCE_OUT_BITPACKED) return launch_positions<POSITIONS_BITS>(q, l.grid, l.smem, s);
        return launch_positions<POSITIONS_FUSED>(q, l.grid, l.smem, s);
    }
    if (p.out_type == LCE_OUT_FLOAT32 && (residual || out_packed || !out || p.activation != LCE_ACT_NONE))
        return launch_mx<EPI_FLOAT_FUSED>(p, l.grid, l.smem, s);
    return launch_mx<EPI_PLAIN>(p, l.grid, l.smem, s);
}

// ---- status of the bounded waits ----------------------------------------------------------------------
namespace {
// One CTA waits, with the kernels' own helper and the given limit, on a barrier that nobody arrives
// at, and reports the expiry the way the convolution kernels do.  Touches no tensor-core state.
__global__ void mx_wait_probe_kernel(uint64_t limit_ns, int *host_flag)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!mbar_wait_bounded(&bar, 0, limit_ns)) mx_report_timeout(host_flag);
    }
}
}  // namespace

lce_status tensor_wait_probe(uint64_t limit_ns, cudaStream_t s)
{
    mx_wait_probe_kernel<<<1, 32, 0, s>>>(limit_ns, mx_flag_for_launch(s));
    return launch_status();
}

// 0 = no bounded wait has given up on the current device since the library was loaded (or since the reset).
lce_status tensor_device_status(int *status)
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_mx_status, sizeof(int)) != cudaSuccess) return LCE_ERR_CUDA;
    *status = v;
    return LCE_OK;
}

lce_status tensor_device_status_reset()
{
    const int zero = 0;
    if (cudaMemcpyToSymbol(g_mx_status, &zero, sizeof(int)) != cudaSuccess) return LCE_ERR_CUDA;
    const int dev = current_device_index();
    int *arr = g_flag_host.load(std::memory_order_acquire);
    if (arr && dev >= 0) *reinterpret_cast<volatile int *>(arr + dev) = 0;
    return LCE_OK;
}

// Host-side look at the mapped word: no synchronisation, no CUDA call beyond cudaGetDevice.
bool tensor_timeout_flagged()
{
    int *arr = g_flag_host.load(std::memory_order_acquire);
    if (!arr) return false;
    const int dev = current_device_index();
    return dev >= 0 && *reinterpret_cast<volatile int *>(arr + dev) != 0;
}

}  // namespace lce
