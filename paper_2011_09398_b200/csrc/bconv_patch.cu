// LceBConv2d for very few input channels (an RGB first layer): when KH*KW*Cin <= 32 the whole
// receptive field of an output pixel fits in ONE 32-bit word.  The paper pads the channel axis to
// a multiple of 32 (Section 3.2, LceQuantize), which for Cin = 3 spends nine word operations per
// output on 27 useful bits; here the taps' Cin bits are first gathered into a single "patch"
// word per pixel (im2col at bit granularity), the weights of a channel into a matching word, and
// the accumulator is K - 2*popcount(patch XOR weight word): one XOR + POPC per output.
//
// Bit-packed output (the stem of a binarized network) runs on the warp-level integer matrix instruction: a patch word
// is exactly its depth of 32, so one m16n8k32 gives 128 popcount(a AND w) for 16 channels x 8 pixels (the bit encoding
// of bconv_small.cu, with lane q of a quad taking the bits q and q + 4 of every byte).  Up to 27 bits (3x3x3) leave
// five bits of the word free: they carry popcount(a) in binary, with weights that take 64 of it off, and the
// threshold is the instruction's third operand, so an output bit is the sign of a matrix result with no arithmetic
// behind it.  What bounds it is the logic pipe: the gather (nine words per pixel) and collecting those signs.
// 224x224x3 -> 32, stride 2: batch 256 43 -> 36 us (the popcount loop before it was bound by the popcount unit), with all
// signs of a lane in one register 36 -> 28.6; batch 64 17 -> 11.4 -> 9.5 us, one image 4.6 -> 2.0 us.
// Other outputs and zero-padding: a thread owns one output pixel and walks all output channels, 32 at a time.
#include "common.cuh"
#include "mx_common.cuh"
#include "u8_mma.cuh"

namespace lce {
namespace {

constexpr int kThreads = 256;

struct PatchParams {
    const uint32_t *in;
    const uint32_t *w;
    const float *mult;
    const float *bias;
    const int32_t *thr;
    void *out;
    int32_t N, H, W, Cin, Cout, Cow, KH, KW, sh, sw, OH, OW, pt, pl;
    int32_t M, padding, out_type, activation;
};

__global__ void __launch_bounds__(kThreads)
bconv_patch_kernel(const PatchParams p)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int taps = p.KH * p.KW;
    const int cout_pad = p.Cow * 32;
    uint32_t *sWord = smem;                                             // [cout_pad] weight patch words
    int32_t *sThr = reinterpret_cast<int32_t *>(smem + cout_pad);       // [cout_pad]
    int32_t *sWsum = reinterpret_cast<int32_t *>(smem + 2 * cout_pad);  // [cout_pad][taps], zero-padding only
    const uint32_t mask = p.Cin >= 32 ? 0xffffffffu : ((1u << p.Cin) - 1u);

    for (int o = threadIdx.x; o < cout_pad; o += kThreads) {
        uint32_t word = 0u;
        if (o < p.Cout)
            for (int t = 0; t < taps; ++t) word |= (__ldg(p.w + (int64_t)o * taps + t) & mask) << (t * p.Cin);
        sWord[o] = word;
        sThr[o] = (o < p.Cout && p.out_type == LCE_OUT_BITPACKED) ? __ldg(p.thr + o) : INT32_MIN;  // pad bits -> 0
    }
    if (p.padding == LCE_PAD_SAME_ZERO) {
        for (int e = threadIdx.x; e < cout_pad * taps; e += kThreads) {
            const int o = e / taps, t = e - o * taps;
            // sum of one tap's weights over the true channels
            sWsum[e] = o < p.Cout ? p.Cin - 2 * __popc(__ldg(p.w + (int64_t)o * taps + t) & mask) : 0;
        }
    }
    __syncthreads();

    const int K = taps * p.Cin;

    for (int m = blockIdx.x * kThreads + threadIdx.x; m < p.M; m += gridDim.x * kThreads) {
        const int r = m / p.OW, ow = m - r * p.OW;
        const int n = r / p.OH, oh = r - n * p.OH;
        const int iy0 = oh * p.sh - p.pt, ix0 = ow * p.sw - p.pl;
        // gather the patch: tap t contributes its Cin bits at bit position t*Cin; taps outside the
        // image contribute zero bits (= +1.0, one-padding)
        uint32_t patch = 0u, oob = 0u;
        const uint32_t *img = p.in + (int64_t)n * p.H * p.W;
        for (int ky = 0; ky < p.KH; ++ky) {
            const int iy = iy0 + ky;
            for (int kx = 0; kx < p.KW; ++kx) {
                const int ix = ix0 + kx;
                const int t = ky * p.KW + kx;
                if (iy >= 0 && iy < p.H && ix >= 0 && ix < p.W)
                    patch |= (__ldg(img + iy * p.W + ix) & mask) << (t * p.Cin);
                else
                    oob |= 1u << t;
            }
        }
        const bool zero_fix = p.padding == LCE_PAD_SAME_ZERO && oob != 0u;
        for (int wd = 0; wd < p.Cow; ++wd) {
            uint32_t bits = 0u;
#pragma unroll 8
            for (int j = 0; j < 32; ++j) {
                const int o = wd * 32 + j;
                int32_t v = K - 2 * __popc(patch ^ sWord[o]);
                if (zero_fix) {
                    // zero-padding: the out-of-image taps counted as +1 * w; take them out again
                    for (int t = 0; t < taps; ++t)
                        if ((oob >> t) & 1u) v -= sWsum[o * taps + t];
                }
                if (p.out_type == LCE_OUT_BITPACKED) {
                    bits |= (v < sThr[o] ? 1u : 0u) << j;
                } else if (o < p.Cout) {
                    if (p.out_type == LCE_OUT_FLOAT32) {
                        const int32_t a = (p.activation == LCE_ACT_RELU && v < 0) ? 0 : v;
                        static_cast<float *>(p.out)[(int64_t)m * p.Cout + o] =
                            __fmaf_rn((float)a, __ldg(p.mult + o), __ldg(p.bias + o));
                    } else {
                        static_cast<int32_t *>(p.out)[(int64_t)m * p.Cout + o] = v;
                    }
                }
            }
            if (p.out_type == LCE_OUT_BITPACKED) static_cast<uint32_t *>(p.out)[(int64_t)m * p.Cow + wd] = bits;
        }
    }
}

// The taps' Cin bits of one output pixel as one word: tap t at bit t * Cin, taps outside the image zero (= +1.0).
// 3x3 filters: the nine words are asked for (PatchWords) well before they are put together, so that the loads of a
// warp's next pixels are in flight while it works on these.
struct PatchWords {
    uint32_t v[9];
};

__device__ __forceinline__ PatchWords load_patch3(const PatchParams &p, int n, int oh, int ow, bool exists)
{
    const int y = oh * p.sh - p.pt, x = ow * p.sw - p.pl;
    const uint32_t *at = p.in + ((int64_t)n * p.H + y) * p.W + x;
    PatchWords w;
    if (__all_sync(0xffffffffu, exists && (unsigned)y < (unsigned)max(0, p.H - 2) && (unsigned)x < (unsigned)max(0, p.W - 2))) {  // nothing to test
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
            w.v[kx] = __ldg(at + kx);
            w.v[3 + kx] = __ldg(at + p.W + kx);
            w.v[6 + kx] = __ldg(at + 2 * p.W + kx);
        }
        return w;
    }
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
        const bool row = exists && (unsigned)(y + ky) < (unsigned)p.H;
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) w.v[3 * ky + kx] = row && (unsigned)(x + kx) < (unsigned)p.W ? __ldg(at + kx) : 0u;
        at += p.W;
    }
    return w;
}

// Horner with `scale` = 2^Cin: tap t ends at bit t * Cin (pad bits of a word are 0).  Multiply-adds: the logic pipe is the
// busy one.
__device__ __forceinline__ uint32_t put_together(const PatchWords &w, uint32_t scale)
{
    uint32_t patch = w.v[8];
#pragma unroll
    for (int t = 7; t >= 0; --t) asm("mad.lo.u32 %0, %0, %1, %2;" : "+r"(patch) : "r"(scale), "r"(w.v[t]));
    return patch;
}

__device__ __forceinline__ uint32_t gather_patch(const PatchParams &p, int n, int oh, int ow, uint32_t mask)
{
    const int iy0 = oh * p.sh - p.pt, ix0 = ow * p.sw - p.pl;
    const uint32_t *img = p.in + (int64_t)n * p.H * p.W;
    uint32_t patch = 0u;
    for (int ky = 0; ky < p.KH; ++ky) {
        const int iy = iy0 + ky;
        for (int kx = 0; kx < p.KW; ++kx) {
            const int ix = ix0 + kx;
            if (iy >= 0 && iy < p.H && ix >= 0 && ix < p.W) patch |= (__ldg(img + iy * p.W + ix) & mask) << ((ky * p.KW + kx) * p.Cin);
        }
    }
    return patch;
}

__device__ __forceinline__ void compare_operands(const uint4 &c, int (&c0)[4], int (&c1)[4])
{
    asm("mov.b32 %0, %4;\n\tmov.b32 %1, %4;\n\tmov.b32 %2, %5;\n\tmov.b32 %3, %5;" : "=r"(c0[0]), "=r"(c0[1]), "=r"(c0[2]), "=r"(c0[3]) : "r"(c.x), "r"(c.y));
    asm("mov.b32 %0, %4;\n\tmov.b32 %1, %4;\n\tmov.b32 %2, %5;\n\tmov.b32 %3, %5;" : "=r"(c1[0]), "=r"(c1[1]), "=r"(c1[2]), "=r"(c1[3]) : "r"(c.z), "r"(c.w));
}

// Bit-packed output, one-padding or none.  A warp takes 32 consecutive output pixels at a time: lane = pixel for the
// gather, then four groups of 8 pixels x 32 channels.  Row r of matrix tile t is channel 4 (r % 8) + 2 t + r / 8 of the
// word, so that a lane's four sums of a pixel are four neighbouring bits, its 32 sums a register of eight nibbles, and one
// transpose of nibbles over eight lanes leaves every lane with the word of one of the 32 pixels (group by group, by a
// product, three exchanges and selections each, this took 110 of 270 instructions).  COUNTED: K <= 27, popcount(a) travels in the word.
constexpr int kLaneWords = 12;  // per lane and 32 channels: eight operand registers, four compare constants

template <bool ONE_WORD, bool COUNTED>
__global__ void __launch_bounds__(kThreads, 4)
bconv_patch_bits_kernel(const PatchParams p, int packed)
{
    extern __shared__ __align__(16) uint32_t smem[];  // [Cow][3][32 lanes][4]
    const int taps = p.KH * p.KW, K = taps * p.Cin;
    const uint32_t mask = p.Cin >= 32 ? 0xffffffffu : ((1u << p.Cin) - 1u);
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // load-time packed weights are constants of the model; plain words may come from the kernel before
    if (!packed) asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int wd = threadIdx.x >> 5; wd < p.Cow; wd += kThreads / 32) {
        uint32_t a[8];
        int32_t c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int o = wd * 32 + 4 * g + i;
            uint32_t word = 0u;
            int32_t thr = -K - 1;  // pad channels: bit 0
            if (o < p.Cout) {
                for (int t = 0; t < taps; ++t) word |= (__ldg(p.w + (int64_t)o * taps + t) & mask) << (t * p.Cin);
                thr = max(-K - 1, min(K + 1, __ldg(p.thr + o)));
            }
            // K - 2 popc(a) - 2 popc(w) + 4 popc(a AND w) < thr  <=>  0 < L + 64 popc(a) - 128 popc(a AND w), all
            // multiples of 32, so the output bit is the complement of the sign of that minus one
            c[i] = 32 * (thr - K) + 64 * __popc(word) - 1;
            // minus 2^(7 - b) for bit b of a byte, as signed bytes; the five count bits 27 .. 31 (bits 3 .. 7 of the last
            // byte, 2^(3 + i) for the digit 2^i): 8
            const auto operand = [&](int b) {
                uint32_t v = 0u;
                for (int byte = 0; byte < 4; ++byte) {
                    const int bit = 8 * byte + b;
                    const uint32_t x = bit >= 27 ? 8u : (word >> bit & 1u) ? (uint32_t)(-(1 << (7 - b))) & 0xFFu : 0u;
                    v |= x << (8 * byte);
                }
                return v;
            };
            a[(i >> 1) * 4 + (i & 1)] = COUNTED ? operand(q) : reverse_in_bytes(word) & (0x80808080u >> q);
            a[(i >> 1) * 4 + 2 + (i & 1)] = COUNTED ? operand(q + 4) : reverse_in_bytes(word) & (0x08080808u >> q);
        }
        uint4 *slot = reinterpret_cast<uint4 *>(smem) + wd * 96 + lane;
        slot[0] = make_uint4(a[0], a[1], a[2], a[3]);
        slot[32] = make_uint4(a[4], a[5], a[6], a[7]);
        slot[64] = make_uint4((uint32_t)c[0], (uint32_t)c[1], (uint32_t)c[2], (uint32_t)c[3]);
    }
    const uint32_t a_lo = 0x01010101u << q, a_hi = 0x10101010u << q;
    // image, row and column of the lane's pixel, advanced by the grid's stride with carries
    const int step = gridDim.x * kThreads;
    const int step_ow = step % p.OW, step_rows = step / p.OW, step_oh = step_rows % p.OH, step_n = step_rows / p.OH;
    uint32_t m0 = blockIdx.x * kThreads + (threadIdx.x & ~31u);  // at most 2^31 + a step: unsigned
    const uint32_t M = (uint32_t)p.M;
    int n, oh, ow;
    {
        const int m = (int)m0 + lane, r = m / p.OW;
        ow = m - r * p.OW;
        n = r / p.OH;
        oh = r - n * p.OH;
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint4 *slots = reinterpret_cast<const uint4 *>(smem) + lane;
    uint4 w0 = slots[0], w1 = slots[32], c = slots[64];
    int c0[4], c1[4];  // the third operands as the instruction wants them, in registers of their own (no moves in the loop)
    compare_operands(c, c0, c1);
    const uint32_t scale = 1u << p.Cin;
    // the transpose's steps: a lane without the bit keeps its low halves and takes the partner's low halves above them, a
    // lane with it the high ones
    const uint32_t by_16 = g & 4 ? 0x3276u : 0x5410u, by_8 = g & 2 ? 0x3715u : 0x6240u, keep_4 = g & 1 ? 0xF0F0F0F0u : 0x0F0F0F0Fu, rot_4 = g & 1 ? 28u : 4u;
    const bool square3 = p.KH == 3 && p.KW == 3;
    PatchWords next{};
    if (square3) next = load_patch3(p, n, oh, ow, m0 + lane < M);
    for (; m0 < M; m0 += step) {
        const uint32_t patch = square3 ? put_together(next, scale) : m0 + lane < M ? gather_patch(p, n, oh, ow, mask) : 0u;
        ow += step_ow;
        oh += step_oh;
        n += step_n;
        if (ow >= p.OW) { ow -= p.OW; ++oh; }
        if (oh >= p.OH) { oh -= p.OH; ++n; }
        if (square3) next = load_patch3(p, n, oh, ow, m0 + step + lane < M);
        const int ones = __popc(patch);
        const uint32_t operand = COUNTED ? patch | (uint32_t)ones << 27 : patch;
        const uint32_t pixel = m0 + (g >> 1) * 8 + 2 * q + (g & 1);
        // Several words one at a time: unrolled, they spill, and two and three words were slower than before the sums of a lane were
        // transposed at once (224x224x2 -> 40 at stride 2, 16 images 8.4 -> 8.7 us, now 8.0; 56x56x3 -> 96, 64 images 10.05 ->
        // 10.25, 9.6; 224x224x3 -> 64 at stride 2 18.6 -> 17.5, 16.5; 112x112x1 -> 64, 5x5 38.3 -> 36.1, 36.6).
#pragma unroll 1
        for (int wd = 0; wd < (ONE_WORD ? 1 : p.Cow); ++wd) {
            if (!ONE_WORD) { w0 = slots[wd * 96]; w1 = slots[wd * 96 + 32]; c = slots[wd * 96 + 64]; compare_operands(c, c0, c1); }
            // this lane's four neighbouring channels of the pixels 8 i + 2 q and 8 i + 2 q + 1, a nibble of sign bits each
            uint32_t half[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t v = 0u;
#pragma unroll
                for (int i = 2 * h + 1; i >= 2 * h; --i) {
                    const uint32_t word = __shfl_sync(0xffffffffu, operand, 8 * i + g), b0 = word & a_lo, b1 = word & a_hi;
                    int d0[4], d1[4];
                    if (COUNTED) {
                        mma_s8u8(d0, w0.x, w0.y, w0.z, w0.w, b0, b1, c0[0], c0[1], c0[2], c0[3]);
                        mma_s8u8(d1, w1.x, w1.y, w1.z, w1.w, b0, b1, c1[0], c1[1], c1[2], c1[3]);
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k) d0[k] = d1[k] = 0;
                        const int p0 = __shfl_sync(0xffffffffu, 64 * ones, 8 * i + 2 * q), p1 = __shfl_sync(0xffffffffu, 64 * ones, 8 * i + 2 * q + 1);
                        mma_u8(d0, w0.x, w0.y, w0.z, w0.w, b0, b1);
                        mma_u8(d1, w1.x, w1.y, w1.z, w1.w, b0, b1);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int more = k & 1 ? p1 : p0;
                            d0[k] = (int)(k & 2 ? c.y : c.x) + more - d0[k];
                            d1[k] = (int)(k & 2 ? c.w : c.z) + more - d1[k];
                        }
                    }
#pragma unroll
                    for (int b = 1; b >= 0; --b) {  // the lowest channel last
                        v = __funnelshift_l((uint32_t)d1[2 + b], v, 1);
                        v = __funnelshift_l((uint32_t)d1[b], v, 1);
                        v = __funnelshift_l((uint32_t)d0[2 + b], v, 1);
                        v = __funnelshift_l((uint32_t)d0[b], v, 1);
                    }
                }
                half[h] = v;
            }
            // nibble s of lane (g, q) belongs to pixel s of the quad's column q: transposed over the eight g, lane (g, q) holds
            // all eight nibbles of pixel s = g
            uint32_t v = __byte_perm(half[0], half[1], 0x5410);
            v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 16), by_16);
            v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 8), by_8);
            const uint32_t y = __shfl_xor_sync(0xffffffffu, v, 4);
            const uint32_t mine = ~((v & keep_4) | (__funnelshift_l(y, y, rot_4) & ~keep_4));
            if (pixel < M) static_cast<uint32_t *>(p.out)[ONE_WORD ? pixel : (uint64_t)pixel * (uint32_t)p.Cow + wd] = mine;
        }
    }
}

}  // namespace

bool patch_covers(const ConvGeom &g)
{
    return g.Cw == 1 && g.KH * g.KW > 1 && g.KH * g.KW * g.Cin <= 32 && g.M < (1ll << 31) - 4096 && g.Cow <= 256;
}

lce_status launch_bconv_patch(const ConvGeom &g, const uint32_t *in, const uint32_t *w, bool packed, const float *mult,
                              const float *bias, const int32_t *thr, void *out, cudaStream_t s)
{
    if (!patch_covers(g)) return LCE_ERR_UNSUPPORTED;
    PatchParams p{};
    p.in = in; p.w = w; p.mult = mult; p.bias = bias; p.thr = thr; p.out = out;
    p.N = g.N; p.H = g.H; p.W = g.W; p.Cin = g.Cin; p.Cout = g.Cout; p.Cow = g.Cow;
    p.KH = g.KH; p.KW = g.KW; p.sh = g.sh; p.sw = g.sw; p.OH = g.OH; p.OW = g.OW; p.pt = g.pt; p.pl = g.pl;
    p.M = (int32_t)g.M; p.padding = g.padding; p.out_type = g.out_type; p.activation = g.activation;
    if (g.out_type == LCE_OUT_BITPACKED && g.padding != LCE_PAD_SAME_ZERO) {
        // the blocks that fit at once (64 registers: four per SM), grid-stride beyond that: a block begins with its operands
        const int64_t bits_blocks = (g.M + kThreads - 1) / kThreads;
        const dim3 grid((unsigned)(bits_blocks < 148 * 4 ? bits_blocks : 148 * 4));
        const size_t bits_smem = (size_t)g.Cow * 32 * kLaneWords * 4;
        const bool counted = g.KH * g.KW * g.Cin <= 27;
        if (g.Cow == 1)
            return counted ? launch_dependent(bconv_patch_bits_kernel<true, true>, grid, kThreads, bits_smem, s, p, (int)packed)
                           : launch_dependent(bconv_patch_bits_kernel<true, false>, grid, kThreads, bits_smem, s, p, (int)packed);
        static SmemOptIn opted, opted_counted;
        if (counted) {
            if (!opted_counted.ensure(bconv_patch_bits_kernel<false, true>, bits_smem)) return LCE_ERR_CUDA;
            return launch_dependent(bconv_patch_bits_kernel<false, true>, grid, kThreads, bits_smem, s, p, (int)packed);
        }
        if (!opted.ensure(bconv_patch_bits_kernel<false, false>, bits_smem)) return LCE_ERR_CUDA;
        return launch_dependent(bconv_patch_bits_kernel<false, false>, grid, kThreads, bits_smem, s, p, (int)packed);
    }
    const size_t smem = (size_t)g.Cow * 32 * (2 + g.KH * g.KW) * 4;
    if (smem > 48 * 1024) return LCE_ERR_UNSUPPORTED;
    // one wave of resident blocks (8 x 256 threads per SM), grid-stride beyond that: every block pays
    // for building the weight words in shared memory, so fewer, longer-lived blocks are cheaper
    int64_t blocks = (g.M + kThreads - 1) / kThreads;
    if (blocks > 148 * 8) blocks = 148 * 8;
    bconv_patch_kernel<<<(unsigned)blocks, kThreads, smem, s>>>(p);
    return launch_status();
}

}  // namespace lce
