// LceQuantize / LceDequantize (paper Section 3.2): sign-binarize and pack 32 channels per
// word, and the inverse.  Both are single-pass HBM streaming kernels, launched as programmatic dependents: they
// wait for the previous kernel before their first access.  LceQuantize lets its own dependent start early, so that
// the convolution behind it fetches its weights meanwhile.
#include "common.cuh"

namespace lce {
namespace {

constexpr int kPackThreads = 256;
constexpr int kWordsPerWarpPass = 32;  // one warp turns 32x32 floats (4 KB) into 32 words per pass

// channels % 32 == 0: the flat float array is a sequence of 32-float groups, each giving one
// word.  A warp reads group g with one coalesced 128-byte load (lane = channel within the
// group); __ballot_sync(x < 0) is the packed word (lane order = bit order, LSB = lowest
// channel).  All 32 loads of a pass are in flight before the first ballot; the 32 ballots are
// handed out four per lane to lanes 0..7, which write them with one 128-bit store each (128
// contiguous bytes per warp).  Passes are small so that even a 100K-word tensor gives every SM
// several warps of work: the kernel is latency-bound otherwise.
template <bool KEEP>
__global__ void __launch_bounds__(kPackThreads)
bitpack_aligned_kernel(const float *__restrict__ x, uint32_t *__restrict__ out, int64_t n_words)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * kPackThreads + threadIdx.x) >> 5;
    const int64_t n_warps = ((int64_t)gridDim.x * kPackThreads) >> 5;
    for (int64_t w0 = warp * kWordsPerWarpPass; w0 < n_words; w0 += n_warps * kWordsPerWarpPass) {
        if (w0 + kWordsPerWarpPass <= n_words) {
            float v[kWordsPerWarpPass];
#pragma unroll
            for (int u = 0; u < kWordsPerWarpPass; ++u) v[u] = KEEP ? __ldg(x + (w0 + u) * 32 + lane) : __ldcs(x + (w0 + u) * 32 + lane);
            uint32_t mine[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int u = 0; u < kWordsPerWarpPass; ++u) {
                const uint32_t word = __ballot_sync(0xffffffffu, v[u] < 0.0f);
                if ((u >> 2) == lane) mine[u & 3] = word;
            }
            // out + w0 is 16-byte aligned: w0 is a multiple of 32 words and out is checked on the host
            if (lane < kWordsPerWarpPass / 4)
                reinterpret_cast<uint4 *>(out + w0)[lane] = make_uint4(mine[0], mine[1], mine[2], mine[3]);
        } else {  // ragged last pass of the tensor
            for (int64_t w = w0; w < n_words; ++w) {
                const uint32_t word = __ballot_sync(0xffffffffu, x[w * 32 + lane] < 0.0f);
                if (lane == 0) out[w] = word;
            }
        }
    }
}

// Any channel count: a block takes a run of whole rows.  Its warps turn the run's floats into a stream of sign bits,
// 32 consecutive floats per ballot whatever the row length (coalesced, 16 loads in flight), kept in shared memory;
// then every output word is a funnel shift out of that stream.  (One thread per word reading its channels one after
// the other ran at a sixth of the bandwidth; this takes 21.6 us for 64x56x56x100, 3.8 TB/s.)
constexpr int kStreamFloats = 8192;   // floats of a run, at most; a longer row is cut into segments of as many

// What a block works on: `run` whole rows, or segment `s` of one row.
struct StreamUnit {
    int64_t first_float, first_word;
    int floats, words;
};
__device__ __forceinline__ StreamUnit stream_unit(int64_t unit, int64_t rows, int32_t channels, int32_t words, int32_t run, int32_t segments)
{
    StreamUnit u;
    if (segments == 1) {
        const int64_t r0 = unit * run;
        const int n = (int)min((int64_t)run, rows - r0);
        u.first_float = r0 * channels;
        u.first_word = r0 * words;
        u.floats = n * channels;
        u.words = n * words;
    } else {
        const int64_t row = unit / segments;
        const int s = (int)(unit - row * segments);
        u.first_float = row * channels + (int64_t)s * kStreamFloats;
        u.first_word = row * words + s * (kStreamFloats / 32);
        u.floats = min(kStreamFloats, channels - s * kStreamFloats);
        u.words = (u.floats + 31) / 32;
    }
    return u;
}
constexpr int kStreamLoads = 16;

__global__ void __launch_bounds__(kPackThreads)
bitpack_stream_kernel(const float *__restrict__ x, uint32_t *__restrict__ out, int64_t rows, int32_t channels, int32_t words, int32_t run,
                      int32_t segments, int64_t units, uint32_t words_mul, uint32_t words_sh)
{
    extern __shared__ uint32_t bits[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = kPackThreads / 32;
    for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
        const StreamUnit u = stream_unit(unit, rows, channels, words, run, segments);
        const int floats = u.floats, groups = (floats + 31) / 32;
        const float *src = x + u.first_float;
        for (int g0 = warp * kStreamLoads; g0 < groups; g0 += warps * kStreamLoads) {
            float v[kStreamLoads];
#pragma unroll
            for (int u = 0; u < kStreamLoads; ++u) {
                const int i = (g0 + u) * 32 + lane;
                v[u] = i < floats ? __ldcs(src + i) : 0.0f;
            }
            uint32_t mine = 0u;
#pragma unroll
            for (int u = 0; u < kStreamLoads; ++u) {
                const uint32_t word = __ballot_sync(0xffffffffu, v[u] < 0.0f);
                if (lane == u) mine = word;
            }
            if (lane < kStreamLoads && g0 + lane <= groups) bits[g0 + lane] = mine;  // one word past the last: read by the funnel shift
        }
        if (threadIdx.x == 0 && groups % kStreamLoads == 0) bits[groups] = 0u;
        __syncthreads();
        uint32_t *dst = out + u.first_word;
        for (int e = threadIdx.x; e < u.words; e += kPackThreads) {
            int at = e * 32, nc = floats - at;
            if (segments == 1) {
                const int r = (int)(((uint64_t)(uint32_t)e * words_mul) >> words_sh), j = e - r * words;
                at = r * channels + j * 32;
                nc = channels - j * 32;
            }
            const uint32_t word = __funnelshift_r(bits[at >> 5], bits[(at >> 5) + 1], at & 31);
            dst[e] = nc >= 32 ? word : word & ((1u << nc) - 1u);  // pad bits stay 0
        }
        __syncthreads();
    }
}

// Very few channels (an RGB image: C = 3): one word per pixel.  A thread takes four consecutive
// pixels = 4*C floats = C aligned 128-bit loads, all in flight together, and writes its four words
// with one 128-bit store; the `rest` rows past the last whole group of four are one thread each.
template <int C>
__global__ void __launch_bounds__(kPackThreads)
bitpack_few_channels_kernel(const float4 *__restrict__ x, uint4 *__restrict__ out, int64_t groups, int32_t rest)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t i = (int64_t)blockIdx.x * kPackThreads + threadIdx.x; i < groups;
         i += (int64_t)gridDim.x * kPackThreads) {
        float v[4 * C];
#pragma unroll
        for (int q = 0; q < C; ++q) {
            const float4 f = __ldcs(x + i * C + q);
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
        uint32_t w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            w[r] = 0u;
#pragma unroll
            for (int c = 0; c < C; ++c) w[r] |= (v[r * C + c] < 0.0f ? 1u : 0u) << c;
        }
        out[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (blockIdx.x == 0 && (int)threadIdx.x < rest) {
        const float *row = reinterpret_cast<const float *>(x + groups * C) + threadIdx.x * C;
        uint32_t w = 0u;
#pragma unroll
        for (int c = 0; c < C; ++c) w |= (row[c] < 0.0f ? 1u : 0u) << c;
        reinterpret_cast<uint32_t *>(out + groups)[threadIdx.x] = w;
    }
}

template <int C>
lce_status launch_few_channels(const float *x, uint32_t *out, int64_t rows, int max_blocks, cudaStream_t s)
{
    const int64_t groups = rows / 4;
    int64_t b = (groups + kPackThreads - 1) / kPackThreads;
    if (b > max_blocks) b = max_blocks;
    return launch_dependent(bitpack_few_channels_kernel<C>, dim3((unsigned)b), kPackThreads, 0, s, reinterpret_cast<const float4 *>(x), reinterpret_cast<uint4 *>(out), groups, (int32_t)(rows - 4 * groups));
}

// LceDequantize, any channel count: a block takes a run of whole rows (as many as make whole 16-byte pieces of
// output), brings their words into shared memory and writes the run's floats four at a time; the row of a float is
// divided out once per four.
__global__ void __launch_bounds__(kPackThreads)
unpack_stream_kernel(const uint32_t *__restrict__ in, float *__restrict__ out, int64_t rows, int32_t channels, int32_t words, int32_t run,
                     int32_t segments, int64_t units, uint32_t channels_mul, uint32_t channels_sh, int32_t vec)
{
    extern __shared__ uint32_t bits[];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
        const StreamUnit un = stream_unit(unit, rows, channels, words, run, segments);
        const int floats = un.floats;
        for (int e = threadIdx.x; e < un.words; e += kPackThreads) bits[e] = __ldcs(in + un.first_word + e);
        __syncthreads();
        float *dst = out + un.first_float;
        for (int e = threadIdx.x * 4; e < floats; e += kPackThreads * 4) {
            int r = segments == 1 ? (int)(((uint64_t)(uint32_t)e * channels_mul) >> channels_sh) : 0, c = e - r * channels;
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                v[u] = (bits[min(r * words + (c >> 5), un.words - 1)] >> (c & 31)) & 1u ? -1.0f : 1.0f;
                if (++c == channels) { c = 0; ++r; }
            }
            if (vec && e + 4 <= floats) {
                __stcs(reinterpret_cast<float4 *>(dst + e), make_float4(v[0], v[1], v[2], v[3]));
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e + u < floats) dst[e + u] = v[u];
            }
        }
        __syncthreads();
    }
}

// channels % 32 == 0 and a 16-byte aligned output: thread t writes the four floats of bits
// 4*(t%8) .. +3 of word t/8 with one 128-bit store (a warp stores 512 contiguous bytes and reads four
// words); no divisions.
__global__ void __launch_bounds__(kPackThreads)
unpack_aligned_kernel(const uint32_t *__restrict__ in, float4 *__restrict__ out, int64_t n_quads)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t t = (int64_t)blockIdx.x * kPackThreads + threadIdx.x; t < n_quads; t += (int64_t)gridDim.x * kPackThreads) {
        const uint32_t nib = (__ldg(in + (t >> 3)) >> (4 * (int)(t & 7))) & 0xFu;
        __stcs(out + t, make_float4((nib & 1u) ? -1.0f : 1.0f, (nib & 2u) ? -1.0f : 1.0f, (nib & 4u) ? -1.0f : 1.0f,
                                    (nib & 8u) ? -1.0f : 1.0f));
    }
}

int grid_for(int64_t work_items, int per_block, int max_blocks)
{
    int64_t b = (work_items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

// rows of a block's run: up to kStreamFloats floats, fewer where the tensor would not give every SM a few runs, a
// multiple of 4 where there are that many (whole 16-byte pieces whatever the channel count)
int64_t stream_run(int64_t rows, int32_t channels)
{
    int64_t run = kStreamFloats / channels;
    const int64_t spread = rows / (148 * 4);
    if (run > spread) run = spread;
    if (run >= 4) run &= ~3ll;
    return run < 1 ? 1 : run;
}

}  // namespace
}  // namespace lce

extern "C" lce_status lce_bitpack(const float *x, uint32_t *out, int64_t rows, int32_t channels, void *stream)
{
    using namespace lce;
    if (rows < 0 || channels <= 0) return LCE_ERR_INVALID_ARG;
    if (rows == 0) return LCE_OK;
    if (!x || !out) return LCE_ERR_INVALID_ARG;
    if (!aligned(x, 4) || !aligned(out, 4)) return LCE_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int32_t words = (channels + 31) / 32;
    const int64_t n_words = rows * words;
    // up to 148 SMs x 8 resident blocks of 256 threads x 4 passes in the queue; grid-stride loops cover the rest
    const int max_blocks = 148 * 8 * 4;
    if (channels % 32 == 0 && aligned(out, 16)) {
        const int64_t passes = (n_words + kWordsPerWarpPass - 1) / kWordsPerWarpPass;
        // A tensor that fits in the L2 stays there: it is a shortcut's operand or comes back as one (51 MB, quantized and then
        // added to another tensor, new ones each time: 30.7 -> 27.5 us); a larger one would only push out what is there (205 MB: 30.1 us, 31.8 if kept; the residual stack 217 and 225).
        const auto kernel = n_words * 128 <= (64ll << 20) ? bitpack_aligned_kernel<true> : bitpack_aligned_kernel<false>;
        return launch_dependent(kernel, dim3(grid_for(passes, kPackThreads / 32, max_blocks)), kPackThreads, 0, s, x, out, n_words);
    }
    if (channels <= 4 && rows >= 4 && aligned(x, 16) && aligned(out, 16)) {
        if (channels == 1) return launch_few_channels<1>(x, out, rows, max_blocks * 4, s);
        if (channels == 2) return launch_few_channels<2>(x, out, rows, max_blocks * 4, s);
        if (channels == 3) return launch_few_channels<3>(x, out, rows, max_blocks * 4, s);
        return launch_few_channels<4>(x, out, rows, max_blocks * 4, s);
    }
    const int64_t run = stream_run(rows, channels), segments = (channels + kStreamFloats - 1) / kStreamFloats, units = segments == 1 ? (rows + run - 1) / run : rows * segments;
    uint32_t mul, sh;
    fast_div_constants((uint32_t)words, &mul, &sh);
    return launch_dependent(bitpack_stream_kernel, dim3(grid_for(units, 1, max_blocks)), kPackThreads, (kStreamFloats / 32 + 1) * 4, s, x, out, rows, channels, words,
                            (int32_t)run, (int32_t)segments, units, mul, sh);
}

extern "C" lce_status lce_unpack(const uint32_t *in, float *out, int64_t rows, int32_t channels, void *stream)
{
    using namespace lce;
    if (rows < 0 || channels <= 0) return LCE_ERR_INVALID_ARG;
    if (rows == 0) return LCE_OK;
    if (!in || !out) return LCE_ERR_INVALID_ARG;
    if (!aligned(in, 4) || !aligned(out, 4)) return LCE_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int32_t words = (channels + 31) / 32;
    if (channels % 32 == 0 && aligned(out, 16)) {
        const int64_t n_quads = rows * channels / 4;
        return launch_dependent(unpack_aligned_kernel, dim3(grid_for(n_quads, kPackThreads, 148 * 32)), kPackThreads, 0, s, in, reinterpret_cast<float4 *>(out), n_quads);
    }
    const int64_t run = stream_run(rows, channels), segments = (channels + kStreamFloats - 1) / kStreamFloats, units = segments == 1 ? (rows + run - 1) / run : rows * segments;
    uint32_t mul, sh;
    fast_div_constants((uint32_t)channels, &mul, &sh);
    const int32_t vec = aligned(out, 16) && (segments == 1 ? run * channels : (int64_t)channels) % 4 == 0;  // every run / segment starts on 16 bytes
    const size_t smem = segments == 1 ? (size_t)run * words * 4 : kStreamFloats / 32 * 4;                  // at most 32 KB: 8192 one-channel rows
    return launch_dependent(unpack_stream_kernel, dim3(grid_for(units, 1, 148 * 32)), kPackThreads, smem, s, in, out, rows, channels, words, (int32_t)run,
                            (int32_t)segments, units, mul, sh, vec);
}
