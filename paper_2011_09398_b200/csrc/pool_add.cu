// LceBMaxPool2d (paper Section 3.2: max-pool on packed bits is the bitwise AND of the window,
// because a 0 bit is +1 and max(sign X) = sign(max X)) and the fp32 residual add that the
// shortcut pattern of Section 5.3 places between a float-output conv and the next LceQuantize.  Launched as
// programmatic dependents: they wait for the previous kernel before their first access.
#include "common.cuh"

#include <string.h>

namespace lce {
namespace {

constexpr int kThreads = 256;

// n / d for 0 <= n < 2^31 (fast_div_constants)
struct FastDiv {
    uint32_t mul, sh;
    __device__ __forceinline__ int32_t operator()(int32_t n) const { return (int32_t)(((uint64_t)(uint32_t)n * mul) >> sh); }
};

struct PoolParams {
    const uint32_t *in;
    uint32_t *out;
    int32_t total, row0, H, W, Cw, OH, OW, PH, PW, sh, sw, pt, pl;  // total: output vectors of the launch, from output row row0 of all images on
    FastDiv by_cv, by_ow, by_oh;                                    // cv: vectors of a pixel
};

template <int VEC>
struct Words;
template <>
struct Words<1> { using type = uint32_t; };
template <>
struct Words<2> { using type = uint2; };
template <>
struct Words<4> { using type = uint4; };

__device__ __forceinline__ uint32_t both(uint32_t a, uint32_t b) { return a & b; }
__device__ __forceinline__ uint2 both(const uint2 &a, const uint2 &b) { return make_uint2(a.x & b.x, a.y & b.y); }
__device__ __forceinline__ uint4 both(const uint4 &a, const uint4 &b) { return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w); }

// A thread takes output vectors, VEC words of a pixel (the widest of 1, 2, 4 that divides a pixel's words), wherever rows
// and images end: a block to an output row left most of its threads idle on the narrow tensors behind a network's first stages
// (56x56x64, 128 images: 28 pixels of two words; 3.9 us, now 1.9; 56x56x128 4.5, now 2.5).  Out-of-image taps are skipped (AND identity = all
// ones); channel-pad bits stay 0 because they are 0 in every input word.
template <int VEC>
__global__ void __launch_bounds__(kThreads) bmaxpool_kernel(const __grid_constant__ PoolParams p)
{
    using V = typename Words<VEC>::type;
    const int32_t cv = p.Cw / VEC, H = p.H, W = p.W;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // Behind the wait: the next convolution reads its per-channel arrays before it waits, and those may come from a kernel in
    // front of the pool, which is complete from here on.  Residual stack, 128 images of 56x56 / 3 of 35x35: released here 212.0 /
    // 47.6 us, at the entry 212.9 / 47.0, not at all 212.1 / 49.3.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const V *const in = reinterpret_cast<const V *>(p.in);
    V *const out = reinterpret_cast<V *>(p.out);
    for (uint32_t e = blockIdx.x * kThreads + threadIdx.x; e < (uint32_t)p.total; e += gridDim.x * kThreads) {
        const int32_t pixel = p.by_cv((int32_t)e), local = p.by_ow(pixel), row = p.row0 + local, n = p.by_oh(row);
        const int32_t iy0 = (row - n * p.OH) * p.sh - p.pt, ix0 = (pixel - local * p.OW) * p.sw - p.pl;
        const V *at = in + ((int64_t)n * H + iy0) * W * cv + (int64_t)ix0 * cv + ((int32_t)e - pixel * cv);
        if (p.PH == 2 && p.PW == 2 && iy0 >= 0 && iy0 + 1 < H && ix0 >= 0 && ix0 + 1 < W) {
            // the usual 2x2 window, inside the image: four independent loads in flight, three ANDs
            const V *below = at + (int64_t)W * cv;
            __stcs(out + e, both(both(__ldcs(at), __ldcs(at + cv)), both(__ldcs(below), __ldcs(below + cv))));
            continue;
        }
        V acc;
        memset(&acc, 0xff, sizeof(acc));
        // the window's part inside the image, so that nothing is tested between the loads
        const int32_t ky0 = max(0, -iy0), kx0 = max(0, -ix0), rows = min(p.PH - ky0, H - max(0, iy0)), columns = min(p.PW - kx0, W - max(0, ix0));
        const V *line = at + ((int64_t)ky0 * W + kx0) * cv;
        for (int32_t y = 0; y < rows; ++y, line += (int64_t)W * cv)
            for (int32_t x = 0; x < columns; ++x) acc = both(acc, __ldg(line + (int64_t)x * cv));
        out[e] = acc;
    }
}

template <int VEC>
lce_status launch_pool(PoolParams p, int32_t batch, cudaStream_t s)
{
    // so many rows at a time that a launch has fewer than 2^31 vectors (a thread's index, a step of the grid more at the end of
    // its loop, is unsigned)
    constexpr int64_t kMost = (1ll << 31) - 1;
    const int64_t row = (int64_t)p.OW * (p.Cw / VEC), rows = (int64_t)batch * p.OH;
    if (row > kMost) return LCE_ERR_UNSUPPORTED;
    const int64_t most = kMost / row;
    fast_div_constants((uint32_t)(p.Cw / VEC), &p.by_cv.mul, &p.by_cv.sh);
    fast_div_constants((uint32_t)p.OW, &p.by_ow.mul, &p.by_ow.sh);
    fast_div_constants((uint32_t)p.OH, &p.by_oh.mul, &p.by_oh.sh);
    for (int64_t r = 0; r < rows; r += most) {
        PoolParams q = p;
        q.row0 = (int32_t)r;
        q.total = (int32_t)((rows - r < most ? rows - r : most) * row);
        q.out += r * p.OW * p.Cw;
        const int64_t blocks = (q.total + (int64_t)kThreads - 1) / kThreads;
        const lce_status st = launch_dependent(bmaxpool_kernel<VEC>, dim3((unsigned)(blocks < 148 * 16 ? blocks : 148 * 16)), kThreads, 0, s, q);
        if (st != LCE_OK) return st;
    }
    return LCE_OK;
}

// HBM-bound.  Forwards, both operands streamed: what is left in the L2 is the sum, which LceQuantize reads next (Section 5.3).
// From the last element to the first with the first operand kept, the add was faster only where the same tensors came
// again and again (quantize, pool, dequantize and add of one 205 MB tensor 164.7 us, 169.0 as it is); with new ones each time it
// was slower: the four 170.0 us against 169.4 (51 MB 46.5 and 46.2), add and quantize of the sum 126.5 against 121.7 (103 MB 62.4
// and 59.1; 13 MB the other way, 8.4 and 8.7).
__global__ void __launch_bounds__(kThreads)
add_f32_vec4_kernel(const float4 *a, const float4 *b, float4 *out, int64_t n4)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n4; i += (int64_t)gridDim.x * kThreads) {
        const float4 u = __ldcs(a + i), v = __ldcs(b + i);
        out[i] = make_float4(__fadd_rn(u.x, v.x), __fadd_rn(u.y, v.y), __fadd_rn(u.z, v.z), __fadd_rn(u.w, v.w));
    }
}

__global__ void __launch_bounds__(kThreads)
add_f32_scalar_kernel(const float *a, const float *b, float *out, int64_t begin, int64_t n)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t i = begin + (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
        out[i] = __fadd_rn(a[i], b[i]);
}

int grid_for(int64_t items, int max_blocks)
{
    int64_t b = (items + kThreads - 1) / kThreads;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

}  // namespace
}  // namespace lce

extern "C" lce_status lce_bmaxpool(const uint32_t *in, uint32_t *out, int32_t batch, int32_t in_h, int32_t in_w,
                                   int32_t channels, int32_t pool_h, int32_t pool_w, int32_t stride_h,
                                   int32_t stride_w, int32_t padding, void *stream)
{
    using namespace lce;
    if (!in || !out) return LCE_ERR_INVALID_ARG;
    if (batch <= 0 || in_h <= 0 || in_w <= 0 || channels <= 0 || pool_h <= 0 || pool_w <= 0 || stride_h <= 0 ||
        stride_w <= 0)
        return LCE_ERR_INVALID_ARG;
    if (padding != LCE_PAD_VALID && padding != LCE_PAD_SAME_ONE) return LCE_ERR_INVALID_ARG;
    if (!aligned(in, 4) || !aligned(out, 4)) return LCE_ERR_ALIGNMENT;
    const Axis ah = axis_geometry(in_h, pool_h, stride_h, padding);
    const Axis aw = axis_geometry(in_w, pool_w, stride_w, padding);
    if (ah.out <= 0 || aw.out <= 0) return LCE_ERR_INVALID_ARG;
    const int32_t Cw = (channels + 31) / 32;
    if ((int64_t)batch * ah.out >= (1ll << 31)) return LCE_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const PoolParams p{in, out, 0, 0, in_h, in_w, Cw, ah.out, aw.out, pool_h, pool_w, stride_h, stride_w, ah.pad_before, aw.pad_before, {}, {}, {}};
    if (Cw % 4 == 0 && aligned(in, 16) && aligned(out, 16)) return launch_pool<4>(p, batch, s);
    if (Cw % 2 == 0 && aligned(in, 8) && aligned(out, 8)) return launch_pool<2>(p, batch, s);
    return launch_pool<1>(p, batch, s);
}

extern "C" lce_status lce_add_f32(const float *a, const float *b, float *out, int64_t n, void *stream)
{
    using namespace lce;
    if (n < 0) return LCE_ERR_INVALID_ARG;
    if (n == 0) return LCE_OK;
    if (!a || !b || !out) return LCE_ERR_INVALID_ARG;
    if (!aligned(a, 4) || !aligned(b, 4) || !aligned(out, 4)) return LCE_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int64_t done = 0;
    if (aligned(a, 16) && aligned(b, 16) && aligned(out, 16) && n >= 4) {
        const int64_t n4 = n / 4;
        const lce_status st = launch_dependent(add_f32_vec4_kernel, dim3(grid_for(n4, 148 * 8)), kThreads, 0, s, reinterpret_cast<const float4 *>(a),
                                               reinterpret_cast<const float4 *>(b), reinterpret_cast<float4 *>(out), n4);
        done = n4 * 4;
        if (st != LCE_OK || done == n) return st;
    }
    return launch_dependent(add_f32_scalar_kernel, dim3(grid_for(n - done, 148 * 8)), kThreads, 0, s, a, b, out, done, n);
}
