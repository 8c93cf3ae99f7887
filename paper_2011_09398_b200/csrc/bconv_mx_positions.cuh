// The tensor-core kernel for few output channels (bit-packed; float with a shortcut or a re-quantised copy) with the roles of the
// operands exchanged: positions are the M dimension (a TMEM lane each), channels the N dimension (32, 64 or 96 columns).  Part of
// bconv_mx.cu, whose loaders, weight image, grid of positions and barriers it shares, and whose mx_positions_pay says when it is taken.
//
// What bounds these layers with channels on the lanes is their finishers (56x56x64: 1620 clocks a tile of 208 positions, its
// matrix instructions 950), who turn 32 channels x 32 positions of signs around with shuffles and all work on one of two
// accumulators.  With positions on the lanes a lane has all the channels of its pixel: the signs of 32 columns are the finished
// word, its words leave in one store, and an accumulator is small enough (128 positions x 64 channels: 64 columns) that several are in
// flight, read out by four warps each.  The tensor pipe loses nothing: 51 - 59 clocks for 128 x 64 x 64 against 105 for
// 208 positions x 128 rows, half of which are copies of the channels.  As a graph of ten launches: 56x56x64, 256 images 26.6 -> 22.0 us,
// 64 images 9.8 -> 8.5; 112x112x32 -> 64 at stride 2, 256 images 30.6 -> 25.6; 56x56x32, 64 images 9.2 -> 7.6.
//   * tile: 256 positions, two accumulators, issued side by side (the two share the weights' descriptor), handed to the
//     finishers and back to the loaders with one commit; two to four tiles' accumulators in TMEM;
//   * finishers: warps 0 - 7 take the even tiles of the CTA, 8 - 15 the odd ones, four warps (lane quarters) to an accumulator;
//   * issuers: four warps take the tiles in turn, since the loop around the matrix instructions costs as much as they do;
//   * loops are not unrolled: 28 warps run three different ones, and what bounds them now is how much code that is (two pairs of matrix
//     instructions written out three times: 23.1 us on 56x56x64, 256 images, once: 22.1);
//   * thresholds lie in shared memory, one per column.
// What bounds it now (56x56x64, 128 images, ncu): bits 46% of the issue slots, the tensor pipe 25% of the cycles; per issue 4.6 warps wait for
// TMEM, shared or global memory, 2 for the next step of their own chain, 2 for instructions.  A tile takes 0.84 us (128 to 256 images: 12.5 ->
// 21.8 us, 12 -> 23 tiles a CTA), its 36 matrix instructions 0.55.  With shortcut and copy 57% of the issue slots, 110 MB in 25.0 us.
#pragma once

namespace lce {
namespace {

constexpr int kPositionsChannels = 96;                      // at most: with 128 two tiles' accumulators do not fit TMEM
constexpr int kUnit = 128;                                  // positions of an accumulator
constexpr int kPositionsTile = 2 * kUnit;
constexpr int kPositionsIssuers = 4;
constexpr int kPositionsThreads = kFinishers + kLoaders + 32 * kPositionsIssuers;
constexpr int kShortcutBytes = kFinishers / 32 * 8192;       // two buffers of 32 positions x 32 channels a finisher warp
constexpr int kPositionsColumns = 480;                      // TMEM columns in front of the block scales
constexpr int BAR_EMPTY_TILE0 = BAR_EMPTY_W0;               // ring of kEmptyRing: the weights are resident, their ring's barriers unused
static_assert(kEmptyRing <= kMaxStages, "the accumulators' barriers are in place of the weight ring's");
static_assert(kPositionsThreads * 72 <= 65536, "registers of a CTA");

struct MxPositionsParams {
    MxParams m;
    int32_t n_dim;   // channels of a block, rounded up to whole words
    int32_t slots;   // tiles whose accumulators TMEM has room for (2..4)
    int32_t wide;    // words per store of bit-packed output: 2 or 1
    int32_t off_shortcut;  // in shared memory: [finisher warp][2][4 KB]
};

// 16 TMEM lanes x 32 columns by quads of threads: v[4 j + 2 i + e] is lane (thread / 4) + 8 i, column 8 j + 2 (thread % 4) + e
__device__ __forceinline__ void tmem_ld_quads(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// v[j] + c[j] < 0 for 16 columns, a bit each
__device__ __forceinline__ uint32_t mx_column_signs(float (&v)[16], const float *c)
{
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
        const float4 t = *reinterpret_cast<const float4 *>(c + j);  // the same for every lane
        asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}" : "+f"(v[j]), "+f"(v[j + 1]) : "f"(t.x), "f"(t.y));
        asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}" : "+f"(v[j + 2]), "+f"(v[j + 3]) : "f"(t.z), "f"(t.w));
    }
    uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
    for (int j = 7; j >= 0; --j) {
        m0 = __funnelshift_l(__float_as_uint(v[j]), m0, 1);
        m1 = __funnelshift_l(__float_as_uint(v[8 + j]), m1, 1);
    }
    return m0 | m1 << 8;
}

__device__ __forceinline__ bool mx_positions_finish(const MxPositionsParams &p, uint64_t *bars, const float *thresholds, uint32_t tmem_base, int warp, int lane,
                                                    int first_tile, int tile_step)
{
    MxGrid g;
    g.N = p.m.N; g.OH = p.m.OH; g.OW = p.m.OW; g.Wg = p.m.Wg; g.Hg = p.m.Hg;
    g.Wg_mul = p.m.Wg_mul; g.Wg_sh = p.m.Wg_sh; g.Hg_mul = p.m.Hg_mul; g.Hg_sh = p.m.Hg_sh;
    MxColumns tile_columns;
    tile_columns.Nt = kPositionsTile;
    const int T = p.m.T, n_tiles = p.m.n_tiles, n_super = p.m.n_super, slots = p.slots, cow = p.m.Cow, wide = p.wide, words = p.n_dim >> 5;
    uint32_t *const out = static_cast<uint32_t *>(p.m.out);
    const int half = warp >> 3, column = (warp & 7) * 32 + lane;
    const uint32_t tile_cols = (uint32_t)(2 * p.n_dim), tmem = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + ((warp & 4) ? (uint32_t)p.n_dim : 0u);
    int it = 0, slot = 0;
    for (int st = first_tile; st < n_super; st += tile_step) {
        const int end = min(st * T + T, n_tiles);
#pragma unroll 1
        for (int tile = st * T; tile < end; ++tile, ++it) {
            const uint32_t d = tmem + slot * tile_cols;
            if (++slot == slots) slot = 0;
            if ((it & 1) != half) continue;
            const int pixel = mx_out_pixel(tile_columns, g, tile, column);
            uint32_t *const at = out + (int64_t)pixel * cow;
            // the warp goes on together
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&bars[BAR_TILE_DONE0 + mx_ring_slot(it, kTileRing)], mx_ring_parity(it, kTileRing)))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t before = 0u;
#pragma unroll 1
            for (int w = 0; w < words; ++w) {
                float v[16];
                tmem_ld16(d + w * 32, v);
                uint32_t m = mx_column_signs(v, thresholds + w * 32);
                tmem_ld16(d + w * 32 + 16, v);
                if (w + 1 == words) mx_hand_back(&bars[BAR_EMPTY_TILE0 + mx_ring_slot(it, kEmptyRing)], lane);
                m |= mx_column_signs(v, thresholds + w * 32 + 16) << 16;
                if (pixel >= 0) {
                    if (wide == 1) at[w] = m;
                    else if (w) *reinterpret_cast<uint2 *>(at) = make_uint2(before, m);
                }
                before = m;
            }
        }
    }
    return true;
}

// Float output (Section 3.2) with the shortcut add and the re-quantised copy of Section 5.3; whole words of channels.  The accumulator
// is read in quads: a thread has two neighbouring channels of every eight of four positions, 8 apart, so that the four threads of
// a quad fill a 32-byte sector with one 8-byte store each, at addresses that differ by constants, and a value costs half a
// multiply-add and half a store (32 channels of a position as a 128-byte store: an address, a compare and a store each).
// The shortcut comes through shared memory: a warp copies 32 channels of its 32 positions (4 KB) two steps ahead, 16 bytes a thread,
// pieces of a row exchanged so that the quads' reads meet every bank once.  Loaded into registers before the accumulator is there
// it is bound by what the L1 can have under way beside 200 KB of shared memory: 56x56x64, 128 images, shortcut and copy 31.8 us,
// 25.0 now (34.1 with channels on the lanes; the shortcut's 103 MB take 15.7 at HBM rate).
template <bool RES, bool PACK, bool WRITE>
__device__ __forceinline__ bool mx_positions_values(const MxPositionsParams &p, uint64_t *bars, const float *scales, uint8_t *staged, uint32_t tmem_base, int warp, int lane, int first_tile, int tile_step)
{
    MxGrid g;
    g.N = p.m.N; g.OH = p.m.OH; g.OW = p.m.OW; g.Wg = p.m.Wg; g.Hg = p.m.Hg;
    g.Wg_mul = p.m.Wg_mul; g.Wg_sh = p.m.Wg_sh; g.Hg_mul = p.m.Hg_mul; g.Hg_sh = p.m.Hg_sh;
    MxColumns tile_columns;
    tile_columns.Nt = kPositionsTile;
    const int T = p.m.T, n_tiles = p.m.n_tiles, n_super = p.m.n_super, slots = p.slots, cout = p.n_dim;
    const int half = warp >> 3, column = (warp & 7) * 32 + lane, quad = lane & 3;
    const uint32_t tile_cols = (uint32_t)(2 * cout), tmem = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + ((warp & 4) ? (uint32_t)cout : 0u);
    float *const out = static_cast<float *>(p.m.out) + 2 * quad;
    const float floor_v = p.m.activation == LCE_ACT_RELU ? 0.f : -INFINITY;
    scales += 4 * quad;  // multiplier, multiplier, bias, bias of two channels
    // the shortcut's way: this warp's two buffers, and its next tile's pixels
    const uint32_t stage = RES ? smem_u32(staged) + (uint32_t)warp * 8192u : 0u;
    const auto pixel_of = [&](int st, int tile) { return mx_pixel_ahead(tile_columns, g, st, tile, column, T, tile_step, n_super, n_tiles); };
    const auto copy = [&](int px, int c, uint32_t buffer) {  // 32 channels from c on
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = 4 * i + (lane >> 3), from = __shfl_sync(0xffffffffu, px, row);
            const uint32_t to = buffer + row * 128 + (((lane & 7) ^ (2 * (row & 3))) << 4);
            const float *src = p.m.residual + (int64_t)from * cout + c + 4 * (lane & 7);
            if (from >= 0) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(src) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int it = 0, slot = 0, next_pixel = -1, step = 0;
    if (RES) {
        next_pixel = pixel_of(first_tile, first_tile * T + half);
        copy(next_pixel, 0, stage);
        if (cout > 32) copy(next_pixel, 32, stage + 4096);
        else copy(pixel_of(first_tile, first_tile * T + half + 2), 0, stage + 4096);
    }
    for (int st = first_tile; st < n_super; st += tile_step) {
        const int end = min(st * T + T, n_tiles);
#pragma unroll 1
        for (int tile = st * T; tile < end; ++tile, ++it) {
            const uint32_t d = tmem + slot * tile_cols;
            if (++slot == slots) slot = 0;
            if ((it & 1) != half) continue;
            const int pixel = RES ? next_pixel : mx_out_pixel(tile_columns, g, tile, column);
            if (RES) next_pixel = pixel_of(st, tile + 2);
            int64_t at[4];  // of the thread's four positions, -1: no output
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int px = __shfl_sync(0xffffffffu, pixel, (lane >> 2) + 8 * i);
                at[i] = px < 0 ? -1 : (int64_t)px * cout;
            }
            // the warp goes on together
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&bars[BAR_TILE_DONE0 + mx_ring_slot(it, kTileRing)], mx_ring_parity(it, kTileRing)))) {
                if (RES) asm volatile("cp.async.wait_all;" ::: "memory");  // nothing in flight at the end
                return false;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int c = 0; c < cout; c += 32, ++step) {
                uint32_t bits[4];
                const uint32_t from = stage + (uint32_t)(step & 1) * 4096u + (lane >> 2) * 128 + (uint32_t)(quad & 1) * 8u;
                if (RES) {
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    __syncwarp();
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v[16];
                    tmem_ld_quads(d + c + ((uint32_t)(16 * h) << 16), v);
                    if (h == 1 && c + 32 == cout) mx_hand_back(&bars[BAR_EMPTY_TILE0 + mx_ring_slot(it, kEmptyRing)], lane);
                    uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
                    for (int j = 3; j >= 0; --j) {
                        const float4 t = *reinterpret_cast<const float4 *>(scales + 2 * c + 16 * j);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            float y0 = v[4 * j + 2 * i], y1 = v[4 * j + 2 * i + 1];
                            y0 = fmaxf(y0, floor_v);
                            y1 = fmaxf(y1, floor_v);
                            asm("{\n\t.reg .b64 y, s, b;\n\tmov.b64 y, {%0, %1};\n\tmov.b64 s, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tfma.rn.f32x2 y, y, s, b;\n\tmov.b64 {%0, %1}, y;\n\t}" : "+f"(y0), "+f"(y1) : "f"(t.x), "f"(t.y), "f"(t.z), "f"(t.w));
                            if (RES) {
                                float r0, r1;
                                asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r0), "=f"(r1) : "r"(from + (16 * h + 8 * i) * 128 + (((2 * j + (quad >> 1)) ^ (2 * ((lane >> 2) & 3))) << 4)));
                                y0 = __fadd_rn(y0, r0);
                                y1 = __fadd_rn(y1, r1);
                            }
                            if (WRITE && at[2 * h + i] >= 0) *reinterpret_cast<float2 *>(out + at[2 * h + i] + c + 8 * j) = make_float2(y0, y1);
                            if (PACK) {  // the sign of y + 0, which makes -0.0 and NaN positive
                                uint32_t &m = i ? m1 : m0;
                                m = __funnelshift_l(__float_as_uint(y1 + 0.f), m << 6, 1);
                                m = __funnelshift_l(__float_as_uint(y0 + 0.f), m, 1);
                            }
                        }
                    }
                    bits[2 * h] = m0;
                    bits[2 * h + 1] = m1;
                }
                if (RES) {  // two steps ahead: the same channels or those of this warp's next tile
                    __syncwarp();
                    const int ahead = c + 64;
                    const bool here = ahead < cout;
                    copy(here ? pixel : cout == 32 ? pixel_of(st, tile + 4) : next_pixel, here ? ahead : ahead - (cout == 32 ? 64 : cout), stage + (uint32_t)(step & 1) * 4096u);
                }
                if (PACK) {
                    uint32_t word = 0u;
                    int64_t where = -1;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t m = bits[i] << (2 * quad);
                        m |= __shfl_xor_sync(0xffffffffu, m, 1);
                        m |= __shfl_xor_sync(0xffffffffu, m, 2);
                        if (quad == i) { word = m; where = at[i]; }
                    }
                    if (where >= 0) p.m.out_packed[(where + c) >> 5] = word;
                }
            }
        }
    }
    if (RES) asm volatile("cp.async.wait_all;" ::: "memory");
    return true;
}

__device__ __forceinline__ bool mx_positions_issue(const MxPositionsParams &p, const uint8_t *smem, uint64_t *bars, uint32_t tmem_base, int mine,
                                                   int first_tile, int tile_step)
{
    const uint2 *tbl = reinterpret_cast<const uint2 *>(smem + p.m.off_tbl);
    // descriptors: see bconv_mx_kernel; here A is the positions and B the weights, N channels
    const uint32_t idesc = (1u << 7) | (1u << 10) | ((uint32_t)(p.n_dim >> 3) << 17) | (1u << 23) | ((uint32_t)(kUnit >> 4) << 24);
    const uint32_t desc_hi = 8u | (1u << 14);
    const int T = p.m.T, n_tiles = p.m.n_tiles, n_super = p.m.n_super, n_xbuf = p.m.n_xbuf, pairs = p.m.pairs, slots = p.slots;
    const uint32_t w_lo = ((uint32_t)p.m.off_w >> 4) + (smem_u32(smem) >> 4) + (128u << 16);
    const uint32_t x_lo0 = ((uint32_t)p.m.off_x >> 4) + (smem_u32(smem) >> 4), x_units = (uint32_t)p.m.x_bytes >> 4;
    const uint32_t n_dim = (uint32_t)p.n_dim, sfa = tmem_base + kSfaCol, sfb = tmem_base + kSfbCol;
    bool ok = mbar_wait_bounded(&bars[BAR_SCALES], 0) && mbar_wait_bounded(&bars[BAR_FULL_W0], 0);
    int it = 0, xbuf = 0, slot = 0;
    for (int st = first_tile; st < n_super; st += tile_step, xbuf = xbuf + 1 == n_xbuf ? 0 : xbuf + 1) {
        const int end = min(T, n_tiles - st * T);
#pragma unroll 1
        for (int k = 0; k < end; ++k, ++it) {
            const uint32_t d = tmem_base + slot * 2 * n_dim;
            if (++slot == slots) slot = 0;
            if ((it & (kPositionsIssuers - 1)) != mine) continue;
            ok = ok && mbar_wait_bounded(&bars[BAR_FULL_X0 + mx_ring_slot(it, kTileRing)], mx_ring_parity(it, kTileRing));
            ok = ok && mx_wait_read_out(it, slots, [&](int tile) {
                return mbar_wait_bounded(&bars[BAR_EMPTY_TILE0 + mx_ring_slot(tile, kEmptyRing)], mx_ring_parity(tile, kEmptyRing));
            });
            if (!__all_sync(0xffffffffu, ok)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) {
                const uint32_t x_lo = x_lo0 + (uint32_t)xbuf * x_units + (uint32_t)(k * kPositionsTile);
#pragma unroll 1
                for (int e = 0; e < pairs; ++e) {
                    const uint2 o = tbl[e];
                    mx_mma(d, x_lo + o.y, w_lo + o.x, desc_hi, idesc, sfa, sfb, e > 0);
                    mx_mma(d + n_dim, x_lo + kUnit + o.y, w_lo + o.x, desc_hi, idesc, sfa, sfb, e > 0);
                }
                mma_commit(&bars[BAR_TILE_DONE0 + mx_ring_slot(it, kTileRing)]);  // to the finishers and to the loaders
            }
            __syncwarp();
        }
    }
    return ok;
}

enum { POSITIONS_BITS, POSITIONS_FUSED };  // bit-packed output; float output with a shortcut or a re-quantised copy

template <int FORM>
__global__ void __launch_bounds__(kPositionsThreads, 1) bconv_mx_positions_kernel(const __grid_constant__ MxPositionsParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBars);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kOffSlot);
    float *thresholds = reinterpret_cast<float *>(smem + kOffPix);      // of the CTA's channels, negated
    uint32_t *raw0 = reinterpret_cast<uint32_t *>(smem + kOffDyn);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int first_tile = blockIdx.x, tile_step = gridDim.x;

    // the next kernel of the stream may start setting itself up as soon as every CTA of this one has got here
    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- set-up, side by side, as in bconv_mx_kernel ------------------------------------------------------
    if (warp == kIssuerWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp == kIssuerWarp + 1) {
        for (int b = lane; b < BAR_COUNT; b += 32)
            mbar_init(&bars[b], b <= BAR_FULL_X3 ? kLoaders : b >= BAR_EMPTY_TILE0 && b < BAR_EMPTY_TILE0 + kEmptyRing ? 8 : b == BAR_SCALES ? 4 : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncwarp();  // the weights' barrier is another lane's
        if (lane == 0) mbar_expect_tx(&bars[BAR_FULL_W0], (uint32_t)(p.m.pairs * kPairBytes));
        __syncwarp();
        const int share = (p.m.pairs + 31) >> 5, first = lane * share, n = min(share, p.m.pairs - first);
        if (n > 0) bulk_copy_g2s(smem + p.m.off_w + (size_t)first * kPairBytes, p.m.wimg + (size_t)first * kPairBytes, (uint32_t)(n * kPairBytes), &bars[BAR_FULL_W0]);
    } else if (tid < kFinishers) {
        uint2 *tbl = reinterpret_cast<uint2 *>(smem + p.m.off_tbl);
        const int even = p.m.Cw & ~1, paired = p.m.KH * p.m.KW * even, words = p.m.KH * p.m.KW * p.m.Cw;
        for (int e = tid; e < p.m.pairs; e += kFinishers) {
            const uint32_t first = word_b_offset(p.m, 2 * e, even, paired);
            const uint32_t apart = 2 * e < paired ? (uint32_t)p.m.P : 2 * e + 1 < words ? word_b_offset(p.m, 2 * e + 1, even, paired) - first : 1u;
            tbl[e] = make_uint2((uint32_t)e * (kPairBytes >> 4), first | apart << 16);
        }
    }
    MxLoad ld;
    MxPos stage{0, 0, 0};
    int form = 0;
    const int ltid = tid - kFinishers;  // a loader's number
    const bool loader = ltid >= 0 && ltid < kLoaders;
    if (loader) {
        form = mx_load_setup(p.m, ld);
        stage = mx_position(first_tile * p.m.T * kPositionsTile + ltid, p.m);
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the activations may come from the previous kernel
        if (first_tile < p.m.n_super) {
            if (p.m.n_phase == 1) mx_prefetch<0, MX_S1>(ld, stage, kPositionsTile + p.m.halo, raw0, ltid, p.m.cp_words);
            else mx_prefetch<0, MX_S2>(ld, stage, kPositionsTile + p.m.halo, raw0, ltid, p.m.cp_words);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    if (warp < 4) {
        // block scales: every byte 0x7F = 2^0
        const uint32_t one = 0x7F7F7F7Fu;
        const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16) + kSfaCol;
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
        uint8_t *sX0 = smem + p.m.off_x;
#define LCE_MX_LOAD_POSITIONS(CW, FORM) ok = mx_load_tiles<CW, FORM>(p.m, ld, stage, bars, raw0, sX0, ltid, first_tile, tile_step)
        LCE_MX_FORMS(LCE_MX_LOAD_POSITIONS)
    } else if (tid < kFinishers) {
        if (FORM != POSITIONS_BITS) {  // by pairs of channels: two multipliers, two biases
            if (tid < p.n_dim) {
                thresholds[4 * (tid >> 1) + (tid & 1)] = __ldg(p.m.mult + tid);
                thresholds[4 * (tid >> 1) + 2 + (tid & 1)] = __ldg(p.m.bias + tid);
            }
        } else if (tid < p.n_dim)  // constants of the model.  acc < thr is unchanged by clamping thr to [-K-1, K+1] (|acc| <= K), and then thr is exact in fp32
            thresholds[tid] = tid < p.m.Cout ? -(float)max(-p.m.K - 1, min(p.m.K + 1, __ldg(p.m.thr + tid))) : INFINITY;
        asm volatile("bar.sync 1, %0;" ::"n"(kFinishers) : "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory");  // outputs: only after the previous kernel
#define LCE_MX_VALUES(...) mx_positions_values<__VA_ARGS__>(p, bars, thresholds, smem + p.off_shortcut, tmem_base, warp, lane, first_tile, tile_step)
        if (FORM == POSITIONS_BITS) {
            ok = mx_positions_finish(p, bars, thresholds, tmem_base, warp, lane, first_tile, tile_step);
        } else {
            switch ((p.m.residual ? 4 : 0) | (p.m.out_packed ? 2 : 0) | (p.m.write_float ? 1 : 0)) {
                case 2: ok = LCE_MX_VALUES(false, true, false); break;
                case 3: ok = LCE_MX_VALUES(false, true, true); break;
                case 5: ok = LCE_MX_VALUES(true, false, true); break;
                case 6: ok = LCE_MX_VALUES(true, true, false); break;
                default: ok = LCE_MX_VALUES(true, true, true); break;
            }
        }
    } else {
        ok = mx_positions_issue(p, smem, bars, tmem_base, warp - kIssuerWarp, first_tile, tile_step);
    }
    if (!ok) mx_report_timeout(p.m.host_flag);

    // ---- tear-down: nothing of this CTA may still be in flight when its TMEM and shared memory go ----
    // When no wait gave up, the finishers have waited for the matrix instructions of every tile and the issuers for the weights.
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (!__syncthreads_and(ok)) {
        if (warp >= kIssuerWarp && elect_one()) {
            uint64_t *done = &bars[BAR_FULL_W0 + 1 + warp - kIssuerWarp];  // of the unused ring
            mma_commit(done);                                              // arrives when every MMA this lane issued has finished
            bool drained = mbar_wait_bounded(done, 0);
            if (warp == kIssuerWarp) drained = mbar_wait_bounded(&bars[BAR_FULL_W0], 0) && drained;
            if (!drained) mx_report_timeout(p.m.host_flag);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == kIssuerWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
}

}  // namespace
}  // namespace lce
