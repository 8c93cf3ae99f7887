// Which channels, columns and output pixels a finisher warp of the tensor-core kernel works on: plain arithmetic, no CUDA
// headers, so that every address it leads to can be checked without a GPU.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define LCE_MX_BOTH __host__ __device__ __forceinline__
#else
#define LCE_MX_BOTH inline
#endif

namespace lce {

constexpr int kColGroups = 4;  // finisher warps per TMEM lane quarter

// n / d for 0 <= n < 2^31 with (mul, sh) from the host: floor(n * mul / 2^sh), exact
LCE_MX_BOTH int fast_div(int n, uint32_t mul, uint32_t sh) { return (int)(((uint64_t)(uint32_t)n * mul) >> sh); }

// The part of a tile that is a warp's.  TMEM lane quarter of the warp = warp % 4; with few output channels the 128 rows
// hold 1 << dup_log2 copies of the channel block, and the warps of copy `sub` take other columns than those of copy 0, so
// that no finisher warp is idle.
struct MxColumns {
    int Nt, n_chunks;        // tile width (0 for a warp without a chunk: no column is below it); 32-column chunks of a tile
    int group, n_groups;     // this warp takes chunks group, group + n_groups, ...
    int last_chunk;          // its last one (-1: none, because no channel of its quarter or no such column exists)
    int word;                // its 32 channels, as a word of the channel block
};

LCE_MX_BOTH void mx_columns(MxColumns &f, int Nt, int Cout, int ch0, int dup_log2, int warp)
{
    const int quarter = warp & 3;
    f.word = quarter & ((4 >> dup_log2) - 1);
    f.n_chunks = (Nt + 31) >> 5;
    f.group = ((warp >> 2) << dup_log2) + (quarter >> (2 - dup_log2));
    f.n_groups = kColGroups << dup_log2;  // 4, 8 or 16
    const bool real = ch0 + f.word * 32 < Cout && f.group < f.n_chunks;
    f.Nt = real ? Nt : 0;
    f.last_chunk = real ? f.group + ((f.n_chunks - 1 - f.group) & ~(f.n_groups - 1)) : -1;
}

// grid positions -> output pixels
struct MxGrid {
    int N, OH, OW, Wg, Hg;
    uint32_t Wg_mul, Wg_sh, Hg_mul, Hg_sh;
};

// Output pixel of column `column` of a tile, -1 where that is no output
LCE_MX_BOTH int mx_out_pixel(const MxColumns &f, const MxGrid &g, int tile, int column)
{
    const int q = tile * f.Nt + column;
    const int row = fast_div(q, g.Wg_mul, g.Wg_sh), c = q - row * g.Wg;
    const int n = fast_div(row, g.Hg_mul, g.Hg_sh), r = row - n * g.Hg;
    return column < f.Nt && n < g.N && r < g.OH && c < g.OW ? (n * g.OH + r) * g.OW + c : -1;
}

// Output pixel of a lane's position in the first or second of the warp's chunks of a tile, -1 also where the warp has no such
// chunk: shortcut values are read from these pixels before anything else is asked, and a warp whose channels do not exist
// (the channel block's last quarters where out_c is not a multiple of 128) would read the next pixels' values, behind the
// last pixel what lies past the tensor.  Its width of 0 says so at no cost (a test of last_chunk here: 366.5 -> 368.7 us on
// seventeen layers at 256 images).
LCE_MX_BOTH int mx_chunk_pixel(const MxColumns &f, const MxGrid &g, int tile, int second, int lane)
{
    if (second && f.last_chunk <= f.group) return -1;
    return mx_out_pixel(f, g, tile, (f.group + (second ? f.n_groups : 0)) * 32 + lane);
}

// Output pixel of a column of a tile that may lie behind the super-tile at hand (tiles st * T .. st * T + T - 1): the CTA's next ones are
// tile_step super-tiles apart.  -1 where that is no output, or the CTA has no such tile.
LCE_MX_BOTH int mx_pixel_ahead(const MxColumns &f, const MxGrid &g, int st, int tile, int column, int T, int tile_step, int n_super, int n_tiles)
{
    while (tile >= st * T + T && st < n_super) { tile += (tile_step - 1) * T; st += tile_step; }
    return st < n_super && tile < n_tiles ? mx_out_pixel(f, g, tile, column) : -1;
}

}  // namespace lce
