// Which phases of which barriers the issuers and finishers of the tensor-core kernel with positions on the lanes wait for
// (bconv_mx_positions.cuh): plain arithmetic, no CUDA headers, so that every order in which the roles can take their steps
// can be walked through without a GPU.
//
// A wait on an mbarrier looks at one bit: it returns while the number of finished phases is odd (parity 0) or even
// (parity 1).  So the barrier may be neither a phase behind nor two phases on when somebody asks for one: either way the bit
// is the wrong one.  Tiles are numbered as the CTA takes them; S = tiles whose accumulators TMEM has room for (2 - 4).  Each
// of four issuers has every fourth tile, each half of the finishers every second one, in order; the loaders have all of
// them in order, and start on tile t when tile t - ahead is done, ahead <= 4.
//
//   FULL_X, TILE_DONE: rings of four, phase t / 4 of barrier t % 4 is tile t's.  Never a phase behind: who waits for tile t
//   has waited for tile t - 4.  Never two on: tile t + 4 is loaded when tile t is done, so that issuer t is through with its
//   FULL_X, and the loaders with its TILE_DONE.  The finishers are through with the latter when issuer t + 4 knows that tile
//   t is read out: directly with S = 4, from tile t + 2 of the same half with S = 2, by a second wait with S = 3.
//
//   EMPTY_TILE: a ring of eight, phase t / 8 of barrier t % 8.  Issuer t waits for tile t - S, and with S = 3 for tile t - 4.
//   Never a phase behind: it has waited for those eight tiles before, at tile t - 8.  Never two on: the barrier's next tile
//   is t - S + 8 or t + 4, loaded when tile t is done.  In a ring of four the next tile would be t + 1 with S = 3: another
//   issuer's and the other half's, which needs tiles t - 2 and t - 3 to be read out, not tile t to be issued, and can be
//   through before issuer t looks.
#pragma once
#include "mx_columns.cuh"

namespace lce {

constexpr int kTileRing = 4;   // FULL_X, TILE_DONE
constexpr int kEmptyRing = 8;  // EMPTY_TILE

LCE_MX_BOTH int mx_ring_slot(int tile, int ring) { return tile & (ring - 1); }
LCE_MX_BOTH uint32_t mx_ring_parity(int tile, int ring) { return ((uint32_t)tile / (uint32_t)ring) & 1u; }

// Calls wait(tile) for each tile that must have been read out of its accumulators before tile `tile` is issued
template <class Wait>
LCE_MX_BOTH bool mx_wait_read_out(int tile, int slots, const Wait &wait)
{
    bool ok = true;
    if (tile >= slots) ok = wait(tile - slots);                       // the accumulators this tile takes
    if (slots == 3 && tile >= kTileRing) ok = ok && wait(tile - kTileRing);  // the barrier this tile is done on
    return ok;
}

}  // namespace lce
