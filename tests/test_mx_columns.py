"""Which output pixels and channels the finisher warps of the tensor-core kernel work on: the arithmetic of
csrc/mx_columns.cuh, compiled for the host and walked through for every warp, tile, chunk and lane of a launch.  No warp may
form the address of a shortcut value outside the tensor or of a channel that does not exist, and every output belongs to
one warp."""
import ctypes
import subprocess
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2011_09398_b200" / "csrc"

SHIM = """
#include "mx_columns.cuh"
// reads: shortcut loads of each element (and of 1024 behind the last one); stores: of each pixel's words; foreign: loads by
// lanes whose channel does not exist
extern "C" void walk(int N, int OH, int OW, int Wg, int Hg, int Nt, int Cout, int dup_log2, int32_t *reads, int32_t *stores, int32_t *foreign)
{
    using namespace lce;
    const auto constants = [](uint32_t d, uint32_t *mul, uint32_t *sh) {
        uint32_t l = 0;
        while ((1ull << l) < d) ++l;
        *sh = 31 + l;
        *mul = (uint32_t)(((1ull << (31 + l)) / d) + 1);
    };
    MxGrid g{N, OH, OW, Wg, Hg, 0, 0, 0, 0};
    constants(Wg, &g.Wg_mul, &g.Wg_sh);
    constants(Hg, &g.Hg_mul, &g.Hg_sh);
    const int tiles = (int)(((int64_t)N * Hg * Wg + Nt - 1) / Nt), words = (Cout + 31) / 32;
    for (int ch0 = 0; ch0 < Cout; ch0 += 128)
        for (int warp = 0; warp < 4 * kColGroups; ++warp) {
            MxColumns f;
            mx_columns(f, Nt, Cout, ch0, dup_log2, warp);
            const int channel = ch0 + 32 * f.word;
            for (int tile = 0; tile < tiles; ++tile)
                for (int second = 0; second < 2; ++second)
                    for (int position = 0; position < 32; ++position) {
                        const int pixel = mx_chunk_pixel(f, g, tile, second, position);
                        if (pixel < 0) continue;
                        for (int lane = 0; lane < 32; ++lane) {
                            ++reads[(int64_t)pixel * Cout + channel + lane];
                            *foreign += channel + lane >= Cout;
                        }
                        if (channel < Cout) ++stores[(int64_t)pixel * words + channel / 32];
                    }
        }
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    where = tmp_path_factory.mktemp("mx_columns")
    (where / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(where / "shim.so"), str(where / "shim.cpp")], check=True)
    return ctypes.CDLL(str(where / "shim.so")).walk


# whole words of channels, as the fused form takes them: blocks of 128 that are full, and with one, two or three words missing
@pytest.mark.parametrize("cout", [32, 64, 96, 128, 160, 192, 224, 256, 288, 352])
@pytest.mark.parametrize("grid", [(1, 1, 1, 0), (2, 5, 7, 1), (3, 14, 14, 2), (1, 9, 30, 4)])  # n, oh, ow, pad positions a row and rows an image
def test_every_output_has_one_warp_and_no_address_is_outside(walk, cout, grid):
    n, oh, ow, pad = grid
    dup_log2 = 2 if cout <= 32 else 1 if cout <= 64 else 0
    for nt in range(16, 225, 16):
        reads = np.zeros(n * oh * ow * cout + 1024, np.int32)
        stores = np.zeros((n * oh * ow, cout // 32), np.int32)
        foreign = ctypes.c_int32(0)
        walk(n, oh, ow, ow + pad, oh + pad, nt, cout, dup_log2, reads.ctypes.data_as(ctypes.c_void_p), stores.ctypes.data_as(ctypes.c_void_p), ctypes.byref(foreign))
        assert foreign.value == 0 and not reads[n * oh * ow * cout:].any(), nt
        assert (reads[:n * oh * ow * cout] == 1).all() and (stores == 1).all(), nt


POSITIONS_SHIM = SHIM + """
// The tiles of 256 with positions on the lanes: how often each pixel's words are stored, and how often the pixel looked up ahead (two tiles
// of the CTA on for two words and more, four on for one) differs from the one of the tile when its turn comes
extern "C" int walk_positions(int N, int OH, int OW, int Wg, int Hg, int T, int ctas, int ahead, int32_t *stores)
{
    using namespace lce;
    const auto constants = [](uint32_t d, uint32_t *mul, uint32_t *sh) {
        uint32_t l = 0;
        while ((1ull << l) < d) ++l;
        *sh = 31 + l;
        *mul = (uint32_t)(((1ull << (31 + l)) / d) + 1);
    };
    MxGrid g{N, OH, OW, Wg, Hg, 0, 0, 0, 0};
    constants(Wg, &g.Wg_mul, &g.Wg_sh);
    constants(Hg, &g.Hg_mul, &g.Hg_sh);
    MxColumns f{};
    f.Nt = 256;
    const int n_tiles = (int)(((int64_t)N * Hg * Wg + 255) / 256), n_super = (n_tiles + T - 1) / T;
    int wrong = 0;
    for (int cta = 0; cta < ctas; ++cta) {
        int order[4096][2], count = 0;  // the CTA's tiles in turn, with their super-tiles
        for (int st = cta; st < n_super; st += ctas)
            for (int tile = st * T; tile < st * T + T && tile < n_tiles; ++tile) { order[count][0] = st; order[count++][1] = tile; }
        for (int column = 0; column < 256; ++column) {
            for (int i = 0; i < count; ++i) {
                const int pixel = mx_out_pixel(f, g, order[i][1], column);
                if (pixel >= 0) ++stores[pixel];
                const int next = i + ahead < count ? mx_out_pixel(f, g, order[i + ahead][1], column) : -1;
                wrong += mx_pixel_ahead(f, g, order[i][0], order[i][1] + ahead, column, T, ctas, n_super, n_tiles) != next;
            }
        }
    }
    return wrong;
}
"""


@pytest.mark.parametrize("grid", [(1, 1, 1, 0), (1, 16, 16, 0), (1, 1, 257, 0), (2, 5, 7, 1), (9, 28, 28, 1), (40, 13, 14, 2)])  # n, oh, ow, pad positions a row and rows an image
def test_tiles_of_256_positions_store_each_pixel_once_and_look_ahead_to_the_right_one(tmp_path, grid):
    (tmp_path / "shim.cpp").write_text(POSITIONS_SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(tmp_path / "shim.so"), str(tmp_path / "shim.cpp")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "shim.so"))
    n, oh, ow, pad = grid
    for T in range(1, 9):
        for ctas in (1, 3, 148):
            for ahead in (2, 4):
                stores = np.zeros(n * oh * ow, np.int32)
                assert lib.walk_positions(n, oh, ow, ow + pad, oh + pad, T, ctas, ahead, stores.ctypes.data_as(ctypes.c_void_p)) == 0, (T, ctas, ahead)
                assert (stores == 1).all(), (T, ctas)
