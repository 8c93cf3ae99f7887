"""The barriers of the tensor-core kernel with positions on the lanes: the ring arithmetic of csrc/mx_rings.cuh, compiled for the
host and walked through in every order in which loaders, issuers, matrix instructions and finishers can take their steps.  No
order may get stuck, no wait may return for another phase than its own."""
import ctypes
import re
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2011_09398_b200" / "csrc"

MODEL = """
#include <unordered_set>
#include <vector>
#include "mx_rings.cuh"
using namespace lce;

// Two threads stand for the loaders and two warps for each half of the finishers: enough for one to be ahead of another.
struct State {
    uint8_t loaded[2], issued[4], waits[4], finished[2][2];  // tiles, of its own, that a role is through with; waits an issuer is through with
    uint32_t done;                                           // tiles whose matrix instructions have finished
    uint64_t key() const  // up to 18 tiles
    {
        uint64_t k = done;
        for (int i = 0; i < 2; ++i) k = k << 5 | loaded[i];
        for (int i = 0; i < 4; ++i) k = (k << 3 | issued[i]) << 2 | waits[i];
        for (int i = 0; i < 4; ++i) k = k << 4 | finished[i >> 1][i & 1];
        return k;
    }
};

struct Model {
    int slots, ahead, tiles, ring;

    static bool has(uint64_t mask, int t) { return mask >> t & 1; }
    // finished phases of a barrier: its arrivals by the number it counts to
    int full(const State &s, int t) const
    {
        int n = 0;
        for (int l = 0; l < 2; ++l)
            for (int u = t % kTileRing; u < s.loaded[l]; u += kTileRing) ++n;
        return n / 2;
    }
    int done(const State &s, int t) const
    {
        int n = 0;
        for (int u = t % kTileRing; u < tiles; u += kTileRing) n += has(s.done, u);
        return n;
    }
    int empty(const State &s, int t) const
    {
        int n = 0;
        for (int h = 0; h < 2; ++h)
            for (int w = 0; w < 2; ++w)
                for (int u = h; u < 2 * s.finished[h][w]; u += 2) n += mx_ring_slot(u, ring) == mx_ring_slot(t, ring);
        return n / 2;
    }
    // what a wait for tile t on a ring's barrier with that many finished phases does; `wrong`: it returns too early
    static bool passes(int phases, int t, int ring, bool *wrong)
    {
        const bool pass = (uint32_t)(phases & 1) != mx_ring_parity(t, ring);
        if (pass && phases <= t / ring) *wrong = true;
        return pass;
    }

    // 0: every order ends; 1: one gets stuck; 2: a wait returned too early
    int walk(int64_t *states) const
    {
        std::unordered_set<uint64_t> seen;
        std::vector<State> stack{State{}};
        seen.insert(stack[0].key());
        bool wrong = false;
        while (!stack.empty() && !wrong) {
            const State s = stack.back();
            stack.pop_back();
            int steps = 0;
            const auto go = [&](const State &n) {
                ++steps;
                if (seen.insert(n.key()).second) stack.push_back(n);
            };
            bool end = true;
            for (int l = 0; l < 2; ++l) {
                const int t = s.loaded[l];
                if (t >= tiles) continue;
                end = false;
                if (t < ahead || passes(done(s, t - ahead), t - ahead, kTileRing, &wrong)) {
                    State n = s;
                    ++n.loaded[l];
                    go(n);
                }
            }
            for (int i = 0; i < 4; ++i) {
                const int t = 4 * s.issued[i] + i;
                if (t >= tiles) continue;
                end = false;
                int waits = 0, at = s.waits[i];
                bool pass = true;
                if (at == waits++) pass = passes(full(s, t), t, kTileRing, &wrong);
                mx_wait_read_out(t, slots, [&](int u) {
                    if (at == waits++) pass = passes(empty(s, u), u, ring, &wrong);
                    return true;
                });
                if (!pass) continue;
                State n = s;
                if (at + 1 < waits) ++n.waits[i];
                else { ++n.issued[i]; n.waits[i] = 0; }
                go(n);
            }
            for (int t = 0; t < tiles; ++t)
                if (!has(s.done, t) && t < 4 * s.issued[t & 3] + (t & 3)) {
                    end = false;
                    State n = s;
                    n.done |= 1u << t;
                    go(n);
                }
            for (int h = 0; h < 2; ++h)
                for (int w = 0; w < 2; ++w) {
                    const int t = 2 * s.finished[h][w] + h;
                    if (t >= tiles) continue;
                    end = false;
                    if (!passes(done(s, t), t, kTileRing, &wrong)) continue;
                    State n = s;
                    ++n.finished[h][w];
                    go(n);
                }
            if (!steps && !end) { *states = (int64_t)seen.size(); return 1; }
        }
        *states = (int64_t)seen.size();
        return wrong ? 2 : 0;
    }
};

extern "C" int walk(int slots, int ahead, int tiles, int ring, int64_t *states) { return Model{slots, ahead, tiles, ring ? ring : kEmptyRing}.walk(states); }
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    where = tmp_path_factory.mktemp("mx_rings")
    (where / "model.cpp").write_text(MODEL)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(where / "model.so"), str(where / "model.cpp")], check=True)
    lib, states = ctypes.CDLL(str(where / "model.so")), ctypes.c_int64(0)
    return lambda *args: (lib.walk(*args, ctypes.byref(states)), states.value)


@pytest.mark.parametrize("ahead", [2, 3, 4])
@pytest.mark.parametrize("slots", [2, 3, 4])
def test_no_order_of_steps_gets_stuck(walk, slots, ahead):
    result, states = walk(slots, ahead, 18, 0)
    assert result == 0 and states > 1000


def test_a_ring_of_four_and_three_slots_would(walk):
    """The model sees the order in which tile t + 1 is read out before issuer t has looked at tile t - 3."""
    assert walk(3, 4, 18, 4)[0] == 1


def test_barriers_initialised_by_lanes_are_there_for_the_warp_before_it_announces_bytes():
    """Barrier b is initialised by lane b % 32: another lane may use it only behind a __syncwarp()."""
    seen = 0
    for source in sorted(CSRC.glob("*.cu*")):
        text = source.read_text()
        for at in re.finditer(r"b \+= 32\)\s*\{?[^}]*?mbar_init\(&bars\[b\]", text):
            announced = text.index("mbar_expect_tx(", at.end())
            assert "__syncwarp();" in text[at.end():announced], source.name
            seen += 1
    assert seen == 2
