"""Which layers the tensor-core kernel takes (host arithmetic, no GPU): the line is drawn by the room that the smallest tile
once needed, the plan by what the kernel needs now.  Every layer inside the line has a plan that fits, none outside is taken."""
import random

import pytest

import paper_2011_09398_b200 as lce

SHARED = 227 * 1024


def extent(size, k, stride, padding):
    """(output size, padding in front)"""
    if padding == lce.PAD_VALID:
        return ((size - k) // stride + 1 if size >= k else 0), 0
    out = -(-size // stride)
    return out, max(0, (out - 1) * stride + k - size) // 2


def covered(n, h, w, cin, kh, kw, stride, padding):
    (oh, pt), (ow, pl) = extent(h, kh, stride, padding), extent(w, kw, stride, padding)
    words, taps = -(-cin // 32), kh * kw
    if words > 32 or taps > 64:
        return False
    if stride == 1:
        wg, hg = w + max(pl, ow - 1 + kw - w - pl, 0), h + max(pt, oh - 1 + kh - h - pt, 0)
        halo = (kh - 1) * wg + kw - 1
        wide = max(wg, kw) if words & 1 else wg
        wide_halo = (kh - 1) * wide + kw - 1
    else:
        wg, hg = ow + (kw - 1) // 2, oh + (kh - 1) // 2
        halo, wide = (kh - 1) // 2 * wg + (kw - 1) // 2, wg
        wide_halo = halo
    if n * hg * wide >= 2 ** 31 - 4096 or wide_halo > 16383:
        return False
    even, phases, rows = words + (words & 1), 1 if taps == 1 else stride * stride, 16 + halo
    raw, table = (phases * rows * words + 3) // 4 * 16, taps * even // 2 * 8
    return (8192 + raw + table + 127) // 128 * 128 + 2 * phases * even * rows * 16 + 256 + (2 if taps > 1 else 1) * even * 2048 <= SHARED


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("padding", [lce.PAD_VALID, lce.PAD_SAME_ONE, lce.PAD_SAME_ZERO])
def test_covered_layers_have_a_plan_and_no_others(stride, padding):
    rng, seen = random.Random(stride + 10 * padding), [0, 0]
    while min(seen) < 150 or sum(seen) < 800:
        kh, kw = rng.choice([(1, 1), (2, 2), (3, 3), (3, 3), (5, 5), (7, 7), (8, 8), (9, 9), (1, 7), (7, 1), (4, 11)])
        n, h, w = rng.choice([1, 2, 17, 256]), rng.randint(1, 64), int(2 ** rng.uniform(0, 9))
        cin = rng.choice([rng.randint(1, 1100), 32 * rng.randint(1, 33)])
        if min(extent(h, kh, stride, padding)[0], extent(w, kw, stride, padding)[0]) <= 0:
            continue
        desc = lce.make_desc(n, h, w, cin, rng.choice([1, 64, 200]), (kh, kw), (stride, stride), padding, lce.OUT_BITPACKED, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1)
        inside = covered(n, h, w, cin, kh, kw, stride, padding)
        seen[inside] += 1
        if inside:
            plan = lce.lce_bconv2d_plan(desc)
            assert plan["kernel"] == lce.KERNEL_TENSOR and 0 < plan["shared_bytes"] <= SHARED, (n, h, w, cin, kh, kw)
        else:
            with pytest.raises(lce.LceError):
                lce.lce_bconv2d_plan(desc)
