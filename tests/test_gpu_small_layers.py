"""The latency kernel (small layers with load-time packed weights) against the oracle, every element, at the
sizes where its tiling can go wrong: one pixel, tiles of 8 pixels that end, start or straddle images, channel
blocks of 32 with one channel more or less, words and steps with remainders, every copy width, filters that are
not square, every padding mode, and the three output forms."""
import numpy as np
import pytest

import oracle
import paper_2011_09398_b200 as lce
from gpu_util import run_bconv, to_dev, to_dev_words, words_to_host

pytestmark = pytest.mark.gpu

ONE, ZERO, VALID = lce.PAD_SAME_ONE, lce.PAD_SAME_ZERO, lce.PAD_VALID
# n, h, w, cin, cout, kh, kw, stride, padding
SHAPES = [
    (1, 1, 1, 1, 1, 1, 1, 1, ONE), (1, 1, 1, 33, 1, 3, 3, 1, ZERO), (1, 7, 1, 31, 31, 3, 1, 1, ONE), (1, 1, 9, 32, 32, 1, 3, 1, ZERO),
    (2, 3, 3, 64, 33, 3, 3, 1, ONE), (5, 3, 5, 96, 65, 3, 3, 1, ZERO), (3, 7, 7, 512, 96, 3, 3, 1, ONE), (1, 14, 14, 256, 40, 3, 3, 1, ZERO),
    (4, 9, 11, 160, 72, 2, 4, 1, ONE), (2, 13, 10, 288, 64, 3, 3, 2, ONE), (3, 8, 8, 128, 130, 5, 5, 2, ZERO), (2, 12, 9, 60, 64, 5, 5, 1, VALID),
    (1, 29, 31, 3, 32, 3, 3, 2, ONE), (7, 5, 5, 224, 100, 1, 1, 1, VALID), (2, 16, 16, 64, 64, 3, 3, 3, VALID), (6, 17, 19, 100, 64, 3, 3, 1, ZERO),
    (1, 8, 8, 1024, 32, 3, 3, 1, ONE), (2, 15, 15, 64, 128, 7, 7, 2, ONE), (10, 60, 60, 32, 64, 3, 3, 3, ZERO), (20, 60, 60, 32, 64, 3, 3, 3, ONE),
]

# tiles of 16 pixels (shallow: two slices; deeper: more), 32 (shallow, just below and above the depth at which slices are
# kept, deep) and 64, the last one of each cut short
TILES = [
    (1, 38, 37, 64, 60, 3, 3, 1, ONE), (3, 21, 25, 96, 70, 3, 3, 1, ZERO), (1, 57, 56, 64, 60, 3, 3, 1, ZERO), (16, 12, 12, 252, 90, 3, 3, 1, ONE),
    (16, 12, 12, 288, 66, 3, 3, 1, ONE), (17, 10, 10, 383, 109, 3, 3, 1, ONE), (41, 14, 13, 64, 64, 1, 1, 1, VALID), (53, 8, 8, 160, 155, 1, 1, 1, ZERO),
]


def is_small(n, h, w, cin, cout, kh, kw, s, pad, out_type):
    plan = lce.lce_bconv2d_plan(lce.make_desc(n, h, w, cin, cout, (kh, kw), (s, s), pad, out_type, weights_packed=1))
    return plan["kernel"] == lce.KERNEL_TILED and not plan["patch"] and plan["pixels_per_thread"] == 0 and plan["tile_pixels"] % 8 == 0


@pytest.mark.parametrize("shape", SHAPES + TILES, ids=lambda s: "x".join(map(str, s)))
def test_small_layers_match_the_oracle(shape):
    n, h, w, cin, cout, kh, kw, s, pad = shape
    assert is_small(*shape, lce.OUT_INT32)
    rng = np.random.default_rng(sum(shape))
    a = (2 * rng.integers(0, 2, size=(n, h, w, cin)) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(cout, kh, kw, cin)) - 1).astype(np.int8)
    aw, ww = oracle.bitpack_pm1(a), oracle.bitpack_pm1(wt)
    kwargs = dict(in_c=cin, padding=pad, stride=(s, s))
    acc = oracle.bconv2d_acc(a, wt, (s, s), pad)
    np.testing.assert_array_equal(run_bconv(aw, ww, dict(kwargs, out_type=lce.OUT_INT32), packed=True), acc)
    thr = np.rint(np.sqrt(kh * kw * cin) * rng.standard_normal(cout)).astype(np.int32)
    thr[: 2] = (np.iinfo(np.int32).max, np.iinfo(np.int32).min)[: len(thr[: 2])]
    np.testing.assert_array_equal(run_bconv(aw, ww, dict(kwargs, out_type=lce.OUT_BITPACKED), thr=thr, packed=True), oracle.transform_bits(acc, thr))
    mult = rng.uniform(0.5, 1.5, cout).astype(np.float32)
    bias = (0.1 * rng.standard_normal(cout)).astype(np.float32)
    for act in (lce.ACT_NONE, lce.ACT_RELU):
        got = run_bconv(aw, ww, dict(kwargs, out_type=lce.OUT_FLOAT32, activation=act), mult=mult, bias=bias, packed=True)
        np.testing.assert_array_equal(got, oracle.transform_float(acc, mult, bias, act))


@pytest.mark.parametrize("cout", [32, 40])
@pytest.mark.parametrize("parts", ["shortcut+float", "packed", "shortcut+float+packed"])
def test_small_fused_layers_match_the_oracle(cout, parts):
    shape = (3, 9, 7, 64, cout, 3, 3, 1, ONE)
    assert is_small(*shape, lce.OUT_FLOAT32)
    rng = np.random.default_rng(cout)
    a = (2 * rng.integers(0, 2, size=shape[:4]) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(cout, 3, 3, 64)) - 1).astype(np.int8)
    mult = rng.uniform(0.5, 1.5, cout).astype(np.float32)
    bias = (0.1 * rng.standard_normal(cout)).astype(np.float32)
    residual = rng.standard_normal((3, 9, 7, cout)).astype(np.float32) if "shortcut" in parts else None
    want = oracle.transform_float(oracle.bconv2d_acc(a, wt, (1, 1), ONE), mult, bias)
    if residual is not None:
        want = oracle.add_f32(want, residual)
    desc = lce.make_desc(*shape[:5], out_type=lce.OUT_FLOAT32, weights_packed=1)
    wd = lce.lce_bconv2d_pack_weights(desc, to_dev_words(oracle.bitpack_pm1(wt)))
    out = to_dev(np.full_like(want, 7.0)) if "float" in parts else None
    packed = to_dev_words(np.full((3, 9, 7, (cout + 31) // 32), 0xFFFFFFFF, dtype=np.uint32)) if "packed" in parts else None
    lce.lce_bconv2d_fused(desc, to_dev_words(oracle.bitpack_pm1(a)), wd, to_dev(mult), to_dev(bias),
                          to_dev(residual) if residual is not None else None, out, packed)
    if out is not None:
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    if packed is not None:
        np.testing.assert_array_equal(words_to_host(packed), oracle.bitpack(want))


# n, h, w, cin, cout, k, stride: a kernel covers them under some padding modes only (the latency kernel 7x7 not under
# zero-padding, the tensor-core kernel the other two under VALID alone: longer rows leave it no room)
@pytest.mark.parametrize("shape", [(1, 14, 14, 64, 64, 7, 1), (1, 4, 30, 1000, 40, 3, 1), (2, 6, 13, 1000, 40, 5, 1)], ids=lambda s: "x".join(map(str, s)))
def test_weights_packed_under_one_padding_mode_run_under_every_other(shape):
    n, h, w, cin, cout, k, s = shape
    rng = np.random.default_rng(sum(shape))
    a = (2 * rng.integers(0, 2, size=(n, h, w, cin)) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(cout, k, k, cin)) - 1).astype(np.int8)
    x, plain = to_dev_words(oracle.bitpack_pm1(a)), to_dev_words(oracle.bitpack_pm1(wt))
    desc = lambda pad, choice: lce.make_desc(n, h, w, cin, cout, (k, k), (s, s), pad, lce.OUT_INT32, lce.ACT_NONE, choice, 1)
    choices, covered = (lce.KERNEL_AUTO, lce.KERNEL_TENSOR, lce.KERNEL_TILED), set()
    packed = {pad: lce.lce_bconv2d_pack_weights(desc(pad, lce.KERNEL_AUTO), plain) for pad in (VALID, ONE, ZERO)}
    for pad in (VALID, ONE, ZERO):
        want = oracle.bconv2d_acc(a, wt, (s, s), pad)
        for choice in choices:
            try:
                lce.lce_bconv2d_plan(desc(pad, choice))
            except lce.LceError as e:
                assert e.status == 2
                continue
            covered.add((pad, choice))
            for under in (VALID, ONE, ZERO):
                got = lce.lce_bconv2d(desc(pad, choice), x, packed[under])
                np.testing.assert_array_equal(got.cpu().numpy(), want, err_msg=f"packed under {under}, run under {pad}, kernel {choice}")
    assert (VALID, lce.KERNEL_AUTO) in covered
    if k != 7:
        assert (VALID, lce.KERNEL_TENSOR) in covered and (ONE, lce.KERNEL_TENSOR) not in covered
    assert lce.lce_device_status() == 0


@pytest.mark.parametrize("cin,cout,k", [(1, 1, 1), (33, 31, 1), (64, 64, 3), (3, 32, 3), (512, 40, 3), (96, 130, 5), (7300, 5, 3), (4000, 33, 1)])
def test_packed_weights_begin_with_the_plain_words(cin, cout, k):
    """With the latency kernel's image its packing kernel copies them, without (the last but one) the copy engine does."""
    rng = np.random.default_rng(cin + cout)
    plain = to_dev_words(oracle.bitpack_pm1((2 * rng.integers(0, 2, size=(cout, k, k, cin)) - 1).astype(np.int8)))
    desc = lce.make_desc(1, 9, 9, cin, cout, (k, k), weights_packed=1)
    words = lce.lce_bconv2d_packed_weights_bytes(desc) // 4
    whole = to_dev(np.full(words + 128, 0x5A5A5A5A, dtype=np.int32))
    packed = lce.lce_bconv2d_pack_weights(desc, plain, whole[64:64 + words])
    assert bool((packed[:plain.numel()] == plain.reshape(-1)).all().item())
    assert bool((whole[:64] == 0x5A5A5A5A).all().item()) and bool((whole[64 + words:] == 0x5A5A5A5A).all().item())
