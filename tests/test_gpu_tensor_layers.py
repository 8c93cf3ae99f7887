"""Tensor-core kernel, layers whose operands are staged in a form of their own, against the oracle: 1x1 filters at
stride 2 (one phase grid of four), odd and even image sizes, channel remainders, several tiles and images; odd numbers
of channel words, whose last ones pair up across taps."""
import numpy as np
import pytest
import torch

import oracle
import paper_2011_09398_b200 as lce
from gpu_util import guarded, guards_intact, run_bconv, to_dev, to_dev_words, words_to_host

pytestmark = pytest.mark.gpu

# n, h, w, cin, cout, k, stride, padding
SHAPES = [
    (1, 1, 1, 1, 1, 1, 2, lce.PAD_SAME_ONE), (3, 7, 9, 40, 33, 1, 2, lce.PAD_SAME_ZERO), (2, 8, 8, 64, 64, 1, 2, lce.PAD_SAME_ONE),
    (5, 13, 10, 128, 130, 1, 2, lce.PAD_VALID), (40, 28, 27, 96, 32, 1, 2, lce.PAD_SAME_ZERO), (9, 56, 56, 256, 256, 1, 2, lce.PAD_SAME_ONE),
]

# odd numbers of words: 1, 3, 5, 31 a tap; odd and even in all; one and two phases of taps; images narrower than the
# filter; filters that stream
ODD_WORDS = [
    (1, 1, 1, 32, 40, 1, 1, lce.PAD_SAME_ONE), (3, 11, 9, 32, 64, 3, 1, lce.PAD_SAME_ZERO), (2, 3, 1, 20, 33, 5, 1, lce.PAD_SAME_ONE),
    (2, 1, 2, 96, 32, 4, 1, lce.PAD_SAME_ZERO), (70, 30, 31, 32, 64, 3, 2, lce.PAD_SAME_ONE), (4, 13, 12, 96, 130, 3, 2, lce.PAD_SAME_ZERO),
    (3, 9, 10, 96, 32, 2, 2, lce.PAD_VALID), (2, 8, 9, 160, 160, 5, 1, lce.PAD_SAME_ONE), (30, 16, 16, 160, 200, 5, 1, lce.PAD_SAME_ZERO),
    (2, 7, 7, 480, 64, 5, 2, lce.PAD_VALID), (1, 5, 4, 990, 40, 3, 1, lce.PAD_VALID), (2, 9, 9, 992, 32, 1, 1, lce.PAD_SAME_ONE),
]

# CTAs with a single super-tile, and so one position buffer: of one tile whose weights stream, of seven tiles (more than the
# barriers of a ring), of tiles that the last CTA has fewer of
ONE_BUFFER = [(64, 28, 28, 256, 40, 3, 2, lce.PAD_SAME_ZERO), (64, 56, 56, 32, 20, 3, 1, lce.PAD_SAME_ONE), (37, 56, 55, 40, 33, 3, 1, lce.PAD_SAME_ZERO)]


# few channels, bits: one, two and three words; one tile of 256 positions, one position more than that, and enough tiles that every
# ring comes round
POSITIONS = [(1, 16, 16, 64, 32, 1, 1, lce.PAD_VALID), (1, 1, 257, 40, 64, 1, 1, lce.PAD_VALID), (80, 56, 56, 32, 32, 1, 1, lce.PAD_SAME_ONE), (80, 56, 56, 64, 64, 1, 1, lce.PAD_SAME_ONE),
             (80, 56, 56, 33, 96, 1, 1, lce.PAD_SAME_ZERO), (70, 55, 56, 32, 41, 3, 1, lce.PAD_SAME_ZERO), (90, 112, 112, 3, 65, 3, 2, lce.PAD_SAME_ONE)]


@pytest.mark.parametrize("shape", SHAPES + ODD_WORDS + ONE_BUFFER + POSITIONS, ids=lambda s: "x".join(map(str, s)))
def test_tensor_layers_match_the_oracle(shape):
    n, h, w, cin, cout, k, s, pad = shape
    rng = np.random.default_rng(sum(shape))
    a = (2 * rng.integers(0, 2, size=(n, h, w, cin)) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(cout, k, k, cin)) - 1).astype(np.int8)
    aw, ww = oracle.bitpack_pm1(a), oracle.bitpack_pm1(wt)
    kwargs = dict(in_c=cin, padding=pad, stride=(s, s))
    acc = oracle.bconv2d_acc(a, wt, (s, s), pad)
    np.testing.assert_array_equal(run_bconv(aw, ww, dict(kwargs, out_type=lce.OUT_INT32), kernel_choice=lce.KERNEL_TENSOR, packed=True), acc)
    thr = np.rint(np.sqrt(k * k * cin) * rng.standard_normal(cout)).astype(np.int32)
    got = run_bconv(aw, ww, dict(kwargs, out_type=lce.OUT_BITPACKED), thr=thr, kernel_choice=lce.KERNEL_TENSOR, packed=True)
    np.testing.assert_array_equal(got, oracle.transform_bits(acc, thr))
    assert lce.lce_device_status() == 0


@pytest.mark.parametrize("cout,offset", [(64, 0), (64, 1), (64, 2), (40, 1), (96, 1), (32, 3)])
def test_bits_of_few_channels_at_any_word(cout, offset):
    """Output words that start on 4 and on 8 bytes, thresholds on, beside and far beyond the accumulators' range."""
    rng = np.random.default_rng(cout + offset)
    a, wt = ((2 * rng.integers(0, 2, size=s) - 1).astype(np.int8) for s in ((3, 19, 20, 64), (cout, 3, 3, 64)))
    acc = oracle.bconv2d_acc(a, wt, (1, 1), lce.PAD_SAME_ONE)
    thr = rng.choice(np.array([-2**31, -577, -576, -2, 0, 1, 2, 576, 577, 2**31 - 1]), cout).astype(np.int32)
    desc = lce.make_desc(3, 19, 20, 64, cout, out_type=lce.OUT_BITPACKED, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1)
    weights = lce.lce_bconv2d_pack_weights(desc, to_dev_words(oracle.bitpack_pm1(wt)))
    count = acc.shape[0] * acc.shape[1] * acc.shape[2] * ((cout + 31) // 32)
    whole = torch.full((count + 8,), 0x5A5A5A5A, dtype=torch.int32, device="cuda:0")
    out = whole[offset:offset + count].view(*acc.shape[:3], -1)
    lce.lce_bconv2d(desc, to_dev_words(oracle.bitpack_pm1(a)), weights, None, None, to_dev(thr), out)
    np.testing.assert_array_equal(words_to_host(out.contiguous()), oracle.transform_bits(acc, thr))
    assert (whole[:offset] == 0x5A5A5A5A).all() and (whole[offset + count:] == 0x5A5A5A5A).all()
    assert lce.lce_device_status() == 0


@pytest.mark.parametrize("n,h,w,c", [(1, 9, 9, 64), (40, 15, 13, 128), (9, 20, 17, 256)])
def test_fused_words_of_special_values(n, h, w, c):
    """The re-quantised copy is y < 0: 0 for -0.0 and for a NaN of either sign; tiles with one and with two chunks a warp."""
    rng = np.random.default_rng(n + c)
    a = (2 * rng.integers(0, 2, size=(n, h, w, c)) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(c, 3, 3, c)) - 1).astype(np.int8)
    acc = oracle.bconv2d_acc(a, wt, (1, 1), lce.PAD_SAME_ONE)
    mult, bias = np.where(rng.integers(0, 2, c), -1.0, 0.0).astype(np.float32), np.full(c, -0.0, np.float32)
    nan = np.array([0x7FC00000, 0xFFC00000], np.uint32).view(np.float32)
    special = np.concatenate([nan, np.array([np.inf, -np.inf, -0.0, 0.0, 1e-45, -1e-45, -1.0], np.float32)])
    residual = rng.choice(special, size=acc.shape).astype(np.float32)
    desc = lce.make_desc(n, h, w, c, c, out_type=lce.OUT_FLOAT32, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1)
    weights = lce.lce_bconv2d_pack_weights(desc, to_dev_words(oracle.bitpack_pm1(wt)))
    with np.errstate(invalid="ignore"):
        want = oracle.transform_float(acc, mult, bias)
        for shortcut in (None, residual):
            y = want if shortcut is None else oracle.add_f32(want, shortcut)
            for floats in (False, True):
                out = torch.empty(acc.shape, device="cuda:0") if floats else None
                words = torch.empty((n, h, w, c // 32), dtype=torch.int32, device="cuda:0")
                lce.lce_bconv2d_fused(desc, to_dev_words(oracle.bitpack_pm1(a)), weights, to_dev(mult), to_dev(bias),
                                      None if shortcut is None else to_dev(shortcut), out, words)
                np.testing.assert_array_equal(words_to_host(words), oracle.bitpack(y))
                if floats:
                    np.testing.assert_array_equal(out.cpu().numpy(), y)  # NaN equal to NaN
    assert lce.lce_device_status() == 0


@pytest.mark.parametrize("n,h,cout,offset", [(1, 16, 32, 0), (1, 17, 64, 4), (2, 15, 96, 0), (70, 56, 64, 4), (80, 56, 32, 0), (60, 57, 96, 4)])
def test_fused_of_few_channels(n, h, cout, offset):
    """Float tensors that start on 16 and on 32 bytes; one tile and so many that every ring comes round; with ReLU."""
    rng = np.random.default_rng(n + cout + offset)
    a, wt = ((2 * rng.integers(0, 2, size=s) - 1).astype(np.int8) for s in ((n, h, h, 32), (cout, 1, 1, 32)))
    acc = oracle.bconv2d_acc(a, wt, (1, 1), lce.PAD_SAME_ONE)
    mult, bias = rng.uniform(-1.5, 1.5, cout).astype(np.float32), rng.standard_normal(cout).astype(np.float32)
    desc = lce.make_desc(n, h, h, 32, cout, (1, 1), out_type=lce.OUT_FLOAT32, activation=lce.ACT_RELU, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1)
    x, weights = to_dev_words(oracle.bitpack_pm1(a)), lce.lce_bconv2d_pack_weights(desc, to_dev_words(oracle.bitpack_pm1(wt)))
    shortcut = torch.randn(acc.size + 8, device="cuda:0")
    residual = shortcut[offset:offset + acc.size].view(acc.shape)
    plain = oracle.transform_float(acc, mult, bias, oracle.ACT_RELU)
    for res in (None, residual):
        y = plain if res is None else oracle.add_f32(plain, res.cpu().numpy())
        for floats, packed in ((True, False), (False, True), (True, True)):
            whole = torch.full((acc.size + 8,), 12345.0, device="cuda:0")
            out = whole[offset:offset + acc.size].view(acc.shape)
            whole_w, words = guarded(acc.shape[:3] + (cout // 32,), torch.int32, 0x5A5A5A5A)
            lce.lce_bconv2d_fused(desc, x, weights, to_dev(mult), to_dev(bias), res, out if floats else None, words if packed else None)
            if floats:
                np.testing.assert_array_equal(out.cpu().numpy(), y)
                assert (whole[:offset] == 12345.0).all() and (whole[offset + acc.size:] == 12345.0).all()
            if packed:
                np.testing.assert_array_equal(words_to_host(words), oracle.bitpack(y))
                assert guards_intact(whole_w, 0x5A5A5A5A)
    assert lce.lce_device_status() == 0


# n, h, w, cin, cout, k, stride: channel blocks with one, two or three words missing, one tile and several tiles a CTA
RAGGED_BLOCKS = [(40, 28, 27, 64, 96, 3, 1), (30, 16, 15, 96, 160, 3, 1), (2, 9, 10, 64, 192, 3, 2), (70, 14, 13, 40, 224, 1, 1), (1, 5, 5, 32, 96, 5, 1)]


@pytest.mark.parametrize("shape", RAGGED_BLOCKS, ids=lambda s: "x".join(map(str, s)))
def test_fused_on_channel_blocks_that_are_partly_empty(shape):
    """Shortcut add, re-quantised copy and float output, each there and not there: exact, and nothing written beside them."""
    n, h, w, cin, cout, k, s = shape
    rng = np.random.default_rng(sum(shape))
    a = (2 * rng.integers(0, 2, size=(n, h, w, cin)) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(cout, k, k, cin)) - 1).astype(np.int8)
    acc = oracle.bconv2d_acc(a, wt, (s, s), lce.PAD_SAME_ONE)
    mult, bias = rng.uniform(0.5, 1.5, cout).astype(np.float32), rng.standard_normal(cout).astype(np.float32)
    residual = (rng.standard_normal(acc.shape) * np.sqrt(k * k * cin)).astype(np.float32)
    desc = lce.make_desc(n, h, w, cin, cout, (k, k), (s, s), out_type=lce.OUT_FLOAT32, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1)
    x, weights = to_dev_words(oracle.bitpack_pm1(a)), lce.lce_bconv2d_pack_weights(desc, to_dev_words(oracle.bitpack_pm1(wt)))
    plain = oracle.transform_float(acc, mult, bias)
    for shortcut in (None, residual):
        y = plain if shortcut is None else oracle.add_f32(plain, shortcut)
        for floats, packed in ((True, False), (False, True), (True, True)):
            whole_f, out = guarded(acc.shape, torch.float32, 12345.0)
            whole_w, words = guarded(acc.shape[:3] + (cout // 32,), torch.int32, 0x5A5A5A5A)
            lce.lce_bconv2d_fused(desc, x, weights, to_dev(mult), to_dev(bias), None if shortcut is None else to_dev(shortcut),
                                  out if floats else None, words if packed else None)
            if floats:
                np.testing.assert_array_equal(out.cpu().numpy(), y)
            if packed:
                np.testing.assert_array_equal(words_to_host(words), oracle.bitpack(y))
            assert guards_intact(whole_f, 12345.0) and guards_intact(whole_w, 0x5A5A5A5A)
    assert lce.lce_device_status() == 0
