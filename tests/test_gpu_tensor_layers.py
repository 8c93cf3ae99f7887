"""Tensor-core kernel, layers whose operands are staged in a form of their own, against the oracle: 1x1 filters at
stride 2 (one phase grid of four), odd and even image sizes, channel remainders, several tiles and images; odd numbers
of channel words, whose last ones pair up across taps."""
import numpy as np
import pytest

import oracle
import paper_2011_09398_b200 as lce
from gpu_util import run_bconv

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


@pytest.mark.parametrize("shape", SHAPES + ODD_WORDS, ids=lambda s: "x".join(map(str, s)))
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
