"""LceQuantize and LceDequantize at channel counts that are not whole words, against the oracle: rows shorter and longer
than a word, runs of rows that end inside a 16-byte piece or a group of sixteen loads, rows longer than a block's run,
outputs that are only 4-byte aligned, and LceQuantize straight before a convolution that reads its output as weights."""
import numpy as np
import pytest
import torch

import oracle
import paper_2011_09398_b200 as lce
from gpu_util import DEV, guarded, guards_intact, run_bconv, to_dev, words_to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("rows,channels", [(1, 1), (5, 3), (7, 4), (3, 5), (1, 31), (9, 33), (4001, 7), (2500, 100), (700, 513), (30000, 38), (2, 8191),
                                           (3, 8193), (2, 20001), (5000, 16)])
def test_quantize_and_back(rows, channels, offset):
    rng = np.random.default_rng(rows * 7 + channels)
    x = rng.standard_normal((rows, channels)).astype(np.float32)
    x[0, 0] = -0.0
    words = (channels + 31) // 32
    src = torch.empty(rows * channels + 1, dtype=torch.float32, device=DEV)[offset:offset + rows * channels].view(rows, channels)
    src.copy_(torch.from_numpy(x))
    whole, out = guarded((rows, words), torch.int32, 0x5A5A5A5A)
    if offset:
        whole = torch.full((rows * words + 129,), 0x5A5A5A5A, dtype=torch.int32, device=DEV)
        out = whole[65:65 + rows * words].view(rows, words)
    lce.lce_bitpack(src, out)
    assert guards_intact(whole, 0x5A5A5A5A)
    want = oracle.bitpack(x)
    np.testing.assert_array_equal(words_to_host(out), want)
    whole_f = torch.full((rows * channels + 129,), 7.0, dtype=torch.float32, device=DEV)
    back = whole_f[64 + offset:64 + offset + rows * channels].view(rows, channels)
    lce.lce_unpack(out, channels, back)
    assert guards_intact(whole_f, 7.0)
    np.testing.assert_array_equal(back.cpu().numpy(), np.where(x < 0, -1.0, 1.0).astype(np.float32))


@pytest.mark.parametrize("cin,k", [(64, 3), (96, 1)])
def test_weights_quantized_right_before_the_convolution(cin, k):
    """Plain weights may be the output of the kernel just launched: many rounds, other weights each time."""
    rng = np.random.default_rng(cin)
    a = (2 * rng.integers(0, 2, size=(2, 12, 12, cin)) - 1).astype(np.int8)
    ws = [(2 * rng.integers(0, 2, size=(160, k, k, cin)) - 1).astype(np.int8) for _ in range(6)]
    desc = lce.make_desc(2, 12, 12, cin, 160, (k, k), out_type=lce.OUT_INT32)
    x, floats = lce.lce_bitpack(to_dev(a.astype(np.float32))), [to_dev(w.astype(np.float32)) for w in ws]
    words = torch.zeros(ws[0].shape[:3] + ((cin + 31) // 32,), dtype=torch.int32, device=DEV)
    outs = []
    for f in floats:
        lce.lce_bitpack(f, words)
        outs.append(lce.lce_bconv2d(desc, x, words))
    for w, out in zip(ws, outs):
        np.testing.assert_array_equal(out.cpu().numpy(), oracle.bconv2d_acc(a, w))


# widths of 1, 2, 3, 4 and 6 words (vectors of one, two and four), windows inside and across the edge, buffers that are only
# 4-byte aligned; windows that reach past both edges and over whole images
@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("n,h,w,c,pool,stride,pad", [(3, 9, 7, 32, (2, 2), (2, 2), lce.PAD_VALID), (2, 8, 11, 50, (2, 2), (2, 2), lce.PAD_SAME_ONE), (5, 7, 6, 96, (2, 2), (1, 1), lce.PAD_SAME_ONE),
                                                     (2, 13, 5, 128, (3, 2), (2, 3), lce.PAD_SAME_ONE), (1, 1, 1, 180, (2, 2), (2, 2), lce.PAD_SAME_ONE), (2, 5, 3, 96, (9, 11), (2, 2), lce.PAD_SAME_ONE), (3, 14, 14, 256, (14, 14), (14, 14), lce.PAD_VALID), (70, 56, 56, 64, (2, 2), (2, 2), lce.PAD_VALID)])
def test_maxpool_matches_the_oracle(n, h, w, c, pool, stride, pad, offset):
    rng = np.random.default_rng(n * h + c)
    x = np.where(rng.random((n, h, w, c)) < 0.8, -1.0, 1.0).astype(np.float32)
    words = oracle.bitpack(x)
    want = oracle.bmaxpool(words, c, pool, stride, pad)
    src = torch.empty(words.size + offset, dtype=torch.int32, device=DEV)[offset:].view(words.shape)
    src.copy_(torch.from_numpy(words.view(np.int32)))
    whole = torch.full((want.size + 128 + offset,), 0x5A5A5A5A, dtype=torch.int32, device=DEV)
    out = whole[64 + offset:64 + offset + want.size].view(want.shape)
    lce.lce_bmaxpool(src, c, pool, stride, pad, out)
    assert guards_intact(whole, 0x5A5A5A5A)
    np.testing.assert_array_equal(words_to_host(out), want)


def test_maxpool_of_a_row_of_almost_2_to_the_31_words():
    """A launch's last indices: threads step past the row's end, and past 2^31."""
    x = torch.randint(-2 ** 31, 2 ** 31, (1, 1, 2 ** 31 - 4096, 1), dtype=torch.int32, device=DEV)
    assert torch.equal(lce.lce_bmaxpool(x, 32, (1, 1), (1, 1), lce.PAD_VALID), x)


@pytest.mark.parametrize("n", [1, 3, 4, 7, 1023, 4 * 148 * 8 * 256 + 5])
def test_add_with_and_without_a_rest_onto_another_tensor_and_onto_an_operand(n):
    rng = np.random.default_rng(n)
    a, b = (rng.standard_normal(n).astype(np.float32) for _ in range(2))
    whole, out = guarded((n,), torch.float32, 9.0)
    lce.lce_add_f32(to_dev(a), to_dev(b), out)
    assert guards_intact(whole, 9.0)
    np.testing.assert_array_equal(out.cpu().numpy(), oracle.add_f32(a, b))
    ad = to_dev(a)
    np.testing.assert_array_equal(lce.lce_add_f32(ad, to_dev(b), ad).cpu().numpy(), oracle.add_f32(a, b))  # onto an operand


@pytest.mark.parametrize("kernel_choice", [lce.KERNEL_AUTO, lce.KERNEL_TENSOR])
def test_a_pool_between_a_convolution_and_the_reader_of_its_output(kernel_choice):
    """A convolution may take its biases from what a convolution before the pool wrote: the pool's dependents start when
    everything in front of the pool is complete."""
    rng = np.random.default_rng(12)
    x = (2 * rng.integers(0, 2, size=(16, 56, 56, 64)) - 1).astype(np.int8)
    w = (2 * rng.integers(0, 2, size=(64, 3, 3, 64)) - 1).astype(np.int8)
    mult, bias = rng.uniform(0.5, 1.5, 64).astype(np.float32), rng.standard_normal(64).astype(np.float32)
    long_desc = lce.make_desc(16, 56, 56, 64, 64, out_type=lce.OUT_FLOAT32, kernel_choice=lce.KERNEL_DIRECT)
    desc = lce.make_desc(1, 14, 14, 64, 64, out_type=lce.OUT_FLOAT32, kernel_choice=kernel_choice, weights_packed=1)
    words = to_dev(oracle.bitpack_pm1(w).view(np.int32))
    packed, xs, mult_d, bias_d = lce.lce_bconv2d_pack_weights(desc, words), to_dev(oracle.bitpack_pm1(x).view(np.int32)), to_dev(mult), to_dev(bias)
    small, pooled = xs[:1, :14, :14].contiguous(), torch.empty((1, 7, 7, 2), dtype=torch.int32, device=DEV)
    tensor_desc = lce.make_desc(16, 56, 56, 64, 64, out_type=lce.OUT_FLOAT32, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1)
    tensor_packed = lce.lce_bconv2d_pack_weights(tensor_desc, words)
    first = oracle.transform_float(oracle.bconv2d_acc(x[-1:], w), mult, bias)
    want = oracle.transform_float(oracle.bconv2d_acc(x[:1, :14, :14], w), mult, first[0, -1, -1])
    for d, weights in ((long_desc, words), (tensor_desc, tensor_packed)) * 5:
        biases = torch.full((16, 56, 56, 64), 1e9, device=DEV)
        lce.lce_bconv2d(d, xs, weights, mult_d, bias_d, None, biases)
        lce.lce_bmaxpool(small, 64, out=pooled)
        got = lce.lce_bconv2d(desc, small, packed, mult_d, biases[-1, -1, -1])
        np.testing.assert_array_equal(got.cpu().numpy(), want)
