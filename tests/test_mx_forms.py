"""Which form of the tensor-core kernel a layer of few output channels gets: positions on the TMEM lanes in tiles of 256, or
channels on the lanes in narrower tiles, which keep more SMs busy where there are few."""
import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

import oracle
import paper_2011_09398_b200 as lce
from gpu_util import guarded, guards_intact, to_dev, to_dev_words, words_to_host


def _plan(shape, out_type):
    n, h, cin, cout, k, s = shape
    return lce.lce_bconv2d_plan(lce.make_desc(n, h, h, cin, cout, (k, k), (s, s), lce.PAD_SAME_ONE, out_type, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1))


# n, h, cin, cout, k, stride
SMALL_GRIDS = [(8, 28, 128, 64, 3, 1), (4, 28, 128, 64, 3, 1), (16, 28, 128, 64, 3, 1), (32, 14, 256, 64, 3, 1), (16, 14, 256, 64, 3, 1), (64, 14, 256, 64, 3, 1),
               (64, 14, 512, 96, 1, 1), (32, 14, 512, 96, 1, 1), (8, 28, 64, 64, 3, 1), (16, 28, 96, 96, 3, 1), (64, 28, 64, 64, 3, 2)]
FULL_GRIDS = [(8, 56, 64, 64, 3, 1), (64, 56, 64, 64, 3, 1), (256, 56, 64, 64, 3, 1), (128, 14, 256, 64, 3, 1), (128, 14, 512, 96, 1, 1), (1, 14, 32, 32, 3, 1),
              (16, 14, 256, 64, 1, 1), (64, 112, 32, 64, 3, 2)]


@pytest.mark.parametrize("shape", SMALL_GRIDS, ids=lambda s: "x".join(map(str, s)))
def test_bits_on_a_small_grid_keep_the_narrow_tiles(shape):
    """The plan of the same layer with int32 output, which has channels on the lanes throughout."""
    assert _plan(shape, lce.OUT_BITPACKED) == _plan(shape, lce.OUT_INT32)


@pytest.mark.parametrize("shape", FULL_GRIDS, ids=lambda s: "x".join(map(str, s)))
def test_bits_on_a_full_grid_have_positions_on_the_lanes(shape):
    bits, other = _plan(shape, lce.OUT_BITPACKED), _plan(shape, lce.OUT_INT32)
    assert bits["tile_pixels"] == 128 and bits["weights_resident"] and bits["shared_bytes"] != other["shared_bytes"]


def _kernels(call):
    call()  # set up
    torch.cuda.synchronize()
    for _ in range(3):  # a profile may come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            call()
            torch.cuda.synchronize()
        names = [e.key for e in p.key_averages() if "bconv" in e.key]
        if names:
            break
    assert len(names) == 1, names
    return names[0]


# n, h, cin, cout, k, stride; positions on the lanes with bits, copy, copy and floats, shortcut and copy, shortcut and floats, all three
FORMS = [((1, 28, 96, 96, 3, 1), "......"), ((32, 14, 96, 96, 3, 1), "......"), ((16, 28, 64, 64, 3, 1), "......"), ((64, 28, 64, 64, 3, 2), "......"),
         ((8, 56, 64, 64, 3, 1), "P....."), ((128, 56, 64, 64, 3, 1), "PPPPPP"), ((128, 28, 32, 32, 3, 1), "PPPPPP"), ((16, 28, 64, 64, 1, 1), "PP...."),
         ((32, 56, 96, 96, 3, 1), "PPP..."), ((24, 56, 64, 64, 3, 1), "P..P..")]


@pytest.mark.gpu
@pytest.mark.parametrize("shape,want", FORMS, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
def test_the_form_that_runs(shape, want):
    """Few tiles, or few in the last wave: channels on the lanes.  A shortcut from 96 to 96 channels has no room beside the weights."""
    n, h, cin, cout, k, s = shape
    oh, dev = -(-h // s), "cuda:0"
    descs = [lce.make_desc(n, h, h, cin, cout, (k, k), (s, s), lce.PAD_SAME_ONE, o, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1) for o in (lce.OUT_BITPACKED, lce.OUT_FLOAT32)]
    x = torch.zeros((n, h, h, cin // 32), dtype=torch.int32, device=dev)
    w = lce.lce_bconv2d_pack_weights(descs[0], torch.zeros((cout, k, k, cin // 32), dtype=torch.int32, device=dev))
    ones, thr = torch.ones(cout, device=dev), torch.zeros(cout, dtype=torch.int32, device=dev)
    res, out = torch.zeros((n, oh, oh, cout), device=dev), torch.empty((n, oh, oh, cout), device=dev)
    words = torch.empty((n, oh, oh, cout // 32), dtype=torch.int32, device=dev)
    names = [_kernels(lambda: lce.lce_bconv2d(descs[0], x, w, None, None, thr, words))]
    for shortcut, floats, packed in ((None, None, words), (None, out, words), (res, None, words), (res, out, None), (res, out, words)):
        names.append(_kernels(lambda: lce.lce_bconv2d_fused(descs[1], x, w, ones, ones, shortcut, floats, packed)))
    assert "".join("P" if "positions" in name else "." for name in names) == want
    assert "positions" not in _kernels(lambda: lce.lce_bconv2d_fused(descs[1], x, w, ones, ones, None, out, None))
    assert lce.lce_device_status() == 0


# n, h, cin, cout, k, stride, padding: bits and fused outputs with every ring coming round; strides and filters beside 1x1, odd words over
# several taps, both paddings.  A shortcut beside the weights of 96 -> 32 channels, 3x3, has no room for two position buffers
LAYERS = [((240, 56, 32, 64, 3, 2, lce.PAD_SAME_ZERO), "PPPPPP"), ((70, 55, 32, 96, 3, 1, lce.PAD_SAME_ZERO), "PPPPPP"), ((70, 56, 96, 32, 3, 1, lce.PAD_SAME_ONE), "PPP..."),
          ((70, 56, 32, 32, 5, 1, lce.PAD_SAME_ONE), "PPPPPP"), ((70, 55, 96, 40, 3, 1, lce.PAD_SAME_ONE), "P")]


@pytest.mark.gpu
@pytest.mark.parametrize("shape,want", LAYERS, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
def test_positions_on_the_lanes_match_the_oracle(shape, want):
    """Bits at words that start on 4 and on 8 bytes, thresholds on, beside and far beyond the accumulators' range; the fused outputs, exact."""
    n, h, cin, cout, k, s, pad = shape
    rng = np.random.default_rng(sum(shape))
    a, wt = ((2 * rng.integers(0, 2, size=d) - 1).astype(np.int8) for d in ((n, h, h, cin), (cout, k, k, cin)))
    acc, K = oracle.bconv2d_acc(a, wt, (s, s), pad), k * k * cin
    x, plain_w = to_dev_words(oracle.bitpack_pm1(a)), to_dev_words(oracle.bitpack_pm1(wt))
    desc = [lce.make_desc(n, h, h, cin, cout, (k, k), (s, s), pad, o, kernel_choice=lce.KERNEL_TENSOR, weights_packed=1) for o in (lce.OUT_BITPACKED, lce.OUT_FLOAT32)]
    w, names = lce.lce_bconv2d_pack_weights(desc[0], plain_w), []
    thr = rng.choice(np.array([-2**31, -K - 1, -K, -2, 0, 1, 2, K, K + 1, 2**31 - 1]), cout).astype(np.int32)
    count, thr_d = acc.size // cout * -(-cout // 32), to_dev(thr)
    for offset in (0, 1, 2):
        whole = torch.full((count + 8,), 0x5A5A5A5A, dtype=torch.int32, device="cuda:0")
        out = whole[offset:offset + count].view(*acc.shape[:3], -1)
        names[:] = [_kernels(lambda: lce.lce_bconv2d(desc[0], x, w, None, None, thr_d, out))]
        np.testing.assert_array_equal(words_to_host(out.contiguous()), oracle.transform_bits(acc, thr))
        assert (whole[:offset] == 0x5A5A5A5A).all() and (whole[offset + count:] == 0x5A5A5A5A).all()
    if cout % 32 == 0:
        mult, bias = rng.uniform(-1.5, 1.5, cout).astype(np.float32), rng.standard_normal(cout).astype(np.float32)
        res = (rng.standard_normal(acc.shape, dtype=np.float32) * np.float32(np.sqrt(K)))
        plain, mult_d, bias_d, res_d = oracle.transform_float(acc, mult, bias), to_dev(mult), to_dev(bias), to_dev(res)
        summed = oracle.add_f32(plain, res)
        for shortcut, floats, packed in ((0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0), (1, 1, 1)):
            whole_f, out = guarded(acc.shape, torch.float32, 12345.0)
            whole_w, words = guarded(acc.shape[:3] + (cout // 32,), torch.int32, 0x5A5A5A5A)
            names.append(_kernels(lambda: lce.lce_bconv2d_fused(desc[1], x, w, mult_d, bias_d, res_d if shortcut else None, out if floats else None, words if packed else None)))
            y = summed if shortcut else plain
            if floats:
                np.testing.assert_array_equal(out.cpu().numpy(), y)
            if packed:
                np.testing.assert_array_equal(words_to_host(words), oracle.bitpack(y))
            assert guards_intact(whole_f, 12345.0) and guards_intact(whole_w, 0x5A5A5A5A)
    assert "".join("P" if "positions" in name else "." for name in names) == want
    assert lce.lce_device_status() == 0
