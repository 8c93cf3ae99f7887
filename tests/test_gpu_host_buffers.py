"""lce_bconv2d_host against the oracle, every element, over the ways an array can reach the device and an output can come
back: by the copy engine or by a kernel, or written by the convolution itself."""
import concurrent.futures
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2011_09398_b200 as lce
from gpu_util import DEV

pytestmark = pytest.mark.gpu

ONE, ZERO = lce.PAD_SAME_ONE, lce.PAD_SAME_ZERO
FILL = 0xA5
READ_ONLY = 8   # cudaHostRegisterReadOnly


class Buffer:
    """Host memory that starts `offset` bytes past a page boundary, guard bytes on both sides.  How: "pinned", "pageable",
    or "registered" / "read-only": pageable memory of which the array's bytes and no others are registered."""

    def __init__(self, nbytes, how, offset=0):
        self.whole = torch.full((nbytes + 3 * 4096,), FILL, dtype=torch.uint8)
        if how == "pinned":
            self.whole = self.whole.pin_memory()
        self.first = -self.whole.data_ptr() % 4096 + 4096 + offset
        self.nbytes, self.ptr = nbytes, self.whole.data_ptr() + self.first
        self.registered = how in ("registered", "read-only")
        if self.registered:
            assert int(torch.cuda.cudart().cudaHostRegister(self.ptr, nbytes, READ_ONLY if how == "read-only" else 0)) == 0

    def release(self):
        if self.registered:
            assert int(torch.cuda.cudart().cudaHostUnregister(self.ptr)) == 0

    @classmethod
    def of(cls, array, how, offset=0):
        b = cls(array.nbytes, how, offset)
        b.whole[b.first:b.first + b.nbytes] = torch.from_numpy(np.ascontiguousarray(array).view(np.uint8).reshape(-1).copy())
        return b

    def read(self, dtype, shape):
        return self.whole[self.first:self.first + self.nbytes].numpy().copy().view(dtype).reshape(shape)

    def guards_intact(self):
        return bool((self.whole[:self.first] == FILL).all()) and bool((self.whole[self.first + self.nbytes:] == FILL).all())


def least_workspace(n, h, w, cin, cout, k, out_words):
    up = lambda b: (b + 255) // 256 * 256
    words = (cin + 31) // 32
    return up(n * h * w * words * 4) + up(cout * k * k * words * 4) + 3 * up(cout * 4) + up(out_words * 4)


def check(shape, out_type, place=lambda name: ("pinned", 0), workspace="full", entry="lce_bconv2d_host"):
    """One call; `place` gives (how, offset) of an array by its name; `workspace`: what the call asks for, or the least
    it accepts (no room to pack weights)."""
    n, h, w, cin, cout, k, s, pad = shape
    rng = np.random.default_rng(sum(shape) + out_type)
    a = (2 * rng.integers(0, 2, size=(n, h, w, cin)) - 1).astype(np.int8)
    wt = (2 * rng.integers(0, 2, size=(cout, k, k, cin)) - 1).astype(np.int8)
    acc = oracle.bconv2d_acc(a, wt, (s, s), pad)
    arrays = dict(input=oracle.bitpack_pm1(a), weights=oracle.bitpack_pm1(wt), multiplier=None, bias=None, thresholds=None)
    if out_type == lce.OUT_FLOAT32:
        arrays.update(multiplier=rng.uniform(0.5, 1.5, cout).astype(np.float32), bias=(0.1 * rng.standard_normal(cout)).astype(np.float32))
        want = oracle.transform_float(acc, arrays["multiplier"], arrays["bias"])
    elif out_type == lce.OUT_BITPACKED:
        arrays.update(thresholds=np.rint(np.sqrt(k * k * cin) * rng.standard_normal(cout)).astype(np.int32))
        want = oracle.transform_bits(acc, arrays["thresholds"])
    else:
        want = acc
    held = {name: None if v is None else Buffer.of(v, *place(name)) for name, v in arrays.items()}
    out = Buffer(want.nbytes, *place("output"))
    desc = lce.make_desc(n, h, w, cin, cout, (k, k), (s, s), pad, out_type)
    asked = lce.lce_bconv2d_host_workspace_bytes(desc)
    least = least_workspace(n, h, w, cin, cout, k, want.size)
    room = asked if workspace == "full" else least
    assert least <= asked
    ws = torch.full((room + 256,), FILL, dtype=torch.uint8, device=DEV)
    fn = getattr(lce.library(), entry)
    args = [ctypes.byref(desc), *(None if b is None else b.ptr for b in held.values()), out.ptr]
    if entry != "lce_bconv2d_host_noalloc":
        assert fn(*args, ws.data_ptr(), least - 1, None) == 6      # LCE_ERR_WORKSPACE, nothing done
        args += [ws.data_ptr(), room]
    torch.cuda.synchronize()
    assert fn(*args, None) == 0
    np.testing.assert_array_equal(out.read(want.dtype, want.shape), want)
    assert out.guards_intact() and all(b is None or b.guards_intact() for b in held.values())
    assert bool((ws[room:] == FILL).all().item()), "wrote past the workspace"
    assert lce.lce_device_status() == 0
    for b in (out, *held.values()):
        if b is not None:
            b.release()
    return asked > least


@pytest.mark.parametrize("offset", [1, 2, 3, 4, 6, 8, 12])
@pytest.mark.parametrize("which", ["input", "weights", "multiplier", "bias", "thresholds", "output", "all"])
def test_pinned_arrays_that_start_on_any_byte(which, offset):
    out_type = lce.OUT_BITPACKED if which == "thresholds" else lce.OUT_FLOAT32
    check((2, 9, 11, 40, 36, 3, 1, ONE), out_type, lambda name: ("pinned", offset if which in (name, "all") else 0))
    if which in ("output", "all"):
        check((2, 9, 11, 40, 36, 3, 1, ONE), lce.OUT_BITPACKED, lambda name: ("pinned", offset if which in (name, "all") else 0))


@pytest.mark.parametrize("offset", [0, 4, 100])
def test_arrays_the_caller_has_registered(offset):
    for out_type in (lce.OUT_FLOAT32, lce.OUT_BITPACKED):
        check((2, 9, 11, 40, 36, 3, 1, ONE), out_type, lambda name: ("registered", offset))
        check((2, 9, 11, 40, 36, 3, 1, ONE), out_type, lambda name: ("registered" if name == "output" else "read-only", offset))


# n, h, w, cin, cout, k, stride, padding: arrays of 1, 2 and 3 words past a 16-byte piece, one word in all, and more
RAGGED = [(1, 1, 1, 1, 1, 1, 1, ONE), (1, 1, 5, 32, 3, 1, 1, ONE), (1, 3, 5, 40, 5, 3, 1, ZERO), (1, 7, 1, 96, 2, 1, 1, ONE), (3, 5, 7, 70, 33, 3, 2, ONE)]


@pytest.mark.parametrize("out_type", [lce.OUT_FLOAT32, lce.OUT_BITPACKED, lce.OUT_INT32])
@pytest.mark.parametrize("shape", RAGGED, ids=lambda s: "x".join(map(str, s)))
def test_arrays_that_are_not_whole_pieces(shape, out_type):
    check(shape, out_type)


NAMES = ("input", "weights", "multiplier", "bias", "thresholds", "output")


@pytest.mark.parametrize("entry", ["lce_bconv2d_host", "lce_bconv2d_host_noalloc"])
@pytest.mark.parametrize("pageable", [{n} for n in NAMES] + [set(NAMES), {"input", "bias", "output"}, {"weights", "multiplier", "thresholds"}],
                         ids=lambda s: "+".join(n for n in NAMES if n in s) if len(s) < 6 else "all")
def test_pageable_arrays_beside_pinned_ones(pageable, entry):
    for out_type in (lce.OUT_FLOAT32, lce.OUT_BITPACKED):
        check((2, 9, 11, 40, 36, 3, 1, ONE), out_type, lambda name: ("pageable" if name in pageable else "pinned", 0), entry=entry)


# around the limits of the two ways for small arrays: copied by a kernel up to 2 MB, outputs written in place up to 256 KB
# of floats and 32 KB of bit-packed words; exactly at a limit and one word past it
LIMITS = [(1, 512, 1024, 32, 1, lce.OUT_BITPACKED), (1, 1, 524289, 32, 1, lce.OUT_BITPACKED), (1, 512, 1024, 32, 1, lce.OUT_FLOAT32),
          (1, 1, 524289, 32, 1, lce.OUT_INT32), (1, 2, 2, 8192, 2048, lce.OUT_FLOAT32), (1, 2, 2, 8192, 2049, lce.OUT_BITPACKED),
          (1, 64, 128, 32, 32, lce.OUT_BITPACKED), (1, 3, 2731, 32, 32, lce.OUT_BITPACKED), (1, 256, 256, 32, 1, lce.OUT_FLOAT32),
          (1, 1, 65537, 32, 1, lce.OUT_FLOAT32), (1, 1, 65537, 32, 1, lce.OUT_INT32)]


@pytest.mark.parametrize("how", ["pinned", "pageable"])
@pytest.mark.parametrize("case", LIMITS, ids=lambda c: "x".join(map(str, c)))
def test_arrays_around_the_limits_of_the_copy_kernel_and_of_outputs_written_in_place(case, how):
    n, h, w, cin, cout, out_type = case
    check((n, h, w, cin, cout, 1, 1, ONE), out_type, lambda name: (how, 0))


@pytest.mark.parametrize("out_type", [lce.OUT_FLOAT32, lce.OUT_BITPACKED, lce.OUT_INT32])
@pytest.mark.parametrize("shape", [(16, 28, 28, 128, 128, 3, 1, ONE), (64, 27, 25, 100, 72, 3, 2, ZERO)], ids=lambda s: "x".join(map(str, s)))
def test_workspace_with_and_without_room_for_packed_weights(shape, out_type):
    assert check(shape, out_type, workspace="full") and check(shape, out_type, workspace="least")


def test_built_in_workspace_without_room_for_packed_weights():
    """The built-in array is enough for the call and not for the packed weights beside it: the call runs all the same."""
    shape = (124, 16, 16, 64, 64, 3, 1, ONE)
    limit = lce.lce_bconv2d_host_noalloc_max_bytes()
    assert least_workspace(*shape[:6], 124 * 16 * 16 * 64) <= limit
    assert lce.lce_bconv2d_host_workspace_bytes(lce.make_desc(*shape[:5])) > limit
    check(shape, lce.OUT_FLOAT32, entry="lce_bconv2d_host_noalloc")


def test_calls_from_fresh_host_threads():
    """A thread's first CUDA call may be this one; several at a time, each with arrays and a workspace of its own."""
    shapes = [(2, 9, 11, 40, 36, 3, 1, ONE), (16, 28, 28, 128, 128, 3, 1, ONE), (1, 512, 1024, 32, 1, 1, 1, ONE), (3, 5, 7, 70, 33, 3, 2, ONE)]
    with concurrent.futures.ThreadPoolExecutor(len(shapes)) as pool:
        for done in [pool.submit(check, shape, out_type, workspace=room) for shape in shapes
                     for out_type, room in ((lce.OUT_FLOAT32, "full"), (lce.OUT_BITPACKED, "least"))]:
            done.result()
