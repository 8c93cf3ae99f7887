"""lce_bconv2d_host against the oracle, every element, over the ways an array can reach the device and an output can come
back: by the copy engine or by a kernel, or written by the convolution itself."""
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
