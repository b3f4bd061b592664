"""The Python binding's argument handling: what it takes, and that a failure of torch underneath is an exception."""
import ctypes
import subprocess
import sys

import pytest
import torch

from paper_2609_28568_b200 import binding as nb
from paper_2609_28568_b200 import build, synth

FAKE = """
import sys
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2609_28568_b200 import binding as nb
bf = dict(dtype=torch.bfloat16, device="cuda")
with FakeTensorMode():
    x, w, d = torch.empty((4, 8), **bf), torch.empty((16, 8), **bf), torch.empty((4, 16), **bf)
    for call in (lambda: nb.linear_forward(x, w), lambda: nb.linear_backward(d, x, w),
                 lambda: nb.nb_linear_forward_ex(d, None, x, w, None, 4, 8, 16, 0)):
        try:
            call()
        except RuntimeError as e:
            print("raised:", type(e).__name__)
"""


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def test_tensors_without_storage_raise():
    """Tensors whose address cannot be had (as while a program is traced): an exception, in a process of its
    own because an exception thrown without the interpreter's lock ends the process."""
    r = subprocess.run([sys.executable, "-c", FAKE], capture_output=True, text=True, timeout=300, stdin=subprocess.DEVNULL)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    assert r.stdout.count("raised:") == 3, r.stdout


class _Carrier:
    def __init__(self, p):
        self._as_parameter_ = p


class _LikeATensor:
    is_cuda = True

    def __init__(self, address):
        self.address = address

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return self.address


def test_kinds_of_streams_and_pointers():
    """Calls on no rows or elements return before the device is touched: only the arguments are looked at."""
    P = 0x10000
    for stream in (0, 7, ctypes.c_void_p(7), ctypes.c_void_p(), _Carrier(ctypes.c_void_p(7)), _Carrier(_Carrier(7))):
        nb.nb_cast_f32_to_bf16(P, P, 0, stream)
        nb.nb_linear_forward_ex(P, None, P, P, None, 0, 8, 8, nb.ACT_NONE, stream=stream)
    with pytest.raises(TypeError):
        nb.nb_cast_f32_to_bf16(P, P, 0, object())
    nb.nb_cast_f32_to_bf16(_LikeATensor(P), _LikeATensor(P), 0, 0)
    with pytest.raises(nb.NbError):  # the address gets there
        nb.nb_cast_f32_to_bf16(_LikeATensor(P), _LikeATensor(P + 4), 8, 0)
    with pytest.raises(AssertionError):
        nb.nb_cast_f32_to_bf16(torch.zeros(8), P, 0, 0)


@pytest.mark.gpu
def test_kinds_of_arguments_of_the_allocating_calls():
    """Addresses in the place of tensors, a weight with its columns in two dimensions, gradients that are not asked
    for, a stream object: the results of the plain call."""
    BT, C, OC = 40, 72, 136
    x, w, b = (synth.normal(i, s, 0.1, "cuda") for i, s in ((1, (BT, C)), (2, (OC, C)), (3, (OC,))))
    out, pre = nb.linear_forward(x, w, b, nb.ACT_GELU)
    for weight in (w.view(OC, 9, 8), w.view(OC, C, 1)):
        o2, p2 = nb.linear_forward(x, weight, b.data_ptr(), nb.ACT_GELU)
        assert torch.equal(o2, out) and torch.equal(p2, pre)
    with pytest.raises(ValueError):
        nb.linear_forward(x.view(BT, 9, 8), w)
    dinp, dw, db = nb.linear_backward(out, x, w, pre, act=nb.ACT_GELU)
    mine = torch.empty_like(dw)
    other = torch.zeros(3)  # on the CPU: never looked at
    got = nb.linear_backward(out.view(BT, 17, 8), x.data_ptr(), w, pre.data_ptr(), act=nb.ACT_GELU, dweight=mine, dbias=other,
                             need_dbias=False)
    assert torch.equal(got[0], dinp) and got[1] is mine and got[2] is other
    assert torch.equal(mine, dw)
    address = mine.zero_().data_ptr()
    assert nb.linear_backward(out, x, w, pre, act=nb.ACT_GELU, dweight=address, need_dinp=False)[:2] == (None, address)
    assert torch.equal(mine, dw)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    o3 = torch.empty_like(out)
    nb.nb_linear_forward_ex(o3, torch.empty_like(pre), x, w, b, BT, C, OC, nb.ACT_GELU, side)
    torch.cuda.synchronize()
    assert torch.equal(o3, out)
