"""The Python binding's argument handling: what it takes, and that a failure of torch underneath is an exception."""
import subprocess
import sys

import pytest

from paper_2609_28568_b200 import build

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
