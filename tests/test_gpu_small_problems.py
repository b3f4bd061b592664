"""The kernels for small problems at the sizes where they change form: the row kernel (1 to 16 rows, K
shared by a cluster or not, several CTAs of features per SM). Every element against the oracle,
canaries around every buffer; the bounds are those of the other parity tests (one rounding to bf16,
fp32 sums)."""
import pytest
import torch

import oracle
from paper_2609_28568_b200 import binding as nb
from paper_2609_28568_b200 import synth
from parity import Guarded, check_bf16, f32

pytestmark = pytest.mark.gpu
DEV = "cuda"


def gen(seed, shape, std):
    return synth.normal(seed, shape, std, DEV)


@pytest.mark.parametrize("act", [nb.ACT_NONE, nb.ACT_GELU, nb.ACT_SWIGLU])
@pytest.mark.parametrize("BT,C,OC", [
    (1, 8, 16), (8, 3080, 208), (9, 1032, 80), (16, 4096, 48),   # rows: K in one CTA / shared by 2, 4 and 8
    (3, 72, 7200), (16, 40, 7200),                                # rows: several CTAs of features per SM
])
def test_small_forward(BT, C, OC, act):
    inp, w, b = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (OC,), 0.05)
    out = Guarded((BT, OC // 2 if act == nb.ACT_SWIGLU else OC), torch.bfloat16)
    pre = Guarded((BT, OC), torch.bfloat16) if act else None
    o_ref, p_ref = oracle.linear_forward(f32(inp), f32(w), f32(b), act)
    for _ in range(2):   # back to back: a second launch may start while the first drains
        nb.nb_linear_forward_ex(out.t, pre.t if pre else None, inp, w, b, BT, C, OC, act)
    check_bf16(out.t, o_ref, "out")
    out.check("out")
    if pre:
        check_bf16(pre.t, p_ref, "pre_act")
        pre.check("pre_act")
    nb.nb_check_status()
