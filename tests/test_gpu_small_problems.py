"""The kernels for small problems at the sizes where they change form: the row kernel (1 to 16 rows, K
shared by a cluster or not, several CTAs of features per SM), the tile kernel (every tile width, one
row past a tile, K split over 2, 4 and 8 CTAs, ragged K and columns), both products of a backward in
one launch, the adapter's two launches. The tests whose name ends in `forms` state the form that each case is
there for and check it by the host's view of the route. Every element against the oracle, canaries around every buffer; the bounds are those of
the other parity tests (one rounding to bf16, fp32 sums)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2609_28568_b200 import binding as nb
from paper_2609_28568_b200 import synth
from parity import Guarded, check_bf16, check_f32, f32

pytestmark = pytest.mark.gpu
DEV = "cuda"


def gen(seed, shape, std):
    return synth.normal(seed, shape, std, DEV)


@pytest.mark.parametrize("act", [nb.ACT_NONE, nb.ACT_GELU, nb.ACT_SWIGLU])
@pytest.mark.parametrize("BT,C,OC", [
    (1, 8, 16), (8, 3080, 208), (9, 1032, 80), (16, 4096, 48),   # rows: K in one CTA / shared by 2, 4 and 8
    (3, 72, 7200), (16, 40, 7200),                                # rows: several CTAs of features per SM (not SwiGLU)
    (17, 264, 144), (64, 1544, 80), (128, 3072, 96),              # tiles: fewer rows than a tile, K split
    (129, 776, 400), (300, 2056, 272), (1000, 328, 1424),         # tiles: one row past, several row tiles
    (1030, 72, 2608),                                             # tiles of 192 columns
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


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("BT,C,OC", [
    (1, 8, 16), (8, 136, 3072), (64, 776, 200), (128, 264, 2056),   # dinp's K split over 4, or not
    (129, 72, 136), (256, 520, 1544), (257, 520, 1544),              # the last split, the first without
    (384, 768, 776), (1000, 264, 328),                               # more k-blocks than stages for dweight
    (1030, 2608, 72),                                                # dinp alone in tiles of 192 columns
    (1500, 776, 3080), (1030, 1000, 6152),                           # the persistent launch, or (second, from zero) tiles
])
def test_small_backward(BT, C, OC, fused):
    inp, w, dout = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (BT, OC), 1e-3)
    ipre = gen(4, (BT, C), 1.0) if fused else None
    r = oracle.linear_backward(f32(dout), f32(inp), f32(w), inp_pre=f32(ipre) if fused else None)
    dinp = Guarded((BT, C), torch.bfloat16)
    dw, db = Guarded((OC, C), torch.float32, fill=7.0), Guarded((OC,), torch.float32, fill=-7.0)
    for acc in range(2):
        nb.nb_linear_backward_ex(dinp.t, dw.t, db.t, dout, inp, w, None, ipre, BT, C, OC, nb.ACT_NONE, acc)
    check_bf16(dinp.t, r["dinp"], "dinp")
    check_f32(dw.t, 2 * r["dweight"], "dweight")
    check_f32(db.t, 2 * r["dbias"], "dbias")
    for g, n in ((dinp, "dinp"), (dw, "dweight"), (db, "dbias")):
        g.check(n)
    # dinp has one value, whatever else is asked for
    alone = torch.empty_like(dinp.t)
    nb.nb_linear_backward_ex(alone, None, None, dout, None, w, None, ipre, BT, C, OC, nb.ACT_NONE, 0)
    assert torch.equal(alone, dinp.t)
    # dweight alone, and without a bias gradient
    dw2 = Guarded((OC, C), torch.float32, fill=3.0)
    nb.nb_linear_backward_ex(None, dw2.t, None, dout, inp, None, None, None, BT, C, OC, nb.ACT_NONE, 0)
    check_f32(dw2.t, r["dweight"], "dweight alone")
    dw2.check("dweight alone")
    nb.nb_check_status()


@pytest.mark.parametrize("BT,C,OC,r", [
    (1, 8, 8, 8), (100, 72, 2056, 16), (129, 1544, 136, 40), (519, 1024, 776, 8), (640, 264, 3072, 64),
])
def test_small_adapter_layer(BT, C, OC, r):
    scale = 32.0 / math.sqrt(r)
    inp, w, dout = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.02), gen(3, (BT, OC), 1e-3)
    a, b = gen(4, (r, C), 0.02), gen(5, (OC, r), 0.02)
    out, t, u = (Guarded((BT, n), torch.bfloat16) for n in (OC, r, r))
    dinp = Guarded((BT, C), torch.bfloat16)
    dA, dB = Guarded((r, C), torch.float32, fill=7.0), Guarded((OC, r), torch.float32, fill=-7.0)
    nb.nb_lora_linear_forward(out.t, t.t, inp, w, None, a, b, scale, BT, C, OC, r)
    for acc in range(2):
        nb.nb_lora_linear_backward(dinp.t, dA.t, dB.t, u.t, dout, inp, w, a, b, t.t, scale, BT, C, OC, r, acc)
    t_ref = scale * oracle.linear_forward(f32(inp), f32(a))[0]
    u_ref = scale * oracle.linear_backward(f32(dout), None, f32(b), want=("dinp",))["dinp"]
    di_ref, dA_ref, dB_ref = oracle.lora_backward(f32(dout), f32(inp), f32(w), f32(a), f32(b), scale)
    check_bf16(t.t, t_ref, "t")
    check_bf16(u.t, u_ref, "u")
    # t and u are rounded to bf16 once (2^-9 of each element), which the other factor passes on
    check_bf16(out.t, oracle.lora_forward(f32(inp), f32(w), None, f32(a), f32(b), scale), "out",
               extra=2.0 ** -9 * (np.abs(t_ref) @ np.abs(f32(b).T.astype(np.float64))))
    check_bf16(dinp.t, di_ref, "dinp", extra=2.0 ** -9 * (np.abs(u_ref) @ np.abs(f32(a).astype(np.float64))))
    check_f32(dA.t, 2 * dA_ref, "dA")
    check_f32(dB.t, 2 * dB_ref, "dB")
    for g, n in ((out, "out"), (t, "t"), (u, "u"), (dinp, "dinp"), (dA, "dA"), (dB, "dB")):
        g.check(n)
    nb.nb_check_status()


@pytest.mark.parametrize("BT,Vp,V", [
    (1, 8, 1), (700001, 8, 5),           # a vector per row; more vectors than one pass of the grid takes
    (40000, 136, 129), (7, 50304, 50257),
    (3, 2 * 148 * 2048 * 8 + 24, 2 * 148 * 2048 * 8 + 1),  # rows longer than a pass
])
def test_dlogits_row_and_column_carried_along(BT, Vp, V):
    logits = gen(1, (BT, Vp), 2.0)
    targets = ((torch.arange(BT, device="cuda", dtype=torch.int64) * 7919 + V - 1) % V).to(torch.int32)
    lse = torch.logsumexp(logits[:, :V].double(), 1).float()
    _, _, ref = oracle.cross_entropy(f32(logits), targets.cpu().numpy(), V, 0.5)
    out = Guarded((BT, Vp), torch.bfloat16)
    nb.nb_ce_backward(out.t, logits, lse, targets, 0.5, BT, Vp, V)
    check_bf16(out.t, ref, "dlogits")
    out.check("dlogits")
    assert torch.all(out.t[:, V:] == 0)
    nb.nb_ce_backward(logits, logits, lse, targets, 0.5, BT, Vp, V)
    assert torch.equal(logits, out.t)


@pytest.mark.parametrize("act", [nb.ACT_NONE, nb.ACT_GELU])
@pytest.mark.parametrize("BT,C,OC,r", [(1990, 136, 3080, 8), (1800, 72, 3264, 64), (4500, 200, 2120, 16)])
def test_forward_in_192_column_pair_tiles(act, BT, C, OC, r):
    """Several waves of the CTA pairs, as many as with 256 columns: one column past a tile, a full last
    tile, a ragged one; with an adapter term, whose k-blocks go through the same boxes."""
    inp, w, bias = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (OC,), 0.1)
    ref, pre_ref = oracle.linear_forward(f32(inp), f32(w), f32(bias), act=act)
    out, pre = Guarded((BT, OC), torch.bfloat16), Guarded((BT, OC), torch.bfloat16)
    nb.nb_linear_forward_ex(out.t, pre.t if act else None, inp, w, bias, BT, C, OC, act)
    check_bf16(out.t, ref, "out")
    out.check("out")
    if act:
        check_bf16(pre.t, pre_ref, "pre")
        pre.check("pre")
        return
    a, b, scale = gen(4, (r, C), 0.02), gen(5, (OC, r), 0.02), 4.0
    t = Guarded((BT, r), torch.bfloat16)
    nb.nb_lora_linear_forward(out.t, t.t, inp, w, bias, a, b, scale, BT, C, OC, r)
    t_ref = scale * oracle.linear_forward(f32(inp), f32(a))[0]
    check_bf16(out.t, oracle.lora_forward(f32(inp), f32(w), f32(bias), f32(a), f32(b), scale), "out with adapter",
               extra=2.0 ** -9 * (np.abs(t_ref) @ np.abs(f32(b).T.astype(np.float64))))
    out.check("out with adapter")
    nb.nb_check_status()


def _layers_loop(BT, C, H, fused, sync):
    """Two layers, forward and backward, over and over on two alternating sets of buffers: every tensor a
    launch reads was written by one of the launches just before it, over what it held two passes earlier.
    The weights shrink what goes through them, so the values settle where the biases put them."""
    w1, w2 = gen(11, (H, C), 0.4 * C ** -0.5), gen(12, (C, H), 0.4 * H ** -0.5)
    b1, b2 = gen(13, (H,), 0.1), gen(14, (C,), 0.1)
    bf = dict(dtype=torch.bfloat16, device=DEV)
    x = [gen(15, (BT, C), 1.0), torch.empty((BT, C), **bf)]
    h, pre, dh = ([torch.empty((BT, H), **bf) for _ in range(2)] for _ in range(3))
    y = [torch.empty((BT, C), **bf) for _ in range(2)]
    dw = [torch.empty((C, H), device=DEV) for _ in range(2)]
    wc = [torch.empty((C, H), **bf) for _ in range(2)]
    for i in range(24):
        k = i & 1
        calls = (
            lambda: nb.nb_linear_forward_ex(h[k], pre[k], x[k], w1, b1, BT, C, H, nb.ACT_GELU),
            lambda: nb.nb_linear_forward_ex(y[k], None, h[k], w2, b2, BT, H, C, nb.ACT_NONE),
            lambda: nb.nb_linear_backward_ex(dh[k], dw[k], None, y[k], h[k], w2, None, pre[k] if fused else None, BT, H, C,
                                             nb.ACT_NONE, 0),
            lambda: nb.nb_cast_f32_to_bf16(wc[k], dw[k], C * H),
            lambda: nb.nb_linear_backward_ex(x[1 - k], None, None, dh[k], None, w1, None if fused else pre[k], None, BT, C, H,
                                             nb.ACT_NONE if fused else nb.ACT_GELU, 0),
        )
        for call in calls:
            call()
            if sync:
                torch.cuda.synchronize()
    torch.cuda.synchronize()
    for a, b in zip(wc, dw):
        assert torch.equal(a, b.to(torch.bfloat16))
    return x + h + pre + y + dh


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("BT,C,H", [(8, 768, 3072), (3, 1032, 520), (72, 768, 776), (300, 520, 1544), (2100, 776, 1032)])
def test_chained_launches_over_two_alternating_buffers(BT, C, H, fused):
    """A launch may start while its producer runs; what it then reads has to be what that one wrote, not what
    the buffer held before: the same bits as with the device idle between launches."""
    for a, b in zip(_layers_loop(BT, C, H, fused, False), _layers_loop(BT, C, H, fused, True)):
        assert torch.isfinite(a).all() and a.any()
        assert torch.equal(a, b)
    nb.nb_check_status()


@pytest.mark.parametrize("BT", [5, 300])
def test_chained_head_over_two_alternating_buffers(BT):
    C, Vp, V = 264, 1016, 1009
    w = gen(21, (Vp, C), C ** -0.5)
    targets = (torch.arange(BT, device=DEV) * 31 % V).to(torch.int32)
    got = []
    for sync in (False, True):
        x = [gen(22, (BT, C), 1.0), torch.empty((BT, C), dtype=torch.bfloat16, device=DEV)]
        logits = [torch.empty((BT, Vp), dtype=torch.bfloat16, device=DEV) for _ in range(2)]
        loss, lse = ([torch.empty(BT, device=DEV) for _ in range(2)] for _ in range(2))
        for i in range(24):
            k = i & 1
            for call in (
                lambda: nb.nb_lm_head_ce_forward(logits[k], loss[k], lse[k], x[k], w, targets, BT, C, Vp, V),
                lambda: nb.nb_ce_backward(logits[k], logits[k], lse[k], targets, 2.0, BT, Vp, V),
                lambda: nb.nb_linear_backward_ex(x[1 - k], None, None, logits[k], None, w, None, None, BT, C, Vp,
                                                 nb.ACT_NONE, 0),
            ):
                call()
                if sync:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        got.append(x + logits + loss + lse)
    for a, b in zip(*got):
        assert torch.isfinite(a).all() and a.any()
        assert torch.equal(a, b)
    nb.nb_check_status()


def _seen(route, form):
    assert route == [form], (route, form)


@pytest.mark.parametrize("act", [nb.ACT_NONE, nb.ACT_GELU])
@pytest.mark.parametrize("BT,C,OC,form", [
    (2, 1048, 24, ("rows", 16, 2, 2)), (7, 2248, 40, ("rows", 16, 4, 2)), (13, 4152, 24, ("rows", 16, 8, 2)),
    (9, 136, 7208, ("rows", 16, 1, 4)),
    (60, 840, 1616, ("tile", 32, 2, 1)), (139, 1208, 560, ("tile", 32, 2, 1)), (129, 672, 48, ("tile", 32, 4, 1)),
    (144, 40, 2448, ("tile", 64, 1, 1)), (35, 856, 2512, ("tile", 64, 2, 1)), (130, 1440, 560, ("tile", 64, 4, 1)),
    (134, 2896, 48, ("tile", 64, 8, 1)), (139, 40, 5520, ("tile", 128, 1, 1)), (26, 1112, 5008, ("tile", 128, 2, 1)),
    (135, 3272, 1200, ("tile", 128, 4, 1)), (25, 1296, 1136, ("tile", 128, 8, 1)), (296, 40, 6320, ("tile", 192, 1, 1)),
    (552, 40, 6384, ("gemm", 192, 1, 1)), (419, 40, 7200, ("gemm", 256, 1, 1)),
])
def test_forward_forms(BT, C, OC, form, act):
    _seen(nb.nb_debug_route(nb.CALL_FORWARD, BT, C, OC, act=act), form)
    test_small_forward(BT, C, OC, act)


@pytest.mark.parametrize("BT,C,OC,form", [
    (5, 136, 14256, ("rows", 16, 1, 4)), (11, 136, 14256, ("rows", 16, 1, 2)), (3, 1048, 48, ("rows", 16, 2, 2)),
    (16, 4152, 32, ("rows", 16, 8, 2)), (17, 264, 144, ("tile", 128, 1, 1)), (300, 40, 6480, ("gemm", 256, 1, 1)),
])
def test_forward_swiglu_forms(BT, C, OC, form):
    _seen(nb.nb_debug_route(nb.CALL_FORWARD, BT, C, OC, act=nb.ACT_SWIGLU), form)
    test_small_forward(BT, C, OC, nb.ACT_SWIGLU)


@pytest.mark.parametrize("BT,C,OC,fused,form", [
    (139, 3312, 96, False, ("tile_pair", 64, 1, 2)), (139, 3312, 96, True, ("tile_pair", 64, 1, 2)),
    (9, 2024, 2448, False, ("tile_pair", 64, 2, 2)), (142, 1272, 1712, True, ("tile_pair", 64, 2, 2)),
    (205, 536, 8080, False, ("tile_pair", 64, 2, 1)), (205, 536, 8080, True, ("tile_pair", 64, 2, 1)),
    (135, 40, 1008, True, ("tile_pair", 64, 4, 1)),
    (131, 552, 1040, False, ("tile_pair", 64, 4, 2)), (131, 552, 1040, True, ("tile_pair", 64, 4, 2)),
    (130, 3184, 48, False, ("tile_pair", 128, 1, 1)), (130, 3184, 48, True, ("tile_pair", 128, 1, 1)),
    (133, 3808, 288, False, ("tile_pair", 128, 1, 2)),
    (134, 800, 5552, False, ("tile_pair", 128, 2, 1)), (134, 800, 5552, True, ("tile_pair", 128, 2, 1)),
    (36, 2616, 880, False, ("tile_pair", 128, 2, 2)),
    (9, 72, 4640, False, ("tile_pair", 128, 4, 1)), (9, 72, 4640, True, ("tile_pair", 128, 4, 1)),
    (9, 2104, 560, False, ("tile_pair", 128, 4, 2)),
    # the persistent launch: ragged edges, and dinp in halved tiles
    (1990, 8, 16, False, ("layer_bwd", 256, 1, 1)), (1990, 8, 16, True, ("layer_bwd", 256, 1, 1)),
    (1424, 808, 48, False, ("layer_bwd", 256, 1, 1)), (1424, 808, 48, True, ("layer_bwd", 256, 1, 1)),
    (2300, 72, 136, False, ("layer_bwd", 256, 1, 1)), (2300, 72, 136, True, ("layer_bwd", 256, 1, 1)),
    (1375, 648, 3088, False, ("layer_bwd", 128, 1, 1)),
])
def test_backward_forms(BT, C, OC, fused, form):
    """With a bias gradient, from zero and accumulating: both take the form."""
    for accumulate in (False, True):
        _seen(nb.nb_debug_route(nb.CALL_BACKWARD, BT, C, OC, gelu_grad=fused, accumulate=accumulate), form)
    test_small_backward(BT, C, OC, fused)


@pytest.mark.parametrize("accumulate", [0, 1])
@pytest.mark.parametrize("BT,C,OC,bias", [(1500, 760, 3080, False), (1500, 760, 3080, True), (1030, 760, 6152, True)])
def test_backward_with_halved_dinp_tiles_forms(BT, C, OC, bias, accumulate):
    """Ragged columns in the last halved tile, ragged rows, ragged K, every element."""
    _seen(nb.nb_debug_route(nb.CALL_BACKWARD, BT, C, OC, dbias=bias, accumulate=bool(accumulate)), ("layer_bwd", 128, 1, 1))
    inp, w, dout = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (BT, OC), 1e-3)
    r = oracle.linear_backward(f32(dout), f32(inp), f32(w))
    dinp = Guarded((BT, C), torch.bfloat16)
    dw = Guarded((OC, C), torch.float32, fill=0.5)
    db = Guarded((OC,), torch.float32, fill=-0.25) if bias else None
    nb.nb_linear_backward_ex(dinp.t, dw.t, db.t if bias else None, dout, inp, w, None, None, BT, C, OC, nb.ACT_NONE, accumulate)
    check_bf16(dinp.t, r["dinp"], "dinp")
    check_f32(dw.t - 0.5 * accumulate, r["dweight"], "dweight")
    if bias:
        check_f32(db.t + 0.25 * accumulate, r["dbias"], "dbias")
    for g, n in ((dinp, "dinp"), (dw, "dweight"), (db, "dbias")):
        if g is not None:
            g.check(n)
    nb.nb_check_status()


@pytest.mark.parametrize("BT,C,OC,r,down,up,back", [
    (83, 784, 1168, 24, ("tile", 32, 4, 1), ("tile", 32, 2, 1), ["tile_pair", "tile_pair"]),
    (134, 968, 736, 64, ("tile", 64, 8, 1), ("tile", 32, 1, 1), ["tile_pair", "tile_pair"]),
    (26, 992, 4544, 16, ("tile", 64, 8, 1), ("tile", 64, 2, 1), ["tile_pair", "tile_pair"]),
    (532, 8, 6352, 16, ("tile", 32, 1, 1), ("gemm", 192, 1, 1), ["tile_pair", "tile_pair"]),
    (852, 2496, 32, 8, ("tile", 32, 4, 1), ("tile", 32, 4, 1), ["tile_pair", "tile", "tile_pair"]),
    (1550, 8, 16, 48, ("tile", 64, 1, 1), ("tile", 32, 1, 1), ["lora_udb", "tile"]),
])
def test_adapter_forms(BT, C, OC, r, down, up, back):
    assert nb.nb_debug_route(nb.CALL_LORA_FORWARD, BT, C, OC, r=r) == [down, up]
    for accumulate in (False, True):
        got = nb.nb_debug_route(nb.CALL_LORA_BACKWARD, BT, C, OC, r=r, accumulate=accumulate)
        assert [k[0] for k in got] == back, got
    test_small_adapter_layer(BT, C, OC, r)


@pytest.mark.parametrize("act,BT,C,OC,whole", [
    (nb.ACT_NONE, 1500, 1000, 1544, True),      # every unit of dweight is a tile's whole K: stored, nothing cleared
    (nb.ACT_NONE, 1290, 1032, 4104, True), (nb.ACT_NONE, 2050, 520, 3080, True),  # ragged tiles, one k-block past 32
    (nb.ACT_NONE, 1300, 2056, 1032, False),     # cut: cleared by a launch of its own
    (nb.ACT_GELU, 1300, 2056, 1032, False), (nb.ACT_SWIGLU, 1300, 2056, 1040, False),  # cleared with the activation's pass
    (nb.ACT_GELU, 1290, 1032, 4104, True),
])
def test_fresh_gradients_of_the_persistent_backward(act, BT, C, OC, whole):
    """dweight and dbias start from nothing (over what the buffers held), then a second call adds to them."""
    route = nb.nb_debug_route(nb.CALL_BACKWARD, BT, C, OC, act=act, accumulate=False)
    assert route[0][0] == "layer_bwd", route
    hdr, recs = nb.nb_debug_layer_bwd_plan(BT, C, OC, torch.cuda.get_device_properties(0).multi_processor_count // 2, False,
                                           launched=True, fresh=True)
    assert all(k1 - k0 == hdr[5] for _, is_w, _, _, k0, k1 in recs if is_w) == whole
    inp, w, dout = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (BT, OC // 2 if act == nb.ACT_SWIGLU else OC), 1e-3)
    pre = gen(4, (BT, OC), 1.0) if act else None
    r = oracle.linear_backward(f32(dout), f32(inp), f32(w), pre=f32(pre) if act else None, act=act)
    dinp = Guarded((BT, C), torch.bfloat16)
    dw, db = Guarded((OC, C), torch.float32, fill=7.0), Guarded((OC,), torch.float32, fill=float("nan"))
    for acc in range(2):
        nb.nb_linear_backward_ex(dinp.t, dw.t, db.t, dout, inp, w, pre, None, BT, C, OC, act, acc)
        check_bf16(dinp.t, r["dinp"], "dinp")
        check_f32(dw.t, (acc + 1) * r["dweight"], "dweight")
        check_f32(db.t, (acc + 1) * r["dbias"], "dbias")
    for g, n in ((dinp, "dinp"), (dw, "dweight"), (db, "dbias")):
        g.check(n)
    nb.nb_check_status()


@pytest.mark.parametrize("fused,bias", [(False, False), (True, True), (True, False)])
@pytest.mark.parametrize("BT,C,OC,whole", [(1500, 1000, 1544, True), (1290, 1032, 4104, True), (2050, 520, 3080, True),
                                           (1300, 2056, 1032, False)])
def test_fresh_gradients_of_the_other_forms(fused, bias, BT, C, OC, whole):
    """The same for the kernels with the producer's GELU derivative, whose fp32 results leave through a single box, and for
    those without a bias gradient: stored or added to, in one part or several."""
    assert nb.nb_debug_route(nb.CALL_BACKWARD, BT, C, OC, dbias=bias, gelu_grad=fused, accumulate=False)[0][0] == "layer_bwd"
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    hdr, recs = nb.nb_debug_layer_bwd_plan(BT, C, OC, pairs, fused, launched=True, fresh=True)
    assert all(k1 - k0 == hdr[5] for _, is_w, _, _, k0, k1 in recs if is_w) == whole
    inp, w, dout = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (BT, OC), 1e-3)
    ipre = gen(4, (BT, C), 1.0) if fused else None
    r = oracle.linear_backward(f32(dout), f32(inp), f32(w), inp_pre=f32(ipre) if fused else None)
    dinp, dw = Guarded((BT, C), torch.bfloat16), Guarded((OC, C), torch.float32, fill=7.0)
    db = Guarded((OC,), torch.float32, fill=float("nan")) if bias else None
    for acc in range(2):
        nb.nb_linear_backward_ex(dinp.t, dw.t, db.t if bias else None, dout, inp, w, None, ipre, BT, C, OC, nb.ACT_NONE, acc)
        check_bf16(dinp.t, r["dinp"], "dinp")
        check_f32(dw.t, (acc + 1) * r["dweight"], "dweight")
        if bias:
            check_f32(db.t, (acc + 1) * r["dbias"], "dbias")
            db.check("dbias")
    dinp.check("dinp")
    dw.check("dweight")
    nb.nb_check_status()


@pytest.mark.parametrize("BT,C,OC", [(4096, 768, 3072), (8192, 768, 3072), (5000, 776, 2056)])
def test_long_sums_of_the_persistent_backward(BT, C, OC):
    """The error of a sum in a tensor core's accumulator goes with its length, and the schedule promises sums of at most 32
    k-blocks at these sizes: dweight is at most twice as far from its value in 64 bits as when the same rows are
    added up 1024 at a time, in sums of 16 (by a kernel that does not cut K)."""
    for rows, accumulate, kernel in ((BT, False, "layer_bwd"), (1024, False, "tile_pair"), (1024, True, "tile_pair")):
        assert nb.nb_debug_route(nb.CALL_BACKWARD, rows, C, OC, dbias=False, accumulate=accumulate)[0][0] == kernel
    inp, w, dout = gen(1, (BT, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (BT, OC), 1e-3)
    ref = dout.double().t() @ inp.double()
    dinp = torch.empty((BT, C), dtype=torch.bfloat16, device="cuda")
    error = {}
    for rows in (BT, 1024):
        dw = torch.empty((OC, C), dtype=torch.float32, device="cuda")
        for m in range(0, BT, rows):
            n = min(rows, BT - m)
            nb.nb_linear_backward_ex(dinp[m:m + n], dw, None, dout[m:m + n], inp[m:m + n], w, None, None, n, C, OC, nb.ACT_NONE,
                                     int(m > 0))
        error[rows] = float((dw.double() - ref).norm() / ref.norm())
    nb.nb_check_status()
    assert error[BT] <= 2 * error[1024], error


def test_many_row_counts_of_the_persistent_backward():
    """More sizes than the schedules that are kept, each twice over, so that the first ones are found again."""
    C, OC, most = 1032, 2056, 2600
    inp, w, dout = gen(1, (most, C), 1.0), gen(2, (OC, C), 0.05), gen(3, (most, OC), 1e-3)
    dinp = torch.empty((most, C), dtype=torch.bfloat16, device="cuda")
    dw = torch.empty((OC, C), dtype=torch.float32, device="cuda")
    for BT in list(range(most - 8 * 69, most + 1, 8)) * 2:
        assert nb.nb_debug_route(nb.CALL_BACKWARD, BT, C, OC, dbias=False, accumulate=False)[0][0] == "layer_bwd"
        nb.nb_linear_backward_ex(dinp[:BT], dw, None, dout[:BT], inp[:BT], w, None, None, BT, C, OC, nb.ACT_NONE, 0)
        ref, dref = dout[:BT].double().t() @ inp[:BT].double(), dout[:BT].double() @ w.double()
        # fp32 sums of at most 41 k-blocks: 1e-7 a k-block; dinp rounded to bf16 besides, 2^-9 at most
        assert torch.dist(dw.double(), ref) <= 5e-6 * torch.linalg.norm(ref), BT
        assert torch.dist(dinp[:BT].double(), dref) <= 2e-3 * torch.linalg.norm(dref), BT
    nb.nb_check_status()
