"""The C-ABI library loads without a GPU, exports what the header declares, and rejects
malformed requests before touching the device."""
import os
import re

import pytest

from paper_2609_28568_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    build.build()
    return binding.lib()


def test_exports_match_header(L):
    header = open(os.path.join(ROOT, "include", "nb_linear.h")).read()
    header = re.sub(r"/\*.*?\*/", "", header, flags=re.S)
    declared = set(re.findall(r"\b(nb_[a-z0-9_]+)\s*\(", header))
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert hasattr(L, name), name


def test_version_and_out_elems(L):
    assert L.nb_version() == 100
    assert L.nb_linear_out_elems(128, 3072, binding.ACT_NONE) == 128 * 3072
    assert L.nb_linear_out_elems(128, 3072, binding.ACT_GELU) == 2 * 128 * 3072
    assert L.nb_linear_out_elems(16, 6144, binding.ACT_SWIGLU) == 16 * 3072 + 16 * 6144
    assert L.nb_linear_out_elems(16, 7, binding.ACT_SWIGLU) == -1
    assert L.nb_linear_out_elems(-1, 8, binding.ACT_NONE) == -1
    assert L.nb_linear_out_elems(1, 8, 9) == -1


def test_stream_is_per_thread_state(L):
    assert L.nb_get_stream() in (None, 0)
    L.nb_set_stream(0x1000)
    assert L.nb_get_stream() == 0x1000
    L.nb_set_stream(None)


def test_malformed_requests_are_rejected_without_a_device(L):
    P = 0x10000  # a fake, aligned device address: never dereferenced by a rejected call
    fwd = L.nb_linear_forward_ex
    assert fwd(None, None, P, P, None, 8, 8, 8, 0, None) == binding.NB_ERR_INVALID_ARG
    assert b"NULL" in L.nb_last_error()
    assert fwd(P, None, P, P, None, 8, 8, 8, 7, None) == binding.NB_ERR_INVALID_ARG
    assert fwd(P, None, P, P, None, -1, 8, 8, 0, None) == binding.NB_ERR_INVALID_ARG
    assert fwd(P, None, P, P, None, 8, 12, 8, 0, None) == binding.NB_ERR_UNSUPPORTED
    assert fwd(P, None, P, P, None, 8, 8, 20, 0, None) == binding.NB_ERR_UNSUPPORTED
    assert fwd(P + 2, None, P, P, None, 8, 8, 8, 0, None) == binding.NB_ERR_INVALID_ARG
    assert fwd(P, None, P, P, None, 8, 8, 24, binding.ACT_SWIGLU, None) == binding.NB_ERR_UNSUPPORTED
    assert fwd(P, None, P, P, None, 1 << 31, 8, 8, 0, None) == binding.NB_ERR_UNSUPPORTED
    bwd = L.nb_linear_backward_ex
    assert bwd(P, P, P, None, P, P, None, None, 8, 8, 8, 0, 0, 0, None) == binding.NB_ERR_INVALID_ARG
    assert bwd(P, P, P, P, P, P, None, None, 8, 8, 8, 1, 0, 0, None) == binding.NB_ERR_INVALID_ARG
    assert bwd(P, P, P, P, None, P, None, None, 8, 8, 8, 0, 0, 0, None) == binding.NB_ERR_INVALID_ARG
    assert bwd(P, P, P, P, P, None, None, None, 8, 8, 8, 0, 0, 0, None) == binding.NB_ERR_INVALID_ARG
    assert bwd(None, P, P, P, P, P, None, P, 8, 8, 8, 0, 0, 0, None) == binding.NB_ERR_INVALID_ARG
    assert bwd(P, P, P, P, P, P, None, None, 8, 8, 8, 0, 1, 1, None) == binding.NB_ERR_UNSUPPORTED
    assert bwd(P, P, P, P, P, P, None, None, 8, 8, 8, 0, 0, 5, None) == binding.NB_ERR_INVALID_ARG
    assert L.nb_reduce_dbias(None, P, 8, 8, 0) == binding.NB_ERR_INVALID_ARG
    assert L.nb_reduce_dbias(P, P, 8, 12, 0) == binding.NB_ERR_UNSUPPORTED
    assert L.nb_debug_wait_timeout(0) == binding.NB_ERR_INVALID_ARG
    assert L.nb_workspace_reserve(-5) == binding.NB_ERR_INVALID_ARG


def test_forward_with_zero_rows_is_a_no_op_everywhere(L):
    P = 0x10000
    assert L.nb_linear_forward_ex(P, None, P, P, None, 0, 8, 8, 0, None) == binding.NB_OK


def test_binding_has_no_cpu_path(monkeypatch, tmp_path):
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", str(tmp_path / "missing.so"))
    with pytest.raises(RuntimeError, match="missing"):
        binding.lib()


def test_wgrad_split_plan_covers_every_k_block_once(L):
    """Host logic: whatever split-K factor is chosen, the units partition (tile, k-block) space."""
    shapes_ = [(2304, 768, 16384), (768, 768, 16384), (3072, 768, 16384), (768, 3072, 16384),
               (50304, 768, 16384), (1024, 1024, 16384), (6144, 1024, 16384), (200, 72, 136),
               (3072, 768, 128), (8, 8, 1), (776, 328, 5000)]
    for M, N, K in shapes_:
        for slots, tile_m in ((148, 128), (74, 256)):
            tm, tn, splits, kps, kblocks = binding.nb_debug_split_plan(M, N, K, slots, tile_m)
            assert tm == -(-M // tile_m) and tn == -(-N // 256) and kblocks == -(-K // 64)
            assert 1 <= splits <= kblocks and kps >= 1
            covered = [0] * kblocks
            for s in range(splits):
                lo, hi = s * kps, min((s + 1) * kps, kblocks)
                assert lo < hi, "empty split"
                for kb in range(lo, hi):
                    covered[kb] += 1
            assert covered == [1] * kblocks
            # the chosen factor never leaves more than a wave's worth of imbalance on big problems
            if kblocks >= 64 and tm * tn <= slots:
                assert tm * tn * splits >= slots // 2


def test_layer_backward_plan_covers_every_unit_once(L):
    """Host logic of the one-launch layer backward: over all CTA pairs, every dinp tile appears once
    with its whole K range, and every (dweight tile, k-block) is covered exactly once, whatever
    the interleaving and the balancing cuts; no pair is much dearer than the mean."""
    cases = [  # BT, C, OC
        (16384, 768, 2304), (16384, 768, 768), (16384, 768, 3072), (16384, 3072, 768),
        (16384, 768, 50304), (4096, 768, 3072), (4096, 3072, 768), (16384, 1024, 2048),
        (16384, 3072, 1024), (384, 768, 768), (136, 72, 200), (5000, 328, 776), (256, 8, 8),
    ]
    for BT, C, OC in cases:
        for pairs in (74, 66, 1):
            for gelu in (False, True):
                try:
                    hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, pairs, gelu)
                except binding.NbError as e:
                    assert e.code == binding.NB_ERR_UNSUPPORTED and pairs == 1
                    continue
                dtm, dtn, dkb, wtm, wtn, wkb, kbc, rounds = hdr
                assert (dtm, dtn, dkb) == (-(-BT // 256), -(-C // 256), -(-OC // 64))
                assert (wtm, wtn, wkb) == (-(-OC // 256), -(-C // 256), -(-BT // 64))
                assert 1 <= kbc <= wkb and rounds <= 64
                d_seen = {}
                w_cov = {}
                load = [0] * pairs   # in the planner's cost units: k-blocks, 5 for a unit of dweight, 1 (gelu' 2) for one of dinp
                for pr, is_w, m, n, kb0, kb1 in recs:
                    assert 0 <= pr < pairs and kb0 < kb1
                    load[pr] += kb1 - kb0 + (5 if is_w else (2 if gelu else 1))
                    if is_w:
                        assert 0 <= m < wtm and 0 <= n < wtn and kb1 <= wkb
                        cov = w_cov.setdefault((m, n), [0] * wkb)
                        for kb in range(kb0, kb1):
                            cov[kb] += 1
                    else:
                        assert 0 <= m < dtm and 0 <= n < dtn and (kb0, kb1) == (0, dkb)
                        d_seen[(m, n)] = d_seen.get((m, n), 0) + 1
                assert len(d_seen) == dtm * dtn and set(d_seen.values()) == {1}
                assert len(w_cov) == wtm * wtn
                assert all(c == [1] * wkb for c in w_cov.values())
                if pairs > 1 and BT >= 4096:
                    # the dearest pair is what counts: it has a few k-blocks more than the mean, as a range is worth its own
                    # allowance and a piece at least (a pair with less, or nothing, is fewer pieces for all)
                    assert max(load) <= sum(load) / pairs + 10, (BT, C, OC, pairs, gelu, max(load), sum(load) / pairs)


def test_layer_backward_plan_on_drawn_shapes(L):
    """The same partition property on 200 drawn problems (seeded): row counts from just past one tile to
    70,000, widths from 8 to 6144, several pair counts. Either the planner declines (more rounds than its
    order mask holds) or every dinp tile appears once and every (dweight tile, k-block) exactly once."""
    import numpy as np
    rng = np.random.default_rng(20260928)
    declined = 0
    for case in range(200):
        BT = int(rng.integers(129, 70_000)) if case % 4 else int(rng.choice((129, 256, 257, 4096, 16384, 65536)))
        C = 8 * int(rng.integers(1, 769))
        OC = 8 * int(rng.integers(1, 769))
        pairs = int(rng.choice((74, 66, 33, 7)))
        gelu = bool(rng.integers(0, 2))
        try:
            hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, pairs, gelu)
        except binding.NbError as e:
            assert e.code == binding.NB_ERR_UNSUPPORTED
            declined += 1
            continue
        dtm, dtn, dkb, wtm, wtn, wkb, kbc, rounds = hdr
        tag = (BT, C, OC, pairs, gelu)
        assert (dtm, dtn, dkb) == (-(-BT // 256), -(-C // 256), -(-OC // 64)), tag
        assert (wtm, wtn, wkb) == (-(-OC // 256), -(-C // 256), -(-BT // 64)), tag
        d_seen = np.zeros((dtm, dtn), dtype=np.int64)
        w_cov = np.zeros((wtm, wtn, wkb), dtype=np.int64)
        for pr, is_w, m, n, kb0, kb1 in recs:
            assert 0 <= pr < pairs and kb0 < kb1, tag
            if is_w:
                assert kb1 <= wkb, tag
                w_cov[m, n, kb0:kb1] += 1
            else:
                assert (kb0, kb1) == (0, dkb), tag
                d_seen[m, n] += 1
        assert (d_seen == 1).all(), tag
        assert (w_cov == 1).all(), tag
    assert declined < 100   # the drawn set mostly exercises the planner, not its refusal


def _check_partition(hdr, recs, pairs, tag):
    """Every dinp tile once over its whole K, every (dweight tile, k-block) exactly once."""
    import numpy as np
    dtm, dtn, dkb, wtm, wtn, wkb, _, rounds = hdr
    assert rounds <= 64, tag
    d_seen, w_cov = np.zeros((dtm, dtn), dtype=np.int64), np.zeros((wtm, wtn, wkb), dtype=np.int64)
    for pr, is_w, m, n, kb0, kb1 in recs:
        assert 0 <= pr < pairs and 0 <= kb0 < kb1, tag
        if is_w:
            assert kb1 <= wkb, tag
            w_cov[m, n, kb0:kb1] += 1
        else:
            assert (kb0, kb1) == (0, dkb), tag
            d_seen[m, n] += 1
    assert (d_seen == 1).all() and (w_cov == 1).all(), tag


def test_layer_backward_plan_of_fresh_and_launched_forms(L):
    """The partition in the forms that are launched: dinp tiles halved where they are, gradients from nothing or added to, units and
    the sums that they are made in. A plan whose dweight units are all a tile's whole K has one for each tile."""
    import numpy as np
    rng = np.random.default_rng(5)
    whole = cut = 0
    for case in range(160):
        BT = int(rng.integers(129, 30_000)) if case % 3 else int(rng.integers(129, 2100))
        C, OC = 8 * int(rng.integers(1, 400)), 8 * int(rng.integers(1, 700))
        pairs, gelu, fresh = int(rng.choice((74, 66, 33, 7))), bool(rng.integers(0, 2)), bool(rng.integers(0, 4))
        try:
            hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, pairs, gelu, launched=True, fresh=fresh)
        except binding.NbError as e:
            assert e.code == binding.NB_ERR_UNSUPPORTED
            continue
        tag = (BT, C, OC, pairs, gelu, fresh)
        _check_partition(hdr, recs, pairs, tag)
        _check_partition(hdr, binding.nb_debug_layer_bwd_plan(BT, C, OC, pairs, gelu, launched=True, fresh=fresh, sums=True)[1], pairs, tag)
        units = [k1 - k0 for _, is_w, _, _, k0, k1 in recs if is_w]
        if all(u == hdr[5] for u in units):
            assert len(units) == hdr[3] * hdr[4], tag
            whole += 1
        else:
            cut += 1
    assert whole > 20 and cut > 60, (whole, cut)


def test_layer_backward_plan_is_found_quickly(L):
    """A program whose row count changes from step to step pays for a plan on every call: 5 to 20 us, where
    a layer takes 15 or more on the GPU. (The limit leaves room for a slow or busy host.)"""
    import time
    out = (binding._int * (1 << 17))()
    for BT, C, OC, flags in [(4096, 768, 2304, 2), (4096, 3072, 768, 3), (16384, 768, 768, 2), (16384, 768, 2304, 6), (16384, 3072, 768, 3),
                             (16384, 1024, 1024, 2), (200000, 768, 768, 2), (171828, 456, 80, 6)]:
        best = 1.0
        for _ in range(20):
            t0 = time.perf_counter()
            assert L.nb_debug_layer_bwd_plan(BT, C, OC, 74, flags, out, len(out)) > 0
            best = min(best, time.perf_counter() - t0)
        assert best < 100e-6, (BT, C, OC, flags, best)


@pytest.mark.parametrize("fresh", [False, True])
@pytest.mark.parametrize("gelu", [False, True])
def test_sums_of_the_layer_backward_plan(L, gelu, fresh):
    """An accumulator loses accuracy with the length of its sum. No sum of dweight is longer than the chunks of the one-pass
    schedule are, about two units a pair of at least 32 k-blocks, and the sums are as good a partition as the units."""
    for BT, C, OC in [(4096, 768, 2304), (4096, 768, 3072), (4096, 3072, 768), (4096, 1024, 6144), (4096, 3072, 1024), (2021, 768, 3072),
                      (2021, 768, 50304), (8192, 768, 3072), (16384, 768, 768), (16384, 768, 3072), (1500, 1000, 1544), (65536, 768, 768),
                      (2826, 240, 2040), (9000, 136, 264)]:
        tiles, wkb = -(-OC // 256) * -(-C // 256), -(-BT // 64)
        chunks = min(-(-148 // tiles), max(1, wkb // 32))
        hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, 74, gelu, launched=True, fresh=fresh, sums=True)
        _check_partition(hdr, recs, 74, (BT, C, OC, gelu, fresh))
        assert max(kb1 - kb0 for _, is_w, _, _, kb0, kb1 in recs if is_w) <= -(-wkb // chunks), (BT, C, OC, gelu, fresh)


@pytest.mark.parametrize("fresh", [False, True])
@pytest.mark.parametrize("BT,C,OC", [(303169, 256, 512), (606272, 256, 256), (309000, 256, 512)])
def test_layer_backward_plan_where_no_chunk_count_gives_short_chunks(L, BT, C, OC, fresh):
    """Many rows of a narrow layer: the largest number of chunks rounds to fewer, and all smaller ones leave chunks
    longer than 64 k-blocks. Such a size is planned all the same."""
    hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, 74, False, launched=True, fresh=fresh)
    _check_partition(hdr, recs, 74, (BT, C, OC, fresh))


@pytest.mark.parametrize("fresh", [False, True])
@pytest.mark.parametrize("BT,C,OC", [(520, 4096, 151936), (712, 4096, 128256), (2312, 4096, 128256), (648, 8192, 65536),
                                     (136, 12288, 50304), (776, 3072, 256000)])
def test_layer_backward_plan_of_large_heads(L, BT, C, OC, fresh):
    """Heads whose weight gradient has far more tiles than 64 rounds of the pairs hold: what the tail dinp tiles leave
    room for is dealt in rounds, the rest is the line."""
    hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, 74, False, launched=True, fresh=fresh)
    _check_partition(hdr, recs, 74, (BT, C, OC, fresh))
    assert binding.nb_debug_route(binding.CALL_BACKWARD, BT, C, OC, accumulate=not fresh)[0][0] == "layer_bwd"


def test_layer_backward_plan_with_halved_dinp_tiles(L):
    """A few dinp tiles over a long K are 128 columns wide in the launch's own plan: they
    partition the work like whole ones. At most a quarter of the pairs as whole tiles, at least 36 and 12 + two a tile of
    k-blocks, and one tile longer than a pair's share; never with the GELU derivative."""
    import numpy as np
    rng = np.random.default_rng(7)
    cases = [(1500, 760, 3080, 74), (1030, 760, 6152, 74), (1500, 768, 3072, 74), (1024, 1024, 6144, 74), (512, 768, 50304, 74),
             (300, 8, 2304, 66), (257, 136, 4104, 33)]
    while len(cases) < 60:
        cases.append((int(rng.integers(129, 1600)), 8 * int(rng.integers(1, 160)), 8 * int(rng.integers(288, 1500)),
                      int(rng.choice((74, 66, 33)))))
    halved = 0
    for BT, C, OC, pairs in cases:
        tiles, dkb, wkb = -(-BT // 256) * -(-C // 256), -(-OC // 64), -(-BT // 64)
        wt = -(-OC // 256) * -(-C // 256)
        narrow = tiles * 4 <= pairs and dkb >= 36 and dkb >= 12 + 2 * tiles and dkb * pairs > tiles * dkb + wt * wkb
        for gelu in (False, True):
            hdr, recs = binding.nb_debug_layer_bwd_plan(BT, C, OC, pairs, gelu, launched=True)
            width = 128 if narrow and not gelu else 256
            tag = (BT, C, OC, pairs, gelu)
            assert hdr[:6] == (-(-BT // 256), -(-C // width), dkb, -(-OC // 256), -(-C // 256), wkb), tag
            d = sorted((m, n, kb0, kb1) for _, is_w, m, n, kb0, kb1 in recs if not is_w)
            assert d == [(m, n, 0, dkb) for m in range(hdr[0]) for n in range(hdr[1])], tag
            cov = np.zeros((hdr[3], hdr[4], wkb), dtype=np.int64)
            for _, is_w, m, n, kb0, kb1 in recs:
                if is_w:
                    cov[m, n, kb0:kb1] += 1
            assert (cov == 1).all(), tag
        halved += narrow
    assert halved >= 20
    assert all(t in cases for t in ((1500, 760, 3080, 74), (1030, 760, 6152, 74)))  # also on the GPU: test_gpu_small_problems


def test_route_view(L):
    """The view of the kernels that calls take: what it refuses, and the promise on dinp: the number of CTAs that
    share its K, which fixes the order of its sums, does not depend on what else the call is asked for."""
    import numpy as np
    assert L.nb_debug_route(9, 8, 8, 8, 0, 0, 7, 148, (binding.ctypes.c_int * 12)()) == -binding.NB_ERR_INVALID_ARG
    assert L.nb_debug_route(0, 0, 8, 8, 0, 0, 7, 148, (binding.ctypes.c_int * 12)()) == -binding.NB_ERR_INVALID_ARG
    with pytest.raises(binding.NbError):
        binding.nb_debug_route(binding.CALL_LORA_FORWARD, 8, 8, 8, r=12)
    assert binding.nb_debug_route(binding.CALL_FORWARD, 8, 768, 3072) == [("rows", 16, 1, 2)]
    assert binding.nb_debug_route(binding.CALL_FORWARD, 16384, 768, 3072) == [("gemm", 256, 1, 1)]
    assert binding.nb_debug_route(binding.CALL_BACKWARD, 16384, 768, 3072) == [("layer_bwd", 256, 1, 1)]
    assert [k[0] for k in binding.nb_debug_route(binding.CALL_LORA_BACKWARD, 16384, 1024, 2048, r=16)] == ["lora_udb", "gemm"]
    rng = np.random.default_rng(3)
    shared = 0
    for _ in range(1500):
        BT = int(2 ** rng.uniform(0, 11.2))
        C, OC = (8 * int(2 ** rng.uniform(0, 9)) for _ in range(2))
        (alone,) = binding.nb_debug_route(binding.CALL_BACKWARD, BT, C, OC, dweight=False, dbias=False)
        shared += alone[2] > 1
        assert alone[0] in ("tile", "gemm") and alone[2] in (1, 2, 4)
        for gelu in (False, True):
            for dbias in (False, True):
                for accumulate in (False, True):
                    route = binding.nb_debug_route(binding.CALL_BACKWARD, BT, C, OC, dbias=dbias, gelu_grad=gelu,
                                                   accumulate=accumulate)
                    assert route[0][0] in ("tile_pair", "layer_bwd", "tile", "gemm")
                    assert route[0][2] == alone[2], (BT, C, OC, route, alone)
    assert shared > 200


def test_backward_forms_that_count_on_two_ctas_fit_them(L):
    """Where the tile kernel of a backward is planned with two CTAs on an SM, two have to fit: 228 KB of shared
    memory of which each CTA reserves one, counted here from the tiles alone (A of 128 rows of 64 bf16, or only the rows
    there are; B of 64 x width; at least two stages where a CTA has more than one k-block; with K shared, one row more than a tile of fp32
    slices received; results staged in the stages), and registers: the form with gelu' in 128-wide tiles has too many."""
    import numpy as np
    rng = np.random.default_rng(4)

    def kb(rows, mn_major, width, kblocks, shared, staged):
        a = 128 if mn_major or rows >= 128 else -(-rows // 8) * 8
        stages = max(min(2, kblocks), 1 if shared > 1 else -(-staged // (128 * (a + width))))
        return (stages * 128 * (a + width) + (129 * width * 4 if shared > 1 else 0)) / 1024

    two = 0
    for _ in range(6000):
        BT = int(2 ** rng.uniform(0, 10.5))
        C, OC = (8 * int(2 ** rng.uniform(3, 10)) for _ in range(2))
        gelu = bool(rng.integers(0, 2))
        for kernel, width, shared, per_sm in binding.nb_debug_route(binding.CALL_BACKWARD, BT, C, OC, gelu_grad=gelu):
            if kernel != "tile_pair" or per_sm != 2:
                continue
            two += 1
            tag = (BT, C, OC, gelu, width, shared)
            assert not (width == 128 and gelu), tag
            longest = -(-(-(-OC // 64)) // shared)
            quarters = -(-min(BT, 128) // 32)
            dinp = kb(BT, False, width, longest, shared, quarters * 32 * width * 2)
            dweight = kb(OC, True, width, -(-BT // 64), 1, 128 * width * 4)
            assert max(dinp, dweight) + 1 <= 114, tag
    assert two > 500
