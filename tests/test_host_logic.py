"""Host logic of the library (no GPU): ABI exports, workloads, classes, legaliser/validator, selector."""
import ctypes
import itertools
import os
import re

import numpy as np
import pytest

from oracle import oracle as orc
from paper_2201_05587_b200 import binding as B
from paper_2201_05587_b200 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GOLDEN = os.path.join(ROOT, "tests", "golden")


def test_library_exports_every_declared_symbol():
    text = open(os.path.join(ROOT, "include", "tt.h")).read()
    declared = set(re.findall(r"\b(tt_[a-z_]+)\s*\(", text))
    declared -= {"tt_op", "tt_act"}
    assert declared, "no declarations found"
    lib = B.lib()
    for name in sorted(declared):
        assert hasattr(lib, name), f"{name} declared in tt.h but not exported"
        assert name in B.EXPORTS, f"{name} has no binding"
    assert set(B.EXPORTS) <= declared


def test_struct_sizes_match_header_layout():
    assert ctypes.sizeof(B.tt_shapes) == 20 * 4
    assert ctypes.sizeof(B.tt_schedule_record) == 3 * 4 + 80 + 21 * 4
    assert B.status_string(B.TT_ERR_INVALID_SCHEDULE) != B.status_string(B.TT_OK)


def test_split_check_matches_paper_examples_and_oracle():
    with open(os.path.join(GOLDEN, "split_validity.txt")) as f:
        for line in f:
            line = line.strip()
            if not line or line.startswith("#"):
                continue
            extent, form, factors, valid = line.split()
            extent, valid = int(extent), bool(int(valid))
            fs = [int(v) for v in factors.split(",")]
            if form == "fixed":
                assert B.split_check(extent, fs) == valid == orc.split_covers(extent, fs), line
            elif form == "reform":
                assert B.split_check(extent, fs, reformulate=True) == valid, line
    for n in (1, 7, 8, 24, 49, 196, 1000, 4096):
        for f in (1, 2, 3, 8, 16):
            assert B.split_check(n, [f], True) == orc.split_reformulated_valid(n, f)
            assert B.split_check(n, [n // f if n % f == 0 else 1, f]) == orc.split_covers(n, [n // f if n % f == 0 else 1, f])


def test_select_matches_oracle_on_hand_tables():
    t = [5.0, 3.0, -1.0, 3.0, -1.0, -1.0, -1.0, -1.0, 2.0, -1.0, 1.5, 9.0, float("nan"), 4.0, 4.0, -1.0]
    assert B.select(t, 4, 4) == orc.select(t, 4, 4) == [1, -1, 2, 1]
    lat = B.model_latency(t, 4, 4, [1, -1, 2, 1], [2, 5, 3, 1])
    assert lat == pytest.approx(orc.model_latency([2, 5, 3, 1], [0 if v != v else v for v in t], [1, -1, 2, 1], 4))
    # deterministic: same table, same answer
    assert all(B.select(t, 4, 4) == [1, -1, 2, 1] for _ in range(5))


def test_resnet18_inventory_matches_table1():
    rows = []
    with open(os.path.join(GOLDEN, "resnet18_table1.txt")) as f:
        for line in f:
            if line.strip() and not line.startswith("#"):
                i, cls, ic, ihw, oc, ohw, use = line.split()
                rows.append((cls, int(ic), int(ihw), int(oc), int(ohw), int(use)))
    specs = W.resnet18()
    assert len(specs) == 16                               # A 3, E 8, F 4, D 1
    want = {(cls, ic, ihw, oc, ohw): use for cls, ic, ihw, oc, ohw, use in rows}
    got = {}
    for sp in specs:
        s = sp.shapes
        if sp.op == B.TT_OP_DENSE:
            got[("D", s.kk, 1, s.nn, 1)] = sp.use_count
        else:
            p = (s.h + 2 * s.pad_h - s.r) // s.stride_h + 1
            kind = "A" if (s.r == 1 and s.act == B.TT_ACT_NONE) else ("F" if s.has_residual else "E")
            got[(kind, s.c, s.h, s.k, p)] = sp.use_count
    assert got == want
    assert sum(sp.use_count for sp in specs) == 21          # 20 convolutions + 1 dense
    # the residual variants are kernels of their own class and workload ID, although they share their sibling's sizes
    e = [sp for sp in specs if sp.shapes.c == 64 and sp.shapes.k == 64 and sp.shapes.r == 3]
    assert len(e) == 2 and e[0].workload().kernel_class() != e[1].workload().kernel_class()
    assert e[0].workload().key() != e[1].workload().key()


def test_chains_are_consistent_with_their_inventories():
    """A model is written once as wired layers; the inventory is derived from it.  Every wire connects buffers of the
    same element count, every skip tensor has the consumer's output shape, and the use counts are the layer counts."""
    for name, make in W.CHAINS.items():
        specs, steps = make()
        assert [sp.use_count for sp in specs] == [sum(1 for st in steps if st.kernel == i) for i in range(len(specs))], name
        for i, st in enumerate(steps):
            if st.spec is None:
                assert st.shape and st.note, (name, i)
                continue
            xs, ws, bs, rs, ys = W.tensor_shapes(st.spec)
            assert bytes(specs[st.kernel].shapes) == bytes(st.spec.shapes)
            assert 0 <= st.x < i and np.prod(steps[st.x].out_shape()) == np.prod(xs), (name, i)
            if st.w_from is not None:
                assert 0 <= st.w_from < i and np.prod(steps[st.w_from].out_shape()) == np.prod(ws), (name, i)
            assert (st.res is not None) == bool(st.spec.shapes.has_residual), (name, i)
            if st.res is not None:
                assert 0 <= st.res < i and steps[st.res].out_shape() == tuple(ys), (name, i)
    # the ResNet-18-shaped chain: a block's second convolution adds the block's input, or its 1x1 downsample
    specs, steps = W.resnet18_net()
    f = [st for st in steps if st.spec is not None and st.spec.shapes.has_residual]
    assert len(f) == 8 and sum(1 for st in f if steps[st.res].spec is not None and steps[st.res].spec.shapes.r == 1) == 3


def test_unique_kernel_counts_of_table2():
    """Table 2: ResNet50 A4 E16 G4 D1; VGG-16 E9 (+ 3 dense shapes); MobileNetV2 A7+K5 J8 L10 D1; BERT Q3 R2."""
    r50 = W.resnet50()
    convs = [s for s in r50 if s.op == B.TT_OP_CONV2D]
    down = [s for s in convs if s.shapes.act == B.TT_ACT_NONE]
    g = [s for s in convs if s.shapes.has_residual]
    assert len(down) == 4 and len(g) == 4 and len(convs) - len(down) - len(g) == 16 and len(r50) == 25    # A, G, E
    vgg = W.vgg16()
    assert len([s for s in vgg if s.op == B.TT_OP_CONV2D]) == 9 and len(vgg) == 12
    mb = W.mobilenet_v2()
    dw = [s for s in mb if s.op == B.TT_OP_DWCONV2D]
    proj = [s for s in mb if s.op == B.TT_OP_CONV2D and s.shapes.act == B.TT_ACT_NONE]
    relu6 = [s for s in mb if s.op == B.TT_OP_CONV2D and s.shapes.act == B.TT_ACT_RELU6]
    assert (len(dw), len(proj), len(relu6)) == (10, 12, 8)
    assert len([s for s in proj if s.shapes.has_residual]) == 5                 # class K; the other 7 are class A
    bert = W.bert_base()
    assert len([s for s in bert if s.op == B.TT_OP_DENSE]) == 3
    assert len([s for s in bert if s.op == B.TT_OP_BATCH_MATMUL]) == 2


def test_workload_key_and_class():
    a = W._conv(64, 56, 64, 3, 1, 1).workload()
    b = W._conv(64, 56, 64, 3, 1, 1).workload()
    c = W._conv(128, 28, 128, 3, 1, 1).workload()
    d = W._conv(64, 56, 128, 1, 2, 0, act=B.TT_ACT_NONE).workload()
    e = W._dense(1, 512, 1000).workload()
    assert a.key() == b.key() != c.key()
    assert a.kernel_class() == c.kernel_class()          # same operators, other sizes: same class
    assert a.kernel_class() != d.kernel_class()          # conv2d_add is another class than conv2d_bias_relu
    assert a.kernel_class() != e.kernel_class()
    assert a.family() == e.family() == B.TT_FAMILY_GEMM_TC
    v = a.gemm_view()
    assert (v.batch, v.gm, v.gn, v.gk) == (1, 64, 3136, 576)
    assert v.flops == pytest.approx(2 * 64 * 3136 * 576)


def test_workload_create_rejects_bad_shapes():
    for bad in (B.conv2d_shapes(1, 0, 8, 8, 4, 3, 3), B.conv2d_shapes(1, 4, 2, 2, 4, 5, 5), B.conv2d_shapes(1, 4, 8, 8, 4, 3, 3, 0)):
        h = ctypes.c_void_p()
        assert B.lib().tt_workload_create(B.TT_OP_CONV2D, ctypes.byref(bad), ctypes.byref(h)) == B.TT_ERR_INVALID_ARG
    h = ctypes.c_void_p()
    assert B.lib().tt_workload_create(99, ctypes.byref(B.dense_shapes(1, 2, 3)), ctypes.byref(h)) == B.TT_ERR_INVALID_ARG


def test_cross_family_and_cross_class_records_are_invalid():
    conv = W._conv(64, 56, 64, 3, 1, 1).workload()
    dw = W._dw(32, 112, 1).workload()
    dense = W._dense(1, 512, 1000).workload()
    st, _ = dw.check(conv.default_schedule())
    assert st == B.TT_ERR_CLASS_MISMATCH
    st, _ = conv.check(dw.default_schedule())
    assert st == B.TT_ERR_CLASS_MISMATCH
    # the paper's rule: a conv schedule on a dense kernel is always invalid
    rec = conv.default_schedule()
    st, _ = dense.check(rec, strict_class=True)
    assert st == B.TT_ERR_CLASS_MISMATCH
    # with family matching (the stated extension) the same record applies
    st, _ = dense.check(rec, strict_class=False)
    assert st == B.TT_OK
    # same class, other sizes: valid in both
    other = W._conv(256, 14, 256, 3, 1, 1).workload()
    assert other.check(rec, strict_class=True)[0] == B.TT_OK


def test_legaliser_clamps_and_strict_mode_rejects():
    wl = W.single_conv()[0].workload()         # GEMM view 32 x 196 x 144
    for rec in W.single_conv_pool():
        st, info = wl.check(rec)
        assert st == B.TT_OK
        L = info.legal
        assert L.tile_m == 128 and L.tile_n % 16 == 0 and L.tile_k in (8, 16)
        assert info.changed & B.TT_CHG_TILE_M
    big = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=64, stages=2, split_k=64, mma_m_axis=1)
    st, info = wl.check(big)
    assert st == B.TT_OK
    assert info.legal.tile_n == 208 and info.legal.split_k == 3 and info.changed & B.TT_CHG_SPLIT_K
    # strict: a factor larger than the loop, or more splits than reduction tiles, is invalid code
    assert wl.check(big, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    ok = B.make_record(B.TT_FAMILY_GEMM_TC, tile_m=32, tile_n=64, tile_k=16, stages=2, split_k=3, mma_m_axis=1)
    assert wl.check(ok, mode=B.TT_MODE_STRICT)[0] == B.TT_OK
    # resources: 8 stages of 128x256x128 do not fit shared memory
    fat = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=128, stages=8, mma_m_axis=1)
    huge = W._dense(512, 4096, 4096).workload()
    # reformulated: the pipeline is made shallower until it fits (one 192 KB stage); kept as written it is invalid
    st, info = huge.check(fat)
    assert st == B.TT_OK and info.legal.stages == 1 and info.changed & B.TT_CHG_STAGES
    st, info = huge.check(fat, mode=B.TT_MODE_STRICT)
    assert st == B.TT_ERR_RESOURCE and info.smem_bytes > 227 * 1024
    # a 128-pixel x 128-channel tile of a strided 1x1 convolution: its input slab alone exceeds shared memory at any depth
    wide = W._conv(256, 56, 512, 1, 2, 0).workload()
    st, info = wide.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=32, tile_k=128, stages=2, mma_m_axis=2))
    assert st == B.TT_ERR_RESOURCE and info.smem_bytes > 227 * 1024
    # the slab is part of the record: a request for more reduction tiles per staging than fit is lowered
    conv = W._conv(512, 28, 512, 3, 1, 1).workload()
    st, info = conv.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=128, tile_k=32, stages=3, slab_tiles=64, mma_m_axis=1))
    assert st == B.TT_OK and 1 <= info.legal.slab_tiles < 64 and info.changed & B.TT_CHG_SLAB
    # nonsense fields
    for kw in (dict(tile_n=0), dict(stages=0), dict(split_k=-1), dict(raster=5), dict(mma_m_axis=7)):
        assert wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, **kw))[0] == B.TT_ERR_INVALID_SCHEDULE
    bad = B.make_record(B.TT_FAMILY_GEMM_TC)
    bad.version = 77
    assert wl.check(bad)[0] == B.TT_ERR_INVALID_SCHEDULE


def test_gemm_records_transfer_between_512_and_1024():
    """The GEMM example of Section 4.1: records of the 512^3 and 1024^3 kernels apply to each other unchanged."""
    a, b = W._dense(512, 512, 512).workload(), W._dense(1024, 1024, 1024).workload()
    ra = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=128, tile_k=32, stages=4, split_k=2, mma_m_axis=1)
    rb = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=64, stages=2, split_k=1, raster=1, mma_m_axis=1)
    for wl in (a, b):
        for r in (ra, rb):
            st, info = wl.check(r, mode=B.TT_MODE_STRICT)
            assert st == B.TT_OK and info.changed == 0


def test_simt_legalisers():
    dw = W._dw(96, 7, 1).workload()
    r = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=2048, block_y=16, block_x=64, items_per_thread=4, vec_width=4, threads=256)
    st, info = dw.check(r)
    assert st == B.TT_OK
    L = info.legal
    assert L.tile_m == 96 and L.block_y == 7 and L.vec_width == 1 and L.block_x % L.items_per_thread == 0
    assert dw.check(r, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    sm = [s for s in W.bert_base() if s.op == B.TT_OP_SOFTMAX][0].workload()
    st, info = sm.check(B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=24, block_y=3, vec_width=4))
    assert st == B.TT_OK and info.legal.block_x == 16 and info.threads % 32 == 0 and info.legal.vec_width == 4


def test_device_calls_fail_loudly_without_gpu():
    import torch
    if torch.cuda.is_available():
        pytest.skip("GPU present")
    wl = W._dense(8, 16, 8).workload()
    st, _ = wl.try_apply(wl.default_schedule())
    assert st == B.TT_ERR_CUDA                      # no CPU fallback
    t = B.tt_tensors()
    assert B.lib().tt_run(wl.handle, ctypes.byref(t), None) == B.TT_ERR_NOT_APPLIED


def test_rank_pools_matches_the_oracle_on_the_papers_tables():
    """tt_rank_pools (Equation 1) against the oracle on Table 2, target by target, and its argument checks."""
    import test_oracle_pins as pins
    feats, choices = pins._load_tables()
    classes = sorted({c for f in feats.values() for c in f})
    for target in feats:
        cands = [m for m in feats if m != target]
        share_d = {c: pct / 100.0 for c, (_, pct) in feats[target].items()}
        counts_d = [{c: n for c, (n, _) in feats[m].items()} for m in cands]
        want_scores, want_order = orc.rank_pools(share_d, counts_d)
        share = [share_d.get(c, 0.0) for c in classes]
        counts = [[cd.get(c, 0) for c in classes] for cd in counts_d]
        scores, order = B.rank_pools(share, counts)
        assert order == want_order
        assert scores == pytest.approx(want_scores, rel=1e-12, abs=1e-15)
        assert [cands[i] for i in order[:len(choices[target])]] == choices[target]
    with pytest.raises(B.TTError):
        B.rank_pools([0.5], [[-1]])


def test_tap_major_reduction_order_is_legalised_per_kernel():
    """k_order = 1 exists for stride-1 convolutions whose image rows are 16-byte multiples; elsewhere the record is
    reformulated to the stored order (legalise) or invalid (strict)."""
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=128, tile_k=32, stages=3, k_order=1, mma_m_axis=1)
    st, info = W._conv(64, 28, 64, 3, 1, 1).workload().check(rec)
    assert st == B.TT_OK and info.legal.k_order == 1 and info.launches == 2
    assert info.workspace_bytes == 64 * 2 * 9 * 32 * 4        # re-packed filters: 2 blocks of 32 channels x 9 taps
    assert info.grid_x == (28 * 32 + 127) // 128              # padded-linear pixels: 28 rows of 28 + 4
    for sp in (W._conv(64, 56, 128, 3, 2, 1), W._conv(64, 14, 64, 3, 1, 1), W._dense(128, 768, 768)):
        wl = sp.workload()
        st, info = wl.check(rec)
        assert st == B.TT_OK and info.legal.k_order == 0 and info.changed & B.TT_CHG_KORDER and info.launches == 1
        assert wl.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    # the mode fixes tile_k, split_k and the row axis; other values are reformulated
    odd = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=100, tile_k=64, stages=9, split_k=4, k_order=1, mma_m_axis=2)
    st, info = W._conv(64, 28, 64, 3, 1, 1).workload().check(odd)
    L = info.legal
    assert st == B.TT_OK and (L.tile_n, L.tile_k, L.split_k, L.mma_m_axis, L.k_order) == (112, 32, 1, 1, 1) and L.stages <= 8


# ---- refinement of a transferred record: neighbourhood and greedy descent against the oracle's definitions ----
_FAMILY_NAME = {B.TT_FAMILY_GEMM_TC: "gemm_tc", B.TT_FAMILY_DW_SIMT: "dw_simt", B.TT_FAMILY_ROW_SIMT: "row_simt"}


def _rec_key(r):
    return tuple(int(getattr(r, f)) for f in B.tt_schedule_record.FIELDS)


def _legal_neighbours_by_definition(wl, rec):
    """The oracle's raw one-step variations, mapped onto this workload by the validity layer (tt_schedule_check):
    invalid ones, ones that coincide with the legalised start and repeats are dropped, order kept."""
    st, info = wl.check(rec)
    assert st == B.TT_OK
    start = info.legal
    fam = _FAMILY_NAME[int(start.family)]
    out, seen = [], {_rec_key(start)}
    for d in orc.raw_neighbours({f: int(getattr(start, f)) for f in B.tt_schedule_record.FIELDS}, fam):
        r = B.make_record(int(start.family), **d)
        st, info = wl.check(r)
        if st != B.TT_OK or _rec_key(info.legal) in seen:
            continue
        seen.add(_rec_key(info.legal))
        out.append(info.legal)
    return out


def _refine_cases():
    r18 = W.resnet18()
    mb = [s for s in W.mobilenet_v2() if s.op == B.TT_OP_DWCONV2D]
    bert = W.bert_base()
    cases = [(r18[1], B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=32, stages=3, mma_m_axis=1)),
             (r18[1], B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=64, stages=4, split_k=8, mma_m_axis=2, k_order=1)),
             (r18[-1], B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=16, tile_k=8, stages=1, split_k=3, mma_m_axis=1)),
             (mb[0], B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=8, block_x=32, items_per_thread=4, vec_width=4, threads=128, unroll=2)),
             (mb[-1], B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=32, block_y=56, block_x=112, items_per_thread=8, vec_width=4, threads=512, unroll=4,
                                    raster=1, stages=4)),
             ([s for s in bert if s.op == B.TT_OP_SOFTMAX][0], B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=8, block_y=4, vec_width=2))]
    return cases


def test_record_neighbours_are_the_legalised_one_step_variations():
    for spec, rec in _refine_cases():
        wl = spec.workload()
        got = wl.neighbours(rec)
        want = _legal_neighbours_by_definition(wl, rec)
        assert [_rec_key(r) for r in got] == [_rec_key(r) for r in want], spec.name
        assert 0 < len(got) <= 18
        _, info = wl.check(rec)
        for r in got:                                    # each differs from the start, and is legal as written
            assert _rec_key(r) != _rec_key(info.legal)
            st, i2 = wl.check(r)
            assert st == B.TT_OK and _rec_key(i2.legal) == _rec_key(r)
        wl.close()


def test_refine_with_follows_the_oracles_descent_on_synthetic_times():
    import math
    for spec, rec in _refine_cases():
        wl = spec.workload()
        # a deterministic, bumpy "time" per record: separable bowls plus a hash term, some records unable to run
        def cost(key):
            h = (hash(key) % 1000) / 1000.0
            if int(h * 1000) % 7 == 0:
                return -1.0
            return float(np.float32(50.0 + sum(abs(math.log2(v + 1) - 3.0) * (i % 3 + 1) for i, v in enumerate(key)) + 3.0 * h))
        _, info = wl.check(rec)
        start_key = _rec_key(info.legal)
        if cost(start_key) < 0:
            wl.close()
            continue
        by_key = {}
        def nb(key):
            r = by_key.get(key) or info.legal
            out = _legal_neighbours_by_definition(wl, r)
            for x in out:
                by_key[_rec_key(x)] = x
            return [_rec_key(x) for x in out]
        by_key[start_key] = info.legal
        for rounds, gain in ((0, 0.0), (1, 0.0), (6, 0.0), (6, 0.03)):
            want = orc.refine(start_key, nb, cost, rounds, gain)
            best, best_us, start_us, timed = wl.refine_with(rec, lambda r: cost(_rec_key(r)), rounds, gain)
            assert _rec_key(best) == want[0], (spec.name, rounds, gain)
            assert best_us == pytest.approx(want[1]) and start_us == pytest.approx(want[2]) and timed == want[3]
        wl.close()


def test_refine_rejects_bad_arguments_and_needs_a_device_for_device_times():
    spec, rec = _refine_cases()[0]
    wl = spec.workload()
    other = B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=8, block_y=4, vec_width=2)
    with pytest.raises(B.TTError):
        wl.neighbours(other)                             # a record of another family
    with pytest.raises(B.TTError):
        wl.refine_with(rec, lambda r: -1.0, 3, 0.0)      # the start itself cannot run
    with pytest.raises(B.TTError):
        wl.refine_with(rec, lambda r: 1.0, -1, 0.0)
    import torch
    if not torch.cuda.is_available():
        t, best, us = B.tt_tensors(), B.tt_schedule_record(), ctypes.c_float()
        assert B.lib().tt_refine(wl.handle, ctypes.byref(t), None, None, ctypes.byref(rec), 2, 0.0, ctypes.byref(best),
                                 ctypes.byref(us), None, None) == B.TT_ERR_CUDA      # no CPU fallback
    wl.close()


def test_depthwise_tma_records_are_legalised_by_shape():
    """raster = 1 names the TMA-staged persistent depthwise kernel: kept where image rows are 16-byte multiples and the
    filter is one the window kernels cover, with 2..4 staging buffers that fit shared memory; legalised away elsewhere
    (strict mode: invalid)."""
    rec = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=8, block_y=14, block_x=56, items_per_thread=4, vec_width=4, threads=256,
                        unroll=2, raster=1, stages=3)
    ok = W._dw(144, 56, 1).workload()                     # 56-pixel rows: 224 bytes
    st, info = ok.check(rec)
    assert st == B.TT_OK and info.legal.raster == 1 and info.legal.stages == 3 and info.grid_y == 1
    assert 0 < info.smem_bytes <= 227 * 1024 and info.grid_x <= 148 * 8
    assert ok.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_OK
    deep = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=8, block_y=14, block_x=56, items_per_thread=4, vec_width=4, threads=256,
                         unroll=2, raster=1, stages=9)
    st, info = ok.check(deep)
    assert st == B.TT_OK and info.legal.raster == 1 and info.legal.stages == 4 and info.changed & B.TT_CHG_STAGES
    assert ok.check(deep, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    odd = W._dw(96, 14, 1).workload()                     # 14-pixel rows: 56 bytes, no aligned TMA rows
    st, info = odd.check(rec)
    assert st == B.TT_OK and info.legal.raster == 0 and info.changed & B.TT_CHG_BLOCK
    assert odd.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    staged = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=8, block_y=8, block_x=32, items_per_thread=4, vec_width=4, threads=256,
                           unroll=0, raster=1, stages=2)  # unroll 0 asks for the staged kernel: no TMA form of it
    st, info = ok.check(staged)
    assert st == B.TT_OK and info.legal.raster == 0
    bad = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=8, block_y=8, block_x=32, items_per_thread=4, vec_width=4, threads=256,
                        unroll=2, raster=2, stages=2)
    assert ok.check(bad)[0] == B.TT_ERR_INVALID_SCHEDULE
    for w in (ok, odd):
        w.close()


def test_pointwise_convolutions_take_the_whole_row_view():
    """A 1x1, stride-1, unpadded convolution is legalised on rows that tile the CTA's pixels exactly: less shared
    memory than the same record needs on a 3x3 layer's slab geometry would suggest, and never more than the image-row
    view of a layer whose pixel count has no suitable divisor."""
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=32, stages=2, mma_m_axis=2, slab_tiles=1)
    pw = W._conv(256, 56, 64, 1, 1, 0).workload()         # 3136 pixels = 49 rows of 64
    st, info = pw.check(rec)
    assert st == B.TT_OK and info.smem_bytes <= 90 * 1024
    strided = W._conv(256, 56, 64, 1, 2, 0).workload()    # stride 2: the image's own rows
    st2, info2 = strided.check(rec)
    assert st2 == B.TT_OK
    v = pw.gemm_view()
    assert (v.gm, v.gn, v.gk) == (64, 3136, 256)          # the view changes nothing the caller sees
    for w in (pw, strided):
        w.close()


def test_depthwise_record_naming_a_kernel_form_the_shape_lacks_is_a_reformulation():
    """A register-window (unroll >= 1) or TMA-staged (raster = 1) depthwise record on a filter that has no such kernel
    runs the staged kernel instead: legalise mode says so in `changed`, strict mode rejects the record (a primitive
    that does not fit the loop nest is invalid code, Sections 4.1 and 4.2)."""
    dw7 = B.Workload(B.TT_OP_DWCONV2D, B.make_shapes(n=1, c=8, h=20, w=20, k=8, r=7, s=7, stride_h=1, stride_w=1, pad_h=3,
                                                     pad_w=3, has_bias=1, act=B.TT_ACT_RELU), "dw7x7")
    dw3s3 = B.Workload(B.TT_OP_DWCONV2D, B.make_shapes(n=1, c=8, h=20, w=20, k=8, r=3, s=3, stride_h=3, stride_w=3, pad_h=1,
                                                       pad_w=1, has_bias=1, act=B.TT_ACT_RELU), "dw3x3s3")
    dw3 = B.Workload(B.TT_OP_DWCONV2D, B.make_shapes(n=1, c=8, h=20, w=20, k=8, r=3, s=3, stride_h=1, stride_w=1, pad_h=1,
                                                     pad_w=1, has_bias=1, act=B.TT_ACT_RELU), "dw3x3")
    win = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=4, block_x=20, items_per_thread=4, vec_width=4, threads=128, unroll=2)
    for wl in (dw7, dw3s3):
        st, info = wl.check(win)
        assert st == B.TT_OK and info.legal.unroll == 0 and info.changed & B.TT_CHG_FORM
        assert wl.check(win, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    st, info = dw3.check(win)
    assert st == B.TT_OK and info.legal.unroll == 2 and not info.changed & B.TT_CHG_FORM
    assert dw3.check(win, mode=B.TT_MODE_STRICT)[0] == B.TT_OK
    three = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=4, block_x=20, items_per_thread=4, vec_width=4, threads=128, unroll=3)
    st, info = dw3.check(three)
    assert st == B.TT_OK and info.legal.unroll == 2 and info.changed & B.TT_CHG_FORM
    assert dw3.check(three, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    tma = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=4, block_x=20, items_per_thread=4, vec_width=4, threads=256,
                        unroll=2, raster=1, stages=2)
    st, info = dw7.check(tma)
    assert st == B.TT_OK and info.legal.raster == 0 and info.changed & B.TT_CHG_FORM
    assert dw3.check(tma)[1].legal.raster == 1


def test_pool_file_round_trip_and_rejections(tmp_path):
    """Schedules persist as records keyed by the kernel they were tuned on (Section 2): a pool written as text reads
    back bit for bit; a damaged line, an unknown field or another record version is refused, not guessed at."""
    recs = W.single_conv_pool()
    recs[2].origin.scale = 0.125
    recs.append(B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=8, block_y=14, block_x=28, items_per_thread=4, vec_width=4, threads=256,
                              unroll=2, raster=1, stages=2))
    path = str(tmp_path / "pool.txt")
    B.pool_save(path, recs, [1.5, 2.25, -1.0, 7.0, 40.5])
    back, us = B.pool_load(path)
    assert us == [1.5, 2.25, -1.0, 7.0, 40.5]
    assert [bytes(r) for r in back] == [bytes(r) for r in recs]
    B.pool_save(path, [], None)
    assert B.pool_load(path) == ([], [])
    good = open(str(tmp_path / "pool.txt")).read()
    B.pool_save(path, recs[:1], None)
    line = [l for l in open(path).read().splitlines() if not l.startswith("#")][0]
    assert "us=-1" in line
    for bad in (line.replace("tile_n=", "tile_q="), line.replace("version=3", "version=99"), line.replace("stages=2", "stages=two"),
                line.replace("origin=1,", "origin=1;")):
        with open(path, "w") as f:
            f.write(bad + "\n")
        n = ctypes.c_size_t()
        assert B.lib().tt_pool_load(path.encode(), None, None, 0, ctypes.byref(n)) == B.TT_ERR_INVALID_ARG, bad
    n = ctypes.c_size_t()
    assert B.lib().tt_pool_load(str(tmp_path / "missing.txt").encode(), None, None, 0, ctypes.byref(n)) == B.TT_ERR_INVALID_ARG
    del good


def test_bench_counts_algorithmic_work_like_the_library():
    """bench.py's reference arm counts flops and bytes from the shapes alone; they are the library's gemm view."""
    import bench
    for model in ("resnet18", "mobilenet_v2", "bert_base"):
        for sp in W.MODELS[model]():
            v = sp.workload().gemm_view()
            f, b = bench.algorithmic_work(sp)
            assert f == pytest.approx(v.flops) and b == pytest.approx(v.bytes), sp.name


def test_pool_subsample_matches_the_oracle():
    for n, c, seed in ((1, 1, 0), (10, 4, 7), (56, 14, 2024), (111, 111, 5), (50, 0, 9)):
        assert B.pool_subsample(n, c, seed) == orc.pool_subsample(n, c, seed)
    out = (ctypes.c_int32 * 4)()
    assert B.lib().tt_pool_subsample(3, 4, 0, out) == B.TT_ERR_INVALID_ARG


@pytest.mark.parametrize("model", ["resnet18", "resnet50", "mobilenet_v2", "bert_base"])
def test_chain_lanes_order_every_dependency(model):
    """The side-by-side plan of a chain: every producer of a layer (input, skip tensor, second operand, and the layer a
    stand-in tensor replaces) either ran earlier on the layer's own lane or is waited for; kernels declared serial
    never overlap with themselves; the attention projections and the downsample convolutions do leave lane 0."""
    specs, steps = W.CHAINS[model]()
    serial = {0}
    plan = W.chain_lanes(steps, max_lanes=4, serial_kernels=serial)
    assert len(plan) == len(steps)
    seen_on_lane = {}
    last_serial = {}
    for i, (st, pl) in enumerate(zip(steps, plan)):
        assert (pl is None) == (st.spec is None)
        if pl is None:
            continue
        lane, waits = pl
        assert 0 <= lane < 4 and all(w < i and plan[w] is not None for w in waits)
        need = [p for p in (st.x, st.w_from, st.res) if p is not None and steps[p].spec is not None]
        for p in (st.x, st.w_from, st.res):
            if p is not None and p > 0 and steps[p].spec is None:
                need += [q for q in range(p - 1, -1, -1) if steps[q].spec is not None][:1]
        if st.kernel in serial and st.kernel in last_serial:
            need.append(last_serial[st.kernel])
        for p in need:
            assert plan[p][0] == lane or p in waits, (model, i, p)
        seen_on_lane.setdefault(lane, []).append(i)
        last_serial[st.kernel] = i
    lanes_used = len(seen_on_lane)
    assert lanes_used == (1 if model == "mobilenet_v2" else 4)


def test_compensated_precision_is_kept_where_it_exists_and_reported_elsewhere():
    """Record field `precision` = 1 (three TF32 products per step): dense and batch_matmul NT in the one-tile form keep
    it, with twice the shared memory per stage and one accumulator; convolutions, NN products and the persistent form
    legalise it away as a change of form (strict mode: invalid)."""
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=32, stages=2, mma_m_axis=1, precision=1, acc_split=4)
    plain = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=32, stages=2, mma_m_axis=1)
    dense = W._dense(256, 512, 384).workload()
    st, info = dense.check(rec)
    st0, info0 = dense.check(plain)
    assert st == B.TT_OK and st0 == B.TT_OK and info.legal.precision == 1 and info.legal.acc_split == 1
    assert info.smem_bytes - 1024 == 2 * (info0.smem_bytes - 1024)
    assert dense.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE       # (acc_split was changed)
    rec.acc_split = 1
    assert dense.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_OK
    nt = W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(4, 128, 128, 64, True), 1, "nt").workload()
    assert nt.check(rec)[1].legal.precision == 1
    for other in (W._conv(32, 14, 64, 3, 1, 1).workload(), W._conv(64, 28, 64, 1, 1, 0).workload(),
                  W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(4, 128, 64, 128, False), 1, "nn").workload()):
        st, info = other.check(rec)
        assert st == B.TT_OK and info.legal.precision == 0 and info.changed & B.TT_CHG_FORM
        assert other.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    rec.persistent = 1
    st, info = dense.check(rec)
    assert st == B.TT_OK and info.legal.precision == 1 and info.legal.persistent == 0 and info.changed & B.TT_CHG_FORM
    bad = B.make_record(B.TT_FAMILY_GEMM_TC, precision=2)
    assert dense.check(bad)[0] == B.TT_ERR_INVALID_SCHEDULE


@pytest.mark.parametrize("lanes,waits,want", [
    ((0, 0), ((), ()), B.TT_ERR_NOT_APPLIED),       # well formed: stops at the first layer, which has no record applied
    ((0, 1), ((), (1,)), B.TT_ERR_INVALID_ARG),     # a layer that waits for itself
    ((0, 2), ((), (0,)), B.TT_ERR_INVALID_ARG),     # a lane without a stream
])
def test_run_chain_checks_its_arguments(lanes, waits, want):
    wl = W._dense(8, 16, 8).workload()
    t = B.tt_tensors()
    ws = [(ctypes.c_int32 * max(len(w), 1))(*w) for w in waits]
    steps = (B.tt_chain_step * 2)(*[B.tt_chain_step(wl.handle, ctypes.pointer(t), w, len(ids), lane) for w, ids, lane in zip(ws, waits, lanes)])
    at = ctypes.c_size_t(99)
    assert B.lib().tt_run_chain(steps, 2, (ctypes.c_void_p * 2)(), 2, ctypes.byref(at)) == want
    assert at.value == (0 if want == B.TT_ERR_NOT_APPLIED else 1)


DYN_SMEM_LIMIT = 227 * 1024 - 6144      # dynamic shared memory a CTA may ask for beside its barriers


def test_depthwise_plans_fit_shared_memory():
    """A record that is accepted never asks for more shared memory than a launch can have: boxes whose channel groups are
    evened out (38 for 40 of 301 channels, 46 for 48 of 504) and whose rows are then widened, and a sweep of the like."""
    import random
    rng = random.Random(5)
    cases = [((16, 301, 114, 16, 5, 2), (40, 12, 256, 2, 2)), ((47, 504, 11, 16, 5, 1), (48, 16, 16, 2, 2))]
    for _ in range(3000):
        r = rng.choice((3, 5))
        cases.append(((rng.randint(1, 48), rng.randint(1, 520), rng.randint(r, 120), 4 * rng.randint(2, 30), r, rng.choice((1, 2))),
                      (rng.randint(1, 64), rng.randint(1, 56), rng.choice((8, 16, 28, 32, 56, 112, 256)), rng.choice((1, 2, 4)), rng.randint(2, 4))))
    boxes = 0
    for (n, c, h, w, r, st), (tc_, by, bx, un, sg) in cases:
        wl = B.Workload(B.TT_OP_DWCONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=c, r=r, s=r, stride_h=st, stride_w=st, pad_h=r // 2, pad_w=r // 2,
                                                        has_bias=1, act=B.TT_ACT_RELU), "dw")
        rec = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=tc_, block_y=by, block_x=bx, items_per_thread=4, vec_width=1, threads=256, unroll=un,
                            raster=1, stages=sg)
        status, info = wl.check(rec)
        assert status in (B.TT_OK, B.TT_ERR_RESOURCE)
        if status == B.TT_OK:
            assert info.smem_bytes <= DYN_SMEM_LIMIT, ((n, c, h, w, r, st), rec.short(), info.smem_bytes)
            boxes += info.legal.raster
        wl.close()
    assert boxes > 1000


@pytest.mark.parametrize("shape", [
    # n, c, h, w, k, r, stride, residual: rows beyond what the taps' slab can hold
    (2, 8, 5, 1025, 16, 3, 1, 0), (3, 2, 40, 2000, 8, 5, 2, 0), (2, 32, 64, 1028, 64, 3, 1, 1), (4, 8, 9, 701, 24, 5, 1, 0), (1, 8, 9, 1200, 24, 3, 1, 0),
])
def test_tap_major_records_on_wide_images_run_in_the_stored_order(shape):
    """A record that names the tap-major order applies wherever the same record in the stored order does."""
    n, c, h, w, k, r, stride, res = shape
    wl = B.Workload(B.TT_OP_CONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=k, r=r, s=r, stride_h=stride, stride_w=stride, pad_h=r // 2, pad_w=r // 2,
                                                  has_bias=1, has_residual=res, act=B.TT_ACT_RELU), "wide")
    for tn, tk, stages in ((16, 32, 1), (64, 32, 2), (128, 96, 2)):
        stored = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=stages, mma_m_axis=1)
        tap = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=stages, k_order=1, mma_m_axis=1)
        st0, i0 = wl.check(stored)
        st1, i1 = wl.check(tap)
        assert st1 == st0
        if st0 != B.TT_OK:                               # the stored order's own rows do not fit either
            assert tn > 16
            continue
        assert i1.legal.k_order == 0 and i1.changed & B.TT_CHG_KORDER and i1.launches == 1
        assert bytes(i1.legal) == bytes(i0.legal) and (i1.grid_x, i1.grid_z, i1.smem_bytes) == (i0.grid_x, i0.grid_z, i0.smem_bytes)
        assert wl.check(tap, mode=B.TT_MODE_STRICT)[0] != B.TT_OK
    wl.close()


def test_nonsense_fields_are_refused_in_every_reduction_order():
    tap, pointwise, dense = W._conv(64, 28, 64, 3, 1, 1).workload(), W._conv(64, 28, 64, 1, 1, 0).workload(), W._dense(64, 128, 96).workload()
    base = dict(tile_n=64, tile_k=32, stages=2, mma_m_axis=1)
    nonsense = [dict(tile_m=0), dict(tile_n=-16), dict(tile_k=0), dict(stages=-3), dict(stages=0), dict(split_k=0), dict(raster=7), dict(raster=-1),
                dict(mma_m_axis=3), dict(acc_split=-1), dict(persistent=2), dict(ctas_per_sm=3), dict(warp_layout=1), dict(precision=2)]
    for wl in (tap, pointwise, dense):
        for order in (0, 1):
            assert wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, **dict(base, k_order=order)))[0] == B.TT_OK
            for bad in nonsense:
                for mode in (B.TT_MODE_LEGALISE, B.TT_MODE_STRICT):
                    rec = B.make_record(B.TT_FAMILY_GEMM_TC, **dict(base, k_order=order, **{k: v for k, v in bad.items() if k not in base}))
                    for k, v in bad.items():
                        setattr(rec, k, v)
                    assert wl.check(rec, mode=mode)[0] == B.TT_ERR_INVALID_SCHEDULE, (order, bad, mode)
    # a convolution's slab of input rows, whether or not this layer stages one; a dense layer has none
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, slab_tiles=-1, **base)
    assert [wl.check(rec)[0] for wl in (tap, pointwise, dense)] == [B.TT_ERR_INVALID_SCHEDULE, B.TT_ERR_INVALID_SCHEDULE, B.TT_OK]
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, slab_tiles=3, **base)           # (64 channels are two reduction tiles)
    assert pointwise.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE


@pytest.mark.parametrize("tn", range(16, 257, 16))
def test_tensor_memory_covers_what_the_read_out_reads(tn):
    """The read-out takes 32 columns at a time, also from the last accumulator: the last block of a tile whose columns are no
    multiple of 32 has to lie inside the allocation."""
    wl = W._dense(300, 256, 1030).workload()
    for acc in (1, 2, 4, 8):
        for kw in (dict(), dict(persistent=1), dict(split_k=3), dict(persistent=1, cta_group=2)):
            st, info = wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=32, stages=2, mma_m_axis=1, acc_split=acc, **kw))
            assert st == B.TT_OK and info.legal.tile_n == tn
            n_acc = 2 if info.legal.persistent else info.legal.acc_split
            assert (n_acc - 1) * tn + (tn + 31) // 32 * 32 <= info.tmem_cols <= 512 and info.tmem_cols & (info.tmem_cols - 1) == 0


def _launch_of(info):
    """What a launch is made from, as far as the apply info says it."""
    return (info.grid_x, info.grid_y, info.grid_z, info.threads, info.smem_bytes, info.tmem_cols, info.workspace_bytes)


def _check_legal_says_what_runs(wl, recs):
    """The legal record is what runs: legalising it again changes nothing and gives the same launch; every field that was
    replaced is reported; a record taken in strict mode runs as written.  Returns {legal record: launch}."""
    seen = {}
    for rec in recs:
        st, info = wl.check(rec)
        if st != B.TT_OK:
            continue
        st2, again = wl.check(info.legal)
        assert st2 == B.TT_OK and _rec_key(again.legal) == _rec_key(info.legal), (rec.short(), info.legal.short(), again.legal.short())
        assert not again.changed and _launch_of(again) == _launch_of(info), (rec.short(), info.legal.short(), again.changed)
        bits = {"tile_n": B.TT_CHG_TILE_N, "tile_k": B.TT_CHG_TILE_K, "stages": B.TT_CHG_STAGES, "split_k": B.TT_CHG_SPLIT_K,
                "k_order": B.TT_CHG_KORDER, "block_x": B.TT_CHG_BLOCK, "block_y": B.TT_CHG_BLOCK, "threads": B.TT_CHG_BLOCK,
                "items_per_thread": B.TT_CHG_ITEMS, "vec_width": B.TT_CHG_VEC, "unroll": B.TT_CHG_FORM}
        used = ("tile_n", "tile_k", "stages", "split_k", "k_order") if rec.family == B.TT_FAMILY_GEMM_TC else \
            ("block_x", "block_y", "threads", "items_per_thread", "vec_width", "unroll") + (("stages",) if info.legal.raster else ())
        for f in used:
            assert getattr(info.legal, f) == getattr(rec, f) or info.changed & bits[f], (rec.short(), info.legal.short(), f, info.changed)
        if info.legal.k_order and info.legal.cta_group != max(1, rec.cta_group):
            assert info.changed & B.TT_CHG_CLUSTER
        if rec.family == B.TT_FAMILY_DW_SIMT and info.legal.tile_m != rec.tile_m:
            assert info.changed & B.TT_CHG_TILE_M
        st3, strict = wl.check(rec, mode=B.TT_MODE_STRICT)
        if st3 == B.TT_OK:
            for f in used:
                assert getattr(strict.legal, f) == getattr(rec, f) and not strict.changed & ~B.TT_CHG_TILE_M
        seen.setdefault(_rec_key(info.legal), set()).add(_launch_of(info))
    assert all(len(v) == 1 for v in seen.values())
    return seen


def test_tap_major_legal_records_say_what_runs():
    """Columns and clusters that are laid over the SMs, taps in flight: named by the legal record, as written in strict mode."""
    import random
    rng = random.Random(3)
    def conv(n, c, h, w, k, r, st, pad):
        return B.Workload(B.TT_OP_CONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=k, r=r, s=r, stride_h=st, stride_w=st, pad_h=pad, pad_w=pad,
                                                        has_bias=1, act=B.TT_ACT_RELU), "tap")
    shapes = [(32, 128, 28, 28, 128, 3, 1, 1), (32, 512, 7, 7, 512, 3, 1, 1), (1, 64, 28, 28, 64, 3, 1, 1), (2, 16, 9, 9, 24, 1, 1, 0)]
    for _ in range(150):
        r = rng.choice((1, 2, 3, 3, 5, 7))
        shapes.append((rng.choice((2, 3, 8, 32, 70)), 8 * rng.randint(1, 64), rng.randint(7, 64), rng.randint(7, 64), 8 * rng.randint(1, 64), r,
                       rng.choice((1, 1, 2, 3)), rng.randint(0, r - 1)))
    recs = [B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=sg, mma_m_axis=1, k_order=1, persistent=ps, cta_group=cg)
            for tn in (16, 48, 64, 112, 128, 192, 224, 256) for tk in (32, 64, 96, 128) for sg, ps, cg in ((1, 0, 1), (2, 0, 1), (4, 1, 2), (8, 0, 8))]
    for shape in shapes:
        wl = conv(*shape)
        _check_legal_says_what_runs(wl, recs)
        wl.close()
    # the two records that used to be one launch under two names
    wl = conv(32, 128, 28, 28, 128, 3, 1, 1)
    a, b = (wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=sg, mma_m_axis=1, k_order=1))[1] for tn, tk, sg in ((224, 96, 2), (128, 32, 4)))
    assert _rec_key(a.legal) == _rec_key(b.legal) and (a.legal.tile_n, a.legal.stages, a.grid_x) == (192, 6, 141) and a.changed & B.TT_CHG_TILE_N
    st, s = wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=224, tile_k=96, stages=2, mma_m_axis=1, k_order=1), mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and s.legal.tile_n == 224 and s.grid_x == 121 and s.grid_y == 1
    wl.close()
    wl = conv(32, 512, 7, 7, 512, 3, 1, 1)
    info = wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=128, tile_k=32, stages=4, mma_m_axis=1, k_order=1))[1]
    assert (info.legal.tile_n, info.legal.cta_group, info.grid_x, info.grid_y) == (256, 4, 32, 4) and info.changed & B.TT_CHG_CLUSTER
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=32, stages=4, mma_m_axis=1, k_order=1, cta_group=3)
    st, s = wl.check(rec, mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and (s.legal.cta_group, s.grid_x, s.grid_y) == (3, 32, 3)
    rec.cta_group = 8                                    # 32 tiles of 8 CTAs are not resident at once
    assert wl.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    # a cluster of that order on a kernel without it
    st, info = W._dense(128, 256, 128).workload().check(rec)
    assert st == B.TT_OK and info.legal.cta_group == 1 and info.changed & B.TT_CHG_FORM
    rec.k_order = 0
    assert wl.check(rec)[0] == B.TT_ERR_INVALID_SCHEDULE
    wl.close()


def test_compensated_legal_records_say_what_runs():
    """Tiles of twice the columns and stages of 32 are named by the legal record; strict mode runs the record as written."""
    import random
    rng = random.Random(9)
    recs = [B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=sg, split_k=sk, mma_m_axis=ax, precision=1, ctas_per_sm=cps)
            for tn in (16, 32, 64, 128, 256) for tk in (8, 32, 64, 128) for sg, sk in ((1, 1), (2, 4), (3, 3), (4, 12)) for ax in (1, 2) for cps in (0, 2)]
    for m, k, n in [(512, 4096, 1024), (1030, 520, 700), (64, 64, 64)] + [(rng.randint(1, 2000), 4 * rng.randint(1, 500), rng.randint(1, 2000)) for _ in range(20)]:
        wl = W._dense(m, k, n).workload()
        _check_legal_says_what_runs(wl, recs)
        wl.close()
    wl = W._dense(512, 4096, 1024).workload()
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=64, stages=2, split_k=4, mma_m_axis=1, precision=1)
    st, info = wl.check(rec)
    assert st == B.TT_OK and (info.legal.tile_n, info.legal.tile_k, info.grid_x) == (128, 32, 32) and info.changed & B.TT_CHG_TILE_N
    st, info = wl.check(rec, mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and (info.legal.tile_n, info.legal.tile_k, info.grid_x) == (64, 64, 64) and not info.changed & B.TT_CHG_TILE_N
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=64, stages=1, mma_m_axis=1, precision=1)
    st, info = wl.check(rec)
    assert st == B.TT_OK and info.legal.tile_k == 32 and info.legal.stages == 2 and info.changed & B.TT_CHG_TILE_K
    wl.close()


def test_persistent_legal_records_say_what_runs():
    """More stages, or a deeper ring of a row-contiguous operand, than fit: the legal record's launch is the one that runs."""
    recs = [B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=sg, slab_tiles=sl, mma_m_axis=ax, persistent=1, cta_group=cg)
            for tn in (16, 64, 112, 256) for tk in (16, 64, 128) for sg in (1, 2, 5, 8) for sl in (0, 1, 8) for ax in (1, 2) for cg in (1, 2)]
    specs = [W._dense(478, 6 * 8, 484), W._dense(41, 120, 416), W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(105, 10, 88, 44, False), 1, "nn"),
             W._conv(64, 28, 96, 1, 1, 0, residual=True)]
    for sp in specs:
        wl = sp.workload()
        _check_legal_says_what_runs(wl, recs)
        wl.close()


DW_RECORDS = [B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=tm, block_y=by, block_x=bx, items_per_thread=it, vec_width=vw, threads=th, unroll=un, raster=ra, stages=sg)
              for tm, by, bx in ((1, 8, 32), (4, 14, 28), (4, 28, 56), (5, 7, 16), (16, 14, 28), (48, 56, 112)) for it, vw, th in ((4, 4, 64), (4, 1, 256), (8, 2, 256))
              for un in (0, 1, 2, 4, 7) for ra, sg in ((0, 1), (1, 2), (1, 4))]


def _dw_batch(n, c, h, w, r, st):
    return B.Workload(B.TT_OP_DWCONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=c, r=r, s=r, stride_h=st, stride_w=st, pad_h=r // 2, pad_w=r // 2,
                                                      has_bias=1, act=B.TT_ACT_RELU6), "dw")


def test_run_staged_depthwise_is_a_record_form():
    """Batches of ragged rows: every register-window record becomes the one record of the run-staged form, which says what runs;
    strict mode takes that record, or a register-window one as written."""
    for shape in ((256, 480, 14, 14, 5, 1), (64, 480, 14, 14, 5, 1), (64, 144, 55, 55, 3, 1), (40, 96, 33, 31, 3, 2), (3, 9, 253, 253, 5, 1)):
        wl = _dw_batch(*shape)
        window = [r for r in DW_RECORDS if r.unroll >= 1]
        seen = _check_legal_says_what_runs(wl, window)
        assert len(seen) == 1
        legal = wl.check(window[0])[1].legal
        assert legal.raster == 1 and legal.unroll in (2, 4, 7) and legal.items_per_thread in (1, 2) and legal.block_x == wl.check(legal)[1].legal.block_x
        assert wl.check(legal, mode=B.TT_MODE_STRICT)[0] == B.TT_OK
        rec = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=7, block_x=12, items_per_thread=4, vec_width=1, threads=64, unroll=2)
        st, info = wl.check(rec, mode=B.TT_MODE_STRICT)
        assert st == B.TT_OK and info.legal.raster == 0 and info.legal.unroll == 2 and info.threads == 64 and info.smem_bytes == 0
        rec.raster = 1
        assert wl.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
        _check_legal_says_what_runs(wl, [r for r in DW_RECORDS if r.unroll == 0])
        # and away from there it is a record like any other
        other = _dw_batch(4, 32, 28, 28, 3, 1)
        assert other.check(legal)[0] == B.TT_OK
        other.close()
        wl.close()


def test_box_staged_depthwise_legal_records_say_what_runs():
    """Evened channel groups, strips of 7 rows and threads without a strip are named by the legal record; strict mode runs the
    record as written."""
    for shape in ((256, 240, 28, 28, 5, 1), (2, 35, 121, 92, 5, 2), (16, 301, 114, 16, 5, 2), (64, 144, 56, 56, 3, 1), (1, 10, 9, 12, 3, 1)):
        wl = _dw_batch(*shape)
        _check_legal_says_what_runs(wl, DW_RECORDS)
        wl.close()
    wl = _dw_batch(256, 240, 28, 28, 5, 1)
    rec = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=7, block_y=28, block_x=28, items_per_thread=4, vec_width=4, threads=256, unroll=4, raster=1, stages=2)
    st, info = wl.check(rec)                             # 35 groups of 7 channels: 240 = 34 * 7 + 2
    assert st == B.TT_OK and (info.legal.tile_m, info.legal.unroll, info.legal.threads) == (7, 7, 224)
    assert info.changed & B.TT_CHG_FORM and info.changed & B.TT_CHG_BLOCK
    rec.tile_m = 50
    rec.block_y = 4
    st, info = wl.check(rec)                             # 5 groups of 48, not of 50
    assert st == B.TT_OK and (info.legal.tile_m, info.legal.unroll) == (48, 4) and info.changed & B.TT_CHG_TILE_M
    rec.tile_m, rec.block_y = 7, 28
    for unroll in (4, 7):
        rec.unroll = unroll
        st, info = wl.check(rec, mode=B.TT_MODE_STRICT)
        assert st == B.TT_OK and (info.legal.tile_m, info.legal.unroll, info.threads) == (7, unroll, 256) and not info.changed
    wl.close()
    wl = _dw_batch(64, 144, 56, 56, 3, 1)                # (3x3: no such strips)
    assert wl.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_ERR_INVALID_SCHEDULE
    assert wl.check(rec)[1].legal.unroll == 4
    wl.close()


def test_softmax_legal_records_say_what_runs():
    """Ragged rows: warps that fit, single-value accesses and the launch that the rows are staged in; strict mode as written."""
    recs = [B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=bx, block_y=by, vec_width=vw) for bx in (1, 2, 4, 8, 16, 32) for by in (1, 4, 16, 32) for vw in (1, 2, 4)]
    for rows, cols in ((151296, 197), (35, 1), (1000, 2), (4097, 1023), (17, 2046), (17, 2081), (300, 64), (300, 66), (5, 4097)):
        wl = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(1, rows, cols, 1.0), 1, "rows").workload()
        _check_legal_says_what_runs(wl, recs)
        for rec in recs:
            st, info = wl.check(rec)
            assert st == B.TT_OK and info.smem_bytes <= 100 * 1024 and info.threads <= 1024
            assert info.legal.block_x * info.legal.block_y == info.threads
            if info.smem_bytes:
                assert cols % 4 and info.legal.vec_width == 1 and info.smem_bytes % (16 * info.threads // 32) == 0
        wl.close()
    wl = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(1, 300, 66, 1.0), 1, "rows").workload()
    rec = B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=8, block_y=4, vec_width=2)
    assert wl.check(rec)[1].legal.vec_width == 1 and wl.check(rec)[1].changed & B.TT_CHG_VEC
    st, info = wl.check(rec, mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and info.legal.vec_width == 2 and info.smem_bytes == 0
    wl.close()


def test_softmax_threads_leave_their_registers_room():
    """A lane that keeps many values takes many registers: fewer threads per CTA, said by the legal record."""
    for cols, lanes, most in ((2048, 32, 512), (1028, 32, 512), (1024, 32, 1024), (576, 16, 512), (637, 32, 768), (1023, 32, 640), (1537, 32, 256), (47, 1, 256), (577, 32, 1024)):
        wl = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(1, 5000, cols, 1.0), 1, "rows").workload()
        rec = B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=lanes, block_y=1024 // lanes, vec_width=4 if cols % 4 == 0 else 1)
        st, info = wl.check(rec)
        assert st == B.TT_OK and info.threads <= most, (cols, lanes, info.threads)
        assert (info.threads == 1024) == (info.legal.block_y == rec.block_y) and (info.threads == 1024 or info.changed & B.TT_CHG_BLOCK)
        _check_legal_says_what_runs(wl, [rec])
        st, info = wl.check(rec, mode=B.TT_MODE_STRICT)       # as written, in passes over memory
        assert st == B.TT_OK and info.threads == 1024
        wl.close()


def test_chain_is_enqueued_with_its_streams_device_current(monkeypatch):
    """Streams of a device that is not the current one: that device is current while the pass is enqueued, and only then; lanes
    on several devices are enqueued layer by layer, each with its own device current and with the plan's waits."""
    import contextlib
    import torch
    now, log = [0], []

    @contextlib.contextmanager
    def device(d):
        back, now[0] = now[0], torch.device(d).index
        yield
        now[0] = back

    class Stream:
        def __init__(self, index, name):
            self.device_index, self.device, self.cuda_stream, self.name = index, torch.device("cuda", index), 0, name

        def record_event(self):
            log.append(("record", self.name))
            return len(log)

        def wait_event(self, e):
            log.append(("wait", self.name, e))

    class Call:
        @staticmethod
        def run_chain(*args):
            log.append(("native", now[0]))
            return B.TT_OK, -1

    class Kernel:
        def run(self, tt):
            log.append(("run", now[0], tt))

    monkeypatch.setattr(torch.cuda, "current_device", lambda: now[0])
    monkeypatch.setattr(torch.cuda, "device", device)
    monkeypatch.setattr(torch.cuda, "stream", lambda s: device(s.device))
    monkeypatch.setattr(B, "_call", Call)
    node = type("Node", (), {"kernel": 0})()
    plan = [None, (0, ()), (1, ()), (0, (2,))]
    for index in (0, 1):
        B.run_chain([Kernel()], [node] * 4, list("abcd"), plan, [Stream(index, "m"), Stream(index, "s")])
        assert log.pop() == ("native", index) and now == [0] and not log
    B.run_chain([Kernel()], [node] * 4, list("abcd"), plan, [Stream(0, "m"), Stream(1, "s")])
    assert log == [("record", "m"), ("run", 0, "b"), ("wait", "s", 1), ("run", 1, "c"), ("record", "s"), ("wait", "m", 5), ("run", 0, "d"),
                   ("record", "s"), ("wait", "m", 8)] and now == [0]


def test_run_chain_takes_plans_of_any_sequence(monkeypatch):
    """A plan entry is a pair of any kind, the waits any iterable, and the chain as long as the shortest of its lists; a layer
    without an applied record is what the pass then fails on."""
    import torch
    wls = [W._dense(8, 16, 8, name="first").workload(), W._dense(8, 16, 8, name="second").workload()]
    node = lambda k: type("Node", (), {"kernel": k})()
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    stream = type("Stream", (), {"cuda_stream": 0, "device_index": 0})()
    t = B.tt_tensors()
    for plan in ([(0, ()), (0, (0,))], [[0, []], [0, [0]]], ((0, set()), (0, {0})), [None, [0, ()]], [(0, ()), (0, (0,)), (0, (1,))]):
        at = 0 if plan[0] is not None else 1
        with pytest.raises(B.TTError) as err:
            B.run_chain(wls, [node(0), node(1)], [t, t], plan, [stream])
        assert err.value.status == B.TT_ERR_NOT_APPLIED and wls[at].name in str(err.value)
    B.run_chain(wls, [node(0), node(1)], [t, t], [], [stream])
    for bad, kind in (([(0,)], ValueError), ([5], TypeError), ([(0, (0,))], ValueError), ([(0, ()), ("x", ())], TypeError)):
        with pytest.raises(kind):
            B.run_chain(wls, [node(0), node(1)], [t, t], bad, [stream])


def test_nothing_throws_across_the_c_abi():
    """Containers that cannot be made are a status, not an exception through C frames (which ends the process: run in a child)."""
    import subprocess
    import sys
    code = """
import ctypes as C
from paper_2201_05587_b200 import binding as B
lib, huge = B.lib(), 1 << 61
share, counts, order = (C.c_double * 1)(1.0), (C.c_int32 * 1)(1), (C.c_int32 * 1)()
assert lib.tt_rank_pools(share, 1, counts, huge, None, order) == B.TT_ERR_OOM
steps, streams, at = (B.tt_chain_step * 1)(), (C.c_void_p * 1)(), C.c_size_t()
assert lib.tt_run_chain(steps, huge, streams, 1, C.byref(at)) == B.TT_ERR_OOM
assert lib.tt_run_chain(steps, 1, streams, huge, C.byref(at)) == B.TT_ERR_OOM
print("statuses")
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "statuses" in r.stdout, r.stderr


@pytest.mark.parametrize("shape", [(6, 320, 9, 200, 3), (16, 512, 7, 512, 3), (8, 256, 14, 256, 3), (1, 64, 56, 64, 3), (8, 64, 14, 128, 1), (32, 512, 7, 512, 3)])
def test_tap_major_clusters_are_resident_and_worth_their_exchange(shape):
    """CTAs of a cluster keep to one group of SMs: 148 SMs do not hold 20 clusters of 7.  A single tap is not shared."""
    resident = (0, 148, 74, 45, 33, 26, 22, 15, 15)
    n, c, hw, k, r = shape
    wl = B.Workload(B.TT_OP_CONV2D, B.conv2d_shapes(n, c, hw, hw, k, r, r, 1, r // 2, True, B.TT_ACT_RELU), "tap")
    for tn in (32, 64, 96, 128, 192, 256):
        st, info = wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=32, stages=8, mma_m_axis=1, k_order=1))
        assert st == B.TT_OK and info.grid_y == info.legal.cta_group
        assert info.legal.cta_group == 1 or info.grid_x <= resident[info.legal.cta_group]
        if c * r * r <= 64:
            assert info.legal.cta_group == 1
    wl.close()


@pytest.mark.parametrize("m,k,n,rec,tile_n,split", [
    (2419, 888, 1976, dict(tile_n=256, tile_k=32, stages=2, persistent=1), 160, 1),                  # 152 tiles: two rounds of less
    (2419, 888, 1976, dict(tile_n=256, tile_k=32, stages=6, persistent=1, cta_group=2), 160, 1),     # 80 pairs of CTAs
    (1500, 512, 2000, dict(tile_n=256, tile_k=32, stages=2, persistent=1), 256, 1),                  # one round: as the record says
    (4096, 64, 4096, dict(tile_n=64, tile_k=32, stages=2, persistent=1), 64, 1),                     # many rounds: likewise
    (533, 4096, 464, dict(tile_n=64, tile_k=64, stages=3, split_k=4), 64, 3),                        # 40 clusters of 4, of which 33 are resident
    (533, 4096, 464, dict(tile_n=64, tile_k=64, stages=2, split_k=8), 64, 3),
    (128, 768, 768, dict(tile_n=64, tile_k=64, stages=3, split_k=4), 64, 4),                         # all resident
    (128, 256, 768, dict(tile_n=16, tile_k=128, stages=1, split_k=2), 16, 2),
])
def test_tiles_and_splits_follow_the_rounds_of_the_sms(m, k, n, rec, tile_n, split):
    """Columns of a persistent record are dealt evenly over its rounds, splits are as many as pay for their rounds; the legal record
    says so, legalising it again changes nothing, and strict mode runs the record as written."""
    wl = W._dense(m, k, n).workload()
    r = B.make_record(B.TT_FAMILY_GEMM_TC, mma_m_axis=1, **rec)
    st, info = wl.check(r)
    assert st == B.TT_OK and (info.legal.tile_n, info.legal.split_k) == (tile_n, split)
    assert bool(info.changed & B.TT_CHG_TILE_N) == (tile_n != r.tile_n) and bool(info.changed & B.TT_CHG_SPLIT_K) == (split != r.split_k)
    _check_legal_says_what_runs(wl, [r])
    st, info = wl.check(r, mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and (info.legal.tile_n, info.legal.split_k) == (r.tile_n, r.split_k)
    wl.close()


def test_what_runs_as_written_is_not_refused_when_it_may_be_laid_out():
    """A rule that lays a record out otherwise gives way where its plan does not fit: whatever strict mode accepts, legalising accepts,
    and the record's own splits then stay.  Wide 5x5 and 7x7 convolutions, whose table of the reduction is the longest."""
    wide = W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(16, 2048, 13, 13, 256, 5, 5, 1, 2, True, B.TT_ACT_RELU), 1, "wide", "he").workload()
    st, info = wide.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=64, stages=2, split_k=8, mma_m_axis=2))
    assert st == B.TT_OK and info.legal.split_k == 8 and not info.changed & B.TT_CHG_SPLIT_K
    wide.close()
    accepted = 0
    shapes = [W._conv(2048, 13, 256, 5, 1, 2), W._conv(1228, 29, 908, 7, 1, 3), W._conv(185, 31, 190, 1, 1, 0), W._dense(533, 4096, 464), W._dense(70, 8190, 1001)]
    for spec, n in itertools.product(shapes, (1, 16, 28)):
        if spec.op == B.TT_OP_CONV2D:
            spec.shapes.n = n
        wl = spec.workload()
        for tn, tk, st_, sk, axis, sl in itertools.product((16, 64, 96, 128, 256), (16, 64, 128), (1, 2, 6), (3, 6, 8), (1, 2), (0, 2)):
            rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tn, tile_k=tk, stages=st_, split_k=sk, mma_m_axis=axis, slab_tiles=sl if spec.op == B.TT_OP_CONV2D else 0)
            if wl.check(rec, mode=B.TT_MODE_STRICT)[0] == B.TT_OK:
                accepted += 1
                assert wl.check(rec)[0] == B.TT_OK, (spec.name, n, rec.short())
        wl.close()
    assert accepted > 1000


def test_the_scratch_that_clusters_exchange_through_is_reported():
    """A tap-major record in clusters has, beside the re-packed filters, scratch for every CTA's accumulator in whole blocks of 32 columns;
    one without clusters has the filters alone."""
    wl = W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(32, 512, 7, 7, 512, 3, 3, 1, 1, True, B.TT_ACT_RELU, True), 1, "c", "he").workload()
    for tile_n, cluster in ((224, 1), (224, 3), (256, 4), (144, 2)):
        rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tile_n, tile_k=32, stages=4, k_order=1, mma_m_axis=1, persistent=1, cta_group=cluster)
        st, info = wl.check(rec, mode=B.TT_MODE_STRICT)
        assert st == B.TT_OK and info.legal.cta_group == cluster and info.grid_y == cluster
        assert info.workspace_bytes == 512 * 512 * 9 * 4
        assert info.exchange_kib * 1024 == (info.grid_x * cluster * -(-tile_n // 32) * 128 * 32 * 4 if cluster > 1 else 0)
    wl.close()
    st, info = W._dense(128, 768, 768).workload().check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=64, stages=2, split_k=4, mma_m_axis=2))
    assert st == B.TT_OK and info.exchange_kib == 0


def test_a_pointwise_layer_of_wide_tiles_is_shared_by_a_cluster():
    """512 -> 64 channels, 1x1, 8 images of 14 x 14: seven tiles of 256 columns whose 16 channel blocks eight CTAs share (29.9 us by one
    CTA each, 11.6 in eights); a tap of two blocks is not worth the exchange."""
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=256, tile_k=32, stages=8, mma_m_axis=1, k_order=1)
    for c, k, cluster in ((512, 64, 8), (64, 128, 1)):
        wl = B.Workload(B.TT_OP_CONV2D, B.conv2d_shapes(8, c, 14, 14, k, 1, 1, 1, 0, True, B.TT_ACT_RELU), "tap")
        st, info = wl.check(rec)
        assert st == B.TT_OK and info.legal.tile_n == 256 and info.legal.cta_group == cluster
        wl.close()


@pytest.mark.parametrize("m,k,n,rec,tile_n", [
    (785, 384, 1160, dict(tile_n=64, tile_k=32, stages=2, mma_m_axis=1, cta_group=2), 64),           # 76 tiles for 74 pairs: 32 columns cost more
    (3147, 1592, 1352, dict(tile_n=128, tile_k=32, stages=3, mma_m_axis=2, cta_group=2), 128),       # 150 for 74
    (495, 1688, 3648, dict(tile_n=96, tile_k=32, stages=3, mma_m_axis=2, cta_group=2), 64),          # 90 for 74: the last round is a fifth full
    (1160, 384, 4096, dict(tile_n=256, tile_k=32, stages=2, mma_m_axis=1), 160),                     # 160 for 148, wide tiles
])
def test_narrow_tiles_are_not_dealt_for_a_last_round_of_few(m, k, n, rec, tile_n):
    """A record whose last round holds less than an eighth of the SMs keeps its columns, unless those that it would get are still 128."""
    wl = W._dense(m, k, n).workload()
    r = B.make_record(B.TT_FAMILY_GEMM_TC, persistent=1, **rec)
    st, info = wl.check(r)
    assert st == B.TT_OK and info.legal.tile_n == tile_n and bool(info.changed & B.TT_CHG_TILE_N) == (tile_n != r.tile_n)
    _check_legal_says_what_runs(wl, [r])
    wl.close()


@pytest.mark.parametrize("tile_n,tile_k,columns", [(64, 32, 64), (112, 32, 128), (128, 32, 512), (176, 32, 512), (192, 32, 256), (16, 64, 32), (32, 64, 512), (64, 64, 512), (128, 16, 128)])
def test_compensated_products_take_tensor_memory_where_a_stage_is_worth_it(tile_n, tile_k, columns):
    """Stages of 64 of the reduction from 32 columns on, of 32 between 128 and 176: the plan then asks for buffers behind the accumulator."""
    wl = W._dense(300, 2048, 400).workload()
    st, info = wl.check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=tile_n, tile_k=tile_k, stages=2, mma_m_axis=1, precision=1), mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and info.tmem_cols == columns
    st, info = W._dense(300, 480, 400).workload().check(B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=128, tile_k=32, stages=2, mma_m_axis=1, precision=1), mode=B.TT_MODE_STRICT)
    assert st == B.TT_OK and info.tmem_cols == 128                 # a short reduction
    wl.close()


@pytest.mark.parametrize("rows,cols,lanes,chunk", [
    (100000, 33, 32, 8), (30000, 33, 32, 4), (100000, 187, 16, 8), (100000, 190, 16, 4),     # eight short rows, where there are many
    (3000, 330, 16, 2), (3000, 330, 8, 4), (100000, 330, 16, 4), (3000, 46, 16, 4),          # two even ones, where there are few and they are long enough
    (30000, 1174, 32, 2), (30000, 1175, 32, 4),                                              # ... or long
])
def test_rows_that_a_warp_of_the_ragged_softmax_takes(rows, cols, lanes, chunk):
    wl = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(1, rows, cols, 1.0), 1, "s", "bert").workload()
    st, info = wl.check(B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=lanes, block_y=4, vec_width=1))
    assert st == B.TT_OK and info.smem_bytes == info.threads // 32 * chunk * cols * 4
    wl.close()


def test_short_reductions_beside_a_gathered_operand_come_without_boxes():
    """Ragged rows of x in an NN product come by TMA from 33 of the reduction on; those of NT and dense products always do."""
    rec = B.make_record(B.TT_FAMILY_GEMM_TC, tile_n=64, tile_k=32, stages=1, mma_m_axis=1)
    for k, trans_b, boxes in ((31, False, 0), (33, False, 1), (31, True, 2)):
        wl = B.Workload(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(4, 100, 64, k, trans_b), "b")
        st, info = wl.check(rec)
        plain = B.Workload(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(4, 100, 64, 32 if k == 31 else 36, trans_b), "p")
        st2, info2 = plain.check(rec)
        box = lambda r: -(-36 * 4 * r // 128) * 128 * 4
        assert st == st2 == B.TT_OK and info.smem_bytes - info2.smem_bytes == (0, box(32), box(32) + box(16))[boxes]
        wl.close()
        plain.close()
