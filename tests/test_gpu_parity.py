"""GPU parity: the CUDA path, called through the C ABI, against the CPU oracle on the same seeded inputs."""
import ctypes
import itertools
import math
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import oracle as orc
from paper_2201_05587_b200 import binding as B
from paper_2201_05587_b200 import workloads as W
import util

pytestmark = pytest.mark.gpu

INVARIANCE_TOL = 1e-5   # between two valid records on the same precision path


def tc(**kw):
    return B.make_record(B.TT_FAMILY_GEMM_TC, **kw)


GUARD_FLOATS = 16384          # 64 KB of a fixed pattern on either side of every output tensor
GUARD_VALUE = -7.5e37
ELEM_TF32 = 1e-4              # max |y - truncation-mode oracle| / max |oracle|: fp32 accumulation of up to 4608 exact products
ELEM_FP32 = 1e-5              # the same for the fp32 SIMT families against the exact oracle


def guarded_output(spec, device="cuda"):
    """An output tensor that sits between two guard bands: returns (y view, whole buffer)."""
    import torch
    shape = W.tensor_shapes(spec)[4]
    n = int(np.prod(shape))
    buf = torch.full((n + 2 * GUARD_FLOATS,), GUARD_VALUE, dtype=torch.float32, device=device)
    y = buf[GUARD_FLOATS:GUARD_FLOATS + n].view(shape)
    y.fill_(float("nan"))
    return y, buf


def guards_intact(buf):
    return bool((buf[:GUARD_FLOATS] == GUARD_VALUE).all()) and bool((buf[-GUARD_FLOATS:] == GUARD_VALUE).all())


def run_spec(spec, rec, arrays, ref=None, tol=None, mode=B.TT_MODE_LEGALISE, ref_elem=None):
    """Run `spec` under `rec` through the C ABI.  ref: exact oracle (whole-tensor rel-L2, the pass/fail of record).
    ref_elem: the oracle every single output is bounded against -- the truncation-mode oracle for the TF32 families
    (the tensor core reads its operands truncated to TF32), the exact oracle for the fp32 SIMT families -- so that
    one wrong output in a large tensor cannot hide inside the L2 norm.  The output sits between guard bands."""
    wl = spec.workload()
    info = wl.apply(rec, mode=mode)
    if info.legal.precision == 1 and ref is not None:
        ref_elem = ref if ref_elem is not None else None      # compensated products: bounded against the exact oracle
    t, _ = W.device_tensors(spec, arrays)
    t["y"], buf = guarded_output(spec)
    tt = B.tensors(t["x"], t["w"], t["bias"], t["residual"], t["y"])
    wl.run(tt)
    assert wl.status() == B.TT_OK
    y = t["y"].cpu().numpy()
    wl.close()
    assert guards_intact(buf), f"{spec.name} {rec.short()} wrote outside its output tensor"
    assert not np.isnan(y).any(), "kernel left outputs unwritten"
    if ref is not None:
        err = util.rel_l2(y, ref)
        assert err <= (tol or util.tolerance(spec.op)), f"{spec.name} {rec.short()} rel-L2 {err:.3e}"
    if ref_elem is not None:
        bound = (ELEM_FP32 if spec.op in (B.TT_OP_DWCONV2D, B.TT_OP_SOFTMAX) else ELEM_TF32) * max(float(np.abs(ref_elem).max()), 1e-30)
        worst = float(np.abs(y.astype(np.float64) - ref_elem.astype(np.float64)).max())
        assert worst <= bound, f"{spec.name} {rec.short()} max element error {worst:.3e} > {bound:.3e}"
    return y


def elem_ref(spec, arrays, ref):
    """The oracle against which single outputs are bounded (see run_spec)."""
    if spec.op in (B.TT_OP_DWCONV2D, B.TT_OP_SOFTMAX):
        return ref
    return util.oracle_ref(spec, arrays, mode=orc.MODE_TF32_TRUNC)


GEMM_RECORDS = [
    tc(tile_n=128, tile_k=32, stages=4, mma_m_axis=1),
    tc(tile_n=64, tile_k=16, stages=3, mma_m_axis=1),
    tc(tile_n=16, tile_k=8, stages=2, mma_m_axis=1),
    tc(tile_n=256, tile_k=64, stages=2, mma_m_axis=1),
    tc(tile_n=48, tile_k=32, stages=1, raster=1, mma_m_axis=1),
    tc(tile_n=96, tile_k=32, stages=6, split_k=3, mma_m_axis=1),
    tc(tile_n=128, tile_k=64, stages=3, split_k=2, mma_m_axis=2),
    tc(tile_n=32, tile_k=128, stages=2, split_k=1, raster=1, mma_m_axis=2),
    tc(tile_n=192, tile_k=16, stages=4, split_k=5, mma_m_axis=2),
    # convolutions: the input rows are staged for 1, 2 or 3 reduction tiles at a time (double-buffered chunks)
    tc(tile_n=64, tile_k=16, stages=3, slab_tiles=1, mma_m_axis=1),
    tc(tile_n=128, tile_k=32, stages=2, slab_tiles=2, mma_m_axis=2),
    tc(tile_n=32, tile_k=8, stages=4, split_k=2, slab_tiles=3, mma_m_axis=1),
    # more than 8 splits: partial tiles through the global workspace (2..8 splits reduce inside a thread-block cluster)
    tc(tile_n=64, tile_k=16, stages=2, split_k=12, mma_m_axis=1),
    # tap-major reduction order (stride-1 convolutions with 16-byte image rows; elsewhere legalised to the stored order)
    tc(tile_n=128, tile_k=32, stages=3, k_order=1, mma_m_axis=1),
    tc(tile_n=256, tile_k=64, stages=2, k_order=1, split_k=2, mma_m_axis=2),
    tc(tile_n=48, tile_k=32, stages=1, k_order=1, raster=1, mma_m_axis=1),
    tc(tile_n=64, tile_k=96, stages=2, k_order=1, mma_m_axis=1),            # three taps per pipeline stage where 3 divides r*s
    # several accumulators in tensor memory, reduction steps dealt round-robin, summed on read-out
    tc(tile_n=32, tile_k=32, stages=4, acc_split=4, mma_m_axis=1),
    tc(tile_n=48, tile_k=16, stages=3, acc_split=8, split_k=2, mma_m_axis=2),
    tc(tile_n=256, tile_k=64, stages=2, acc_split=2, mma_m_axis=1),
    # the persistent form (tile loop, two alternating accumulators; operands by TMA, row-contiguous ones transposed in
    # shared memory), alone and as CTA pairs; the register-capped two-CTAs-per-SM build of the one-tile form.  Kernels
    # that have no such form legalise these records back
    tc(tile_n=64, tile_k=32, stages=4, persistent=1, mma_m_axis=1),
    tc(tile_n=16, tile_k=16, stages=3, persistent=1, raster=1, mma_m_axis=2),
    tc(tile_n=128, tile_k=64, stages=2, persistent=1, mma_m_axis=2),
    tc(tile_n=96, tile_k=8, stages=8, persistent=1, mma_m_axis=0),
    tc(tile_n=64, tile_k=32, stages=3, persistent=1, cta_group=2, mma_m_axis=1),
    tc(tile_n=256, tile_k=32, stages=2, persistent=1, cta_group=2, mma_m_axis=2),
    tc(tile_n=32, tile_k=128, stages=2, persistent=1, cta_group=2, raster=1, mma_m_axis=1),
    tc(tile_n=128, tile_k=32, stages=3, k_order=1, persistent=1, mma_m_axis=1),          # tap-major in the persistent form
    tc(tile_n=64, tile_k=96, stages=2, k_order=1, persistent=1, raster=1, mma_m_axis=1),
    tc(tile_n=64, tile_k=32, stages=2, ctas_per_sm=2, mma_m_axis=1),
    tc(tile_n=128, tile_k=16, stages=3, ctas_per_sm=1, split_k=2, mma_m_axis=2),
    # error-compensated products (dense, batch_matmul NT; legalised away elsewhere)
    tc(tile_n=64, tile_k=32, stages=2, precision=1, mma_m_axis=1),
    tc(tile_n=128, tile_k=64, stages=3, precision=1, split_k=3, mma_m_axis=2),
]


def check_all_records(spec, seed, records=GEMM_RECORDS):
    a = W.make_inputs(spec, seed)
    ref = util.oracle_ref(spec, a)
    # a record whose tiles (for a convolution: plus the staged input rows) exceed shared memory on this shape is an
    # invalid pair, as in the evaluator; everything that applies must be right, and most records must apply
    probe = spec.workload()
    valid = [r for r in records if probe.check(r)[0] == B.TT_OK]
    assert all(probe.check(r)[0] in (B.TT_OK, B.TT_ERR_RESOURCE) for r in records)
    assert probe.check(probe.default_schedule())[0] == B.TT_OK
    compensated = [probe.check(r)[1].legal.precision == 1 for r in valid]      # (kept only where the kernel has that form)
    probe.close()
    assert len(valid) >= len(records) - 6
    re = elem_ref(spec, a, ref)
    outs = [run_spec(spec, r, a, ref, ref_elem=re) for r in valid]
    # a schedule changes speed, never semantics: every valid record gives the same output up to the order of the
    # fp32 additions (tile_k and split_k regroup them): sqrt(K) * 2^-24 is about 4e-6 at the largest K here.  Records
    # with error-compensated products are another precision path: compared among themselves
    for group in (False, True):
        ys = [y for y, c in zip(outs, compensated) if c == group]
        for y in ys[1:]:
            assert util.rel_l2(y, ys[0]) <= INVARIANCE_TOL
    return outs


@pytest.mark.parametrize("spec", [
    W._dense(128, 768, 768, name="bert_dense"),
    W._dense(200, 300, 100, act=B.TT_ACT_RELU, name="ragged_dense"),        # ragged M, N, K tails; K % 8 != 0
    W._dense(129, 147, 257, act=B.TT_ACT_GELU_ERF, name="odd_dense_gatherK"),   # K % 4 != 0: gathered operands
    W._dense(1, 512, 1000, name="head_m1"),
    W._dense(1, 1, 1, name="one_by_one"),
    W._dense(3, 5, 7, name="tiny"),
], ids=lambda s: s.name)
def test_dense_parity_all_records(spec):
    check_all_records(spec, seed=31)


@pytest.mark.parametrize("spec", [
    W.single_conv()[0],
    W._conv(3, 32, 64, 7, 2, 3, name="stem_like_7x7s2"),                    # reduction 147: gathered filters
    W._conv(24, 15, 40, 3, 2, 1, name="conv3x3s2_odd"),
    W._conv(32, 14, 64, 1, 1, 0, act=B.TT_ACT_RELU6, name="conv1x1_relu6"),
    W._conv(64, 14, 128, 1, 2, 0, act=B.TT_ACT_NONE, name="downsample_1x1s2"),
    W._conv(20, 7, 24, 3, 1, 1, name="conv3x3_7x7"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(2, 8, 9, 11, 12, 3, 3, 1, 1, True, B.TT_ACT_RELU, True), 1, "batch2_residual", "uniform"),
    W.Spec(B.TT_OP_CONV2D, B.make_shapes(n=1, c=6, h=10, w=12, k=9, r=3, s=2, stride_h=2, stride_w=1, pad_h=0, pad_w=1,
                                         has_bias=0, act=B.TT_ACT_NONE), 1, "asym_nobias", "uniform"),
    W._conv(20, 12, 40, 3, 1, 1, name="conv3x3_12x12_tap"),                 # rows of 48 bytes: the tap-major path applies
    W._conv(72, 16, 136, 3, 1, 1, act=B.TT_ACT_NONE, name="conv3x3_72ch_tap"),   # 3 channel blocks (the last one partial), 2 filter tiles
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(2, 33, 8, 20, 10, 5, 3, 1, 2, True, B.TT_ACT_RELU6), 1, "conv5x3_batch2_tap", "uniform"),
    W._conv(20, 10, 40, 1, 1, 0, name="conv1x1_100px_20ch"),
    W._conv(136, 12, 200, 1, 1, 0, act=B.TT_ACT_NONE, name="conv1x1_136ch"),
    # pointwise layers whose pixels are re-viewed as rows that tile the CTA exactly: 400 = 16 x 25, 784 = 16 x 49,
    # 3136 = 64 x 49 (batch 3, a partial last tile, a residual), and one whose pixel count has no such divisor
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(3, 40, 20, 20, 24, 1, 1, 1, 0, True, B.TT_ACT_RELU, True), 1, "conv1x1_400px_batch3_residual", "uniform"),
    W._conv(64, 28, 80, 1, 1, 0, act=B.TT_ACT_RELU6, name="conv1x1_784px"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(2, 24, 56, 56, 40, 1, 1, 1, 0, True, B.TT_ACT_NONE), 1, "conv1x1_3136px_batch2", "uniform"),
    W._conv(48, 18, 32, 1, 1, 0, name="conv1x1_324px_no_row_view"),
    W._conv(96, 9, 48, 3, 1, 1, name="conv3x3_96ch_chunks"),                # 864 reduction indices: many slab chunks
    W._conv(40, 12, 24, 5, 1, 2, act=B.TT_ACT_RELU6, name="conv5x5_pad2"),
    W._conv(32, 17, 16, 1, 3, 0, name="conv1x1s3"),                         # stride beyond the filter: rows are skipped
    W.Spec(B.TT_OP_CONV2D, B.make_shapes(n=2, c=5, h=9, w=13, k=7, r=2, s=4, stride_h=3, stride_w=2, pad_h=1, pad_w=3,
                                         has_bias=1, act=B.TT_ACT_RELU), 1, "asym_2x4_s3x2_p1x3", "uniform"),
], ids=lambda s: s.name)
def test_conv_parity_all_records(spec):
    check_all_records(spec, seed=32)


@pytest.mark.parametrize("spec", [
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(12, 128, 128, 64, True), 1, "qk_nt", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(12, 128, 64, 128, False), 1, "pv_nn", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(3, 50, 70, 36, False), 1, "ragged_nn", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(2, 45, 76, 52, False), 1, "ragged_nn_76", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(2, 33, 17, 10, True), 1, "ragged_nt_k10", "bert"),
], ids=lambda s: s.name)
def test_batch_matmul_parity_all_records(spec):
    check_all_records(spec, seed=33)


def test_config1_every_pool_record_and_selection():
    spec = W.single_conv()[0]
    a = W.make_inputs(spec, 1)
    ref = util.oracle_ref(spec, a)
    pool = W.single_conv_pool()
    outs = [run_spec(spec, r, a, ref) for r in pool]
    for y in outs[1:]:
        assert util.rel_l2(y, outs[0]) <= INVARIANCE_TOL
    wl = spec.workload()
    t, tt = W.device_tensors(spec, a)
    res = B.transfer_tune([wl], [tt], pool)
    assert res["pairs_timed"] == 5 and res["pairs_invalid"] == 0
    times = res["times_us"][0]
    assert all(v > 0 for v in times)
    # selection is the oracle's argmin on the measured table
    assert res["chosen"] == orc.select(times, 1, 5) == B.select(times, 1, 5)
    assert res["best_us"][0] == pytest.approx(min(times))
    # the chosen record is left applied: running now reproduces the oracle
    t["y"].zero_()
    wl.run(tt)
    assert wl.status() == B.TT_OK
    assert util.rel_l2(t["y"].cpu().numpy(), ref) <= util.TOL_TF32


def test_evaluator_records_invalid_pairs_and_falls_back_to_default():
    conv = W._conv(16, 12, 24, 3, 1, 1)
    dw = W._dw(16, 12, 1)
    a1, a2 = W.make_inputs(conv, 7), W.make_inputs(dw, 7, 1)
    w1, w2 = conv.workload(), dw.workload()
    t1, tt1 = W.device_tensors(conv, a1)
    t2, tt2 = W.device_tensors(dw, a2)
    fat = tc(tile_n=256, tile_k=128, stages=8, mma_m_axis=1)           # legal fields, too much shared memory... on big shapes
    nonsense = tc(tile_n=64, tile_k=32, stages=0)
    pool = [tc(tile_n=32, tile_k=16, stages=2), nonsense, B.make_record(B.TT_FAMILY_ROW_SIMT)]
    res = B.transfer_tune([w1, w2], [tt1, tt2], pool)
    st = res["status"]
    assert st[0][0] == B.TT_OK and st[0][1] == B.TT_OK
    assert st[0][2] == B.TT_ERR_INVALID_SCHEDULE and st[0][3] == B.TT_ERR_CLASS_MISMATCH
    assert res["times_us"][0][2] == -1.0 and res["times_us"][0][3] == -1.0
    # the depthwise kernel has no compatible record in this pool: it keeps its default schedule
    assert st[1][1] == st[1][2] == st[1][3] == B.TT_ERR_CLASS_MISMATCH
    assert res["chosen"][1] == 0 and res["best_us"][1] > 0
    assert res["pairs_invalid"] == 5 and res["pairs_timed"] == 3
    w2.run(tt2)
    assert util.rel_l2(t2["y"].cpu().numpy(), util.oracle_ref(dw, a2)) <= util.TOL_FP32
    del fat


@pytest.mark.parametrize("spec", [s for s in W.mobilenet_v2() if s.op == B.TT_OP_DWCONV2D][::3] + [
    W._dw(5, 9, 2), W._dw(40, 28, 1, r=5), W._dw(1, 1, 1),
    W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=3, c=7, h=13, w=10, r=3, s=3, stride_h=1, stride_w=2, pad_h=1, pad_w=0,
                                           has_bias=0, act=B.TT_ACT_RELU), 1, "dw_batch3_asym", "uniform"),
], ids=lambda s: s.name)
def test_depthwise_parity_records(spec):
    a = W.make_inputs(spec, 34)
    ref = util.oracle_ref(spec, a)
    recs = [spec.workload().default_schedule()]
    # unroll 0: shared-memory staged kernel; 1, 2, 4: register-window kernel with that many output rows per thread
    # (3x3 / 5x5 "same" filters; other filters fall back to the staged kernel)
    for tcn, by, bx, it, vw, th, un in ((4, 8, 32, 4, 4, 256, 0), (16, 4, 16, 2, 2, 128, 0), (1, 16, 64, 8, 4, 64, 0),
                                        (32, 7, 7, 1, 1, 512, 0), (3, 5, 24, 8, 1, 96, 0),
                                        (4, 8, 32, 4, 4, 256, 1), (1, 16, 64, 8, 4, 64, 2), (2, 7, 12, 4, 4, 512, 4),
                                        (8, 5, 8, 1, 1, 32, 4), (3, 6, 112, 4, 2, 96, 2), (2, 3, 16, 8, 4, 128, 1), (5, 9, 24, 8, 1, 64, 4)):
        recs.append(B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=tcn, block_y=by, block_x=bx, items_per_thread=it,
                                  vec_width=vw, threads=th, unroll=un))
    # raster = 1: input boxes staged by TMA, persistent CTAs (image rows of 16-byte multiples; elsewhere legalised away)
    for tcn, by, bx, it, vw, th, un, st in ((4, 8, 32, 4, 4, 128, 2, 3), (1, 7, 16, 4, 4, 64, 4, 2), (16, 4, 8, 4, 2, 256, 1, 4),
                                            (3, 5, 28, 4, 4, 96, 2, 2), (8, 6, 56, 8, 4, 256, 2, 2), (5, 3, 16, 8, 4, 32, 1, 3),
                                            (32, 56, 56, 4, 4, 256, 1, 2)):
        recs.append(B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=tcn, block_y=by, block_x=bx, items_per_thread=it, vec_width=vw,
                                  threads=th, unroll=un, raster=1, stages=st))
    outs = [run_spec(spec, r, a, ref, ref_elem=ref) for r in recs]
    for y in outs[1:]:
        np.testing.assert_array_equal(y, outs[0])       # same fp32 operations in the same order: bit-identical


@pytest.mark.parametrize("shape", [(12, 128, 128), (1, 1, 1), (3, 5, 37), (2, 9, 1000), (1, 300, 6)])
def test_softmax_parity_records(shape):
    spec = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(*shape, scale=0.125), 1, "softmax", "bert")
    a = W.make_inputs(spec, 35)
    a["x"] = a["x"] * 6.0
    ref = util.oracle_ref(spec, a)
    for bx, by, vw in ((32, 4, 1), (8, 16, 4), (1, 32, 1), (16, 3, 2), (4, 64, 4)):
        run_spec(spec, B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=bx, block_y=by, vec_width=vw), a, ref, ref_elem=ref)


def test_split_k_is_bit_reproducible():
    spec = W._dense(128, 3072, 768)
    a = W.make_inputs(spec, 36)
    for sk in (8, 16):        # cluster reduction through distributed shared memory; workspace + last-arriving split
        r = tc(tile_n=128, tile_k=32, stages=4, split_k=sk, mma_m_axis=1)
        y1 = run_spec(spec, r, a)
        y2 = run_spec(spec, r, a)
        np.testing.assert_array_equal(y1, y2)


def test_run_requires_apply_and_pointers():
    spec = W._dense(8, 16, 8)
    wl = spec.workload()
    a = W.make_inputs(spec, 37)
    t, tt = W.device_tensors(spec, a)
    assert B.lib().tt_run(wl.handle, ctypes.byref(tt), None) == B.TT_ERR_NOT_APPLIED
    wl.apply(wl.default_schedule())
    bad = B.tensors(t["x"], t["w"], None, None, t["y"])
    assert B.lib().tt_run(wl.handle, ctypes.byref(bad), None) == B.TT_ERR_INVALID_ARG
    # an invalid record leaves the applied one in force
    st, _ = wl.try_apply(tc(stages=0))
    assert st == B.TT_ERR_INVALID_SCHEDULE
    wl.run(tt)
    assert util.rel_l2(t["y"].cpu().numpy(), util.oracle_ref(spec, a)) <= util.TOL_TF32


def test_run_host_matches_oracle():
    import torch
    spec = W._conv(16, 14, 32, 3, 1, 1)
    a = W.make_inputs(spec, 38)
    wl = spec.workload()
    wl.apply(tc(tile_n=64, tile_k=32, stages=3))
    host = {k: (None if v is None else torch.from_numpy(v).pin_memory()) for k, v in a.items()}
    y = torch.empty(W.tensor_shapes(spec)[4], dtype=torch.float32).pin_memory()
    up, down = wl.run_host(B.tensors(host["x"], host["w"], host["bias"], None, y))
    assert up == 4 * (a["x"].size + a["w"].size + a["bias"].size) and down == 4 * y.numel()
    assert util.rel_l2(y.numpy(), util.oracle_ref(spec, a)) <= util.TOL_TF32


def test_run_host_async_on_several_streams_matches_oracle():
    """tt_run_host_async: several workloads enqueued on different streams (each workload always on its own), twice
    each, nothing synchronised in between; after tt_workload_status every output equals the oracle's."""
    import torch
    specs = [W._conv(16, 14, 32, 3, 1, 1), W._dw(24, 28, 1), W._dense(8, 96, 40), W._conv(32, 14, 64, 1, 1, 0)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    jobs = []
    for i, spec in enumerate(specs):
        a = W.make_inputs(spec, 60 + i)
        wl = spec.workload()
        wl.apply(wl.default_schedule())
        host = {k: (None if v is None else torch.from_numpy(v).pin_memory()) for k, v in a.items()}
        y = torch.full(W.tensor_shapes(spec)[4], float("nan"), dtype=torch.float32).pin_memory()
        jobs.append((spec, a, wl, host, y, streams[i % len(streams)]))
    torch.cuda.synchronize()
    for _ in range(2):
        for spec, a, wl, host, y, st in jobs:
            up, down = wl.run_host_async(B.tensors(host["x"], host["w"], host["bias"], None, y), st)
            assert down == 4 * y.numel() and up > 0
    for spec, a, wl, host, y, st in jobs:
        assert wl.status(st) == B.TT_OK                  # synchronises that workload's stream
        assert util.rel_l2(y.numpy(), util.oracle_ref(spec, a)) <= util.tolerance(spec.op), spec.name
        wl.close()


def test_timing_and_grid_tuner_smoke():
    spec = W._conv(32, 14, 64, 3, 1, 1)
    a = W.make_inputs(spec, 39)
    wl = spec.workload()
    t, tt = W.device_tensors(spec, a)
    wl.apply(wl.default_schedule())
    o = B.tt_timing_opts()
    o.batches, o.warmup_batches, o.min_batch_us = 4, 1, 50
    tm = wl.time(tt, o)
    assert 0 < tm.min_us <= tm.median_us <= tm.max_us and tm.batches == 4
    o.use_graph = 1
    tg = wl.time([tt, tt], o)
    assert tg.median_us > 0
    best, tried = wl.grid_tune(tt, o, level=0, top_k=3)
    assert tried > 10 and 1 <= len(best) <= 3
    assert best[0][1] <= best[-1][1]
    assert best[0][0].origin_op == B.TT_OP_CONV2D and best[0][0].origin.c == 32
    wl.run(tt)                                     # the best record is left applied
    assert util.rel_l2(t["y"].cpu().numpy(), util.oracle_ref(spec, a)) <= util.TOL_TF32


@pytest.mark.parametrize("spec,start", [
    (W._conv(128, 28, 128, 3, 1, 1), tc(tile_n=32, tile_k=16, stages=2, split_k=1, mma_m_axis=2)),
    (W._dw(96, 56, 1), B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=1, block_y=2, block_x=8, items_per_thread=1, vec_width=1,
                                     threads=32, unroll=0)),
], ids=lambda v: getattr(v, "name", None) or "start")
def test_refining_a_transferred_record_never_loses_time_and_stays_correct(spec, start):
    """tt_refine: greedy one-field-at-a-time descent from a (deliberately poor) transferred record.  The result is at
    least as fast as the start by the search's own timings, is left applied, and computes what the oracle does."""
    a = W.make_inputs(spec, 41)
    wl = spec.workload()
    t, tt = W.device_tensors(spec, a)
    o = B.tt_timing_opts()
    o.batches, o.warmup_batches, o.min_batch_us, o.use_graph = 5, 1, 100, 1
    best, best_us, start_us, timed = wl.refine(tt, start, o, max_rounds=3, min_gain=0.02)
    assert 0 < best_us <= start_us and timed >= 2
    assert wl.check(best)[0] == B.TT_OK
    if best_us < start_us:                          # a move was made: the record differs from the (legalised) start
        assert best.as_dict() != wl.check(start)[1].legal.as_dict()
    t["y"].fill_(float("nan"))
    wl.run(tt)                                      # the best record is left applied
    assert wl.status() == B.TT_OK
    assert util.rel_l2(t["y"].cpu().numpy(), util.oracle_ref(spec, a)) <= util.tolerance(spec.op)
    wl.close()


def _model_parity(model, seed, recs):
    specs = W.MODELS[model]()
    for i, spec in enumerate(specs):
        a = W.make_inputs(spec, seed, i)
        ref = util.oracle_ref(spec, a)
        re = elem_ref(spec, a, ref)
        rr = [spec.workload().default_schedule()] + (recs if spec.op in (B.TT_OP_CONV2D, B.TT_OP_DENSE, B.TT_OP_BATCH_MATMUL) else [])
        for r in rr:
            run_spec(spec, r, a, ref, ref_elem=re)


def test_resnet18_full_size_every_kernel():
    _model_parity("resnet18", 2, [tc(tile_n=64, tile_k=64, stages=3, split_k=4, mma_m_axis=2),
                                  tc(tile_n=256, tile_k=32, stages=3, split_k=1, raster=1, mma_m_axis=1)])


def test_mobilenet_v2_full_size_every_kernel():
    _model_parity("mobilenet_v2", 4, [tc(tile_n=32, tile_k=16, stages=4, split_k=2, mma_m_axis=2)])


def test_bert_base_full_size_every_kernel():
    _model_parity("bert_base", 5, [tc(tile_n=64, tile_k=32, stages=4, split_k=3, mma_m_axis=1)])


def test_resnet50_full_size_sampled_filters():
    """Full-size kernels under three records, outputs sampled by filter: a convolution restricted to some filters is
    exactly those output channels, so the oracle computes only them (exact mode for the rel-L2 of record, truncation
    mode for the bound on every single sampled output)."""
    specs = W.resnet50()
    recs = [tc(tile_n=128, tile_k=32, stages=4, split_k=2, mma_m_axis=1),
            tc(tile_n=64, tile_k=64, stages=3, split_k=1, raster=1, mma_m_axis=2, slab_tiles=2),
            tc(tile_n=256, tile_k=32, stages=2, split_k=1, mma_m_axis=1, k_order=1)]
    for i, spec in enumerate(specs):
        a = W.make_inputs(spec, 3, i)
        ys = [run_spec(spec, rec, a) for rec in recs if spec.workload().check(rec)[0] == B.TT_OK]
        assert len(ys) >= 2, spec.name
        if spec.op == B.TT_OP_CONV2D:
            ks = sorted({0, spec.shapes.k // 3, spec.shapes.k - 1})
            geo = ((spec.shapes.stride_h,) * 2, (spec.shapes.pad_h,) * 2, spec.shapes.act)
            res = None if a["residual"] is None else np.ascontiguousarray(a["residual"][:, ks])
            sub = orc.conv2d(a["x"], a["w"][ks], a["bias"][ks], *geo, residual=res)
            sub_t = orc.conv2d(a["x"], a["w"][ks], a["bias"][ks], *geo, residual=res, mode=orc.MODE_TF32_TRUNC)
            for y in ys:
                assert util.rel_l2(y[:, ks], sub) <= util.TOL_TF32, spec.name
                assert np.abs(y[:, ks].astype(np.float64) - sub_t).max() <= ELEM_TF32 * np.abs(sub_t).max(), spec.name
        else:
            for y in ys:
                assert util.rel_l2(y, util.oracle_ref(spec, a)) <= util.TOL_TF32
        for y in ys[1:]:
            assert util.rel_l2(y, ys[0]) <= INVARIANCE_TOL, spec.name


def test_largest_dense_sampled_outputs():
    """The largest kernel of the pool sources (25088 -> 4096, 411 MB of weights), checked on sampled out-features."""
    spec = W._dense(1, 25088, 4096, B.TT_ACT_RELU)
    a = W.make_inputs(spec, 40)
    y = run_spec(spec, tc(tile_n=16, tile_k=64, stages=4, split_k=16), a)
    rows = [0, 1, 127, 128, 2047, 4000, 4095]
    sub = orc.dense(a["x"], a["w"][rows], a["bias"][rows], B.TT_ACT_RELU)
    assert util.rel_l2(y[:, rows], sub) <= util.TOL_TF32


def test_chained_kernels_on_one_stream_see_each_others_results():
    """Kernels are launched so that a kernel's set-up may overlap the tail of the one before it in the stream; every
    global access still comes after the previous kernel has finished.  A chain in which each layer reads the output of
    the layer before it (conv3x3 -> conv1x1/2 cluster split-K -> depthwise -> conv3x3 workspace split-K), launched back
    to back without any synchronisation, several times over, must equal the same chain on the oracle."""
    import torch
    layers = [
        (W._conv(16, 20, 32, 3, 1, 1), tc(tile_n=64, tile_k=32, stages=3, mma_m_axis=1)),
        (W._conv(32, 20, 48, 1, 2, 0, act=B.TT_ACT_NONE), tc(tile_n=32, tile_k=8, stages=2, split_k=4, mma_m_axis=2)),
        (W._dw(48, 10, 1), B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=4, block_x=8, items_per_thread=4, vec_width=2,
                                          threads=64, unroll=2)),
        (W._conv(48, 10, 24, 3, 1, 1, act=B.TT_ACT_RELU6), tc(tile_n=48, tile_k=16, stages=2, split_k=12, mma_m_axis=1)),
    ]
    arrays = [W.make_inputs(sp, 61, i) for i, (sp, _) in enumerate(layers)]
    # oracle chain
    x = arrays[0]["x"]
    for (sp, _), a in zip(layers, arrays):
        a = dict(a)
        a["x"] = x
        x = util.oracle_ref(sp, a)
    ref = x
    # device chain: layer i writes the buffer layer i + 1 reads
    wls, tts, keep = [], [], []
    first = cur = torch.from_numpy(arrays[0]["x"]).cuda()      # `first` keeps the chain's input alive
    for (sp, rec), a in zip(layers, arrays):
        wl = sp.workload()
        wl.apply(rec)
        t, _ = W.device_tensors(sp, a)
        assert tuple(cur.shape) == tuple(t["x"].shape)
        tts.append(B.tensors(cur, t["w"], t["bias"], None, t["y"]))
        keep.append(t)
        wls.append(wl)
        cur = t["y"]
    for _ in range(5):
        for t in keep:
            t["y"].fill_(float("nan"))
        for wl, tt in zip(wls, tts):
            wl.run(tt)
        torch.cuda.synchronize()
        y = cur.cpu().numpy()
        assert not np.isnan(y).any()
        assert util.rel_l2(y, ref) <= 3 * util.TOL_TF32      # three TF32 layers in a row
    for wl in wls:
        assert wl.status() == B.TT_OK
        wl.close()
    del first


def _sampled_filters_ok(spec, rec, seed):
    a = W.make_inputs(spec, seed)
    y = run_spec(spec, rec, a)
    ks = sorted({0, spec.shapes.k // 2 + 1, spec.shapes.k - 1})
    sub = orc.conv2d(a["x"], a["w"][ks], a["bias"][ks], (spec.shapes.stride_h,) * 2, (spec.shapes.pad_h,) * 2, spec.shapes.act)
    assert util.rel_l2(y[:, ks], sub) <= util.TOL_TF32, (spec.name, rec.short())


def test_vgg_shaped_pool_source_convs_sampled_filters():
    """The widest images of the pool sources (224 x 224: the slab rows are 228 floats, chunks of a few channels) and a
    512-channel layer whose reduction needs many slab chunks, checked on sampled filters."""
    recs = [tc(tile_n=128, tile_k=32, stages=3, mma_m_axis=1),
            tc(tile_n=256, tile_k=64, stages=2, slab_tiles=2, mma_m_axis=1),
            tc(tile_n=64, tile_k=32, stages=2, split_k=3, mma_m_axis=2)]
    for i, spec in enumerate([W._conv(3, 224, 64, 3, 1, 1), W._conv(64, 224, 64, 3, 1, 1), W._conv(512, 28, 512, 3, 1, 1)]):
        for rec in recs:
            _sampled_filters_ok(spec, rec, 70 + i)


def test_batched_kernels_of_the_saturating_size_points():
    """The batched shapes that bench.py times at saturating size, at a smaller batch, under the records it uses:
    sampled filters for the convolutions, every output for depthwise and softmax."""
    conv = W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(6, 128, 28, 28, 128, 3, 3, 1, 1, True, B.TT_ACT_RELU), 1, "conv3x3_n6_128x28")
    _sampled_filters_ok(conv, tc(tile_n=256, tile_k=32, stages=2, mma_m_axis=1), 80)
    _sampled_filters_ok(conv, tc(tile_n=128, tile_k=64, stages=2, mma_m_axis=2), 80)
    pw = W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(5, 256, 56, 56, 64, 1, 1, 1, 0, True, B.TT_ACT_RELU), 1, "conv1x1_n5_256x56")
    _sampled_filters_ok(pw, tc(tile_n=256, tile_k=32, stages=2, mma_m_axis=1), 81)
    dw = W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=3, c=144, h=56, w=56, k=144, r=3, s=3, stride_h=1, stride_w=1, pad_h=1,
                                                  pad_w=1, has_bias=1, act=B.TT_ACT_RELU6), 1, "dw_n3_144x56")
    a = W.make_inputs(dw, 82)
    ref = util.oracle_ref(dw, a)
    for rec in (B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=8, block_y=56, block_x=56, items_per_thread=8, vec_width=4,
                              threads=128, unroll=2),
                B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=16, block_x=56, items_per_thread=4, vec_width=4,
                              threads=128, unroll=4)):
        run_spec(dw, rec, a, ref)
    sm = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(12 * 8, 128, 128, 0.125), 1, "softmax_96x128x128", "bert")
    a = W.make_inputs(sm, 83)
    run_spec(sm, B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=16, block_y=4, vec_width=4), a, util.oracle_ref(sm, a))


def _random_records(family, n, seed):
    """Seeded draws from the record space the tuner walks (and a little beyond it): any legal record, however ill
    suited to the shape, must still compute the same kernel."""
    import random
    rng = random.Random(seed)
    recs = []
    for _ in range(n):
        if family == B.TT_FAMILY_GEMM_TC:
            recs.append(tc(tile_n=rng.choice([16, 32, 48, 64, 96, 128, 160, 192, 256]), tile_k=rng.choice([8, 16, 32, 64, 96, 128]),
                           stages=rng.choice([1, 2, 3, 4, 6, 8]), split_k=rng.choice([1, 1, 2, 3, 4, 5, 8, 9, 16]),
                           raster=rng.choice([0, 1]), mma_m_axis=rng.choice([0, 1, 2]), slab_tiles=rng.choice([0, 0, 1, 2, 5]),
                           acc_split=rng.choice([1, 1, 2, 4, 8]), k_order=rng.choice([0, 0, 1]),
                           persistent=rng.choice([0, 0, 1]), cta_group=rng.choice([1, 1, 2]), ctas_per_sm=rng.choice([0, 1, 2]),
                           precision=rng.choice([0, 0, 0, 1])))
        else:
            recs.append(B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=rng.choice([1, 2, 4, 8, 16, 32]), block_y=rng.choice([1, 2, 4, 7, 8, 14, 28]),
                                      block_x=rng.choice([4, 8, 16, 28, 32, 56]), items_per_thread=rng.choice([1, 2, 4, 8]),
                                      vec_width=rng.choice([1, 2, 4]), threads=rng.choice([32, 64, 128, 256, 512]),
                                      unroll=rng.choice([0, 1, 2, 4]), raster=rng.choice([0, 1]), stages=rng.choice([1, 2, 3, 4, 6])))
    return recs


@pytest.mark.parametrize("spec,n", [
    (W._conv(48, 20, 80, 3, 1, 1, name="rand_conv3x3"), 40),
    (W._conv(40, 14, 72, 3, 2, 1, act=B.TT_ACT_RELU6, name="rand_conv3x3s2"), 25),
    (W._dense(70, 300, 200, act=B.TT_ACT_GELU_ERF, name="rand_dense"), 25),
    (W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(3, 40, 56, 48, False), 1, "rand_bmm_nn", "bert"), 15),
    (W._dw(24, 28, 1), 25),
], ids=lambda v: getattr(v, "name", str(v)))
def test_a_schedule_changes_speed_never_semantics_random_records(spec, n):
    a = W.make_inputs(spec, 90)
    ref = util.oracle_ref(spec, a)
    fam = B.TT_FAMILY_DW_SIMT if spec.op == B.TT_OP_DWCONV2D else B.TT_FAMILY_GEMM_TC
    re = elem_ref(spec, a, ref)
    probe = spec.workload()
    ran = 0
    for rec in _random_records(fam, n, seed=sum(map(ord, spec.name))):
        st, _ = probe.check(rec)
        assert st in (B.TT_OK, B.TT_ERR_RESOURCE), (rec.short(), st)
        if st == B.TT_OK:
            run_spec(spec, rec, a, ref, ref_elem=re)
            ran += 1
    probe.close()
    assert ran >= n * 2 // 3


def test_sequence_length_transfer_256_tokens_under_records_tuned_on_128():
    """Section 5.4: schedules tuned for one input size of a model reused on another.  The kernels of the 256-token
    encoder run under records natively tuned on the 128-token encoder's kernels (and the reverse for one layer): every
    output within tolerance, element-wise bound included, and the evaluator's selection reproduces the oracle's argmin."""
    o = B.tt_timing_opts()
    o.batches, o.warmup_batches, o.min_batch_us, o.use_graph = 3, 1, 50, 1
    pool = []
    for j, sp in enumerate(W.bert_base()):
        a = W.make_inputs(sp, 105, j)
        wl = sp.workload()
        _, tt = W.device_tensors(sp, a)
        best, _ = wl.grid_tune(tt, o, level=0, top_k=2)
        pool += [r for r, _ in best]
        wl.close()
    assert all(r.origin.m == 128 for r in pool)
    for i, sp in enumerate(W.bert_base_256()):
        a = W.make_inputs(sp, 5, i)
        ref = util.oracle_ref(sp, a)
        re = elem_ref(sp, a, ref)
        probe = sp.workload()
        fam = probe.family()
        ran = 0
        for rec in pool:
            if rec.family != fam or probe.check(rec)[0] != B.TT_OK:
                continue
            run_spec(sp, rec, a, ref, ref_elem=re)
            ran += 1
        probe.close()
        assert ran >= 2, sp.name
    # the evaluator on the 256-token kernels with the 128-token pool: a complete, valid table
    specs = W.bert_base_256()
    arrays = [W.make_inputs(sp, 5, i) for i, sp in enumerate(specs)]
    wls = [sp.workload() for sp in specs]
    keep, tts = zip(*[W.device_tensors(sp, a) for sp, a in zip(specs, arrays)])
    opts = B.tt_tune_opts()
    opts.include_default = 1
    opts.timing = o
    res = B.transfer_tune(list(wls), list(tts), pool, opts)
    n_cols = len(pool) + 1
    flat = [v for row in res["times_us"] for v in row]
    assert res["chosen"] == orc.select(flat, len(wls), n_cols)
    assert all(c >= 0 for c in res["chosen"]) and res["pairs_timed"] >= len(wls) * 3
    for w in wls:
        w.close()


def test_bounded_wait_expires_reports_timeout_and_the_workload_recovers():
    """A wait inside the kernel that can never be satisfied (the first stage's barrier is told to expect more bytes
    than its copies deliver: every copy lands, the barrier never completes) runs into the wait limit: tt_run returns,
    the status word says TT_ERR_TIMEOUT, nothing traps, and the same workload then runs normally.  An invalid pair is
    a result of the search, which goes on (Section 4.3)."""
    import torch
    # (a) one CTA, no split; (b) twelve splits through the workspace, of which only split 0 stalls: the other eleven
    # arrive at the tile counters, which the status path has to clear again or the next run finishes tiles early;
    # (c) three splits as a thread-block cluster: split 0 gives up and sends nothing, its peers send it their bands, then
    # give up waiting for its band, and all three leave together
    for spec, rec in ((W._dense(8, 16, 8, name="stall_one_cta"), tc(tile_n=16, tile_k=16, stages=2, mma_m_axis=1)),
                      (W._dense(96, 1536, 200, name="stall_split12"), tc(tile_n=64, tile_k=32, stages=3, split_k=12, mma_m_axis=1)),
                      (W._dense(96, 768, 200, name="stall_cluster3"), tc(tile_n=64, tile_k=32, stages=3, split_k=3, mma_m_axis=2))):
        a = W.make_inputs(spec, 77)
        ref = util.oracle_ref(spec, a)
        wl = spec.workload()
        info = wl.apply(rec)
        assert info.legal.split_k == rec.split_k
        t, tt = W.device_tensors(spec, a)
        wl.set_wait_limit(2_000_000)                    # 2 ms
        wl.test_stall(64)
        t["y"].fill_(float("nan"))
        wl.run(tt)
        assert wl.status() == B.TT_ERR_TIMEOUT
        assert wl.status() == B.TT_OK                   # reading the status cleared it
        torch.cuda.synchronize()                        # the context is alive
        wl.test_stall(0)
        for _ in range(2):
            t["y"].fill_(float("nan"))
            wl.run(tt)
            assert wl.status() == B.TT_OK
            y = t["y"].cpu().numpy()
            assert not np.isnan(y).any()
            assert util.rel_l2(y, ref) <= util.TOL_TF32, spec.name
        # and after a fresh apply with the default limit
        wl.set_wait_limit(1_000_000_000)
        wl.apply(rec)
        wl.run(tt)
        assert wl.status() == B.TT_OK
        assert util.rel_l2(t["y"].cpu().numpy(), ref) <= util.TOL_TF32
        wl.close()


def _tf32_depth(steps):
    """Per node: the number of TF32 layers on the longest path that leads to it (each may add the TF32 tolerance)."""
    depth = []
    for st in steps:
        if st.spec is None:
            depth.append(0)
            continue
        d = max([depth[i] for i in (st.x, st.res, st.w_from) if i is not None])
        depth.append(d + (1 if st.spec.op in (B.TT_OP_CONV2D, B.TT_OP_DENSE, B.TT_OP_BATCH_MATMUL) else 0))
    return depth


@pytest.mark.parametrize("model,make,seed", [
    ("resnet18", W.resnet18_net, 2),
    ("mobilenet_v2", W.mobilenet_v2_net, 4),
    ("resnet50", W.resnet50_net, 3),
    ("bert_base_2_layers", lambda: W.bert_base_net(layers=2), 5),
], ids=lambda v: v if isinstance(v, str) else "")
def test_data_chained_model_pass_matches_the_oracle_chain(model, make, seed):
    """The whole model as a chain: every layer reads the buffer its producer wrote (and the skip tensor of its block),
    all launched back to back on one stream without synchronisation, three passes.  Every layer's output is compared
    with the same chain on the oracle; a layer k TF32 layers deep may be off by k times the TF32 tolerance.  Run once
    under the default records and once under a record that uses cluster split-K and the other accumulator axis."""
    import torch
    specs, steps = make()
    arrays = W.make_chain_inputs(steps, seed, init="bert" if model.startswith("bert") else "he")
    refs = util.oracle_chain(steps, arrays)
    depth = _tf32_depth(steps)
    alt = tc(tile_n=64, tile_k=32, stages=3, split_k=2, mma_m_axis=2)
    for use_alt in (False, True):
        wls = [sp.workload() for sp in specs]
        for wl in wls:
            rec = alt if use_alt and wl.family() == B.TT_FAMILY_GEMM_TC else wl.default_schedule()
            wl.apply(rec)
            wl.set_constant_weights(use_alt)              # the second pass also fetches the weights early
        bufs, tts = W.chain_device_tensors(steps, arrays)
        for _ in range(3):
            for st, b in zip(steps, bufs):
                if st.spec is not None:
                    b["y"].fill_(float("nan"))
            for st, tt in zip(steps, tts):
                if st.spec is not None:
                    wls[st.kernel].run(tt)
            torch.cuda.synchronize()
        for wl in wls:
            assert wl.status() == B.TT_OK
        for i, (st, b, ref, d) in enumerate(zip(steps, bufs, refs, depth)):
            if st.spec is None:
                continue
            y = b["y"].cpu().numpy()
            assert not np.isnan(y).any(), (model, i, st.spec.name)
            tol = max(d, 1) * util.TOL_TF32 if d else util.TOL_FP32
            assert util.rel_l2(y, ref) <= tol, (model, i, st.spec.name, d, util.rel_l2(y, ref))
        for wl in wls:
            wl.close()


@pytest.mark.parametrize("spec", [
    W._dense(700, 520, 900, act=B.TT_ACT_GELU_ERF, name="ps_dense_many_tiles"),
    W._dense(300, 64, 5000, act=B.TT_ACT_RELU, name="ps_dense_short_k"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(200, 128, 128, 64, True), 1, "ps_bmm_nt_200", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(200, 128, 64, 128, False), 1, "ps_bmm_nn_200", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(7, 150, 76, 52, False), 1, "ps_bmm_nn_ragged", "bert"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(5, 96, 28, 28, 200, 1, 1, 1, 0, True, B.TT_ACT_RELU6), 1, "ps_conv1x1_n5", "uniform"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(3, 40, 14, 14, 24, 1, 1, 1, 0, True, B.TT_ACT_NONE, True), 1, "ps_conv1x1_res", "uniform"),
], ids=lambda s: s.name)
def test_persistent_form_walks_many_tiles(spec):
    """More tiles than SMs (or many batch entries), so that every CTA of the persistent form walks several tiles, both
    accumulators are used over and over and the operand pipeline wraps across tile boundaries; ragged tails in every
    dimension.  The one-tile form under the same tile sizes gives the same values up to the fp32 summation order."""
    a = W.make_inputs(spec, 91)
    ref = util.oracle_ref(spec, a)
    re = elem_ref(spec, a, ref)
    outs = []
    probe = spec.workload()
    for rec in (tc(tile_n=16, tile_k=32, stages=4, mma_m_axis=1),
                tc(tile_n=16, tile_k=32, stages=4, persistent=1, mma_m_axis=1),
                tc(tile_n=32, tile_k=16, stages=7, persistent=1, mma_m_axis=2),
                tc(tile_n=48, tile_k=64, stages=2, persistent=1, raster=1, mma_m_axis=1),
                tc(tile_n=32, tile_k=32, stages=3, persistent=1, cta_group=2, mma_m_axis=1),
                tc(tile_n=64, tile_k=32, stages=5, persistent=1, cta_group=2, raster=1, mma_m_axis=2)):
        st, info = probe.check(rec)
        assert st == B.TT_OK
        if rec.persistent:
            assert info.legal.persistent == 1, "this kernel has the persistent form"
            assert info.grid_y == 1 and info.grid_z == 1
        outs.append(run_spec(spec, rec, a, ref, ref_elem=re))
    probe.close()
    for y in outs[1:]:
        assert util.rel_l2(y, outs[0]) <= INVARIANCE_TOL


def test_constant_weights_are_fetched_early_and_results_do_not_change():
    """With the caller's promise that the weights are constants, a dense or conv2d kernel requests their first tiles
    before it waits for the kernel in front of it.  Layers launched back to back -- each reading its predecessor's
    output, with that promise and without it -- give bit-identical results, equal to the oracle chain."""
    import torch
    layers = [(W._dense(128, 768, 768, name="cw_a"), tc(tile_n=64, tile_k=32, stages=3, split_k=8, mma_m_axis=2)),
              (W._dense(128, 768, 3072, act=B.TT_ACT_GELU_ERF, name="cw_b"), tc(tile_n=32, tile_k=128, stages=2, mma_m_axis=1)),
              (W._dense(128, 3072, 768, name="cw_c"), tc(tile_n=64, tile_k=64, stages=3, split_k=6, mma_m_axis=2)),
              (W._dense(128, 768, 768, name="cw_d"), tc(tile_n=64, tile_k=32, stages=4, persistent=1, mma_m_axis=1))]
    arrays = [W.make_inputs(sp, 95, i) for i, (sp, _) in enumerate(layers)]
    x = arrays[0]["x"]
    for (sp, _), a in zip(layers, arrays):
        a = dict(a)
        a["x"] = x
        x = util.oracle_ref(sp, a)
    ref = x
    results = []
    for promise in (False, True):
        wls, tts, keep = [], [], []
        first = cur = torch.from_numpy(arrays[0]["x"]).cuda()
        for (sp, rec), a in zip(layers, arrays):
            wl = sp.workload()
            wl.apply(rec)
            wl.set_constant_weights(promise)
            t, _ = W.device_tensors(sp, a)
            tts.append(B.tensors(cur, t["w"], t["bias"], None, t["y"]))
            keep.append(t)
            wls.append(wl)
            cur = t["y"]
        for _ in range(4):
            for t in keep:
                t["y"].fill_(float("nan"))
            for wl, tt in zip(wls, tts):
                wl.run(tt)
            torch.cuda.synchronize()
        for wl in wls:
            assert wl.status() == B.TT_OK
            wl.close()
        y = cur.cpu().numpy()
        assert util.rel_l2(y, ref) <= 4 * util.TOL_TF32
        results.append(y)
        del first
    np.testing.assert_array_equal(results[0], results[1])


@pytest.mark.parametrize("spec", [
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(20, 40, 20, 20, 72, 3, 3, 1, 1, True, B.TT_ACT_RELU), 1, "ps_tap_conv3x3_n20", "uniform"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(9, 33, 12, 16, 136, 5, 3, 1, 2, True, B.TT_ACT_RELU6), 1, "ps_tap_conv5x3_n9", "uniform"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(30, 8, 8, 8, 16, 3, 3, 1, 1, False, B.TT_ACT_NONE), 1, "ps_tap_small_n30", "uniform"),
], ids=lambda s: s.name)
def test_persistent_tap_major_convolution_walks_many_tiles(spec):
    """The tap-major reduction order in the persistent form: filter stages, the staging ring and the two pixel-major
    slab buffers all run on across tile boundaries (several tiles per CTA, one or several 32-channel blocks per tile,
    a partial last block, two filter tiles).  Same values as the one-tile form and as the stored reduction order."""
    a = W.make_inputs(spec, 92)
    ref = util.oracle_ref(spec, a)
    re = elem_ref(spec, a, ref)
    outs = []
    probe = spec.workload()
    for rec in (tc(tile_n=32, tile_k=32, stages=3, mma_m_axis=1),
                tc(tile_n=48, tile_k=32, stages=3, k_order=1, mma_m_axis=1),
                tc(tile_n=48, tile_k=32, stages=3, k_order=1, persistent=1, mma_m_axis=1),
                tc(tile_n=16, tile_k=96, stages=2, k_order=1, persistent=1, raster=1, mma_m_axis=1),
                tc(tile_n=96, tile_k=32, stages=6, k_order=1, persistent=1, mma_m_axis=1),
                tc(tile_n=256, tile_k=64, stages=2, k_order=1, persistent=1, mma_m_axis=1)):
        st, info = probe.check(rec)
        assert st == B.TT_OK
        if rec.persistent:
            assert info.legal.persistent == 1 and info.legal.k_order == 1
        outs.append(run_spec(spec, rec, a, ref, ref_elem=re))
    probe.close()
    for y in outs[1:]:
        assert util.rel_l2(y, outs[0]) <= INVARIANCE_TOL


def test_subsampled_evaluator_skips_what_the_rule_says_and_keeps_a_valid_choice():
    """Pool sub-sampling: the seeded subset is evaluated first; with a bar nothing can clear (100 % gain) every record is
    still evaluated, with a bar everything clears (a negative gain) only the subset is, the rest is marked TT_SKIPPED,
    and the chosen record is the argmin over what was evaluated."""
    spec = W._conv(32, 14, 64, 3, 1, 1)
    a = W.make_inputs(spec, 44)
    wl = spec.workload()
    t, tt = W.device_tensors(spec, a)
    pool = [tc(tile_n=tn, tile_k=tk, stages=st) for tn in (32, 64, 128) for tk in (16, 32) for st in (2, 3)]   # 12 records
    o = B.tt_tune_opts()
    o.include_default = 1
    o.timing.warmup_batches, o.timing.batches, o.timing.min_batch_us, o.timing.use_graph = 1, 3, 50, 1
    o.subsample_percent, o.subsample_seed = 25, 11
    first = B.pool_subsample(len(pool), 3, 11)
    assert first == orc.pool_subsample(len(pool), 3, 11)
    o.subsample_gain_percent = 100                       # unreachable: the whole pool gets evaluated
    res = B.transfer_tune([wl], [tt], pool, o)
    assert res["pairs_skipped"] == 0 and res["pairs_timed"] == 13
    o.subsample_gain_percent = -1000                     # any valid subset record ends the search
    res = B.transfer_tune([wl], [tt], pool, o)
    st = res["status"][0]
    evaluated = {0} | {f + 1 for f in first}
    assert {j for j, s in enumerate(st) if s == B.TT_OK} == evaluated
    assert all(st[j] == B.TT_SKIPPED and res["times_us"][0][j] == -1.0 for j in range(13) if j not in evaluated)
    assert res["pairs_skipped"] == 9 and res["pairs_timed"] == 4
    assert res["chosen"] == orc.select(res["times_us"][0], 1, 13) and res["chosen"][0] in evaluated
    wl.run(tt)                                           # the chosen record is left applied
    assert util.rel_l2(t["y"].cpu().numpy(), util.oracle_ref(spec, a)) <= util.TOL_TF32
    wl.close()


@pytest.mark.parametrize("model,make,seed", [("resnet18", W.resnet18_net, 2), ("bert_base", lambda: W.bert_base_net(layers=2), 5)])
def test_chain_on_several_streams_matches_the_oracle_chain(model, make, seed):
    """The same chain with layers that do not depend on one another on side streams (the attention projections, a
    block's downsample beside its first convolution), enqueued directly and replayed as one captured graph: every
    layer's output against the oracle chain.  The projections share one workload object and run beside one another."""
    import torch
    specs, steps = make()
    arrays = W.make_chain_inputs(steps, seed, init="bert" if model.startswith("bert") else "he")
    refs = util.oracle_chain(steps, arrays)
    depth = _tf32_depth(steps)
    wls = [sp.workload() for sp in specs]
    rec = tc(tile_n=64, tile_k=64, stages=2, split_k=4, mma_m_axis=2)
    for wl in wls:
        wl.apply(rec if wl.family() == B.TT_FAMILY_GEMM_TC else wl.default_schedule())
        wl.set_constant_weights(True)
    bufs, tts = W.chain_device_tensors(steps, arrays)
    plan = W.chain_lanes(steps, max_lanes=4)
    assert len({pl[0] for pl in plan if pl}) == 4
    side = [torch.cuda.Stream() for _ in range(3)]

    def clear():
        for st, b in zip(steps, bufs):
            if st.spec is not None:
                b["y"].fill_(float("nan"))

    def check(what):
        for wl in wls:
            assert wl.status() == B.TT_OK
        for i, (st, b, ref, d) in enumerate(zip(steps, bufs, refs, depth)):
            if st.spec is None:
                continue
            y = b["y"].cpu().numpy()
            assert not np.isnan(y).any(), (what, model, i, st.spec.name)
            tol = max(d, 1) * util.TOL_TF32 if d else util.TOL_FP32
            assert util.rel_l2(y, ref) <= tol, (what, model, i, st.spec.name, d, util.rel_l2(y, ref))

    main = torch.cuda.Stream()
    with torch.cuda.stream(main):
        for _ in range(2):
            clear()
            W.run_chain(wls, steps, tts, plan, [main] + side)
        main.synchronize()
    torch.cuda.synchronize()
    check("direct")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        W.run_chain(wls, steps, tts, plan, [torch.cuda.current_stream()] + side)
    for _ in range(3):
        clear()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
    check("graph")
    for wl in wls:
        wl.close()


@pytest.mark.parametrize("spec", [
    W._dense(300, 1024, 520, act=B.TT_ACT_GELU_ERF, name="x3_dense"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(6, 200, 136, 256, True), 1, "x3_bmm_nt", "bert"),
])
def test_compensated_products_come_within_fp32_accumulation_of_the_exact_result(spec):
    """precision = 1: what the tensor core drops of each operand (everything below TF32's ten mantissa bits) is fed
    back through two more products per step, so the result must sit far inside the TF32 tolerance: at least twenty
    times closer to the exact oracle than the same record with plain TF32 products, and within 2e-5 in rel-L2 (fp32
    accumulation of up to 1024 terms plus the dropped second-order term); under a split-K cluster too."""
    a = W.make_inputs(spec, 91)
    ref = util.oracle_ref(spec, a)
    for kw in (dict(tile_n=64, tile_k=32, stages=3, mma_m_axis=1), dict(tile_n=128, tile_k=64, stages=2, split_k=2, mma_m_axis=2)):
        y0 = run_spec(spec, tc(**kw), a, ref)
        y3 = run_spec(spec, tc(precision=1, **kw), a, ref)
        e0, e3 = util.rel_l2(y0, ref), util.rel_l2(y3, ref)
        assert e3 <= 2e-5 and e3 * 20 <= e0, (spec.name, kw, e0, e3)


@pytest.mark.parametrize("tile_n,tile_k,stages", [(32, 64, 2), (64, 64, 2), (128, 32, 2), (176, 32, 2), (32, 128, 1), (16, 64, 2), (64, 16, 4), (32, 8, 4)])
def test_compensated_products_over_an_odd_number_of_tiles(tile_n, tile_k, stages):
    """Long reductions of every depth and swizzle.  The first five multiply A from tensor memory: with stages of 64 there are fewer buffers
    than stages (3 for 4 with tiles of 32 columns), with 128 one for two, which then wrap at different places."""
    spec = W._dense(150, 1060, 200, init="bert", name="x3_1060")
    a = W.make_inputs(spec, 92)
    ref = util.oracle_ref(spec, a)
    for axis in (1, 2):
        if tile_n > 160 and axis == 2:
            continue                                     # (wider than the layer has rows)
        y = run_spec(spec, tc(tile_n=tile_n, tile_k=tile_k, stages=stages, mma_m_axis=axis, precision=1), a, ref, mode=B.TT_MODE_STRICT)
        assert util.rel_l2(y, ref) <= 2e-5, (axis, util.rel_l2(y, ref))


@pytest.mark.parametrize("rows,cols", [(70003, 33), (70001, 186), (300, 330), (299, 94), (303, 1174), (64000, 187)])
def test_softmax_chunks_of_two_four_and_eight_rows(rows, cols):
    """Both sides of the rule for a warp's rows, by few and many lanes; the last rows fill no whole chunk."""
    spec = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(1, rows, cols, scale=0.125), 1, f"softmax_{rows}x{cols}", "bert")
    a = W.make_inputs(spec, 13)
    ref = util.oracle_ref(spec, a)
    for bx in (4, 16, 32):
        run_spec(spec, B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=bx, block_y=8, vec_width=1), a, ref, ref_elem=ref)


@pytest.mark.parametrize("k", [29, 31, 33])
def test_ragged_rows_beside_a_gathered_operand(k):
    """NN products whose x has ragged rows, on both sides of the reduction from which they come by TMA."""
    spec = W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(5, 45, 30, k, False), 1, f"nn_{k}", "bert")
    a = W.make_inputs(spec, 18)
    ref = util.oracle_ref(spec, a)
    for axis in (1, 2):
        run_spec(spec, tc(tile_n=32, tile_k=32, stages=2, mma_m_axis=axis), a, ref, ref_elem=elem_ref(spec, a, ref))


@pytest.mark.parametrize("tile_n", [96, 160, 224])
def test_pairs_of_ctas_with_tiles_between_the_powers_of_two(tile_n):
    """Widths that the columns of a persistent record are dealt in: a CTA of the pair loads 48, 80 or 112 rows of B.  Ragged rows and
    columns, several tiles a pair."""
    spec = W._dense(1301, 68, 2500, act=B.TT_ACT_RELU, name="pairs")
    a = W.make_inputs(spec, 93)
    ref = util.oracle_ref(spec, a)
    for stages in (2, 4):
        run_spec(spec, tc(tile_n=tile_n, tile_k=32, stages=stages, mma_m_axis=1, persistent=1, cta_group=2), a, ref, mode=B.TT_MODE_STRICT, ref_elem=elem_ref(spec, a, ref))


@pytest.mark.parametrize("rows,cols", [(60001, 33), (150003, 5), (40001, 61), (19002, 198), (20003, 1174)])
def test_softmax_of_many_short_ragged_rows(rows, cols):
    """Rows that come several passes at a time, and even ones in chunks of two rows; the last rows fill no whole chunk."""
    spec = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(1, rows, cols, scale=0.125), 1, f"softmax_{rows}x{cols}", "bert")
    a = W.make_inputs(spec, 12)
    ref = util.oracle_ref(spec, a)
    for bx in (8, 32):
        run_spec(spec, B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=bx, block_y=8, vec_width=1), a, ref, ref_elem=ref)


@pytest.mark.parametrize("cols", [1, 2, 3, 5, 31, 33, 63, 127, 129, 197, 255, 257, 1023, 1025, 2045, 2047, 2049, 2051])
def test_softmax_ragged_rows(cols):
    """Rows that start at every offset inside a 16-byte group, up to the longest row that stays in registers and just
    beyond it; lanes per row from 1 to 32; the last rows fill no whole chunk."""
    spec = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(5, 7, cols, scale=0.125), 1, f"softmax_35x{cols}", "bert")
    a = W.make_inputs(spec, 11)
    ref = util.oracle_ref(spec, a)
    for bx in (1, 4, 16, 32):
        run_spec(spec, B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=bx, block_y=8, vec_width=4), a, ref, ref_elem=ref)


@pytest.mark.parametrize("spec", [
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(40, 20, 14, 14, 200, 1, 1, 1, 0, True, B.TT_ACT_RELU, True), 1, "mn_conv1x1_res_n40", "uniform"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(3, 33, 6, 6, 17, 1, 1, 1, 0, True, B.TT_ACT_RELU6, True), 1, "mn_conv1x1_c33", "uniform"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(5, 70, 132, 36, False), 1, "mn_bmm_nn_ragged", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(3, 130, 44, 35, False), 1, "mn_bmm_nn_gathered_a", "bert"),
], ids=lambda s: s.name)
def test_mn_major_operands_and_tma_read_out(spec):
    """Operands whose row index is the contiguous one, multiplied as they lie: boxes of 32 rows with tails in rows and in
    K, tiles of less than a box, split-K through a cluster and through the workspace, several accumulators, the residual
    read ahead through the read-out's ring (several tiles per CTA, both output orders, tiles that are no whole blocks)."""
    a = W.make_inputs(spec, 93)
    ref = util.oracle_ref(spec, a)
    re = elem_ref(spec, a, ref)
    probe = spec.workload()
    recs = [tc(tile_n=tn, tile_k=tk, stages=st, mma_m_axis=ax, persistent=ps, split_k=sk, acc_split=acc, slab_tiles=sl)
            for tn, tk, st, ax, ps, sk, acc, sl in (
                (16, 8, 2, 1, 0, 1, 1, 0), (48, 16, 3, 1, 0, 3, 1, 0), (64, 32, 2, 2, 0, 2, 2, 0), (256, 64, 1, 1, 0, 1, 1, 0),
                (32, 8, 2, 2, 0, 12, 1, 0), (32, 32, 2, 1, 1, 1, 1, 0), (64, 16, 8, 1, 1, 1, 1, 2), (256, 32, 2, 1, 1, 1, 1, 0),
                (48, 32, 2, 1, 1, 1, 1, 3), (32, 64, 2, 2, 1, 1, 1, 0), (160, 32, 1, 2, 1, 1, 1, 1))]
    for rec in recs:
        assert probe.check(rec)[0] == B.TT_OK
        run_spec(spec, rec, a, ref, ref_elem=re)
    probe.close()


@pytest.mark.parametrize("m, k, n, tn, tk, sk", [(512, 1000, 1100, 64, 64, 4), (300, 200, 2000, 32, 128, 2), (1030, 520, 700, 16, 32, 3),
                                                   (129, 68, 513, 128, 64, 1), (515, 260, 1030, 128, 128, 2), (700, 2052, 300, 64, 64, 8)])
def test_compensated_tiles_of_twice_the_columns(m, k, n, tn, tk, sk):
    """Compensated products whose tile runs with twice the record's columns, or whose one stage runs as several: remainders of
    rows, columns and of the reduction, split over a cluster, on either axis."""
    sp = W.Spec(B.TT_OP_DENSE, B.dense_shapes(m, k, n, True, B.TT_ACT_RELU), 1, "x3_wide", "bert")
    a = W.make_inputs(sp, 97)
    ref = util.oracle_ref(sp, a)
    re = elem_ref(sp, a, ref)
    for ax in (1, 2):
        run_spec(sp, tc(tile_n=tn, tile_k=tk, stages=2, mma_m_axis=ax, split_k=sk, precision=1), a, ref, ref_elem=re)


@pytest.mark.parametrize("n, c, h, w, r, stride, act, bias, off", [
    (5, 301, 14, 14, 5, 1, B.TT_ACT_RELU6, True, 0), (29, 190, 7, 7, 3, 1, B.TT_ACT_NONE, False, 0), (80, 47, 17, 18, 3, 2, B.TT_ACT_RELU, True, 0),
    (37, 33, 31, 30, 5, 2, B.TT_ACT_GELU_ERF, True, 0), (3, 9, 111, 109, 3, 1, B.TT_ACT_RELU, True, 0), (2, 11, 130, 131, 5, 1, B.TT_ACT_NONE, True, 0),
    (3, 53, 5, 342, 3, 1, B.TT_ACT_RELU, True, 0), (9, 65, 33, 45, 5, 1, B.TT_ACT_RELU6, True, 1), (4, 403, 13, 14, 3, 1, B.TT_ACT_RELU6, True, 3),
    (1, 131200, 2, 1, 3, 1, B.TT_ACT_RELU, True, 0), (3, 70, 253, 37, 3, 2, B.TT_ACT_NONE, False, 2), (3, 17, 150, 150, 5, 2, B.TT_ACT_NONE, False, 0)])
def test_depthwise_rows_staged_as_runs(n, c, h, w, r, stride, act, bias, off):
    """A batch of images whose rows are no 16-byte multiples: odd and even rows, planes and bands of planes, groups of channels
    with a remainder, a tensor that ends inside 16 bytes, an input that starts inside them.  Each output is bounded against the
    oracle, and the first and the last image equal, bit for bit, what the register-window form makes of them alone."""
    def spec_for(m):
        return W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=m, c=c, h=h, w=w, k=c, r=r, s=r, stride_h=stride, stride_w=stride, pad_h=r // 2,
                                                      pad_w=r // 2, has_bias=int(bias), act=act), 1, "dw_runs", "uniform")
    spec = spec_for(n)
    a = W.make_inputs(spec, 96)
    ref = util.oracle_ref(spec, a)
    rec = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=8, block_x=32, items_per_thread=4, vec_width=4, threads=128, unroll=2)
    probe = spec.workload()
    legal = probe.check(rec)[1].legal                    # (rows of more than 256 outputs have no such form)
    assert legal.raster == ((w - 1) // stride + 1 <= 256), legal.short()
    probe.close()
    y = run_spec(spec, rec, a, ref, ref_elem=ref)
    if off:
        t, _ = W.device_tensors(spec, a)
        import torch
        x = torch.empty(t["x"].numel() + 4, device="cuda")[off:off + t["x"].numel()].view(t["x"].shape).copy_(t["x"])
        wl = spec.workload()
        wl.apply(rec)
        wl.run(B.tensors(x, t["w"], t["bias"], t["residual"], t["y"]))
        assert wl.status() == B.TT_OK
        np.testing.assert_array_equal(t["y"].cpu().numpy(), y)
        wl.close()
    one = spec_for(1)
    for i in {0, n - 1}:
        alone = dict(a, x=np.ascontiguousarray(a["x"][i:i + 1]))
        if n > 1:
            np.testing.assert_array_equal(run_spec(one, rec, alone)[0], y[i])


@pytest.mark.parametrize("k", [8, 22, 72, 136, 263, 1032])
def test_ring_deeper_than_the_record(k):
    """One CTA per SM: the ring takes as many stages as fit, from one up to the kernel's limit, a CTA's whole reduction or a
    part of it, beside a gather table, a compensated operand pair and a cluster's reduction."""
    sp = W.Spec(B.TT_OP_DENSE, B.dense_shapes(37, k, 50, True, B.TT_ACT_RELU), 1, "ring_k%d" % k, "bert")
    a = W.make_inputs(sp, 95)
    ref = util.oracle_ref(sp, a)
    re = elem_ref(sp, a, ref)
    for tn, tk, st, ax, sk, x3 in ((16, 8, 1, 1, 1, 0), (16, 32, 2, 2, 1, 1), (32, 8, 2, 1, 4, 0), (128, 64, 1, 2, 2, 0), (256, 32, 3, 1, 1, 0)):
        run_spec(sp, tc(tile_n=tn, tile_k=tk, stages=st, mma_m_axis=ax, split_k=sk, precision=x3), a, ref, ref_elem=re)


@pytest.mark.parametrize("shape", [
    # n, c, h, w, k, r, s, stride_h, stride_w, pad_h, pad_w, residual
    (3, 33, 7, 7, 40, 3, 3, 1, 1, 1, 1, True), (5, 8, 9, 5, 130, 3, 3, 2, 2, 1, 1, False), (2, 64, 14, 14, 16, 1, 1, 2, 2, 0, 0, True),
    (2, 40, 11, 13, 24, 5, 3, 2, 1, 2, 0, False), (4, 16, 6, 6, 20, 2, 4, 3, 2, 0, 3, True), (2, 70, 23, 8, 150, 7, 7, 1, 1, 3, 3, False),
    (160, 32, 8, 8, 136, 3, 3, 1, 1, 1, 1, True), (70, 40, 9, 9, 40, 3, 3, 2, 2, 1, 1, True), (1, 96, 12, 12, 48, 3, 3, 1, 1, 1, 1, True),
], ids=lambda s: "x".join(map(str, s)))
def test_tap_major_convolutions_of_every_layout(shape):
    """The tap-major order over padded-linear positions of a whole batch: rows that are no 16-byte multiples, tiles that
    cross rows and images, strides (one sub-image per parity class), unequal padding, partial channel blocks, the skip
    tensor, channel blocks shared by a cluster, and tiles that CTAs walk with two accumulators."""
    n, c, h, w, k, r, s, sh, sw, ph, pw, res = shape
    sp = W.Spec(B.TT_OP_CONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=k, r=r, s=s, stride_h=sh, stride_w=sw, pad_h=ph, pad_w=pw, has_bias=1,
                                              has_residual=int(res), act=B.TT_ACT_RELU), 1, "tap", "uniform")
    a = W.make_inputs(sp, 94)
    ref = util.oracle_ref(sp, a)
    re = elem_ref(sp, a, ref)
    probe = sp.workload()
    for tn, tk, st, ps in ((16, 32, 4, 0), (224, 96, 2, 0), (128, 32, 2, 1), (64, 128, 8, 0)):
        rec = tc(tile_n=tn, tile_k=tk, stages=st, k_order=1, persistent=ps, mma_m_axis=1)
        stat, info = probe.check(rec)
        assert stat == B.TT_OK and info.legal.k_order == 1
        run_spec(sp, rec, a, ref, ref_elem=re)
    probe.close()


@pytest.mark.parametrize("cg", [1, 2, 3, 5])
def test_tap_major_records_run_as_written_in_strict_mode(cg):
    """Columns, taps in flight and the CTAs that share a tile's channel blocks (5 blocks, the last one partial) as the record has
    them, where legalise mode would lay them out for the kernel's size."""
    sp = W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(3, 140, 9, 9, 150, 3, 3, 1, 1, True, B.TT_ACT_RELU, True), 1, "tap_strict", "uniform")
    a = W.make_inputs(sp, 98)
    ref = util.oracle_ref(sp, a)
    re = elem_ref(sp, a, ref)
    for tn, tk, st in ((32, 32, 1), (112, 96, 2)):
        rec = tc(tile_n=tn, tile_k=tk, stages=st, k_order=1, mma_m_axis=1, cta_group=cg)
        probe = sp.workload()
        status, info = probe.check(rec, mode=B.TT_MODE_STRICT)
        assert status == B.TT_OK and (info.legal.tile_n, info.legal.stages, info.grid_y) == (tn, st, cg)
        probe.close()
        run_spec(sp, rec, a, ref, mode=B.TT_MODE_STRICT, ref_elem=re)


@pytest.mark.parametrize("shape, kw", [
    ((9, 50, 20, 28, 5, 1), dict(tile_m=7, block_y=20, block_x=28, threads=256, unroll=7, stages=3)),      # 8 groups, the last of one channel
    ((9, 50, 20, 28, 5, 2), dict(tile_m=12, block_y=5, block_x=8, threads=256, unroll=7, stages=2)),       # more threads than strips
    ((5, 33, 17, 36, 3, 1), dict(tile_m=16, block_y=17, block_x=36, threads=64, unroll=4, stages=2)),      # two groups of 16 and one of 1
], ids=str)
def test_box_staged_depthwise_records_run_as_written_in_strict_mode(shape, kw):
    n, c, h, w, r, st = shape
    sp = W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=c, r=r, s=r, stride_h=st, stride_w=st, pad_h=r // 2, pad_w=r // 2, has_bias=1,
                                                act=B.TT_ACT_RELU6), 1, "dw_strict", "uniform")
    a = W.make_inputs(sp, 99)
    ref = util.oracle_ref(sp, a)
    q = (w - 1) // st + 1
    rec = B.make_record(B.TT_FAMILY_DW_SIMT, items_per_thread=4, vec_width=4 if q % 4 == 0 else 2 if q % 2 == 0 else 1, raster=1, **kw)
    y = run_spec(sp, rec, a, ref, mode=B.TT_MODE_STRICT, ref_elem=ref)
    np.testing.assert_array_equal(run_spec(sp, rec, a), y)


@pytest.mark.parametrize("cols", [577, 637, 865, 1023, 1025, 1028, 1535, 2047, 2048, 2081])
def test_softmax_rows_under_the_largest_blocks(cols):
    """1024 threads of lanes that keep up to 16 groups or 65 values of a row each: more registers than an SM has."""
    spec = W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(3, 23, cols, scale=0.125), 1, f"softmax_69x{cols}", "bert")
    a = W.make_inputs(spec, 12)
    ref = util.oracle_ref(spec, a)
    for bx in (8, 32):
        rec = B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=bx, block_y=1024 // bx, vec_width=4 if cols % 4 == 0 else 1)
        for mode in (B.TT_MODE_LEGALISE, B.TT_MODE_STRICT):
            run_spec(spec, rec, a, ref, mode=mode, ref_elem=ref)


@pytest.mark.parametrize("spec, operand", [
    (W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(3, 37, 14, 14, 70, 1, 1, 1, 0, True, B.TT_ACT_RELU, True), 1, "off_conv1x1_14", "uniform"), "x"),
    (W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(2, 64, 6, 6, 40, 1, 1, 1, 0, True, B.TT_ACT_RELU6), 1, "off_conv1x1_6", "uniform"), "x"),
    (W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(4, 70, 132, 36, False), 1, "off_bmm_nn", "bert"), "w"),
    (W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(3, 130, 44, 35, False), 1, "off_bmm_nn_odd_k", "bert"), "w"),
], ids=lambda v: v.name if isinstance(v, W.Spec) else v)
def test_row_contiguous_operands_that_start_anywhere(spec, operand):
    """A pointwise convolution's image, or an NN product's second operand, that starts inside a 16-byte group: no TMA box can fetch
    it, the one-tile form gathers it."""
    import torch
    a = W.make_inputs(spec, 92)
    ref = util.oracle_ref(spec, a)
    re = elem_ref(spec, a, ref)
    for off, rec in ((1, tc(tile_n=16, tile_k=8, stages=2, mma_m_axis=1)), (2, tc(tile_n=64, tile_k=32, stages=3, mma_m_axis=2)),
                     (3, tc(tile_n=48, tile_k=32, stages=2, split_k=2, mma_m_axis=1, acc_split=2)), (1, tc(tile_n=32, tile_k=8, stages=4, split_k=4, mma_m_axis=2))):
        wl = spec.workload()
        wl.apply(rec)
        wl.set_constant_weights(True)
        t, _ = W.device_tensors(spec, a)
        t["y"], buf = guarded_output(spec)
        n = t[operand].numel()
        t[operand] = torch.empty(n + 4, device="cuda")[off:off + n].view(t[operand].shape).copy_(t[operand])
        wl.run(B.tensors(t["x"], t["w"], t["bias"], t["residual"], t["y"]))
        assert wl.status() == B.TT_OK and guards_intact(buf)
        y = t["y"].cpu().numpy()
        assert util.rel_l2(y, ref) <= util.TOL_TF32, (spec.name, rec.short())
        assert float(np.abs(y.astype(np.float64) - re).max()) <= ELEM_TF32 * float(np.abs(re).max())
        wl.close()


FIRST_CALLS = """
import threading
import torch
from paper_2201_05587_b200 import binding as B
from paper_2201_05587_b200 import workloads as W
tc = lambda **kw: B.make_record(B.TT_FAMILY_GEMM_TC, **kw)
dw = lambda **kw: B.make_record(B.TT_FAMILY_DW_SIMT, items_per_thread=4, vec_width=4, **kw)
def dwc(n, hw): return W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=n, c=32, h=hw, w=hw, k=32, r=3, s=3, stride_h=1, stride_w=1, pad_h=1, pad_w=1, has_bias=1), 1, "dw")
kinds = [(W._dense(300, 256, 400), tc(tile_n=128, tile_k=32, stages=3, mma_m_axis=1, persistent=1)), (W._dense(300, 256, 400), tc(tile_n=64, tile_k=32, stages=2, mma_m_axis=1)),
         (W._dense(64, 512, 200), tc(tile_n=64, tile_k=32, stages=2, split_k=4, mma_m_axis=1)), (W._conv(32, 28, 64, 3, 1, 1), tc(tile_n=64, tile_k=32, stages=2, k_order=1, mma_m_axis=1)),
         (dwc(4, 28), dw(tile_m=4, block_y=28, block_x=28, threads=128, unroll=2, raster=1, stages=2)), (dwc(2, 20), dw(tile_m=8, block_y=20, block_x=20, threads=128, unroll=0)),
         (W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(4, 100, 197, 0.1), 1, "rows"), B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=16, block_y=4, vec_width=1))]
torch.zeros(1, device="cuda")
gate, out = threading.Barrier(2 * len(kinds)), [None] * (2 * len(kinds))
def work(i):
    try:
        sp, rec = kinds[i % len(kinds)]
        wl = sp.workload()
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            t, tt = W.device_tensors(sp, W.make_inputs(sp, 7))
            t["y"].fill_(float("nan"))
            gate.wait()
            wl.apply(rec)
            wl.run(tt)
            assert wl.status() == B.TT_OK
            out[i] = t["y"].cpu()
    except BaseException as e:
        out[i] = e
        gate.abort()
threads = [threading.Thread(target=work, args=(i,)) for i in range(2 * len(kinds))]
[t.start() for t in threads]
[t.join() for t in threads]
for i in range(len(kinds)):
    for o in (out[i], out[i + len(kinds)]):
        assert torch.is_tensor(o), (kinds[i][0].name, o)
        assert not torch.isnan(o).any() and torch.equal(o, out[i]), kinds[i][0].name
print("first calls ok")
"""


def test_first_calls_of_several_threads_at_once():
    """Kernels of every form, each set up for the device by whichever thread comes first: a fresh process, all threads at once."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_CALLS], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "first calls ok" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("spec, rec", [
    (W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(2, 512, 14, 14, 512, 3, 3, 1, 1, True, B.TT_ACT_RELU), 1, "lanes_tap", "uniform"),
     tc(tile_n=64, tile_k=32, stages=4, k_order=1, mma_m_axis=1)),
    (W._dense(64, 4096, 512, name="lanes_split12"), tc(tile_n=64, tile_k=32, stages=2, split_k=12, mma_m_axis=1)),
], ids=lambda v: v.name if isinstance(v, W.Spec) else "")
def test_chain_layers_that_share_scratch_on_different_lanes(spec, rec):
    """Layers of one workload with different weights on three lanes of a chain, no wait between them: its scratch (re-packed
    filters; partial sums and counters) serves one layer at a time."""
    import torch
    arrays = [W.make_inputs(spec, 60 + i) for i in range(3)]
    refs = [util.oracle_ref(spec, a) for a in arrays]
    for constant in (False, True):
        wl = spec.workload()
        assert wl.apply(rec).workspace_bytes > 0
        wl.set_constant_weights(constant)
        ts, tts = zip(*[W.device_tensors(spec, a) for a in arrays])
        steps = [type("Node", (), {"kernel": 0})() for _ in arrays]
        streams = [torch.cuda.current_stream()] + [torch.cuda.Stream() for _ in range(2)]
        for _ in range(5):
            for t in ts:
                t["y"].fill_(float("nan"))
            W.run_chain([wl], steps, list(tts), [(0, ()), (1, ()), (2, ())], streams)
            assert wl.status() == B.TT_OK
            for t, ref in zip(ts, refs):
                assert util.rel_l2(t["y"].cpu().numpy(), ref) <= util.TOL_TF32
        wl.close()


def test_repacked_filters_follow_the_promise_and_captured_passes():
    """The re-packed filters of a tap-major convolution: forgotten when the promise of constant weights is switched off, kept for
    the captured pass that reads them while other weights run, and not taken from a capture that has never run."""
    import torch
    sp = W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(2, 96, 14, 14, 200, 3, 3, 1, 1, True, B.TT_ACT_RELU), 1, "filters", "uniform")
    rec = tc(tile_n=64, tile_k=32, stages=4, k_order=1, mma_m_axis=1)
    arrays = [W.make_inputs(sp, 70 + i) for i in range(2)]
    refs = [util.oracle_ref(sp, a) for a in arrays]
    (t0, tt0), (t1, tt1) = [W.device_tensors(sp, a) for a in arrays]

    def right(t, ref):
        torch.cuda.synchronize()
        assert wl.status() == B.TT_OK
        ok = util.rel_l2(t["y"].cpu().numpy(), ref) <= util.TOL_TF32
        t["y"].fill_(float("nan"))
        return ok

    def capture(*tts):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for tt in tts:
                wl.run(tt)
        return g

    # weights written between a run without the promise and one with it
    wl = sp.workload()
    assert wl.apply(rec).legal.k_order == 1
    w0 = t0["w"].clone()
    t0["w"].mul_(3.0)
    wl.run(tt0)
    t0["w"].copy_(w0)
    torch.cuda.synchronize()
    wl.set_constant_weights(True)
    wl.run(tt0)
    assert right(t0, refs[0])
    # ... and while it is switched off
    wl.set_constant_weights(False)
    t0["w"].mul_(3.0)
    torch.cuda.synchronize()
    wl.set_constant_weights(True)
    wl.run(tt0)
    wl.set_constant_weights(False)
    t0["w"].copy_(w0)
    torch.cuda.synchronize()
    wl.set_constant_weights(True)
    wl.run(tt0)
    assert right(t0, refs[0])
    # a captured pass reads the copy in place; other weights in between, run and captured
    g0 = capture(tt0)
    wl.run(tt1)
    assert right(t1, refs[1])
    g0.replay()
    assert right(t0, refs[0])
    both = capture(tt0, tt1, tt0)
    for _ in range(2):
        both.replay()
        assert right(t0, refs[0]) and right(t1, refs[1])
        g0.replay()
        assert right(t0, refs[0])
        wl.run(tt1)
        assert right(t1, refs[1])
        wl.run(tt0)
        assert right(t0, refs[0])
    wl.close()
    # captured before anything has run
    for constant in (True, False):
        wl = sp.workload()
        wl.apply(rec)
        wl.set_constant_weights(constant)
        g0 = capture(tt0)
        wl.run(tt0)
        assert right(t0, refs[0])
        wl.run(tt1)
        g0.replay()
        assert right(t0, refs[0]) and right(t1, refs[1])
        wl.run(tt1)
        assert right(t1, refs[1])
        g0.replay()
        assert right(t0, refs[0])
        # timing captures too, and keeps nothing for its own captures
        opts = B.tt_timing_opts()
        opts.use_graph, opts.batches, opts.min_batch_us = 1, 2, 50
        wl.time([tt0, tt1], opts)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(40):
            wl.time([tt0, tt1], opts)
        assert free - torch.cuda.mem_get_info()[0] < 16 << 20
        wl.run(tt1)
        assert right(t1, refs[1])
        g0.replay()
        assert right(t0, refs[0])
        wl.close()


def test_staged_depthwise_grid_is_settled_when_the_record_is_applied():
    """Two layers that share a kernel instantiation and differ in their launch, run in turn: the apply info has the grid that the
    device holds, and a launch asks the driver nothing."""
    import torch
    sp = [W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=n, c=96, h=28, w=28, k=96, r=3, s=3, stride_h=1, stride_w=1, pad_h=1, pad_w=1, has_bias=1,
                                                 act=B.TT_ACT_RELU6), 1, f"dw_turns_{n}", "uniform") for n in (40, 33)]
    recs = [B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=tm, block_y=by, block_x=28, items_per_thread=4, vec_width=4, threads=256, unroll=2, raster=1, stages=sg)
            for tm, by, sg in ((4, 28, 2), (2, 14, 4))]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wls = [s.workload() for s in sp]
    infos = [wl.apply(r) for wl, r in zip(wls, recs)]
    for wl, rec, info in zip(wls, recs, infos):
        checked = wl.check(rec)[1]
        assert 0 < info.grid_x <= checked.grid_x and info.grid_x <= 32 * sms and (info.threads, info.smem_bytes) == (checked.threads, checked.smem_bytes)
    arrays = [W.make_inputs(s, 80 + i) for i, s in enumerate(sp)]
    bufs = [W.device_tensors(s, a) for s, a in zip(sp, arrays)]
    for _ in range(3):
        for wl, (t, tt) in zip(wls, bufs):
            t["y"].fill_(float("nan"))
            wl.run(tt)
            assert wl.status() == B.TT_OK
    for s, a, (t, _) in zip(sp, arrays, bufs):
        assert util.rel_l2(t["y"].cpu().numpy(), util.oracle_ref(s, a)) <= util.TOL_FP32
    for wl in wls:
        wl.close()


@pytest.mark.parametrize("items", [1, 2])
@pytest.mark.parametrize("rows", [2, 4, 7])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("r", [3, 5])
def test_every_run_staged_instantiation(r, stride, rows, items):
    """Filter, stride, strip height and columns per thread of the run-staged form, each reached by its own batch: planes with a
    partial last strip, rows that end inside a strip's columns, bands of a plane, an input that starts inside 16 bytes.  Bounded against the oracle and
    bit-identical to the register-window form, which strict mode runs as written."""
    import torch
    p = {2: 2, 4: 8, 7: 13}[rows]
    shapes = [(p, 21 if items == 1 else 22)] + ([(131, 77 if items == 1 else 50)] if rows == 7 else [])
    for k, (out_h, w) in enumerate(shapes):
        h = out_h if k or stride == 1 else 2 * out_h - (items - 1)
        ph, q = (h - 1) // stride + 1, (w - 1) // stride + 1
        c = 37
        n = -(-(1 << 18) // (c * ph * q))
        spec = W.Spec(B.TT_OP_DWCONV2D, B.make_shapes(n=n, c=c, h=h, w=w, k=c, r=r, s=r, stride_h=stride, stride_w=stride, pad_h=r // 2, pad_w=r // 2,
                                                      has_bias=1, act=(B.TT_ACT_RELU6, B.TT_ACT_GELU_ERF)[k]), 1, f"runs_{r}{stride}{rows}{items}", "uniform")
        a = W.make_inputs(spec, 100 + k)
        ref = util.oracle_ref(spec, a)
        rec = B.make_record(B.TT_FAMILY_DW_SIMT, tile_m=4, block_y=min(8, ph), block_x=8, items_per_thread=4, vec_width=1, threads=64, unroll=2)
        wl = spec.workload()
        legal = wl.apply(rec).legal
        assert (legal.raster, legal.unroll, legal.items_per_thread) == (1, rows, items), legal.short()
        assert (legal.block_y < ph) == (k == 1)
        y = run_spec(spec, rec, a, ref, ref_elem=ref)
        np.testing.assert_array_equal(run_spec(spec, rec, a, mode=B.TT_MODE_STRICT), y)
        t, _ = W.device_tensors(spec, a)
        size = t["x"].numel()
        x = torch.empty(size + 4, device="cuda")[3:3 + size].view(t["x"].shape).copy_(t["x"])
        t["y"].fill_(float("nan"))
        wl.run(B.tensors(x, t["w"], t["bias"], t["residual"], t["y"]))
        assert wl.status() == B.TT_OK
        np.testing.assert_array_equal(t["y"].cpu().numpy(), y)
        wl.close()


@pytest.mark.parametrize("seq,heads,d", [(1, 2, 64), (31, 3, 64), (32, 12, 64), (33, 2, 32), (64, 1, 128), (97, 12, 64), (130, 12, 64), (192, 3, 36), (255, 12, 64), (256, 12, 64), (257, 2, 64), (129, 48, 16)])
def test_attention_and_projections_of_a_chain(seq, heads, d):
    """One encoder layer as a chained pass, on lanes and on one stream: the three projections run as one launch, scores, softmax and
    context as another (up to 256 keys and 148 CTAs of 32 rows).  Every layer's output against the oracle chain, between guard bands
    and starting as NaN; blocks of 32 rows and keys with remainders of every kind."""
    import torch
    specs, steps = W.bert_base_net(seq=seq, hidden=heads * d, heads=heads, ffn=2 * heads * d, layers=1)
    arrays = W.make_chain_inputs(steps, 9, init="bert")
    refs, depth = util.oracle_chain(steps, arrays), _tf32_depth(steps)
    wls = [sp.workload() for sp in specs]
    for wl in wls:
        wl.apply(tc(tile_n=64, tile_k=64, stages=2, split_k=4, mma_m_axis=2) if wl.family() == B.TT_FAMILY_GEMM_TC else wl.default_schedule())
        wl.set_constant_weights(True)
    bufs, _ = W.chain_device_tensors(steps, arrays)
    tts, guards = [], []
    for st, b in zip(steps, bufs):
        if st.spec is None:
            tts.append(None)
            continue
        b["y"], buf = guarded_output(st.spec)
        guards.append(buf)
        xs, ws, _, _, _ = W.tensor_shapes(st.spec)
        w = b["w"] if st.w_from is None else bufs[st.w_from]["y"].view(ws)
        tts.append(B.tensors(bufs[st.x]["y"].view(xs), w, b["bias"], None, b["y"]))
    fused = seq <= 256 and heads * ((seq + 31) // 32) <= 148
    streams = [torch.cuda.current_stream()] + [torch.cuda.Stream() for _ in range(3)]
    lanes = W.chain_lanes(steps, max_lanes=4)
    for plan in (lanes, [None if pl is None else (0, ()) for pl in lanes]):
        assert B.chain_launches(wls, steps, tts, plan) == (5 if fused else 7)
        for st, b in zip(steps, bufs):
            if st.spec is not None:
                b["y"].fill_(float("nan"))
        torch.cuda.synchronize()
        W.run_chain(wls, steps, tts, plan, streams)
        torch.cuda.synchronize()
        assert all(wl.status() == B.TT_OK for wl in wls) and all(guards_intact(g) for g in guards)
        for i, (st, b, ref, k) in enumerate(zip(steps, bufs, refs, depth)):
            if st.spec is not None:
                y = b["y"].cpu().numpy()
                assert not np.isnan(y).any() and util.rel_l2(y, ref) <= max(k, 1) * util.TOL_TF32, (i, st.spec.name, util.rel_l2(y, ref))
    for wl in wls:
        wl.close()


@pytest.mark.parametrize("residual,per_sm", [(False, 1), (True, 1), (False, 2)], ids=["plain", "skip_tensor", "two_per_sm"])
def test_dense_layers_of_one_input_in_a_chain(residual, per_sm):
    """Three layers of one plan on one input, each with its own weights, bias and skip tensor: one launch where the kernel has that
    form, else three; between them a layer that reads the first one's output.  Each against the layer run by itself."""
    import types
    import torch
    spec = W.Spec(B.TT_OP_DENSE, B.dense_shapes(70, 192, 192, True, B.TT_ACT_RELU), 1, "chain_dense", "he")
    spec.shapes.has_residual = residual
    wl = spec.workload()
    wl.apply(tc(tile_n=64, tile_k=32, stages=2, split_k=2, ctas_per_sm=per_sm))
    wl.set_constant_weights(True)
    rng = torch.Generator().manual_seed(3)
    draw = lambda *s: torch.randn(*s, generator=rng).cuda()
    x, out, tts = draw(70, 192), [], []
    ops = [(draw(192, 192), draw(192), draw(70, 192) if residual else None) for _ in range(4)]
    for i, (w, b, r) in enumerate(ops):
        out.append(torch.full((70, 192), float("nan"), device="cuda"))
        tts.append(B.tensors(x if i < 3 else out[0], w, b, r, out[i]))
    node = types.SimpleNamespace(kernel=0)
    args = ([wl], [node] * 4, tts, [(0, ())] * 4)
    assert B.chain_launches(*args) == (4 if residual or per_sm == 2 else 2)
    B.run_chain(*args, [torch.cuda.current_stream()])
    torch.cuda.synchronize()
    assert wl.status() == B.TT_OK
    got = [y.cpu().numpy() for y in out]
    for i, (y, tt) in enumerate(zip(out, tts)):
        y.fill_(float("nan"))
        wl.run(tt)
        np.testing.assert_array_equal(got[i], y.cpu().numpy(), err_msg=str(i))
    wl.close()


@pytest.mark.parametrize("m,k,n,rec", [
    (128, 768, 768, dict(tile_n=64, tile_k=64, stages=3, split_k=4, mma_m_axis=2)),                 # 36 clusters of 4 as the record has them: other tiles
    (128, 768, 768, dict(tile_n=64, tile_k=64, stages=3, split_k=4, mma_m_axis=1)),
    (256, 768, 768, dict(tile_n=64, tile_k=64, stages=2, split_k=4, mma_m_axis=2)),
    (33, 1000, 500, dict(tile_n=16, tile_k=32, stages=4, split_k=7, mma_m_axis=1, acc_split=2)),    # ragged, two accumulators
    (200, 264, 900, dict(tile_n=32, tile_k=32, stages=2, split_k=1, mma_m_axis=2)),                 # no split: 148 tiles
    (64, 2048, 96, dict(tile_n=32, tile_k=128, stages=1, split_k=8, mma_m_axis=2)),                 # the record's tiles fit
])
def test_layers_in_one_launch_give_the_bits_they_give_alone(m, k, n, rec):
    """Two and three dense layers of one input in a chained pass: the tiles of the group may be others than the record's, its sums are
    the record's.  Then each layer alone, and the group again: neither takes the other's tensor maps."""
    import types
    import torch
    wl = W._dense(m, k, n, act=B.TT_ACT_RELU).workload()
    wl.apply(tc(**rec))
    rng = torch.Generator().manual_seed(4)
    draw = lambda *s: torch.randn(*s, generator=rng).cuda()
    x, ops = draw(m, k), [(draw(n, k), draw(n)) for _ in range(3)]
    for layers in (2, 3):
        out = [torch.empty(m, n, device="cuda") for _ in range(layers)]
        tts = [B.tensors(x, w, b, None, y) for (w, b), y in zip(ops, out)]
        args = ([wl], [types.SimpleNamespace(kernel=0)] * layers, tts, [(0, ())] * layers)
        assert B.chain_launches(*args) == 1
        runs = []
        for chained in (True, False, True):
            for y in out:
                y.fill_(float("nan"))
            if chained:
                B.run_chain(*args, [torch.cuda.current_stream()])
            else:
                for tt in tts:
                    wl.run(tt)
            runs.append(torch.stack(out).cpu().numpy())
        assert wl.status() == B.TT_OK and not np.isnan(runs[1]).any()
        np.testing.assert_array_equal(runs[0], runs[1])
        np.testing.assert_array_equal(runs[2], runs[1])
    wl.close()


_PLAIN = dict(tile_n=64, tile_k=64, stages=2, mma_m_axis=1)


@pytest.mark.parametrize("n,d,qk,lanes,pv,launches", [
    (1, 8, _PLAIN, 32, _PLAIN, 1),
    (31, 64, _PLAIN, 8, _PLAIN, 1),
    (64, 64, dict(tile_n=64, tile_k=64, stages=4, mma_m_axis=2, persistent=1), 16, dict(tile_n=64, tile_k=64, stages=3, mma_m_axis=1, persistent=1), 1),
    (97, 36, dict(_PLAIN, tile_k=16, split_k=2), 16, dict(_PLAIN, tile_k=32, split_k=3), 1),
    (128, 64, dict(_PLAIN, tile_k=16, split_k=3), 4, dict(_PLAIN, tile_k=64, split_k=2), 1),
    (128, 64, dict(_PLAIN, acc_split=2), 32, dict(_PLAIN, acc_split=4, mma_m_axis=2), 1),
    (130, 64, _PLAIN, 4, dict(_PLAIN, tile_n=32, tile_k=8, split_k=8, mma_m_axis=2), 3),                     # 160 + 8 x 64 columns
    (130, 100, _PLAIN, 8, dict(_PLAIN, tile_n=128, tile_k=64, split_k=2), 1),
    (200, 64, _PLAIN, 8, dict(_PLAIN, tile_k=128, split_k=2, mma_m_axis=2), 1),
    (255, 32, dict(_PLAIN, tile_k=8), 32, dict(_PLAIN, tile_k=32, split_k=4), 1),
    (256, 64, _PLAIN, 16, dict(_PLAIN, split_k=4), 1),
    (256, 64, _PLAIN, 32, dict(_PLAIN, acc_split=2), 1),
    (100, 64, _PLAIN, 8, _PLAIN, 1),
    (128, 32, _PLAIN, 8, _PLAIN, 1),
    (129, 64, _PLAIN, 2, _PLAIN, 3),                                                                       # rows of two lanes
    (96, 64, _PLAIN, 16, dict(_PLAIN, tile_k=32, split_k=2, acc_split=2), 3),                               # splits of two accumulators
])
def test_attention_in_one_launch_gives_the_bits_of_its_layers(n, d, qk, lanes, pv, launches):
    """Scores, softmax and context under records of every order of their sums: the one launch of a chained pass against the three
    layers by themselves; orders that it does not know go to the device one by one."""
    import types
    import torch
    heads = 3
    specs = [W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(heads, n, n, d, True), 1, "qk", "bert"),
             W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(heads, n, n, 2.0 / math.sqrt(d)), 1, "softmax", "bert"),
             W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(heads, n, d, n, False), 1, "pv", "bert")]
    wls = [sp.workload() for sp in specs]
    wls[0].apply(tc(**qk))
    wls[1].apply(B.make_record(B.TT_FAMILY_ROW_SIMT, block_x=lanes, block_y=4, vec_width=4))
    wls[2].apply(tc(**pv))
    rng = torch.Generator().manual_seed(6)
    q, k, v = (torch.randn(heads, n, d, generator=rng).cuda() for _ in range(3))
    out = [torch.empty(heads, n, n, device="cuda"), torch.empty(heads, n, n, device="cuda"), torch.empty(heads, n, d, device="cuda")]
    tts = [B.tensors(q, k, None, None, out[0]), B.tensors(out[0], None, None, None, out[1]), B.tensors(out[1], v, None, None, out[2])]
    args = (wls, [types.SimpleNamespace(kernel=i) for i in range(3)], tts, [(0, ())] * 3)
    assert B.chain_launches(*args) == launches
    runs = []
    for chained in (True, False):
        for y in out:
            y.fill_(float("nan"))
        if chained:
            B.run_chain(*args, [torch.cuda.current_stream()])
        else:
            for wl, tt in zip(wls, tts):
                wl.run(tt)
        runs.append([y.cpu().numpy() for y in out])
    assert all(wl.status() == B.TT_OK for wl in wls) and not any(np.isnan(y).any() for y in runs[1])
    for name, a, b in zip(("scores", "probabilities", "context"), *runs):
        np.testing.assert_array_equal(a, b, err_msg=name)
    for wl in wls:
        wl.close()


def test_a_wait_that_gives_up_in_a_shared_launch_is_reported_by_every_layer():
    """Attention as one launch, told to expect more than arrives on behalf of each of its workloads in turn: all three report the
    time-out after the shortest of their wait limits, and the next pass is right.  Then a group of dense layers."""
    import time
    import types
    import torch
    heads, n, d = 2, 96, 32
    specs = [W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(heads, n, n, d, True), 1, "qk", "bert"), W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(heads, n, n, 0.2), 1, "softmax", "bert"),
             W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(heads, n, d, n, False), 1, "pv", "bert"), W._dense(n, 64, 48, name="dense")]
    wls = [sp.workload() for sp in specs]
    for wl in wls:
        wl.apply(tc(tile_n=64, tile_k=32, stages=2) if wl.family() == B.TT_FAMILY_GEMM_TC else wl.default_schedule())
    rng = torch.Generator().manual_seed(7)
    draw = lambda *s: torch.randn(*s, generator=rng).cuda()
    q, k, v, x = draw(heads, n, d), draw(heads, n, d), draw(heads, n, d), draw(n, 64)
    out = [torch.empty(s, device="cuda") for s in ((heads, n, n), (heads, n, n), (heads, n, d), (n, 48), (n, 48))]
    tts = [B.tensors(q, k, None, None, out[0]), B.tensors(out[0], None, None, None, out[1]), B.tensors(out[1], v, None, None, out[2])]
    tts += [B.tensors(x, draw(48, 64), draw(48), None, y) for y in out[3:]]
    stream = [torch.cuda.current_stream()]
    node = lambda kernel: types.SimpleNamespace(kernel=kernel)
    attention, group = (wls, [node(i) for i in range(3)], tts[:3], [(0, ())] * 3), (wls, [node(3)] * 2, tts[3:], [(0, ())] * 2)
    for args, members, outs in ((attention, wls[:3], out[:3]), (group, wls[3:], out[3:])):
        assert B.chain_launches(*args) == 1
        B.run_chain(*args, stream)
        right = [y.clone() for y in outs]
        for i, wl in enumerate(members):
            wl.test_stall(64)
            members[(i + 1) % len(members)].set_wait_limit(2_000_000)
            assert B.chain_launches(*args) == 1
            torch.cuda.synchronize()
            t0 = time.monotonic()
            B.run_chain(*args, stream)
            torch.cuda.synchronize()
            assert time.monotonic() - t0 < 0.5                         # (not the others' second)
            assert [w.status() for w in members] == [B.TT_ERR_TIMEOUT] * len(members)
            wl.test_stall(0)
            members[(i + 1) % len(members)].set_wait_limit(1_000_000_000)
            for y in outs:
                y.fill_(float("nan"))
            B.run_chain(*args, stream)
            assert [w.status() for w in members] == [B.TT_OK] * len(members)
            assert all(torch.equal(y, r) for y, r in zip(outs, right))
    for wl in wls:
        wl.close()


def test_what_a_pass_brings_into_the_l2_ahead_is_bounded():
    """An encoder's launches ask for the weights behind them, whole layers of 10 MB in all at most, whatever the next layers' sizes; a
    pass of single layers asks for nothing; results are those of the layers one by one."""
    import types
    import torch
    stream = [torch.cuda.current_stream()]

    def wired(specs, steps):
        wls = [sp.workload() for sp in specs]
        for wl in wls:
            wl.apply(tc(tile_n=64, tile_k=64, stages=2, split_k=2) if wl.family() == B.TT_FAMILY_GEMM_TC else wl.default_schedule())
        bufs, tts = W.chain_device_tensors(steps, W.make_chain_inputs(steps, 3, init="bert"))
        plan = [None if st.spec is None else (0, ()) for st in steps]
        ahead = B.chain_ahead(wls, steps, tts, plan)
        W.run_chain(wls, steps, tts, plan, stream)
        got = [b["y"].clone() for b in bufs]
        for st, tt in zip(steps, tts):
            if tt is not None:
                wls[st.kernel].run(tt)
        assert all(torch.equal(b["y"], y) for b, y in zip(bufs, got)) and all(wl.status() == B.TT_OK for wl in wls)
        for wl in wls:
            wl.close()
        return ahead

    limit = 10 << 20
    for hidden, ffn in ((768, 3072), (256, 70000), (512, 2500)):          # projections and what comes behind: 2.4 + 9.4, 0.3 + 72, 1 + 5.1 MB
        ahead = wired(*W.bert_base_net(seq=64, hidden=hidden, heads=hidden // 64, ffn=ffn, layers=2))
        assert 0 < max(ahead) <= limit, (hidden, ffn, ahead)
    net = W.Net()
    cur = net.external((3, 256), "rows")
    for a, b in ((256, 256), (256, 40000), (40000, 256)):
        cur = net.add(W._dense(3, a, b, init="bert", name=f"d{a}_{b}"), x=cur)
    assert not any(wired(*net.finish()))


@pytest.mark.parametrize("spec", [
    W._dense(130, 421, 295, act=B.TT_ACT_RELU, name="raw_dense_421"),
    W._dense(3, 7, 6, name="raw_dense_too_few_rows"),
    W._dense(258, 1030, 66, name="raw_dense_1030"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(5, 131, 64, 161, False), 1, "raw_nn_161", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(3, 37, 50, 33, True), 1, "raw_nt_33", "bert"),
    W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(3, 70, 61, 35, False), 1, "raw_nn_61", "bert"),
], ids=lambda s: s.name)
def test_operands_of_ragged_rows(spec):
    """Rows that are no 16-byte multiples, by boxes of four rows' lines: every tile depth, both accumulator axes, splits, the rows
    behind the last whole group of four, and a NaN in one row, which stays in that row's results."""
    import torch
    a = W.make_inputs(spec, 17)
    ref = util.oracle_ref(spec, a)
    re = elem_ref(spec, a, ref)
    for tk in (8, 16, 32, 64, 128):
        for kw in (dict(tile_n=64, stages=2, mma_m_axis=1), dict(tile_n=16, stages=3, split_k=3, mma_m_axis=2), dict(tile_n=128, stages=1, mma_m_axis=1, ctas_per_sm=2)):
            run_spec(spec, tc(tile_k=tk, **kw), a, ref, ref_elem=re)
    wl = spec.workload()
    wl.apply(tc(tile_n=64, tile_k=32, stages=2, mma_m_axis=1))
    t, tt = W.device_tensors(spec, a)
    bad = a["x"].shape[-2] - 2
    t["x"][..., bad, :] = float("nan")
    wl.run(tt)
    y = t["y"].cpu().numpy()
    keep = np.arange(y.shape[-2]) != bad
    assert util.rel_l2(y[..., keep, :], ref.reshape(y.shape)[..., keep, :]) <= util.TOL_TF32
    # an operand that does not start on 16 bytes is gathered value by value
    x2 = torch.empty(t["x"].numel() + 1, device="cuda")[1:].view(t["x"].shape)
    x2.copy_(torch.from_numpy(a["x"]))
    wl.run(B.tensors(x2, t["w"], t["bias"], None, t["y"]))
    assert wl.status() == B.TT_OK and util.rel_l2(t["y"].cpu().numpy(), ref) <= util.TOL_TF32
    wl.close()


@pytest.mark.parametrize("spec", [
    W._conv(64, 7, 48, 1, 1, 0, name="run_64x7x7"),
    W._conv(132, 11, 40, 1, 1, 0, residual=True, name="run_132x11x11_res"),
    W.Spec(B.TT_OP_CONV2D, B.conv2d_shapes(3, 20, 5, 3, 70, 1, 1, 1, 0, True, B.TT_ACT_RELU6), 1, "run_n3_5x3", "uniform"),
    W._conv(30, 7, 16, 1, 1, 0, name="no_run_30_channels"),
], ids=lambda s: s.name)
def test_pointwise_images_of_one_tile(spec):
    """A 1x1 convolution whose image is no multiple of 16 bytes and fits a tile: its channels arrive as runs of memory, in one chunk or
    several, the last one shorter; images that do not start on 16 bytes by smaller copies."""
    import torch
    a = W.make_inputs(spec, 23)
    ref = util.oracle_ref(spec, a)
    re = elem_ref(spec, a, ref)
    for kw in (dict(tile_n=128, tile_k=32, stages=2, mma_m_axis=1), dict(tile_n=16, tile_k=16, stages=3, mma_m_axis=2, slab_tiles=1),
               dict(tile_n=64, tile_k=8, stages=2, split_k=3, mma_m_axis=2), dict(tile_n=32, tile_k=32, stages=2, mma_m_axis=1)):
        run_spec(spec, tc(**kw), a, ref, ref_elem=re)
    wl = spec.workload()
    wl.apply(tc(tile_n=128, tile_k=32, stages=2, mma_m_axis=1))
    t, _ = W.device_tensors(spec, a)
    x2 = torch.empty(t["x"].numel() + 1, device="cuda")[1:].view(t["x"].shape)
    x2.copy_(t["x"])
    wl.run(B.tensors(x2, t["w"], t["bias"], t["residual"], t["y"]))
    assert wl.status() == B.TT_OK and util.rel_l2(t["y"].cpu().numpy(), ref) <= util.TOL_TF32
    wl.close()
