"""What the performance of this framework is measured on: the calls its users make, over the range of sizes they make them at.

A case is one kernel called through ``Workload.run`` under the record that ``transfer_tune`` picks for it from a pool,
one data-chained pass of a model (``workloads.run_chain``, called directly or captured once and replayed, as the
benchmark does), or one search (``transfer_tune`` itself).  ``listed`` gives the fixed ones, ``draw`` more of the same
ranges: batch 1 to 32 for convolutions (256 for the depthwise ones, 3072 heads for attention), image sides 7 to 112,
vectors of one row up to 4096 x 4096 matrices, sizes that are multiples of nothing among them.
"""
import math
import os

import torch

from paper_2201_05587_b200 import binding as B
from paper_2201_05587_b200 import workloads as W

POOL_DIR = os.path.join(os.path.dirname(os.path.abspath(W.__file__)), "pools")
ACT = {"none": B.TT_ACT_NONE, "relu": B.TT_ACT_RELU, "relu6": B.TT_ACT_RELU6, "gelu": B.TT_ACT_GELU_ERF}


# ---- the cases -------------------------------------------------------------------------------------------------------
def _conv(n, c, hw, k, r, stride, act="relu", residual=False):
    return {"kind": "conv", "n": n, "c": c, "hw": hw, "k": k, "r": r, "stride": stride, "act": act, "residual": residual}


def _dw(n, c, hw, r, stride, act="relu6"):
    return {"kind": "dw", "n": n, "c": c, "hw": hw, "r": r, "stride": stride, "act": act}


def _dense(m, kk, nn, act="none", precision=0):
    return {"kind": "dense", "m": m, "kk": kk, "nn": nn, "act": act, "precision": precision}


def _bmm(batch, m, nn, kk, trans_b):
    return {"kind": "bmm", "batch": batch, "m": m, "nn": nn, "kk": kk, "trans_b": trans_b}


def _softmax(batch, m, nn):
    return {"kind": "softmax", "batch": batch, "m": m, "nn": nn}


def listed():
    named = [
        # the smallest call: the single-convolution configuration (16 channels at 14 x 14), where latency is all there is
        ("conv_single", _conv(1, 16, 14, 32, 3, 1)),
        # batched inference of a residual network: a 3x3 layer in the middle of it ...
        ("conv3x3_b32_28", _conv(32, 128, 28, 128, 3, 1)),
        # ... one of its last stage, whose 7-pixel rows are not 16-byte multiples, with the skip tensor added ...
        ("conv3x3_b32_7_res", _conv(32, 512, 7, 512, 3, 1, residual=True)),
        # ... and an expanding 1x1 layer with the skip tensor, bound by memory
        ("conv1x1_b32_56_res", _conv(32, 64, 56, 256, 1, 1, residual=True)),
        # a batched 5x5 depthwise layer, as EfficientNet-B0-shaped networks have
        ("dw5x5_b256_28", _dw(256, 240, 28, 5, 1)),
        # the largest matrix product
        ("dense_4096", _dense(4096, 4096, 4096)),
        # a dense layer for a user who needs fp32-like results: error-compensated products
        ("dense_x3_512", _dense(512, 4096, 1024, precision=1)),
        # attention scores of a large batch of sequences (12 heads x 256 sequences of 128 tokens)
        ("bmm_scores_3072", _bmm(3072, 128, 128, 64, True)),
        # softmax over rows whose length is a multiple of nothing
        ("softmax_ragged_197", _softmax(768, 197, 197)),
        # the benchmark's headline: the BERT-base-shaped encoder at batch 1, captured once and replayed
        ("bert_base_replayed", {"kind": "chain", "model": "bert", "seq": 128, "layers": 12, "graph": True}),
        # a MobileNetV2-shaped pass at batch 1, enqueued call by call: 53 small kernels of every convolution class
        ("mobilenet_v2_direct", {"kind": "chain", "model": "mobilenet_v2", "seq": 0, "layers": 0, "graph": False}),
        # the search: every kernel of the encoder on 256 tokens under every record tuned for it on 128
        ("search_bert_256", {"kind": "search", "seq": 256, "records": 12}),
    ]
    return [dict(c, name=n) for n, c in named]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("conv", "conv", "conv", "dw", "dense", "dense", "bmm", "softmax", "chain", "search"))
    while True:
        if kind == "conv":
            # image sides of the networks' stages and odd ones between them; channels in eights, as networks have them
            hw = rng.choice((7, 14, 28, 56, _log_int(rng, 7, 64)))
            r = rng.choice((1, 1, 3, 3, 5))
            c = _conv(_log_int(rng, 1, 32), 8 * _log_int(rng, 2, 64), hw, 8 * _log_int(rng, 2, 64), r, rng.choice((1, 1, 1, 2)),
                      rng.choice(("none", "relu", "relu", "relu6")), rng.random() < 0.3)
        elif kind == "dw":
            c = _dw(_log_int(rng, 1, 256), 8 * _log_int(rng, 4, 72), rng.choice((7, 14, 28, 56, 112, _log_int(rng, 7, 112))),
                    rng.choice((3, 3, 5)), rng.choice((1, 1, 2)))
        elif kind == "dense":
            odd = rng.random() < 0.3                     # otherwise features come in eights
            f = (lambda lo, hi: _log_int(rng, lo, hi)) if odd else (lambda lo, hi: 8 * _log_int(rng, lo // 8, hi // 8))
            c = _dense(_log_int(rng, 1, 4096), f(64, 4096), f(64, 4096), rng.choice(("none", "relu", "gelu")), int(rng.random() < 0.25 and not odd))
        elif kind == "bmm":
            seq, trans_b = _log_int(rng, 32, 512), rng.random() < 0.5
            heads = 12 * _log_int(rng, 1, 256)
            c = _bmm(heads, seq, seq if trans_b else 64, 64 if trans_b else seq, trans_b)
        elif kind == "softmax":
            c = _softmax(12 * _log_int(rng, 1, 256), _log_int(rng, 16, 512), _log_int(rng, 16, 2048))
        elif kind == "chain":
            c = {"kind": "chain", "model": "bert", "seq": _log_int(rng, 64, 256), "layers": rng.randint(2, 12), "graph": rng.random() < 0.5}
        else:
            c = {"kind": "search", "seq": 8 * _log_int(rng, 8, 32), "records": rng.randint(4, 12)}
        w = work(c)
        if w["bytes"] <= 1.2e9 and w["flops"] <= 1.3e11:
            return c


# ---- kernels and pools -----------------------------------------------------------------------------------------------
def _spec(c):
    k = c["kind"]
    if k == "conv":
        s = B.conv2d_shapes(c["n"], c["c"], c["hw"], c["hw"], c["k"], c["r"], c["r"], c["stride"], c["r"] // 2, True, ACT[c["act"]], c["residual"])
        return W.Spec(B.TT_OP_CONV2D, s, 1, "conv")
    if k == "dw":
        s = B.make_shapes(n=c["n"], c=c["c"], h=c["hw"], w=c["hw"], k=c["c"], r=c["r"], s=c["r"], stride_h=c["stride"], stride_w=c["stride"],
                          pad_h=c["r"] // 2, pad_w=c["r"] // 2, has_bias=1, act=ACT[c["act"]])
        return W.Spec(B.TT_OP_DWCONV2D, s, 1, "dw")
    if k == "dense":
        return W.Spec(B.TT_OP_DENSE, B.dense_shapes(c["m"], c["nn"], c["kk"], True, ACT[c["act"]]), 1, "dense", "bert")
    if k == "bmm":
        return W.Spec(B.TT_OP_BATCH_MATMUL, B.bmm_shapes(c["batch"], c["m"], c["nn"], c["kk"], c["trans_b"]), 1, "bmm", "bert")
    return W.Spec(B.TT_OP_SOFTMAX, B.softmax_shapes(c["batch"], c["m"], c["nn"], 0.125), 1, "softmax", "bert")


def _tc(**kw):
    return B.make_record(B.TT_FAMILY_GEMM_TC, **kw)


def _dwr(**kw):
    return B.make_record(B.TT_FAMILY_DW_SIMT, items_per_thread=4, vec_width=4, **kw)


def _pool(family, precision):
    """A small pool of the forms that the native tuner arrives at over these sizes (split-K for few rows, the persistent
    form and CTA pairs for many, the tap-major order for batched 3x3 layers, ...)."""
    if family == B.TT_FAMILY_ROW_SIMT:
        return [B.make_record(family, block_x=x, block_y=y, vec_width=v) for x, y, v in ((8, 8, 4), (16, 4, 4), (32, 4, 4), (32, 4, 1))]
    if family == B.TT_FAMILY_DW_SIMT:
        return [_dwr(tile_m=1, block_y=8, block_x=32, threads=64, unroll=1), _dwr(tile_m=4, block_y=14, block_x=28, threads=128, unroll=2),
                _dwr(tile_m=4, block_y=8, block_x=56, threads=256, unroll=2, raster=1, stages=2),
                _dwr(tile_m=4, block_y=28, block_x=56, threads=256, unroll=4, raster=1, stages=2),
                _dwr(tile_m=16, block_y=14, block_x=28, threads=256, unroll=2, raster=1, stages=2)]
    pool = [_tc(tile_n=256, tile_k=32, stages=6, mma_m_axis=1, persistent=1, cta_group=2), _tc(tile_n=256, tile_k=32, stages=2, mma_m_axis=1, persistent=1),
            _tc(tile_n=128, tile_k=64, stages=2, mma_m_axis=2, persistent=1), _tc(tile_n=64, tile_k=64, stages=2, mma_m_axis=2, persistent=1),
            _tc(tile_n=64, tile_k=64, stages=3, mma_m_axis=1, persistent=1),
            _tc(tile_n=224, tile_k=96, stages=2, mma_m_axis=1, k_order=1), _tc(tile_n=128, tile_k=32, stages=4, mma_m_axis=1, k_order=1),
            _tc(tile_n=256, tile_k=32, stages=2, mma_m_axis=1), _tc(tile_n=128, tile_k=32, stages=3, mma_m_axis=2),
            _tc(tile_n=64, tile_k=64, stages=3, split_k=4, mma_m_axis=2), _tc(tile_n=64, tile_k=64, stages=2, split_k=8, mma_m_axis=2),
            _tc(tile_n=32, tile_k=64, stages=4, split_k=6, mma_m_axis=1)]
    for r in pool:
        r.precision = precision
    return pool


def _tune_opts(warmup, batches, us, default):
    o = B.tt_tune_opts()
    o.include_default = default
    o.timing.warmup_batches, o.timing.batches, o.timing.min_batch_us, o.timing.use_graph = warmup, batches, us, 1
    return o


def _log_of(name):
    return B.pool_load(os.path.join(POOL_DIR, name + ".txt"))[0]


def _distance(spec, rec):
    """How far a logged record's kernel is from this one: 0 for the same workload, else by the ratio of the sizes."""
    if rec.origin_op != spec.op or rec.origin.trans_b != spec.shapes.trans_b:
        return math.inf
    return sum(abs(math.log2(max(getattr(rec.origin, f), 1) / max(getattr(spec.shapes, f), 1)))
               for f in ("n", "c", "h", "w", "k", "r", "s", "stride_h", "batch", "m", "nn", "kk")) + 0.01 * (rec.origin.has_residual != spec.shapes.has_residual)


# ---- inputs ----------------------------------------------------------------------------------------------------------
class _Inputs:
    """Seeded tensors made on the GPU, with the distributions of workloads.make_inputs."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def uniform(self, shape, lo=-1.0, hi=1.0):
        return torch.empty(shape, device="cuda").uniform_(lo, hi, generator=self.g)

    def normal(self, shape, std=1.0):
        return torch.empty(shape, device="cuda").normal_(0.0, std, generator=self.g)

    def activations(self, shape, init):
        return self.normal(shape) if init == "bert" else self.uniform(shape)

    def params(self, spec):
        """(w, bias) of a layer; a batch_matmul's second operand is an activation."""
        _, ws, bs, _, _ = W.tensor_shapes(spec)
        if spec.op == B.TT_OP_BATCH_MATMUL:
            return self.normal(ws), None
        std = 0.02 if spec.init == "bert" else math.sqrt(2.0 / max(1, math.prod(ws[1:]))) if ws else 0.0
        return self.normal(ws, std) if ws else None, self.uniform(bs, -0.1, 0.1) if bs else None


def _kernel_tensors(spec, inp):
    xs, _, _, rs, ys = W.tensor_shapes(spec)
    w, bias = inp.params(spec)
    t = {"x": inp.activations(xs, spec.init), "w": w, "bias": bias, "residual": inp.activations(rs, spec.init) if rs else None,
         "y": torch.empty(ys, device="cuda")}
    return t, B.tensors(t["x"], t["w"], t["bias"], t["residual"], t["y"])


# ---- prepare, run ----------------------------------------------------------------------------------------------------
def prepare(case, seed):
    inp = _Inputs(seed)
    kind = case["kind"]
    if kind == "chain":
        return _prepare_chain(case, inp)
    if kind == "search":
        specs = W.bert_base(case["seq"])
        wls = [sp.workload() for sp in specs]
        for wl in wls:
            wl.set_constant_weights(True)
        t, tts = zip(*(_kernel_tensors(sp, inp) for sp in specs))
        return {"kind": kind, "wls": wls, "t": t, "tts": list(tts), "pool": _log_of("bert_base")[:case["records"]],
                "opts": _tune_opts(3, 10, 200, 1)}      # three warm-up batches, then the median of ten
    spec = _spec(case)
    t, tt = _kernel_tensors(spec, inp)
    wl = spec.workload()
    wl.set_constant_weights(True)
    precision = case.get("precision", 0)
    # error-compensated results are the user's choice of precision: the default record has none, and is left out there
    B.transfer_tune([wl], [tt], _pool(wl.family(), precision), _tune_opts(2, 5, 100, 1 - precision))
    return {"kind": kind, "wl": wl, "t": t, "tt": tt}


def _prepare_chain(case, inp):
    if case["model"] == "bert":
        specs, steps = W.bert_base_net(seq=case["seq"], layers=case["layers"])
        log, init = _log_of("bert_base") + _log_of("bert_base_256"), "bert"
    else:
        specs, steps = W.CHAINS[case["model"]]()
        log, init = _log_of(case["model"]), "he"
    wls, infos = [], []
    for sp in specs:
        wl = sp.workload()
        wl.set_constant_weights(True)
        infos.append(wl.apply(min(log, key=lambda r: _distance(sp, r))))
        wls.append(wl)
    bufs, tts = [], []
    for st in steps:                                     # wired as workloads.chain_device_tensors wires them
        if st.spec is None:
            bufs.append({"y": inp.activations(st.shape, init)})
            tts.append(None)
            continue
        xs, ws, _, rs, ys = W.tensor_shapes(st.spec)
        w, bias = inp.params(st.spec) if st.w_from is None else (bufs[st.w_from]["y"].view(ws), None)
        t = {"x": bufs[st.x]["y"].view(xs), "w": w, "bias": bias, "residual": bufs[st.res]["y"].view(rs) if rs else None,
             "y": torch.empty(ys, device="cuda")}
        bufs.append(t)
        tts.append(B.tensors(t["x"], t["w"], t["bias"], t["residual"], t["y"]))
    serial = {i for i, inf in enumerate(infos) if inf.launches > 1 or inf.legal.split_k > 8}
    state = {"kind": "chain", "wls": wls, "steps": steps, "tts": tts, "bufs": bufs, "plan": W.chain_lanes(steps, max_lanes=4, serial_kernels=serial),
             "side": [torch.cuda.Stream() for _ in range(3)], "graph": None}
    # what the pass is for: the outputs of the encoder layers, or of the blocks (at most 60, the last ones) and the classifier
    layers = [i for i, st in enumerate(steps) if st.spec is not None]
    state["outs"] = layers[8::9] if case["model"] == "bert" else layers[-60:]
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _enqueue(state)
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            _enqueue(state)
        state["graph"] = graph
    return state


def _enqueue(s):
    W.run_chain(s["wls"], s["steps"], s["tts"], s["plan"], [torch.cuda.current_stream()] + s["side"])


def run(state):
    if state["kind"] == "chain":
        if state["graph"] is not None:
            state["graph"].replay()
        else:
            _enqueue(state)
        return [state["bufs"][i]["y"] for i in state["outs"]]
    if state["kind"] == "search":
        # the search leaves every kernel with its chosen record applied; the pass ends with each kernel run under it
        B.transfer_tune(state["wls"], state["tts"], state["pool"], state["opts"])
        for wl, tt in zip(state["wls"], state["tts"]):
            wl.run(tt)
        return [t["y"] for t in state["t"]]
    state["wl"].run(state["tt"])
    return state["t"]["y"]


# ---- work, tolerance -------------------------------------------------------------------------------------------------
def _kernel_work(spec):
    """(bytes, flops): every tensor once, 4 bytes each; two operations per multiply-add, five per softmax element."""
    xs, ws, bs, rs, ys = W.tensor_shapes(spec)
    by = 4.0 * sum(math.prod(s) for s in (xs, ws, bs, rs, ys) if s is not None)
    s, out = spec.shapes, float(math.prod(ys))
    per = {B.TT_OP_CONV2D: 2.0 * s.c * s.r * s.s, B.TT_OP_DWCONV2D: 2.0 * s.r * s.s, B.TT_OP_SOFTMAX: 5.0}.get(spec.op, 2.0 * s.kk)
    return by, per * out


def work(case):
    if case["kind"] == "chain":
        specs = W.bert_base_net(seq=case["seq"], layers=case["layers"])[0] if case["model"] == "bert" else W.CHAINS[case["model"]]()[0]
        parts = [(sp, sp.use_count) for sp in specs]
    elif case["kind"] == "search":
        # every kernel at least once under every record of its own operators' family, and the default one; the
        # batches that the timing protocol asks for come on top (thirteen of 200 us for each pair)
        parts = [(sp, 1 + case["records"]) for sp in W.bert_base(case["seq"])]
    else:
        parts = [(_spec(case), 1)]
    total = [_kernel_work(sp) + (u,) for sp, u in parts]
    return {"bytes": sum(b * u for b, _, u in total), "flops": sum(f * u for _, f, u in total)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("dw", "softmax"):
        return {"rel": 1e-5}                             # fp32 throughout
    if kind == "dense" and case["precision"]:
        return {"rel": 5e-5}                             # fp32 sums of error-compensated products
    if kind == "chain":
        return {"rel": 1e-2, "max": 0.5}                 # up to 84 contractions on TF32 operands, one after the other
    return {"rel": 2e-3}                                 # one contraction on TF32 operands (ten mantissa bits)
