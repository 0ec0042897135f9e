"""Performance cases: the work that users of this library have it do, through its public calls.

A case has a kind (what the program does), the weight it does it to and, where activations are
multiplied, their shape.  Sizes are those of the benchmark's workloads (inputs.WORKLOADS, the
4096 x 4096 sweep, the projection size sweep), of the tests, or round numbers between them.

  layer        compress a linear layer and run it: mwu_project, mwu_pack, mwu_gemm_ws
  conv         the same for a convolution: mwu_project, mwu_pack, mwu_conv_implicit_ws
  product      inference on weights packed beforehand: mwu_gemm_ws
  conv_product the same for a convolution: mwu_conv_implicit_ws
  project      the Q-step alone: mwu_project
  admm         the Q-step and the dual step of an ADMM iteration: mwu_admm_step
  shape_conv   a 2- or 3-dim block shape on a convolution: mwu_project, Q rounded to bf16 (torch),
               mwu_conv_dense (such shapes have no packed form)
  keep         keep 2 of 4 and multiply: mwu_keep_n_of_m, mwu_gemm_dense

Weights are fp32 N(0, 0.02^2) (convolutions Kaiming-normal), the dual tensor N(0, 0.004^2),
activations bf16 N(0, 1): the distributions of inputs.py, drawn on the GPU.
"""
from __future__ import annotations

import math

import torch

from paper_2106_08301_b200 import binding as B


def _case(kind, rows, cols, block, unified=500, pruned=250, **more):
    c = {"kind": kind, "rows": rows, "cols": cols, "block": block, "unified": unified, "pruned": pruned,
         "l1": False, "m": 0, "fp32_out": False, "group_rows": 0, "group_cols": 0, "block_rows": 0,
         "block_taps": 0, "batch": 0, "cin": 0, "h": 0, "w": 0, "k": 0, "stride": 1, "pad": 0}
    c.update(more)
    return c


def _conv(kind, filters, cin, h, w, k, stride, batch, block, unified, pruned, **more):
    return _case(kind, filters, cin * k * k, block, unified, pruned, batch=batch, cin=cin, h=h, w=w, k=k,
                 stride=stride, pad=k // 2, **more)


def listed():
    out = []

    def add(name, case):
        out.append(dict(case, name=name))

    # one small linear layer, batch 64: launches and latency
    add("linear_small", _case("layer", 256, 256, 4, 500, 250, m=64))
    # a layer whose sizes divide nothing: ragged row tiles, the L1 prune key, fp32 output
    add("linear_ragged", _case("layer", 1000, 1216, 8, 700, 450, m=777, l1=True, fp32_out=True))
    # transformer FFN up-projection over 8192 tokens: compress, then prefill
    add("ffn_layer", _case("layer", 16384, 4096, 16, 800, 600, m=8192))
    # the same layer with whole 256 x 64 groups pruned, which the tensor cores can skip
    add("ffn_layer_grouped", _case("layer", 16384, 4096, 16, 800, 600, m=8192, group_rows=256, group_cols=64))
    # the same layer at decode time: a few tokens against weights packed long ago
    add("ffn_decode", _case("product", 16384, 4096, 16, 800, 600, m=16))
    # a 1x1 convolution as a product: few weights, many pixels, mostly output
    add("conv1x1_product", _case("product", 1024, 256, 8, 750, 500, m=200704))
    # a 3x3 convolution layer: compress, then run
    add("conv3x3", _conv("conv", 128, 128, 28, 28, 3, 1, 32, 4, 600, 300))
    # a strided 3x3 convolution (the first of a stage) on packed weights
    add("conv3x3_stride2", _conv("conv_product", 128, 64, 56, 56, 3, 2, 32, 4, 600, 300))
    # the largest tensor of the projection size sweep
    add("project_large", _case("project", 16384, 16384, 4, 500, 250))
    # one ADMM iteration of training on the FFN weight, the dual tensor in and out
    add("ffn_admm", _case("admm", 16384, 4096, 16, 800, 600))
    # 2x2x2 blocks on a 3x3 convolution, then the convolution
    add("conv3x3_block222", _conv("shape_conv", 128, 128, 28, 28, 3, 1, 32, 2, 600, 300, block_rows=2, block_taps=2))
    # keep 2 of 4 on a square layer, then the product
    add("keep_2_of_4", _case("keep", 4096, 4096, 4, m=2048))
    return out


# ---------------------------------------------------------------------------------------------
# drawn cases: the ranges the listed ones stand for
# ---------------------------------------------------------------------------------------------
_MAX_WEIGHTS = 1 << 26
_MAX_MACS = 5000 << 26


def _log(rng, lo, hi):
    """Log-uniform whole number in [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _fractions(rng):
    pruned = rng.choice([0, 250, 500, 750, 900, rng.randrange(0, 900)])
    return min(1000, pruned + rng.choice([50, 100, 200, 250])), pruned


def _linear(rng, kind, max_m):
    """rows x cols log-uniform, cols in whole 64s (the packed form's unit), rows of any kind."""
    block = rng.choice([2, 4, 8, 16])
    while True:
        rows = _log(rng, 96, 16384)
        cols = 64 * _log(rng, 2, 128)
        if rng.random() < 0.5:
            rows = max(128, rows // 128 * 128)
        m = _log(rng, 1, max_m)
        if rows * cols <= _MAX_WEIGHTS >> (block < 8) and rows * cols * m <= _MAX_MACS and rows * m <= (200 << 20):
            break
    unified, pruned = _fractions(rng)
    return _case(kind, rows, cols, block, unified, pruned, m=m, l1=rng.random() < 0.2,
                 fp32_out=rng.random() < 0.2)


def _conv_draw(rng, kind, stride):
    while True:
        cin = 64 * rng.choice([1, 1, 2, 2, 3, 4])
        k = rng.choice([1, 3, 3, 3, 5]) if stride == 1 else 3
        filters = rng.choice([64, 128, 128, 200, 256, 384, 512])
        h, w = _log(rng, 7, 56), _log(rng, 7, 56)
        if rng.random() < 0.5:
            w = h = rng.choice([7, 14, 28, 56])
        batch = _log(rng, 1, 64)
        pixels = batch * (-(-h // stride)) * (-(-w // stride))
        if cin * k * k <= (2304 if stride == 2 else 6400) and pixels * filters * cin * k * k <= (12 << 30):
            break
    unified, pruned = _fractions(rng)
    if kind == "shape_conv":
        # [2, 2, 2], and [2, 2] (which spans channels and filters, tap by tap)
        filters = min(filters, 256)
        return _conv(kind, filters, cin, h, w, k, 1, batch, 2, unified, pruned, block_rows=2,
                     block_taps=2 if k > 1 and rng.random() < 0.7 else 1)
    return _conv(kind, filters, cin, h, w, k, stride, batch, rng.choice([2, 4, 8, 16]), unified, pruned)


def draw(rng):
    what = rng.choice(["layer", "layer", "grouped", "decode", "product", "conv", "conv_product", "project",
                       "admm", "shape_conv", "keep"])
    if what == "layer":
        return _linear(rng, "layer", 8192)
    if what == "decode":
        return _linear(rng, "product", 64)
    if what == "product":
        return _linear(rng, "product", 200704)
    if what == "grouped":
        gr, gc = rng.choice([128, 256]), rng.choice([16, 32, 64])
        b = rng.choice([x for x in (2, 4, 8, 16) if x <= gc])
        rows, cols = 256 * _log(rng, 1, 64), 64 * _log(rng, 4, 64)
        unified, pruned = _fractions(rng)
        return _case("layer", rows, cols, b, unified, pruned, m=_log(rng, 1, 8192), group_rows=gr, group_cols=gc)
    if what == "conv":
        return _conv_draw(rng, "conv", 1)
    if what == "conv_product":
        return _conv_draw(rng, "conv_product", 2)
    if what == "shape_conv":
        return _conv_draw(rng, "shape_conv", 1)
    if what == "keep":
        return _case("keep", _log(rng, 128, 4096), 8 * _log(rng, 16, 512), 4, m=_log(rng, 1, 2048))
    unified, pruned = _fractions(rng)
    b = rng.choice([2, 4, 8, 16])
    if what == "admm":
        # ADMM trains layers of every size; a reduction axis of any multiple of the block
        n = _log(rng, 1 << 14, _MAX_WEIGHTS)
        rows = _log(rng, 16, 16384)
        return _case("admm", rows, max(b, n // rows // b * b), b, unified, pruned, l1=rng.random() < 0.2)
    n = _log(rng, 1 << 16, 1 << 28)
    rows = _log(rng, 128, 16384)
    cols = max(b, n // rows // b * b)
    return _case("project", rows, cols, max(b, 4) if n > (1 << 27) and cols % max(b, 4) == 0 else b, unified, pruned)


# ---------------------------------------------------------------------------------------------
# one case
# ---------------------------------------------------------------------------------------------
def _taps(c):
    return c["k"] * c["k"] if c["kind"] == "shape_conv" and c["k"] > 1 else 0


def _blocks(c):
    dr, dt, taps = max(c["block_rows"], 1), max(c["block_taps"], 1), max(_taps(c), 1)
    return (c["rows"] // dr) * (c["cols"] // taps // c["block"]) * (-(-taps // dt))


def _counts(c):
    """(k_unify, k_prune): the case's fractions as whole blocks (whole groups of blocks where grouped)."""
    mb = _blocks(c)
    ku, kp = (c["unified"] * mb + 500) // 1000, (c["pruned"] * mb + 500) // 1000
    if c["group_rows"]:
        per = c["group_rows"] * c["group_cols"] // c["block"]
        kp = kp // per * per
    return ku, kp


def _desc(c):
    ku, kp = _counts(c)
    return B.make_desc(c["rows"], c["cols"], c["block"], ku, kp,
                       prune_key=B.MWU_PRUNE_KEY_L1 if c["l1"] else B.MWU_PRUNE_KEY_L2SQ,
                       prune_group=(c["group_rows"], c["group_cols"]) if c["group_rows"] else None,
                       block_rows=c["block_rows"], block_taps=c["block_taps"], taps=_taps(c))


def _out_hw(c):
    return tuple((x + 2 * c["pad"] - c["k"]) // c["stride"] + 1 for x in (c["h"], c["w"]))


def _conv_args(c):
    return c["batch"], c["cin"], c["h"], c["w"], c["k"], c["k"], c["stride"], c["pad"]


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    rows, cols, kind = c["rows"], c["cols"], c["kind"]

    def normal(shape, std, dtype=torch.float32):
        return (torch.randn(shape, generator=gen, device="cuda") * std).to(dtype)

    s = {"case": c}
    W = normal((rows, cols), math.sqrt(2.0 / cols) if c["cin"] else 0.02)
    y_type = torch.float32 if c["fp32_out"] else torch.bfloat16
    if kind == "keep":
        s.update(W=W, X=normal((c["m"], cols), 1.0, torch.bfloat16),
                 Q=torch.empty_like(W), keep_bits=torch.empty((rows * cols + 31) // 32, dtype=torch.int32, device="cuda"),
                 Wd=torch.empty((rows, cols), dtype=torch.bfloat16, device="cuda"),
                 Y=torch.empty((c["m"], -(-rows // 8) * 8), dtype=torch.bfloat16, device="cuda").zero_(),
                 dev_status=torch.zeros(1, dtype=torch.int32, device="cuda"))
        return s
    desc = _desc(c)
    bufs = B.ProjectionBuffers(desc)
    s.update(desc=desc, bufs=bufs, dev_status=bufs.dev_status)
    if kind in ("layer", "product"):
        # rows of Y on 16-byte boundaries: what ldy has to be a multiple of
        s.update(X=normal((c["m"], cols), 1.0, torch.bfloat16),
                 Y=torch.zeros((c["m"], -(-rows // 8) * 8), dtype=y_type, device="cuda"))
        n_ws = B.mwu_gemm_workspace_bytes(desc, c["m"])
    elif kind in ("conv", "conv_product", "shape_conv"):
        s.update(X=normal((c["batch"], c["cin"], c["h"], c["w"]), 1.0, torch.bfloat16),
                 Y=torch.zeros((c["batch"], rows) + _out_hw(c), dtype=y_type, device="cuda"))
        n_ws = (B.mwu_conv_dense_workspace_bytes(rows, *_conv_args(c)) if kind == "shape_conv"
                else B.mwu_conv_workspace_bytes(desc, *_conv_args(c)))
    else:
        n_ws = 0
    s["workspace"] = torch.empty(n_ws, dtype=torch.uint8, device="cuda") if n_ws else None
    if kind in ("product", "conv_product"):
        # compressed long ago: the program keeps the packed weights and nothing else
        bufs.project(W)
        s["packed"] = bufs.pack(W)
        s["bufs"] = None
        return s
    s["W"] = W
    if kind in ("layer", "conv"):
        s["packed"] = torch.empty(B.mwu_packed_bytes(desc), dtype=torch.uint8, device="cuda")
    if kind == "admm":
        s.update(U=normal((rows, cols), 0.004), U_next=torch.empty((rows, cols), device="cuda"),
                 residual=torch.zeros(1, dtype=torch.float64, device="cuda"))
    return s


def run(state):
    s = state
    c = s["case"]
    kind, rows, cols, bufs = c["kind"], c["rows"], c["cols"], s.get("bufs")
    y_dtype = 1 if c["fp32_out"] else 0
    if kind == "keep":
        B.mwu_keep_n_of_m(rows, cols, 2, 4, s["W"], None, s["Q"], s["keep_bits"], s["Wd"], cols, s["dev_status"])
        B.mwu_gemm_dense(rows, cols, s["Wd"], cols, s["X"], c["m"], cols, s["Y"], s["Y"].shape[1], y_dtype, s["dev_status"])
        return {"Q": s["Q"], "keep": s["keep_bits"], "Wd": s["Wd"], "Y": s["Y"], "status": s["dev_status"]}
    out = {"status": s["dev_status"]}
    if kind == "admm":
        bufs.admm_step(s["W"], s["U"], s["U_next"], s["residual"])
        out.update(U_next=s["U_next"], residual=s["residual"])
    elif bufs is not None:
        bufs.project(s["W"])
    if bufs is not None:
        out.update(Q=bufs.Q, u=bufs.u, pruned=bufs.pruned_bitmap, unified=bufs.unified_bitmap, signs=bufs.sign_bits)
    if kind in ("layer", "conv"):
        bufs.pack(s["W"], packed=s["packed"])
        out["packed"] = s["packed"]
    if kind in ("layer", "product"):
        B.mwu_gemm_ws(s["desc"], s["packed"], s["X"], c["m"], cols, s["Y"], s["Y"].shape[1], y_dtype, s["workspace"],
                      s["dev_status"])
        out["Y"] = s["Y"]
    elif kind in ("conv", "conv_product"):
        B.mwu_conv_implicit_ws(s["desc"], s["packed"], s["X"], *_conv_args(c), s["Y"], y_dtype, s["workspace"],
                               s["dev_status"])
        out["Y"] = s["Y"]
    elif kind == "shape_conv":
        Wd = bufs.Q.view(rows, cols).to(torch.bfloat16)
        B.mwu_conv_dense(rows, Wd, cols, s["X"], *_conv_args(c), s["Y"], y_dtype, s["workspace"], s["dev_status"])
        out["Y"] = s["Y"]
    return out


def work(case):
    """Each input read once and each output written once; FLOPs of the blocks that are not pruned."""
    c = case
    n, mb, kind = c["rows"] * c["cols"], _blocks(c), c["kind"]
    y_bytes = 4 if c["fp32_out"] else 2
    if c["cin"]:
        oh, ow = _out_hw(c)
        m = c["batch"] * oh * ow
        x = 2.0 * c["batch"] * c["cin"] * c["h"] * c["w"]
    else:
        m, x = c["m"], 2.0 * c["m"] * c["cols"]
    y = float(y_bytes) * m * c["rows"]
    if kind == "keep":
        return {"bytes": 4.0 * n + 4.0 * n + n / 8 + 2.0 * n + x + y, "flops": 2.0 * m * n / 2}
    ku, kp = _counts(c)
    # W in; Q, u, two bitmaps and the sign plane out
    projection = 8.0 * n + 4.0 * mb + mb / 4 + n / 8
    # per unified block 8 bytes, per dense block its position and bf16 values, per pruned block its position
    b = c["block"]
    packed = 8.0 * (ku - kp) + (2.0 + 2.0 * b) * (mb - ku) + 2.0 * kp
    flops = 2.0 * m * n * (mb - kp) / mb
    return {"project": {"bytes": projection, "flops": 0.0},
            "admm": {"bytes": projection + 8.0 * n, "flops": 0.0},
            "layer": {"bytes": projection + packed + x + y, "flops": flops},
            "conv": {"bytes": projection + packed + x + y, "flops": flops},
            "product": {"bytes": packed + x + y, "flops": flops},
            "conv_product": {"bytes": packed + x + y, "flops": flops},
            "shape_conv": {"bytes": projection + x + y, "flops": flops}}[kind]


def tolerance(case):
    """Projection results are defined bit by bit; the residual is an fp64 sum in no fixed order; the
    products are bf16 x bf16 summed in fp32, rounded to bf16 unless fp32 is asked for.  Measured
    against fp64 products of the same operands: bf16 outputs 1e-4 (a few values round the other way,
    each by one unit: 2^-7 of itself at most), fp32 outputs 6e-7 at a reduction of 1216."""
    if case["kind"] == "project":
        return "exact"
    if case["kind"] == "admm":
        return {"rel": 1e-11, "max": 1e-11}
    if case["fp32_out"]:
        return {"rel": 5e-6, "max": 4e-5}
    return {"rel": 4e-4, "max": 1.6e-2}
