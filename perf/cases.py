"""Performance cases of the quantizer: what its users call, over the sizes they call it with.

Each case is one call (or one call over a list of matrices) through the public entry points of
``paper_2605_12245_b200.api``, with buffers, settings and workspace kept by the caller as a program that
quantizes a model, or an activation per step, keeps them.  ``listed()`` names twelve; ``draw()`` gives more
of the same kinds: matrices from a few blocks to a 28672 x 8192 projection, every preset, both scale layouts,
column shards of a wider matrix (row stride above the column count), the deterministic sums, the weighted
objective, MXFP4, the error of stored outputs, and host memory in and out.

Weights are drawn on the GPU with the distributions of ``paper_2605_12245_b200.workloads`` (heavy tails, outlier
columns or entries), so that making the inputs costs little beside the call.
"""
from __future__ import annotations

import math

import torch

from paper_2605_12245_b200 import api

PRESETS = {"paper": api.PRESET_PAPER, "single_pass": api.PRESET_SINGLE_PASS, "rtn": api.PRESET_RTN,
           "cjso_only": api.PRESET_CJSO_ONLY, "dss_only": api.PRESET_DSS_ONLY,
           "coupled_pair": api.PRESET_COUPLED_PAIR}
DISTS = ("student_t4", "laplace", "gauss_t2mix")
LINEAR, SWIZZLED, BOTH = api.SCALES_LINEAR, api.SCALES_SWIZZLED, api.SCALES_LINEAR | api.SCALES_SWIZZLED

# the largest listed case (a 70B decoder layer, seven matrices) bounds what draw() may ask for
MOST_ELEMENTS = 2 * 8192 * 8192 + 2 * 1024 * 8192 + 3 * 28672 * 8192


def listed():
    return [
        # activations of a 16-token decode step, quantized per step for the block-scaled product: latency is everything
        dict(name="rtn_decode_16x8192", op="quantize", rows=16, cols=8192, preset="rtn", layout=SWIZZLED, shards=1,
             deterministic=False, dist="gauss_t2mix"),
        # one of a model's many small matrices (an expert's or a head's projection) on its own
        dict(name="paper_small_128x2048", op="quantize", rows=128, cols=2048, preset="paper", layout=LINEAR, shards=1,
             deterministic=False, dist="student_t4"),
        # benchmark config 1
        dict(name="paper_2048x2048", op="quantize", rows=2048, cols=2048, preset="paper", layout=LINEAR, shards=1,
             deterministic=False, dist="student_t4"),
        # a column shard of a down projection under tensor parallelism, ragged in both directions, sums reproducible
        dict(name="paper_shard_5003x2352", op="quantize", rows=5003, cols=2352, preset="paper", layout=BOTH, shards=8,
             deterministic=True, dist="laplace"),
        # benchmark config 2: the seven matrices of an 8B decoder layer in one call
        dict(name="paper_layer_8b", op="batch", hidden=4096, kv=1024, ffn=12288, layers=1, preset="paper", layout=LINEAR,
             dist="student_t4"),
        # benchmark config 4 (the default workload): a 70B decoder layer in one call
        dict(name="paper_layer_70b", op="batch", hidden=8192, kv=1024, ffn=28672, layers=1, preset="paper", layout=LINEAR,
             dist="laplace"),
        # benchmark config 5's shape with one candidate per block (the HBM-bound three-pass form)
        dict(name="single_pass_28672x8192", op="quantize", rows=28672, cols=8192, preset="single_pass", layout=LINEAR,
             shards=1, deterministic=False, dist="gauss_t2mix"),
        # activations of a 4096-token prefill
        dict(name="rtn_prefill_4096x8192", op="quantize", rows=4096, cols=8192, preset="rtn", layout=SWIZZLED, shards=1,
             deterministic=False, dist="gauss_t2mix"),
        # an 8B decoder layer under the column-weighted objective
        dict(name="weighted_layer_8b", op="weighted", hidden=4096, kv=1024, ffn=12288, layers=1, preset="paper",
             layout=LINEAR, zero_pct=0, dist="student_t4"),
        # an up projection as MXFP4 with the scale search
        dict(name="mxfp4_12288x4096", op="mxfp4", rows=12288, cols=4096, n_beta=101, dist="student_t4"),
        # checking a stored down projection against its weights
        dict(name="error_4096x12288", op="error", rows=4096, cols=12288, layout=LINEAR, weighted=False, dist="student_t4"),
        # a checkpoint's attention matrices from pinned host memory and back, copies overlapped with the quantizer
        dict(name="host_attention_8b", op="host", hidden=4096, kv=1024, preset="paper", layout=LINEAR, dist="student_t4"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, most, unit=16):
    """Rows from 1 and columns from two blocks, up to ``most`` elements; odd row counts and odd block counts among them."""
    while True:
        rows = _log_uniform(rng, 1, 32768)
        cols = unit * _log_uniform(rng, max(1, 32 // unit), 28672 // unit)
        if 4096 <= rows * cols <= most:
            return rows, cols


def draw(rng):
    op = rng.choice(("quantize", "quantize", "quantize", "quantize", "batch", "batch", "weighted", "mxfp4", "error", "host"))
    dist = rng.choice(DISTS)
    if op == "quantize":
        preset = rng.choice(("paper", "paper", "paper", "single_pass", "rtn", "rtn", "coupled_pair", "cjso_only", "dss_only"))
        rows, cols = _shape(rng, 28672 * 8192)
        shards = rng.choice((1, 1, 1, 2, 4, 8)) if rows * cols <= 1 << 26 else 1
        return dict(op=op, rows=rows, cols=cols, preset=preset, layout=rng.choice((LINEAR, SWIZZLED, BOTH)), shards=shards,
                    deterministic=rng.random() < 0.25, dist=dist)
    if op in ("batch", "weighted"):
        hidden = 64 * _log_uniform(rng, 4, 96 if op == "weighted" else 128)
        kv = 64 * _log_uniform(rng, 2, 16)
        ffn = 16 * int(hidden * rng.uniform(2.5, 3.5) / 16)
        per_layer = 2 * hidden * hidden + 2 * kv * hidden + 3 * ffn * hidden
        most = 1.93e8 if op == "weighted" else MOST_ELEMENTS
        layers = rng.randint(1, max(1, min(4, int(most // per_layer))))
        case = dict(op=op, hidden=hidden, kv=kv, ffn=ffn, layers=layers, dist=dist,
                    layout=rng.choice((LINEAR, SWIZZLED, BOTH)))
        if op == "weighted":
            return dict(case, preset="paper", zero_pct=rng.choice((0, 0, 1)))
        return dict(case, preset=rng.choice(("paper", "paper", "single_pass", "coupled_pair")))
    if op == "mxfp4":
        rows, cols = _shape(rng, 28672 * 8192, 32)
        return dict(op=op, rows=rows, cols=cols, n_beta=rng.choice((0, 101, 101)), dist=dist)
    if op == "error":
        rows, cols = _shape(rng, 28672 * 8192)
        return dict(op=op, rows=rows, cols=cols, layout=rng.choice((LINEAR, SWIZZLED)), weighted=rng.random() < 0.3, dist=dist)
    return dict(op="host", hidden=64 * _log_uniform(rng, 8, 64), kv=64 * _log_uniform(rng, 2, 16),
                preset=rng.choice(("paper", "single_pass")), layout=rng.choice((LINEAR, BOTH)), dist=dist)


def _shapes(case):
    """(rows, cols) of every matrix of the case, in call order."""
    if case["op"] == "host":
        h, kv = case["hidden"], case["kv"]
        return [(h, h), (kv, h), (kv, h), (h, h)]
    if case["op"] in ("batch", "weighted"):
        h, kv, f = case["hidden"], case["kv"], case["ffn"]
        return [(h, h), (kv, h), (kv, h), (h, h), (f, h), (f, h), (h, f)] * case["layers"]
    return [(case["rows"], case["cols"])]


def _fill(W, dist, gen):
    """Random weights in place: W is bf16 on the GPU, drawn in chunks of rows to keep the float32 temporaries small."""
    rows, cols = W.shape
    step = max(1, (1 << 25) // cols)
    for r in range(0, rows, step):
        shape = (min(step, rows - r), cols)
        if dist == "student_t4":      # normal over the root of a chi-square(4) quarter; standard deviation 0.02
            x = torch.randn(shape, device="cuda", generator=gen)
            y = torch.empty(shape, device="cuda").exponential_(generator=gen)
            y += torch.empty(shape, device="cuda").exponential_(generator=gen)
            x = x * torch.rsqrt(y * 0.5) * (0.02 / math.sqrt(2.0))
        elif dist == "laplace":       # 0.05 % of the entries 50 times larger
            x = torch.empty(shape, device="cuda").exponential_(1.0 / 0.015, generator=gen)
            u = torch.rand(shape, device="cuda", generator=gen)
            x = torch.where(u < 0.5, -x, x)
            x = torch.where((u * 1024.0).frac() < 0.0005, 50.0 * x, x)
        else:                         # normal with 1 % Student-t(2)
            x = torch.randn(shape, device="cuda", generator=gen) * 0.02
            y = torch.empty(shape, device="cuda").exponential_(generator=gen)
            u = torch.rand(shape, device="cuda", generator=gen)
            x = torch.where(u < 0.01, x * torch.rsqrt(y), x)
        W[r:r + shape[0]] = x.bfloat16()
    if dist == "student_t4":          # outlier input channels
        n = max(1, cols // 1000)
        W[:, torch.randperm(cols, device="cuda", generator=gen)[:n]] *= 20.0


def _column_weights(cols, gen, zero_pct=0):
    """Second moments of input channels: log-normal, 0.5 % of the channels 10-30 times larger in amplitude, mean 1."""
    s = torch.exp(0.5 * torch.randn(cols, device="cuda", generator=gen, dtype=torch.float64))
    big = torch.rand(cols, device="cuda", generator=gen) < 0.005
    s = torch.where(big, s * (10.0 + 20.0 * torch.rand(cols, device="cuda", generator=gen)), s)
    h = s * s
    h = torch.clamp(h / h.mean(), 2.0 ** -20, 2.0 ** 20)
    if zero_pct:
        h[torch.rand(cols, device="cuda", generator=gen) < zero_pct / 100.0] = 0.0
    return h.float()


def _report(raw):
    """The fields of soar_result(s) as typed views of their bytes: status and iterations, alpha and amax, the three errors,
    the two counters, the traces."""
    return [raw[..., 0:8].view(torch.int32), raw[..., 8:16].view(torch.float32), raw[..., 16:40].view(torch.float64),
            raw[..., 40:56].view(torch.int64), raw[..., 56:56 + 16 * (api.MAX_ITERS + 1)].view(torch.float64)]


def _outputs(b):
    """Everything one quantized matrix consists of."""
    return [t for t in (b.packed, b.scales, b.scales_sw, b.alpha) if t is not None] + _report(b.result)


def _model_buffers(shapes, cfg):
    """Output buffers of a list of matrices, as a quantized checkpoint holds them: one allocation per kind of output with
    each matrix's part on a 256-byte boundary.  Returns the matrices' ``QuantBuffers`` and the allocations."""
    def parts(sizes):
        starts, at = [], 0
        for n in sizes:
            starts.append(at)
            at += (n + 255) // 256 * 256
        flat = torch.zeros(at, dtype=torch.uint8, device="cuda")
        return flat, [flat[a:a + n] for a, n in zip(starts, sizes)]

    packed, p = parts([r * c // 2 for r, c in shapes])
    flats, none = [packed], [None] * len(shapes)
    lin = sw = none
    if cfg.scale_layout & LINEAR:
        flat, lin = parts([r * c // 16 for r, c in shapes])
        flats.append(flat)
    if cfg.scale_layout & SWIZZLED:
        flat, sw = parts([api.soar_swizzled_scale_bytes(r, c) for r, c in shapes])
        flats.append(flat)
    alpha = torch.zeros(len(shapes), dtype=torch.float32, device="cuda")
    results = torch.zeros((len(shapes), 56 + 16 * (api.MAX_ITERS + 1)), dtype=torch.uint8, device="cuda")
    bufs = [api.QuantBuffers(packed=p[i].view(r, c // 2), scales=None if lin[i] is None else lin[i].view(r, c // 16),
                             scales_sw=sw[i], alpha=alpha[i:i + 1], result=results[i], workspace=None)
            for i, (r, c) in enumerate(shapes)]
    return bufs, flats + [alpha] + _report(results)


def prepare(case, seed):
    op = case["op"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    shapes = _shapes(case)
    Ws = []
    for rows, cols in shapes:
        full = torch.empty((rows, cols * case.get("shards", 1)), dtype=torch.bfloat16, device="cuda")
        _fill(full, case["dist"], gen)
        Ws.append(full[:, (case.get("shards", 1) // 2) * cols:][:, :cols])
    s = dict(op=op, Ws=Ws)
    if op == "mxfp4":
        rows, cols = shapes[0]
        out = api.MxBuffers(torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda"),
                            torch.empty((rows, cols // 32), dtype=torch.uint8, device="cuda"),
                            torch.empty(56, dtype=torch.uint8, device="cuda"))
        r = out.result
        s.update(n_beta=case["n_beta"], out=out,
                 outputs=[out.packed, out.scales, r[0:8].view(torch.int32), r[8:12].view(torch.float32),
                          r[16:32].view(torch.float64), r[40:56].view(torch.int64)])
        return s
    if op == "error":
        cfg = api.soar_default_cfg(api.PRESET_SINGLE_PASS, scale_layout=case["layout"])
        b = api.soar_quantize(Ws[0], cfg)
        s.update(packed=b.packed, scales=b.scales if case["layout"] == LINEAR else b.scales_sw, alpha=b.alpha,
                 layout=case["layout"], h=_column_weights(shapes[0][1], gen) if case["weighted"] else None,
                 out=torch.empty(2, dtype=torch.float64, device="cuda"))
        return s
    cfg = api.soar_default_cfg(PRESETS[case["preset"]], scale_layout=case["layout"])
    if case.get("deterministic"):
        cfg.flags |= api.FLAG_DETERMINISTIC
    s["cfg"] = cfg
    if op == "host":
        s["hosts"] = [api.alloc_host_buffers(r, c, cfg) for r, c in shapes]
        for hb, W in zip(s["hosts"], Ws):
            hb.W.copy_(W)
        del s["Ws"]
        s["pipe"] = api.HostPipeline(shapes, cfg, depth=3)
        s["outputs"] = [_outputs(hb) for hb in s["hosts"]]
        return s
    if op == "quantize":
        s["out"] = api.alloc_buffers(*shapes[0], cfg)
        s["outputs"] = _outputs(s["out"])
        return s
    s["outs"], s["outputs"] = _model_buffers(shapes, cfg)
    if op == "weighted":
        s["hs"] = [_column_weights(c, gen, case["zero_pct"]) for _, c in shapes]
        need = sum(api.soar_weighted_workspace_bytes(r, c, cfg) for r, c in shapes)
    else:
        need = api.soar_batch_workspace_bytes(Ws, s["outs"], cfg)
    s["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    op = s["op"]
    if op == "quantize":
        api.soar_quantize(s["Ws"][0], s["cfg"], s["out"])
        return s["outputs"]
    if op == "batch":
        api.soar_quantize_batch(s["Ws"], s["cfg"], s["outs"], s["workspace"])
        return s["outputs"]
    if op == "weighted":
        api.soar_quantize_weighted_batch(s["Ws"], s["hs"], s["cfg"], s["outs"], s["workspace"])
        return s["outputs"]
    if op == "mxfp4":
        api.soar_mx_quantize(s["Ws"][0], n_beta=s["n_beta"], out=s["out"])
        return s["outputs"]
    if op == "error":
        if s["h"] is None:
            return api.soar_dequant_error(s["Ws"][0], s["packed"], s["scales"], s["alpha"], s["layout"], out=s["out"])
        return api.soar_dequant_error_weighted(s["Ws"][0], s["h"], s["packed"], s["scales"], s["alpha"], s["layout"],
                                               out=s["out"])
    s["pipe"].run(s["hosts"])
    s["pipe"].synchronize()
    return s["outputs"]


def work(case):
    """Every weight read once, every code, scale byte and column weight moved once.  Operations: per weight the maximum and
    the square of the first pass, a product and a rounding per code vector tried, and the two sums of each (one trial for
    the max-based rule, four more per iteration of the search, at least one iteration)."""
    bytes_, flops = 0.0, 0.0
    trials = {"rtn": 1, "single_pass": 2, "cjso_only": 2, "coupled_pair": 3}.get(case.get("preset"), 5)
    for rows, cols in _shapes(case):
        n = float(rows) * cols
        bytes_ += 2.0 * n + 0.5 * n
        if case["op"] == "mxfp4":
            bytes_ += n / 32
            flops += n * (3 + 6 * (4 if case["n_beta"] else 1))
            continue
        layout = case["layout"]
        bytes_ += (n / 16 if layout & LINEAR else 0) + (api.soar_swizzled_scale_bytes(rows, cols) if layout & SWIZZLED else 0)
        if case["op"] == "weighted" or case.get("weighted"):
            bytes_ += 4.0 * cols
        flops += n * (6 if case["op"] == "error" else 3 + 6 * trials)
    return dict(bytes=bytes_, flops=flops)


def tolerance(case):
    """Tensor-wide sums are binary64 additions in no fixed order: the errors of the report repeat to about 1e-13.  Where a
    global scale is solved from such sums it is rounded to binary32, and a last bit that falls the other way can move the
    few weights that sit on a rounding boundary."""
    if case["op"] == "error":
        return dict(rel=1e-12)
    if case["op"] == "mxfp4" or case.get("preset") == "rtn":
        return dict(rel=1e-11, differ=0.0)
    return dict(rel=2e-7, differ=1e-5)
