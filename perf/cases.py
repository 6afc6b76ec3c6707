"""Work that users of the N:M library give it, as measurable cases.

Two halves of the path are covered, as in the tests and the benchmark: the integer linear layers that run compressed
weights (single projections, the four GEMMs of an encoder layer, whole chains with dynamically quantised activations),
and the projection that makes those weights (packing a model, the ADMM step with dense outputs, group-wise scales, the
ADMM-Dist scale search).  Shapes are those of BERT-base / BERT-large encoder layers on the batch x sequence grid
(sequences of 128 and 384, batch 1 .. 128) and generic ragged ones between and around them.

A case is a dict of plain values:
  kind = "linear"   one linear layer call: tokens, in, out, fmt, y
         "layer"    the four GEMMs of an encoder layer (QKV, attention output, FFN1, FFN2) back to back: tokens, hidden,
                    fmt, y; with pack = True the layer's weights are projected from fp32 first (as after a training step)
         "chain"    encoder layers in sequence, activations re-quantised between the GEMMs: tokens, hidden, layers, fmt
         "project"  fp32 weights -> N:M low-bit weights: layers, hidden, split (Q, K, V apart), fmt, dual, dense, scale
  fmt  = "n:m/bits" (kept : group, code bits), or "mixed" = formats rotating over the matrices
  y    = "f32", "q8" (8-bit codes at a static scale) or "bf16": what the linear layer writes
  dual = project W + U (ADMM) and not W alone; dense = write Z (and U + W - Z) besides the packed form
  scale = "row", "group" (one scale per 32 output channels) or "dist" (32 candidates per output channel)
"""
import math

import torch

import paper_2206_15014_b200 as nm

# Formats of the heterogeneous chain, of the configuration search, and every format the linear layer takes.
CHAIN_MIX = ("4:4/8", "2:4/8", "2:4/4", "1:4/8", "4:8/8")
SEARCH_MIX = ("2:4/8", "2:4/8", "4:4/8", "4:4/4", "2:4/4", "2:4/4")
FORMATS = ("2:4/8", "2:4/4", "4:4/8", "4:4/4", "1:4/8", "1:4/4", "2:8/8", "2:8/4", "1:8/8", "1:8/4", "4:8/8", "4:8/4")
GROUP_ROWS, CANDIDATES = 32, 32


def listed():
    return [
        # one attention output projection of BERT-base for one sequence of 128: the smallest call, all latency
        {"name": "projection_128tok", "kind": "linear", "tokens": 128, "in": 768, "out": 768, "fmt": "2:4/8", "y": "f32"},
        # BERT-large answering one question: batch 1, sequence 384, all 24 layers
        {"name": "bert_large_batch1", "kind": "chain", "tokens": 384, "hidden": 1024, "layers": 24, "fmt": "2:4/8"},
        # BERT-base with a weight format per GEMM as a configuration search picks them, batch 16 x 384
        {"name": "bert_base_mixed_chain", "kind": "chain", "tokens": 6144, "hidden": 768, "layers": 12, "fmt": "mixed"},
        # compression-aware training: a BERT-large layer's weights projected, then its GEMMs, 16384 tokens
        {"name": "bert_large_step", "kind": "layer", "tokens": 16384, "hidden": 1024, "fmt": "2:4/8", "y": "f32", "pack": True},
        # 4-bit weights x 8-bit activations, batch 32 x 384
        {"name": "bert_large_4bit", "kind": "layer", "tokens": 12288, "hidden": 1024, "fmt": "2:4/4", "y": "f32", "pack": False},
        # the largest batch of the inference grid, 128 x 384, bfloat16 hand-over
        {"name": "bert_large_bf16", "kind": "layer", "tokens": 49152, "hidden": 1024, "fmt": "2:4/8", "y": "bf16", "pack": False},
        # sequences of uneven length packed without padding, 8-bit activations between layers
        {"name": "bert_base_q8_ragged", "kind": "layer", "tokens": 3977, "hidden": 768, "fmt": "2:4/8", "y": "q8", "pack": False},
        # quantised but not pruned layer with a ragged output width
        {"name": "dense_int8_ragged", "kind": "linear", "tokens": 2085, "in": 1024, "out": 1002, "fmt": "4:4/8", "y": "f32"},
        # one configuration of the heterogeneous search: every matrix of BERT-base to its own format
        {"name": "search_projection", "kind": "project", "layers": 12, "hidden": 768, "split": True, "fmt": "mixed",
         "dual": False, "dense": False, "scale": "row"},
        # packing with one scale per 32 neurons (the paper's granularity), 4 bit
        {"name": "grouped_pack", "kind": "project", "layers": 6, "hidden": 1024, "split": False, "fmt": "2:4/4",
         "dual": True, "dense": False, "scale": "group"},
        # the ADMM Z- and U-update of all of BERT-large
        {"name": "admm_bert_large", "kind": "project", "layers": 24, "hidden": 1024, "split": False, "fmt": "2:4/8",
         "dual": True, "dense": True, "scale": "row"},
        # ADMM-Dist scales for BERT-base, 4 bit
        {"name": "dist_bert_base", "kind": "project", "layers": 12, "hidden": 768, "split": False, "fmt": "2:4/4",
         "dual": True, "dense": False, "scale": "dist"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("linear", "linear", "layer", "layer", "chain", "project", "project"))
    if kind == "linear":
        return {"kind": kind, "tokens": _log(rng, 1, 20000), "in": 128 * _log(rng, 1, 32), "out": _log(rng, 64, 4096),
                "fmt": rng.choice(FORMATS), "y": rng.choice(("f32", "f32", "q8", "bf16"))}
    hidden = 128 * rng.randint(2, 8)
    if kind == "layer":
        return {"kind": kind, "tokens": _log(rng, 64, 40000), "hidden": hidden, "fmt": rng.choice(("2:4/8",) * 4 + FORMATS),
                "y": rng.choice(("f32", "f32", "q8", "bf16")), "pack": rng.random() < 0.25}
    if kind == "chain":
        return {"kind": kind, "tokens": _log(rng, 32, 6144), "hidden": min(hidden, 768), "layers": rng.randint(1, 12),
                "fmt": rng.choice(("mixed", "2:4/8", "2:4/4", "4:4/8"))}
    scale = rng.choice(("row", "row", "group", "dist"))
    fmt = rng.choice(FORMATS + ("mixed", "2:4/8", "2:4/4"))
    # the search over candidate scales costs more per weight than the other forms, most of all where nothing is pruned
    most = 24 if scale != "dist" else (6 if fmt.startswith("4:4") else 12)
    return {"kind": kind, "layers": _log(rng, 1, most), "hidden": hidden if scale != "dist" else min(hidden, 768),
            "split": rng.random() < 0.5, "fmt": fmt, "dual": rng.random() < 0.7, "dense": rng.random() < 0.4, "scale": scale}


# ---- shapes ---------------------------------------------------------------------------------------------------------
def _fmt(text):
    pattern, bits = text.split("/")
    n, m = pattern.split(":")
    return int(n), int(m), int(bits)


def _gemms(hidden):
    """(in, out) of the four GEMMs of an encoder layer."""
    return ((hidden, 3 * hidden), (hidden, hidden), (hidden, 4 * hidden), (4 * hidden, hidden))


def _linears(case):
    """(tokens, in, out, n, m, bits) of every GEMM of a pass."""
    if case["kind"] == "linear":
        return [(case["tokens"], case["in"], case["out"]) + _fmt(case["fmt"])]
    got = []
    for layer in range(case.get("layers", 1)):
        for g, (k, out) in enumerate(_gemms(case["hidden"])):
            fmt = CHAIN_MIX[(layer + g) % len(CHAIN_MIX)] if case["fmt"] == "mixed" else case["fmt"]
            got.append((case["tokens"], k, out) + _fmt(fmt))
    return got


def _matrices(case):
    """(out, in, n, m, bits) of every matrix of a projection."""
    h, got = case["hidden"], []
    shapes = [(h, h)] * 4 + [(4 * h, h), (h, 4 * h)] if case.get("split") else [(o, k) for k, o in _gemms(h)]
    for layer in range(case.get("layers", 1)):
        for c, (out, k) in enumerate(shapes):
            fmt = SEARCH_MIX[(c + layer) % len(SEARCH_MIX)] if case["fmt"] == "mixed" else case["fmt"]
            got.append((out, k) + _fmt(fmt))
    return got


# ---- what a program has in hand -----------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(gen, shape, std):
    return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(0.0, std, generator=gen)


def _quantised(x, status):
    """int8 activations and their scale, as the library's own quantiser makes them."""
    amax = torch.zeros(1, dtype=torch.float32, device="cuda")
    sx = torch.empty(1, dtype=torch.float32, device="cuda")
    xq = torch.empty(x.shape, dtype=torch.int8, device="cuda")
    nm.nm_absmax(x, x.numel(), amax)
    nm.nm_quantize_act(x, x.numel(), amax, xq, sx)
    return xq, sx


class _Packed:
    """A packed weight matrix with its buffers."""

    def __init__(self, gen, k, out, n, m, bits, status, keep_dense=False):
        values, meta = nm.nm_packed_sizes(out, k, n, m, bits)
        self.values = torch.zeros(values, dtype=torch.uint8, device="cuda")
        self.meta = torch.zeros(meta // 4, dtype=torch.int32, device="cuda") if meta else None
        self.scales = torch.empty(out, dtype=torch.float32, device="cuda")
        self.bias = _normal(gen, (out,), 0.02)
        W = _normal(gen, (out, k), 0.02)
        nm.nm_project_pack(W, None, out, k, n, m, bits, self.values, self.meta, self.scales, status)
        self.W = W if keep_dense else None
        self.desc = nm.make_packed(out, k, n, m, bits, self.values, self.meta)
        self.k, self.out, self.fmt = k, out, (n, m, bits)


def _output(tokens, out, y):
    dtype = {"f32": torch.float32, "q8": torch.int8, "bf16": torch.bfloat16}[y]
    return torch.zeros((tokens, out), dtype=dtype, device="cuda")


def _prepare_linears(case, seed):
    gen = _generator(seed)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    calls, y = [], case["y"]
    for tokens, k, out, n, m, bits in _linears(case):
        w = _Packed(gen, k, out, n, m, bits, status, keep_dense=bool(case.get("pack")))
        x, sx = _quantised(_normal(gen, (tokens, k), 1.0), status)
        sx, sy = float(sx.item()), 1.0
        if y == "q8":  # the static output scale comes from a look at a few tokens ahead of time
            few = min(tokens, 128)
            probe = torch.empty((few, out), dtype=torch.float32, device="cuda")
            nm.nm_int_linear(x, few, w.desc, sx, w.scales, w.bias, probe)
            sy = max(float(probe.abs().max().item()), 1e-6) * 1.1 / 127.0
        calls.append((w, x, tokens, sx, sy, _output(tokens, out, y)))
    jobs = None
    if case.get("pack"):
        rows = [(w.W, _normal(gen, w.W.shape, 0.002)) + w.fmt + (w.values, w.meta, w.scales) for w, *_ in calls]
        bytes_ = nm.nm_pack_workspace_bytes(len(rows))
        jobs = (nm.make_pack_jobs(rows), len(rows), torch.empty(bytes_, dtype=torch.uint8, device="cuda"), bytes_, rows)
    return {"kind": case["kind"], "y": y, "calls": calls, "jobs": jobs, "status": status}


def _prepare_chain(case, seed):
    gen = _generator(seed)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    tokens, hidden = case["tokens"], case["hidden"]
    weights = [_Packed(gen, k, out, n, m, bits, status) for _, k, out, n, m, bits in _linears(case)]
    wide = 4 * hidden
    x = [torch.empty(tokens * wide, dtype=torch.int8, device="cuda") for _ in range(2)]
    y = torch.empty(tokens * wide, dtype=torch.float32, device="cuda")
    v = torch.empty((tokens, hidden), dtype=torch.float32, device="cuda")
    last = torch.empty((tokens, hidden), dtype=torch.float32, device="cuda")
    h0 = _normal(gen, (tokens, hidden), 1.0)
    n = len(weights)
    amax = torch.zeros(n, dtype=torch.float32, device="cuda")
    sx = torch.empty(n, dtype=torch.float32, device="cuda")
    steps = []
    for i, w in enumerate(weights):
        yi = last if i == n - 1 else y[: tokens * w.out].view(tokens, w.out)
        v_slice = yi[:, 2 * hidden:] if i % 4 == 0 else None  # QKV: the V part goes on
        steps.append((w, x[i & 1][: tokens * w.k].view(tokens, w.k), yi, v_slice, amax[i:i + 1], sx[i:i + 1]))
    return {"kind": "chain", "tokens": tokens, "steps": steps, "h0": h0, "v": v, "amax": amax, "sx": sx, "status": status}


def _prepare_project(case, seed):
    gen = _generator(seed)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    mats = _matrices(case)
    sizes = [nm.nm_packed_sizes(*x) for x in mats]
    up = lambda v: (v + 255) // 256 * 256
    values = torch.zeros(sum(up(v) for v, _ in sizes), dtype=torch.uint8, device="cuda")
    meta = torch.zeros(sum(up(m) for _, m in sizes) // 4, dtype=torch.int32, device="cuda")
    scales = torch.zeros(sum(up(4 * x[0]) for x in mats) // 4, dtype=torch.float32, device="cuda")
    weights = sum(x[0] * x[1] for x in mats)
    W = _normal(gen, (weights,), 0.02)
    U = _normal(gen, (weights,), 0.002) if case["dual"] else None
    Z = torch.zeros(weights, dtype=torch.float32, device="cuda") if case["dense"] else None
    N = torch.zeros(weights, dtype=torch.float32, device="cuda") if case["dense"] and case["dual"] else None
    rows, at_w, at_v, at_m, at_s = [], 0, 0, 0, 0
    for (out, k, n, m, bits), (vb, mb) in zip(mats, sizes):
        dense = lambda t: None if t is None else t[at_w:at_w + out * k].view(out, k)
        packed = (values[at_v:at_v + vb], meta[at_m:at_m + mb // 4] if mb else None, scales[at_s:at_s + out])
        rows.append((dense(W), dense(U), n, m, bits) + ((dense(Z), dense(N)) if case["dense"] else ()) + packed)
        at_w, at_v, at_m, at_s = at_w + out * k, at_v + up(vb), at_m + up(mb) // 4, at_s + up(4 * out) // 4
    jobs = nm.make_admm_jobs(rows) if case["dense"] else nm.make_pack_jobs(rows)
    bytes_ = nm.nm_admm_workspace_bytes(len(rows)) if case["dense"] else nm.nm_pack_workspace_bytes(len(rows))
    ws = torch.empty(bytes_, dtype=torch.uint8, device="cuda")
    call = {("row", False): nm.nm_project_pack_batched, ("row", True): nm.nm_admm_project_batched,
            ("group", False): nm.nm_project_pack_grouped_batched, ("group", True): nm.nm_admm_project_grouped_batched,
            ("dist", False): nm.nm_project_pack_dist_batched, ("dist", True): nm.nm_admm_project_dist_batched}
    more = {"row": (), "group": (GROUP_ROWS,), "dist": (CANDIDATES,)}[case["scale"]]
    args = (jobs, len(rows)) + more + (ws, bytes_, status)
    outs = [t for t in (values, meta, scales, Z, N) if t is not None and t.numel()]
    return {"kind": "project", "call": call[case["scale"], case["dense"]], "args": args, "outs": outs, "keep": (rows, W, U)}


def prepare(case, seed):
    if case["kind"] == "project":
        return _prepare_project(case, seed)
    return _prepare_chain(case, seed) if case["kind"] == "chain" else _prepare_linears(case, seed)


# ---- one pass -------------------------------------------------------------------------------------------------------------
def _run_linears(s):
    status, y = s["status"], s["y"]
    outs = []
    if s["jobs"]:
        arr, n, ws, ws_bytes, rows = s["jobs"]
        nm.nm_project_pack_batched(arr, n, ws, ws_bytes, status)
        outs = [t for r in rows for t in r[5:] if t is not None]
    for w, x, tokens, sx, sy, out in s["calls"]:
        if y == "f32":
            nm.nm_int_linear(x, tokens, w.desc, sx, w.scales, w.bias, out, status=status)
        elif y == "q8":
            nm.nm_int_linear_q8(x, tokens, w.desc, sx, w.scales, w.bias, sy, out, status=status)
        else:
            nm.nm_int_linear_bf16(x, tokens, w.desc, sx, w.scales, w.bias, out, status=status)
        outs.append(out)
    return outs


def _run_chain(s):
    tokens, status, steps, v = s["tokens"], s["status"], s["steps"], s["v"]
    s["amax"].zero_()
    src, absmax = s["h0"], True
    for i, (w, x, y, v_slice, amax, sx) in enumerate(steps):
        if absmax:  # no GEMM has left this tensor's maximum behind
            nm.nm_absmax(src, src.numel(), amax)
        nm.nm_quantize_act(src, src.numel(), amax, x, sx)
        if v_slice is not None or i + 1 == len(steps):
            nm.nm_int_linear_dsx(x, tokens, w.desc, sx, w.scales, w.bias, y, None, status=status)
        else:       # the GEMM's own running max|Y| feeds the next quantiser
            nm.nm_int_linear_dsx(x, tokens, w.desc, sx, w.scales, w.bias, y, steps[i + 1][4], status=status)
        src, absmax = y, v_slice is not None
        if absmax:
            v.copy_(v_slice)
            src = v
    return [y, s["sx"]]


def run(state):
    if state["kind"] == "project":
        state["call"](*state["args"])
        return state["outs"]
    return _run_chain(state) if state["kind"] == "chain" else _run_linears(state)


# ---- what a pass cannot do without ---------------------------------------------------------------------------------------------
def _packed_bytes(out, k, n, m, bits):
    return sum(nm.nm_packed_sizes(out, k, n, m, bits)) + 4 * out


def work(case):
    """Bytes: inputs read once and outputs written once; in a chain the fp32 result of a GEMM is an output of one call and
    the input of the next.  Operations: two per kept weight and token; in a projection two per weight (the sum and the
    division), in the scale search six per kept weight and candidate (quotient, rounding, distance, square, sum)."""
    if case["kind"] == "project":
        mats = _matrices(case)
        weights = sum(x[0] * x[1] for x in mats)
        kept = sum(x[0] * x[1] * x[2] / x[3] for x in mats)
        reads = 1 + (1 if case["dual"] else 0)
        writes = (1 + (1 if case["dual"] else 0)) if case["dense"] else 0
        flops = 2.0 * weights + (6.0 * CANDIDATES * kept if case["scale"] == "dist" else 0.0)
        return {"bytes": 4.0 * weights * (reads + writes) + sum(_packed_bytes(*x) for x in mats), "flops": flops}
    total, flops = 0.0, 0.0
    width = {"f32": 4, "q8": 1, "bf16": 2}[case.get("y", "f32")]
    for i, (tokens, k, out, n, m, bits) in enumerate(_linears(case)):
        total += _packed_bytes(out, k, n, m, bits) + 4.0 * out + tokens * k + width * tokens * out
        flops += 2.0 * tokens * k * out * n / m
        if case["kind"] == "chain":
            total += 4.0 * tokens * k + tokens * k  # the quantiser in front of the GEMM
        if case.get("pack"):
            total += 8.0 * out * k
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Packed values, metadata, scales, integer sums and the roundings behind them are defined bit for bit by the
    interface, and every path to them gives the same.  Only the scale search compares sums of double precision whose
    order is left open: a tie to the last bits may fall to a neighbouring candidate (1/64 of the scale) in a row here
    and there; with the sums in another order none of the 82944 rows of the listed case chose otherwise, and a row or two
    are allowed for."""
    if case["kind"] == "project" and case["scale"] == "dist":
        return {"rel": 1e-4, "max": 0.02, "differ": 1e-4}
    return "exact"
