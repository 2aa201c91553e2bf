"""The work that users of this library have it do, as cases that can be timed and compared.

A GEMV case is one decode step's linear layers (or one of them) through the C ABI or its Python
binding; a quantizer case is one weight matrix through ``qtea_quantize``. Layer shapes are those of
``synth.WORKLOADS``; sizes outside them are generic.

Fields of a GEMV case: ``shapes`` ("NxK" of every matrix of a layer), ``calls`` (which matrices share
a grouped call: "0,1,2;3" is two calls), ``layers``, ``M`` (batch rows), ``storage`` (2bit: one fp16
alpha per row; 2bit_groups: alpha and beta per row and 128 columns; 2bit_groups_fp8: the same with an
FP8 residual; base3: base-3 codes, one alpha per row; paper: base-3 codes, alpha and beta per row and
128 columns, FP8 residual), ``salient`` (share of the columns), ``massive`` (activation columns far above the others, as LLM hidden states show),
``act_bits`` and ``through`` (python: the binding; c: the C ABI with the problem records a program
keeps; graph: the same calls captured once in a CUDA graph and replayed, as a decode loop does).
"""
import ctypes
import math

import torch

import paper_2609_00224_gb300 as qt

# out x in of one decoder layer: q, k, v, o, gate, up, down (synth.LLAMA3_8B, QWEN3_14B, LLAMA3_70B)
LLAMA3_8B = "4096x4096,1024x4096,1024x4096,4096x4096,14336x4096,14336x4096,4096x14336"
QWEN3_14B = "5120x5120,1024x5120,1024x5120,5120x5120,17408x5120,17408x5120,5120x17408"
LLAMA3_70B = "8192x8192,1024x8192,1024x8192,8192x8192,28672x8192,28672x8192,8192x28672"
ONE_CALL = "0,1,2,3,4,5,6"
DECODER_ORDER = "0,1,2;3;4,5;6"  # q, k, v; then o; then gate, up; then down


def _gemv(name, shapes, M, storage="2bit", calls=ONE_CALL, layers=1, salient=0.03, massive=0, act_bits=16, through="c"):
    return dict(name=name, op="gemv", shapes=shapes, M=M, storage=storage, calls=calls, layers=layers, salient=salient,
                massive=massive, act_bits=act_bits, through=through)


def _quantize(name, N, K, group, bias, salient=0.03):
    return dict(name=name, op="quantize", N=N, K=K, group=group, bias=bias, salient=salient, fit_iters=4,
                rescale_iters=2)


def listed():
    return [
        # one small projection called from Python: the call where latency and the host path count
        _gemv("k_proj_m1_python", "1024x4096", 1, calls="0", through="python"),
        # the linear layers of a token through consecutive decoder layers, in the order a decoder can
        # issue them, replayed from a CUDA graph: single-stream decoding
        _gemv("decode_8b_m1_graph", LLAMA3_8B, 1, calls=DECODER_ORDER, layers=4, through="graph"),
        # the largest layer, its seven products in one call
        _gemv("layer_70b_m1", LLAMA3_70B, 1),
        # 2-bit codes with the paper's scales: alpha and beta per row and group of 128 columns
        _gemv("layer_8b_groups_m1", LLAMA3_8B, 1, storage="2bit_groups"),
        # decoding several sequences at once (or checking a few drafted tokens): the low batches
        _gemv("layer_14b_m4", QWEN3_14B, 4),
        _gemv("layer_14b_m16", QWEN3_14B, 16),
        # the paper's own storage (base-3 codes, group scales, FP8 residual) at one row, at a few, and
        # at the largest batch
        _gemv("layer_8b_paper_m1", LLAMA3_8B, 1, storage="paper"),
        _gemv("layer_8b_paper_m4", LLAMA3_8B, 4, storage="paper"),
        _gemv("layer_8b_paper_m16", LLAMA3_8B, 16, storage="paper"),
        # sizes that are multiples of nothing, rows of x unaligned, massive activations
        _gemv("ragged_m3_python", "3028x5003,516x1501", 3, calls="0;1", massive=2, through="python"),
        # quantizing a matrix to the paper's storage, and with the call's defaults (one alpha per row)
        _quantize("quantize_8b_down_groups", 4096, 14336, 128, True),
        _quantize("quantize_8b_q_rows", 4096, 4096, 0, False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.2:
        K = _log_int(rng, 128, 16384)
        N = 4 * max(1, _log_int(rng, 64, min(16384, 60_000_000 // K)) // 4)
        return {k: v for k, v in _quantize("", N, K, rng.choice([0, 128]), rng.random() < 0.6,
                                           round(rng.uniform(0.0, 0.05), 3)).items() if k != "name"}
    storage = rng.choice(["2bit", "2bit", "2bit", "2bit_groups", "2bit_groups_fp8", "base3", "paper", "paper"])
    M = 1 if rng.random() < 0.4 else rng.randint(2, 16)
    n = 1 if rng.random() < 0.5 else rng.randint(2, 4)
    K0 = _log_int(rng, 256, 28672)
    shapes = []
    for _ in range(n):
        K = K0 if rng.random() < 0.7 else _log_int(rng, 256, 28672)
        if rng.random() < 0.6:
            K = max(128, K // 128 * 128)  # real layers; the others are ragged
        N = 4 * max(1, _log_int(rng, 128, min(32768, 100_000_000 // K)) // 4)
        shapes.append("%dx%d" % (N, K))
    calls = ",".join(map(str, range(n))) if rng.random() < 0.6 else ";".join(map(str, range(n)))
    c = _gemv("", ",".join(shapes), M, storage, calls, 1, round(rng.uniform(0.0, 0.06), 3), rng.choice([0, 0, 2]),
              rng.choice([16, 16, 16, 24]), rng.choice(["c", "c", "python"]))
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------- operands

def _shapes(case):
    return [tuple(int(t) for t in s.split("x")) for s in case["shapes"].split(",")]


def _salient_count(K, frac):
    return min(K, 8 * int(math.floor(frac * K / 8 + 0.5)))


def _grouped(case):
    return case["storage"] in ("2bit_groups", "2bit_groups_fp8", "paper")


def _fp8(case):
    return case["storage"] in ("2bit_groups_fp8", "paper")


def _half_uniform(g, shape, lo, hi):
    return (torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo).half()


def _half_normal(g, shape, std):
    return (torch.randn(shape, generator=g, device="cuda") * std).half()


def _matrix(case, seed, index, N, K):
    """The operands of one matrix, from the seed alone: a model's weights as they would be stored
    (P(-1, 0, +1) = 0.3, 0.4, 0.3) and one batch of activations."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 4096 + index)
    M, s = case["M"], _salient_count(K, case["salient"])
    G = (K + 127) // 128 if _grouped(case) else 1
    T = torch.empty((N, K), dtype=torch.int8, device="cuda")
    for r in range(0, N, 4096):
        u = torch.rand((min(N, r + 4096) - r, K), generator=g, device="cuda")
        T[r:r + 4096] = (u > 0.7).to(torch.int8) - (u < 0.3).to(torch.int8)
    alpha = _half_uniform(g, (N, G), 0.01, 0.05)
    scale = torch.stack((alpha, _half_normal(g, (N, G), 0.002)), dim=2) if _grouped(case) else alpha
    v = _half_uniform(g, (K,), 0.8, 1.2)
    x = _half_normal(g, (M, K), 1.0)
    if case["massive"]:
        x[:, torch.randperm(K, generator=g, device="cuda")[:case["massive"]]] *= 100
    sal = torch.randperm(K, generator=g, device="cuda")[:s].sort().values.to(torch.int32)
    rvals = _half_normal(g, (N // 4, s), 0.02)
    if _fp8(case):
        rvals = rvals.to(torch.float8_e4m3fn).view(torch.uint8)
    pos = torch.randint(0, 4, (N // 4, s), generator=g, device="cuda", dtype=torch.uint8)
    quads = torch.zeros((N // 4, (s + 3) // 4 * 4), dtype=torch.uint8, device="cuda")
    quads[:, :s] = pos
    quads = quads.view(N // 4, (s + 3) // 4, 4)
    ridx = quads[..., 0] | (quads[..., 1] << 2) | (quads[..., 2] << 4) | (quads[..., 3] << 6)
    return dict(T=T, alpha=alpha, scale=scale.contiguous(), v=v, x=x, sal=sal, rvals=rvals, pos=pos,
                ridx=ridx.contiguous(), s=s)


class _Record(ctypes.Structure):  # qtea_gemv_problem of include/qtea.h
    _fields_ = [(f, ctypes.c_void_p) for f in ("x", "packed_ternary", "row_scale", "col_scale", "salient_idx",
                                               "residual_vals", "residual_idx", "y")]


def _quant_inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = (torch.randn((case["N"], case["K"]), generator=g, device="cuda") * 0.02).half().float()
    h = torch.randn((case["K"],), generator=g, device="cuda").exp().half().float()
    return W, h


def prepare(case, seed):
    if case["op"] == "quantize":
        W, h = _quant_inputs(case, seed)
        return dict(case=case, W=W, h=h, group=case["group"] or None, s=_salient_count(case["K"], case["salient"]))
    shapes, problems = _shapes(case), []
    for layer in range(case["layers"]):
        for j, (N, K) in enumerate(shapes):
            m = _matrix(case, seed, layer * len(shapes) + j, N, K)
            fmt = qt.QTEA_FMT_BASE3 if case["storage"] in ("base3", "paper") else qt.QTEA_FMT_2BIT
            lay = qt.qtea_pack_layout(m["T"], n_salient=m["s"], group_size=128 if _grouped(case) else None, fmt=fmt)
            options = (qt.QTEA_OPT_BIAS if _grouped(case) else 0) | (
                qt.QTEA_OPT_RESIDUAL_FP8 if _fp8(case) else 0)
            if options:
                lay.set_options(options)
            if case["act_bits"] != 16:
                lay.set_activation_precision(case["act_bits"])
            problems.append(dict(x=m["x"], layout=lay, row_scale=m["scale"], col_scale=m["v"],
                                 salient_idx=m["sal"] if m["s"] else None,
                                 residual_vals=m["rvals"] if m["s"] else None,
                                 residual_idx=m["ridx"] if m["s"] else None,
                                 y=torch.empty((case["M"], N), dtype=torch.float32, device="cuda")))
    calls = [[layer * len(shapes) + int(j) for j in call.split(",")]
             for layer in range(case["layers"]) for call in case["calls"].split(";")]
    state = dict(case=case, problems=problems, calls=[[problems[j] for j in call] for call in calls])
    state["records"] = []
    for call in state["calls"]:
        recs = (_Record * len(call))()
        for r, p in zip(recs, call):
            ptr = lambda k: p[k].data_ptr() if p[k] is not None else None
            r.x, r.packed_ternary, r.y = ptr("x"), p["layout"].handle.value, ptr("y")
            r.row_scale, r.col_scale, r.salient_idx = ptr("row_scale"), ptr("col_scale"), ptr("salient_idx")
            r.residual_vals, r.residual_idx = ptr("residual_vals"), ptr("residual_idx")
        state["records"].append(recs)
    state["out"] = [p["y"] for p in problems]
    if case["through"] == "graph":
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"], stream=stream):
            _c_calls(state)
    return state


def _c_calls(state):
    lib, stream, M = qt.load(), torch.cuda.current_stream().cuda_stream, state["case"]["M"]
    for recs in state["records"]:
        rc = lib.qtea_gemv_grouped(recs, len(recs), M, stream)
        if rc:
            raise qt.QteaError(rc, "qtea_gemv_grouped")


def run(state):
    case = state["case"]
    if case["op"] == "quantize":
        return qt.qtea_quantize(state["W"], state["h"], group_size=state["group"], n_salient=state["s"],
                                bias=case["bias"], fit_iters=case["fit_iters"], rescale_iters=case["rescale_iters"])
    if case["through"] == "graph":
        state["graph"].replay()
    elif case["through"] == "c":
        _c_calls(state)
    else:
        for call in state["calls"]:
            if len(call) == 1:
                qt.qtea_gemv(**call[0])
            else:
                qt.qtea_gemv_grouped(call)
    return state["out"]


def work(case):
    if case["op"] == "quantize":
        N, K = case["N"], case["K"]
        g = case["group"] or K
        s, G = _salient_count(K, case["salient"]), (K + g - 1) // g
        passes = 2 + 2 * case["fit_iters"] + 5 * case["rescale_iters"]  # per weight: mean, |W - beta|, refits, rescales
        return {"bytes": 5 * N * K + 4 * K + 2 * N * G * (2 if case["bias"] else 1) + 2 * K + 4 * s
                + (N // 4) * (2 * s + (s + 3) // 4), "flops": passes * N * K}
    total, flops, M = 0, 0, case["M"]
    for N, K in _shapes(case):
        s, groups = _salient_count(K, case["salient"]), (K + 127) // 128
        codes = N * groups * 26 if case["storage"] in ("base3", "paper") else N * ((K + 63) // 64) * 16
        scales = 4 * N * groups if _grouped(case) else 2 * N
        value = 1 if _fp8(case) else 2
        total += codes + scales + 2 * K + 4 * s + (N // 4) * (value * s + (s + 3) // 4) + 2 * M * K + 4 * M * N
        flops += 2 * M * N * K
    return {"bytes": total * case["layers"], "flops": flops * case["layers"]}


def exact(case, seed):
    if case["op"] == "quantize":
        return None  # codes, indices and binary16 patterns: whole numbers, which stay equal
    out = []
    for layer in range(case["layers"]):
        for j, (N, K) in enumerate(_shapes(case)):
            m = _matrix(case, seed, layer * len(_shapes(case)) + j, N, K)
            x, v, s = m["x"].double(), m["v"].double(), m["s"]
            y = torch.empty((case["M"], N), dtype=torch.float64, device="cuda")
            for r in range(0, N, 4096):  # dense rows of the weight matrix, a block at a time
                e = min(N, r + 4096)
                W = m["T"][r:e].double() * v
                if _grouped(case):
                    sc = m["scale"][r:e].double().repeat_interleave(128, dim=1)[:, :K]
                    W = W * sc[..., 0] + sc[..., 1]
                else:
                    W = W * m["alpha"][r:e].double()
                if s:
                    R = m["rvals"][r // 4:e // 4]
                    R = R.view(torch.float8_e4m3fn).float().double() if _fp8(case) else R.double()
                    rows = 4 * torch.arange((e - r) // 4, device="cuda")[:, None] + m["pos"][r // 4:e // 4].long()
                    W.index_put_((rows, m["sal"].long()[None, :].expand_as(rows)), R, accumulate=True)
                y[:, r:e] = x @ W.T
            out.append(y)
    return out
