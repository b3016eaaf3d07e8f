"""The workloads this library's speed is judged by.

Each case is a dict of plain values; `prepare` builds on the GPU what a
program holds before the call (packed weights, activations, output buffers,
workspaces, and for a decode loop the captured CUDA graph of its calls), `run`
is one pass through the public entry points of paper_2607_08779_gb300.sss.

kind        what it is in use
gemv        one sss_gemv call on one matrix, called eagerly: the smallest unit
            a program calls, where the call's latency is what counts
decode      one decode step through a stack of decoder layers, captured once
            as a CUDA graph and replayed, as a serving loop does.  Batch 1:
            four sss_gemv_multi launches per layer in dependency order
            ({q,k,v}, o, {gate,up}, down) with programmatic dependent launch,
            optionally on Q8_0 activations.  Batch 2..16: sss_gemv on each of
            the seven matrices
prefill     a prompt of m tokens through one decoder layer: four eager
            sss_gemm_multi calls, or with Q8_0 activations seven sss_gemm_q8
gemm        one eager sss_gemm
quantize    casting a decoder layer: sss_quantize on its seven fp32 matrices
rotate      sss_quantize_rotated on one matrix (rotation and casting in one)
lsq         sss_quantize_lsq on one matrix

Layer shapes are Llama3-8B's and Qwen3-32B's (the shapes of the benchmark and
its sweeps), and generic ones in the drawn cases.  Weights are heavy-tailed
with outlier input channels, activations N(0, 1) in bf16.
"""
import math

import torch

from paper_2607_08779_gb300 import sss

GRIDS = {"signed": 1, "unsigned": 0, "asym": 2}

LLAMA = {"d": 4096, "heads": 4096, "kv": 1024, "ffn": 14336}
QWEN = {"d": 5120, "heads": 8192, "kv": 1024, "ffn": 25600}


def listed():
    return [
        # the smallest call a program makes: one k_proj at batch 1
        dict(name="gemv_k_proj_q4", kind="gemv", n=1024, k=4096, q=4, group=32, grid="signed", batch=1),
        # single-user decoding at the three widths of the paper's formats; q=2
        # with the Q8_0 activations the paper's runtime pairs the formats with,
        # on the larger model
        dict(name="decode_llama_q4", kind="decode", layers=4, q=4, group=32, grid="signed", batch=1, act_q8=False, **LLAMA),
        dict(name="decode_llama_q3", kind="decode", layers=4, q=3, group=32, grid="signed", batch=1, act_q8=False, **LLAMA),
        dict(name="decode_qwen_q2_act8", kind="decode", layers=2, q=2, group=32, grid="signed", batch=1, act_q8=True, **QWEN),
        # a few users together, and a full batch on the min-max grid
        dict(name="decode_llama_q4_b4", kind="decode", layers=2, q=4, group=32, grid="signed", batch=4, act_q8=False, **LLAMA),
        dict(name="decode_llama_q2_b16_minmax", kind="decode", layers=2, q=2, group=64, grid="asym", batch=16, act_q8=False, **LLAMA),
        # prompts: the benchmark's 512 tokens through a layer, a long chunk of
        # 2048 on one large matrix (q=3, min-max), a short ragged prompt
        dict(name="prefill_llama_q4_m512", kind="prefill", m=512, q=4, group=32, grid="signed", act_q8=False, **LLAMA),
        dict(name="gemm_gate_q3_minmax_m2048", kind="gemm", n=14336, k=4096, m=2048, q=3, group=32, grid="asym"),
        dict(name="prefill_llama_q2_act8_m77", kind="prefill", m=77, q=2, group=64, grid="signed", act_q8=True, **LLAMA),
        # casting a layer, and the two pipelines composed with it: a rotation
        # of whole rows, and learned scales
        dict(name="quantize_llama_q4", kind="quantize", q=4, group=32, grid="signed", **LLAMA),
        dict(name="rotate_gate_q3", kind="rotate", n=14336, k=4096, block=4096, q=3, group=32, grid="signed"),
        dict(name="lsq_o_proj_q4", kind="lsq", n=4096, k=4096, q=4, group=32, grid="signed", steps=20, lr=0.01),
    ]


def _log_int(rng, lo, hi, step=1):
    """An integer from lo to hi, spread over its logarithm, in steps."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi, max(lo, round(v / step) * step)))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["gemv", "decode", "decode", "decode_b", "decode_b", "prefill", "gemm", "quantize", "rotate", "lsq"])
    q = rng.choice([2, 3, 4])
    group = rng.choice([32, 32, 64, 128])
    grid = rng.choice(["signed", "signed", "unsigned", "asym"])
    fmt = dict(q=q, group=group, grid=grid)
    if kind == "gemv":
        # rows of any number; mostly the common widths, sometimes one that is
        # a multiple of the group only
        k = _log_int(rng, 512, 16384, 256) if rng.random() < 0.7 else _log_int(rng, 4, 96) * group
        return dict(kind="gemv", n=_log_int(rng, 64, 16384), k=k, batch=rng.choice([1, 1, 2, 4, 7, 16]), **fmt)
    if kind in ("decode", "decode_b", "prefill", "quantize"):
        d = _log_int(rng, 1024, 5120, 256)
        layer = dict(d=d, heads=_log_int(rng, max(1024, d // 2), 2 * d, 256), kv=rng.choice([256, 512, 1024]),
                     ffn=_log_int(rng, 2 * d, 14336, 256))
        if kind == "decode":
            return dict(kind="decode", layers=rng.choice([1, 2, 4]), batch=1, act_q8=rng.random() < 0.3, **fmt, **layer)
        if kind == "decode_b":
            return dict(kind="decode", layers=rng.choice([1, 2]), batch=_log_int(rng, 2, 16), act_q8=False, **fmt, **layer)
        if kind == "prefill":
            return dict(kind="prefill", m=_log_int(rng, 17, 512), act_q8=rng.random() < 0.3, **fmt, **layer)
        return dict(kind="quantize", **fmt, **layer)
    n, k = _log_int(rng, 256, 14336, 4), _log_int(rng, 1024, 8192, 256)
    if kind == "gemm":
        return dict(kind="gemm", n=n, k=min(k, 4096), m=_log_int(rng, 17, 2048), **fmt)
    if kind == "rotate":
        block = rng.choice([64, 128, 256, 1024, 4096])
        return dict(kind="rotate", n=n, k=max(block, k // block * block), block=block, **fmt)
    return dict(kind="lsq", n=_log_int(rng, 256, 4096), k=min(k, 4096), q=q, group=group,
                grid="unsigned" if grid == "unsigned" else "signed", steps=rng.choice([4, 10, 20]), lr=0.01)


# ---------------------------------------------------------------------------
# inputs, in plain torch
# ---------------------------------------------------------------------------

def _gen(seed, i):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1009 + i)
    return g


def _weights(n, k, seed, i):
    """fp32 [n, k]: Student-t with 4 degrees of freedom, scaled by 0.02, with
    0.5 % of the input channels 20 times larger."""
    g = _gen(seed, i)
    w = torch.empty((n, k), device="cuda").normal_(generator=g)
    v = torch.empty_like(w).uniform_(1e-6, 1.0, generator=g).log_()
    v += torch.empty_like(w).uniform_(1e-6, 1.0, generator=g).log_()  # chi2_4 = -2 (ln u1 + ln u2)
    w *= v.mul_(-0.5).rsqrt_().mul_(0.02)
    w[:, torch.randperm(k, generator=g, device="cuda")[: round(0.005 * k)]] *= 20.0
    return w


def _acts(m, k, seed, i):
    return torch.empty((m, k), device="cuda").normal_(generator=_gen(seed, 1000 + i)).to(torch.bfloat16)


def _cast(w, q, group, grid):
    """Integer codes [n, k/g, g] (0 .. 2^q - 1) and the fp16 scale and min of
    each group, as the formats define them."""
    n, k = w.shape
    w = w.view(n, k // group, group)
    mx, mn = w.amax(2, keepdim=True), w.amin(2, keepdim=True)
    if grid == "asym":
        s = (mx - mn) / (2 ** q - 1)
        u = torch.where(s > 0, ((w - mn) / s).round_(), 0.0).clamp_(0, 2 ** q - 1)
        return u.to(torch.uint8), s.squeeze(2).half(), mn.squeeze(2).half()
    half = 2 ** (q - 1)
    s = torch.maximum(mx, -mn) / half
    if grid == "signed":
        s = torch.where(mx > -mn, -s, s)
    u = torch.where(s != 0, (w / s).round_(), 0.0).clamp_(-half, half - 1).add_(half)
    return u.to(torch.uint8), s.squeeze(2).half(), None


def _pack(u, q):
    """The library's code layout: [n, k*q/8] bytes."""
    n, ng, g = u.shape

    def plane(v, bits):
        v = v.view(n, ng, -1, 8 // bits)
        out = v[..., 0].clone()
        for e in range(1, 8 // bits):
            out |= v[..., e] << (bits * e)
        return out

    if q == 3:
        return torch.cat([plane(u & 3, 2), plane(u >> 2, 1)], dim=2).reshape(n, -1)
    return plane(u, q).reshape(n, -1)


def _qtensor(n, k, c, seed, i):
    u, s, m = _cast(_weights(n, k, seed, i), c["q"], c["group"], c["grid"])
    return sss.QTensor(n, k, c["q"], c["group"], GRIDS[c["grid"]], _pack(u, c["q"]), s.view(torch.int16),
                       None if m is None else m.view(torch.int16))


def _dequantized(n, k, c, seed, i):
    """The same weights' values in 64 bits."""
    u, s, m = _cast(_weights(n, k, seed, i), c["q"], c["group"], c["grid"])
    s = s.double().unsqueeze(2)
    if m is None:
        return ((u.double() - 2 ** (c["q"] - 1)) * s).view(n, k)
    return (u.double() * s + m.double().unsqueeze(2)).view(n, k)


def _q8(x, wide):
    """bf16 x on the Q8_0 grid (blocks of 32), in 64 bits; the scale that the
    codes are taken with is fp32's, the stored one fp16's.  wide: the product
    of both is an fp16 operand of the tensor cores."""
    b = x.float().view(x.shape[0], -1, 32)
    m = b.abs().amax(2, keepdim=True)
    d = m / torch.full_like(m, 127.0)  # by a tensor: a scalar divisor would become a multiplication
    code = torch.where(d > 0, (b.double() / d.double()).round_(), 0.0).clamp_(-127, 127)
    v = code * d.half().double()
    return (v.half().double() if wide else v).view(x.shape)


def _groups(c):
    """The matrices of a layer by what they share: {q,k,v}, o, {gate,up}, down."""
    return [[(c["heads"], c["d"]), (c["kv"], c["d"]), (c["kv"], c["d"])], [(c["d"], c["heads"])],
            [(c["ffn"], c["d"]), (c["ffn"], c["d"])], [(c["d"], c["ffn"])]]


def _plan(c):
    """[(x index, rows of x, [(n, k, weight index)])] of one pass: each entry
    shares one x."""
    if c["kind"] == "gemv":
        return [(0, c["batch"], [(c["n"], c["k"], 0)])]
    if c["kind"] == "gemm":
        return [(0, c["m"], [(c["n"], c["k"], 0)])]
    out, w = [], 0
    for _ in range(c.get("layers", 1)):
        for mats in _groups(c):
            out.append((len(out), c.get("m", c.get("batch")), [(n, k, w + j) for j, (n, k) in enumerate(mats)]))
            w += len(mats)
    return out


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def prepare(case, seed):
    c = case
    st = {"case": c}
    if c["kind"] in ("quantize", "rotate", "lsq"):
        shapes = [s for grp in _groups(c) for s in grp] if c["kind"] == "quantize" else [(c["n"], c["k"])]
        st["w"] = [_weights(n, k, seed, i) for i, (n, k) in enumerate(shapes)]
        st["out"] = [sss.empty_qtensor(n, k, c["q"], c["group"], GRIDS[c["grid"]]) for n, k in shapes]
        return st
    st["calls"] = []
    for xi, rows, mats in _plan(c):
        x = _acts(rows, mats[0][1], seed, xi)
        qts = [_qtensor(n, k, c, seed, wi) for n, k, wi in mats]
        one = c["kind"] == "decode" and c["batch"] == 1
        ys = [torch.empty((n,) if one else (rows, n), device="cuda") for n, _, _ in mats]
        ws = None
        if c["kind"] in ("prefill", "gemm"):
            if c.get("act_q8") or len(qts) == 1:
                need = max(sss.sss_workspace_bytes(qt, rows, sss.OP_GEMM) for qt in qts)
            else:
                need = sss.sss_gemm_multi_workspace_bytes(qts, rows)
            ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        st["calls"].append((qts, x, ys, ws))
    if c["kind"] == "decode":
        # a serving loop's step: warmed up, then captured once
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode_calls(c, st["calls"])
        torch.cuda.current_stream().wait_stream(side)
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"]):
            _decode_calls(c, st["calls"])
    return st


def _decode_calls(c, calls):
    flags = sss.GEMV_PDL | sss.GEMV_WEIGHTS_READY | (sss.GEMV_ACT_Q8 if c["act_q8"] else 0)
    for qts, x, ys, _ in calls:
        if c["batch"] == 1:
            sss.sss_gemv_multi(qts, x[0], ys=ys, flags=flags)
        else:
            for qt, y in zip(qts, ys):
                sss.sss_gemv(qt, x, y=y)


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "decode":
        state["graph"].replay()
    elif kind in ("quantize", "rotate", "lsq"):
        grid = GRIDS[c["grid"]]
        for w, out in zip(state["w"], state["out"]):
            if kind == "quantize":
                sss.sss_quantize(w, c["q"], c["group"], grid, out=out)
            elif kind == "rotate":
                sss.sss_quantize_rotated(w, c["block"], c["q"], c["group"], grid, out=out)
            else:
                sss.sss_quantize_lsq(w, c["q"], c["group"], grid, c["steps"], c["lr"], out=out)
        return [[t for t in (o.codes, o.scales, o.mins) if t is not None] for o in state["out"]]
    else:
        for qts, x, ys, ws in state["calls"]:
            if kind == "gemv":
                sss.sss_gemv(qts[0], x, y=ys[0])
            elif kind == "gemm":
                sss.sss_gemm(qts[0], x, y=ys[0], workspace=ws)
            elif c["act_q8"]:
                for qt, y in zip(qts, ys):
                    sss.sss_gemm_q8(qt, x, y=y, workspace=ws)
            else:
                sss.sss_gemm_multi(qts, x, ys=ys, workspace=ws)
    return [ys for _, _, ys, _ in state["calls"]]


def _weight_bytes(n, k, c):
    return n * k * c["q"] / 8 + n * (k // c["group"]) * (4 if c["grid"] == "asym" else 2)


def work(case):
    c = case
    if c["kind"] in ("quantize", "rotate", "lsq"):
        shapes = [s for grp in _groups(c) for s in grp] if c["kind"] == "quantize" else [(c["n"], c["k"])]
        nbytes = sum(4 * n * k + _weight_bytes(n, k, c) for n, k in shapes)
        # per weight: max, min and rounding; the butterfly's stages; about nine
        # operations of a scale step
        per = 4 + (math.log2(c["block"]) + 1 if c["kind"] == "rotate" else 0) + 9 * c.get("steps", 0)
        return {"bytes": nbytes, "flops": per * sum(n * k for n, k in shapes)}
    nbytes = flops = 0
    for _, rows, mats in _plan(c):
        nbytes += 2 * rows * mats[0][1]
        for n, k, _ in mats:
            nbytes += _weight_bytes(n, k, c) + 4 * rows * n
            flops += 2 * rows * n * k
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    c = case
    if c["kind"] in ("quantize", "rotate", "lsq"):
        return "exact"  # codes and scales are defined bit for bit
    if c.get("m") or c.get("batch", 1) > 1:
        # one rounding of each weight to fp16, the tensor cores' operand:
        # 1.5e-4 measured against 64 bits
        return {"rel": 6e-4}
    return {"rel": 8e-6}  # exact products, 32-bit sums: 2e-6 measured


def exact(case, seed):
    c = case
    if c["kind"] in ("quantize", "rotate", "lsq"):
        return None  # whole numbers
    out = []
    for xi, rows, mats in _plan(c):
        x = _acts(rows, mats[0][1], seed, xi)
        x = _q8(x, bool(c.get("m"))) if c.get("act_q8") else x.double()
        ys = [x @ _dequantized(n, k, c, seed, wi).T for n, k, wi in mats]
        out.append([y[0] for y in ys] if c["kind"] == "decode" and c["batch"] == 1 else ys)
    return out
