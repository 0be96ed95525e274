"""Timed cases of the fused M+Adam step, through the package's public entry points.

A case is one optimizer step (or one run of the matrix-fitting diagnostic) of
a program that holds its parameters, gradients and moments on the GPU: a
parameter list's shapes, its storage formats, its rounding, its Algorithm 2
options, where its arrays lie in memory, and the entry point that it calls.
Shapes are those of the repository's workloads (GPT-2 small, LLaMA-style
decoders of 1.5B and 7B parameters with fewer layers where the whole list is
not needed, a ragged list, a flat buffer) and generic ones of the same kind.

Values are mid-training ones: moments are not zero, the step number starts at
1000, gradients have a standard deviation of their own in every tensor.
Every result of the library is defined bit for bit, so outputs are compared
exactly.
"""
import math
import random

import torch

from paper_2607_10611_gb300 import _native as N
from paper_2607_10611_gb300.optimizer import MPAdam
from paper_2607_10611_gb300.toy import ToyDiagnostic

FIRST_STEP = 1000
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
BLOCK, FP4_BLOCK = 32, 16  # weights per block scale


# ---------------------------------------------------------------------------
# Parameter lists: (elements, role) per tensor
# ---------------------------------------------------------------------------
def _gpt2(layers, d, vocab, ctx):
    s = [(vocab * d, "embedding"), (ctx * d, "embedding")]
    for _ in range(layers):
        s += [(d, "norm"), (d, "bias"), (3 * d * d, "matrix"), (3 * d, "bias"), (d * d, "matrix"), (d, "bias"),
              (d, "norm"), (d, "bias"), (4 * d * d, "matrix"), (4 * d, "bias"), (4 * d * d, "matrix"), (d, "bias")]
    return s + [(d, "norm"), (d, "bias")]


def _llama(layers, d, ffn, vocab):
    s = [(vocab * d, "embedding")]
    for _ in range(layers):
        s += [(d * d, "matrix")] * 4 + [(d * ffn, "matrix")] * 3 + [(d, "norm")] * 2
    return s + [(d, "norm"), (vocab * d, "head")]


def _ragged(tensors, max_log2, list_seed):
    r = random.Random(list_seed)
    return [(max(1, round(math.exp(r.random() * max_log2 * math.log(2.0)))), "flat") for _ in range(tensors)]


def shapes(case):
    kind = case["list"]
    if kind == "flat":
        s = [(case["n"], "flat")]
    elif kind == "gpt2":
        s = _gpt2(case["layers"], case["d"], case["vocab"], case["ctx"])
    elif kind == "llama":
        s = _llama(case["layers"], case["d"], case["ffn"], case["vocab"])
    else:
        s = _ragged(case["tensors"], case["max_log2"], case["list_seed"])
    # "vectors": the group that trains without weight decay; "matrices": the one with it
    if case.get("group") == "vectors":
        s = [x for x in s if x[1] in ("norm", "bias")]
    elif case.get("group") == "matrices":
        s = [x for x in s if x[1] not in ("norm", "bias")]
    return s


def formats(case):
    wd = case["weights"]
    if wd in ("fp8_regime", "fp4_regime"):  # linear layers in the low format, the rest BF16
        low = "e4m3_b32" if wd == "fp8_regime" else "nvfp4"
        return [low if role == "matrix" else "bf16" for _, role in shapes(case)]
    return [wd] * len(shapes(case))


def listed():
    base = {"entry": "step", "grads": "bf16", "moments": "f32", "rounding": "stochastic", "layout": "separate"}
    gpt2 = {"list": "gpt2", "layers": 12, "d": 768, "vocab": 50257, "ctx": 1024}
    return [
        # The smallest call: the norms and biases of GPT-2 small, which train in a group without weight decay.
        dict(base, **gpt2, name="gpt2_vectors", group="vectors", weights="bf16", rounding="nearest"),
        # A flat buffer of 1 Mi parameters with binary32 gradients: a small model, or one shard of a larger one.
        dict(base, name="flat_1m", list="flat", n=1 << 20, weights="bf16", grads="f32", rounding="nearest", zeros=0.01),
        # The whole GPT-2 small list, its arrays in flat buffers.
        dict(base, **gpt2, name="gpt2", weights="bf16", layout="flat"),
        # The matrices of GPT-2 small in their group with AdamW's decay (the usual way to train it).
        dict(base, **gpt2, name="gpt2_matrices_decay", group="matrices", weights="bf16", wd_add=0.1),
        # A 7B-width decoder shard, everything BF16: the ordinary large-model step.
        dict(base, name="llama7_bf16", list="llama", layers=4, d=4096, ffn=11008, vocab=32000, weights="bf16",
             moments="bf16", layout="flat"),
        # The same width with Algorithm 2's clamps and decay on.
        dict(base, name="llama7_bf16_options", list="llama", layers=1, d=4096, ffn=11008, vocab=32000, weights="bf16",
             moments="bf16", wd_add=0.1, g_max=10.0, w_max=8.0),
        # The same width through the entry for programs whose device memory belongs to their own allocator.
        dict(base, name="llama7_noalloc", entry="noalloc", list="llama", layers=1, d=4096, ffn=11008, vocab=32000,
             weights="bf16", moments="bf16", rounding="nearest"),
        # The largest call: the 1.5B list in E4M3 with a scale per tensor.
        dict(base, name="llama15_e4m3", list="llama", layers=24, d=2048, ffn=5632, vocab=32000, weights="e4m3",
             layout="flat"),
        # FP8 training: block-scaled linears with their BF16 copy for the next forward pass, the rest BF16.
        dict(base, name="llama15_fp8_regime", list="llama", layers=8, d=2048, ffn=5632, vocab=32000,
             weights="fp8_regime", compute=True),
        # NVFP4 training, with stochastic rounding.
        dict(base, name="llama15_fp4_regime", list="llama", layers=8, d=2048, ffn=5632, vocab=32000,
             weights="fp4_regime", compute=True),
        # Ragged sizes, and gradients as a reducer leaves them: packed one after another in one bucket, so that most
        # of them start at odd elements.
        dict(base, name="ragged_bucket", list="ragged", tensors=4000, max_log2=18, list_seed=1, weights="bf16",
             layout="bucket", zeros=0.3),
        # The matrix-fitting diagnostic, 256 steps of the mixed regime at its full size.
        dict(name="toy_run", entry="toy", n=4096 * 4096, batch=65536, steps=256, mode="combined", split=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if rng.random() < 0.08:  # n, batch: powers of two, as the diagnostic wants them
        n = 1 << rng.randint(14, 24)
        split = rng.random() < 0.5
        return {"entry": "toy", "n": n, "batch": min(1 << rng.randint(8, 16), n // 4), "steps": log_int(1, 300),
                "mode": rng.choice(["additive", "multiplicative", "combined"]), "split": split}
    kind = rng.choice(["flat", "gpt2", "gpt2", "llama", "llama", "ragged"])
    case = {"entry": "step", "list": kind}
    if kind == "flat":
        case["n"] = log_int(1000, 200_000_000)
    elif kind == "gpt2":
        case.update(layers=rng.randint(2, 24), d=64 * rng.randint(2, 20), vocab=log_int(1000, 50257), ctx=log_int(128, 2048))
        case["group"] = rng.choice(["all", "all", "matrices", "vectors"])
    elif kind == "llama":
        d = 128 * rng.randint(1, 20)
        case.update(layers=rng.randint(1, 8), d=d, ffn=8 * round(d * rng.uniform(2.5, 4.0) / 8), vocab=log_int(1000, 32000))
        case["group"] = rng.choice(["all", "all", "all", "matrices", "vectors"])
    else:
        case.update(tensors=log_int(30, 6000), max_log2=rng.randint(10, 19), list_seed=rng.randrange(1 << 20), zeros=0.3)
    whole = kind in ("gpt2", "llama") and case["group"] != "vectors"
    case["weights"] = rng.choice(["bf16", "bf16", "bf16", "e4m3"] + (["fp8_regime", "fp4_regime"] if whole else []))
    if case["weights"] in ("fp8_regime", "fp4_regime"):
        case["compute"] = rng.random() < 0.8
    case["grads"] = rng.choice(["bf16", "bf16", "f32"])
    case["moments"] = rng.choice(["f32", "f32", "bf16"])
    case["rounding"] = rng.choice(["stochastic", "stochastic", "nearest"])
    case["layout"] = rng.choice(["separate", "flat", "bucket"])
    if case.get("group") != "vectors" and rng.random() < 0.35:
        case["wd_add"] = rng.choice([0.01, 0.1])
        if rng.random() < 0.3:
            case.update(g_max=10.0, w_max=8.0)
    if case["weights"] == "bf16" and rng.random() < 0.15:
        case["entry"] = "noalloc"
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _toy_prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, half = case["n"], case["n"] // 2
    z = torch.randn(n, generator=g, device="cuda")
    if case["split"]:  # mixed scales: small targets from zero, large ones from 100
        ws = torch.cat([1e-4 * z[:half], 900.0 * z[half:].abs().clamp(min=1.0 / 900.0)])
        w = torch.cat([torch.zeros(half, device="cuda"), torch.full((n - half,), 100.0, device="cuda")])
        c = (1e8, 1e-7)
    else:  # sign flip
        ws = torch.where(z < 0, -1.0, 1.0)
        w, c = -ws, (1.0, 1.0)
    lr = 3072.0 * case["batch"] / 65536  # the gradient of one sample goes as 1 / batch
    toy = ToyDiagnostic(w.to(torch.bfloat16), ws, mode=case["mode"], lr_add=lr, lr_mul=lr, batch=case["batch"],
                        c_lo=c[0], c_hi=c[1], split=case["split"], seed=seed)
    return {"toy": toy, "t": 1, "losses": torch.zeros(case["steps"], dtype=torch.float64, device="cuda")}


def _split(buf, ns, pad):
    """Views of the tensors in a buffer, each starting at a multiple of `pad` elements."""
    views, o = [], 0
    for n in ns:
        views.append(buf[o:o + n])
        o = -(-(o + n) // pad) * pad
    return views


def _views(ns, pad, dtype):
    """A zeroed buffer for a list of tensors, and their views."""
    o = 0
    for n in ns:
        o = -(-(o + n) // pad) * pad
    buf = torch.zeros(o, dtype=dtype, device="cuda")
    return buf, _split(buf, ns, pad)


# "separate": every array starts where an allocator puts it (a 256-element boundary of a pool); "flat": tensors
# follow one another at multiples of 8 elements, as in the library's own index space; "bucket": as "separate", but
# the gradients are packed without padding.
def _pad(case, grads=False):
    return 8 if case["layout"] == "flat" else 1 if grads and case["layout"] == "bucket" else 256


def _fill(bufs, parts, sizes, pad, dtype):
    """Copies the tensors' parts (None: the tensor has none) into one buffer; the views, None where there is none."""
    buf, views = _views([n if p is not None else 0 for n, p in zip(sizes, parts)], pad, dtype)
    for v, p in zip(views, parts):
        if p is not None:
            v.copy_(p)
    bufs.append(buf)
    return [v if p is not None else None for v, p in zip(views, parts)]


def _block_codes(w):
    """E4M3 codes and FP16 power-of-two scales of 32-weight blocks."""
    n = w.numel()
    x = torch.nn.functional.pad(w, (0, -n % BLOCK)).view(-1, BLOCK)
    a = x.abs().amax(1)
    k = torch.where(a > 0, torch.ceil(torch.log2(a / 448.0)), torch.full_like(a, -12.0)).clamp_(-24, 15)
    sc = torch.exp2(k)
    q = (x / sc[:, None]).clamp_(-448.0, 448.0).reshape(-1)[:n].to(torch.float8_e4m3fn).view(torch.uint8)
    return q, sc.to(torch.float16)


FP4_SCALE = 2.0 ** -12  # tensor scale of the NVFP4 weights: block scales of a 0.02 draw near 112 of 448


def _fp4_codes(w):
    """Packed E2M1 codes and E4M3 scale codes of 16-weight blocks."""
    n = w.numel()
    vals = torch.arange(1, 127, dtype=torch.uint8, device=w.device).view(torch.float8_e4m3fn).float()
    x = torch.nn.functional.pad(w, (0, -n % FP4_BLOCK)).view(-1, FP4_BLOCK)
    i = torch.bucketize(x.abs().amax(1) / (6.0 * FP4_SCALE), vals).clamp_(max=125)
    x = (x / (vals[i] * FP4_SCALE)[:, None]).reshape(-1)[:n]
    mid = torch.tensor([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0], device=w.device)
    c = torch.bucketize(x.abs(), mid, out_int32=True).to(torch.uint8) + 8 * (x < 0).to(torch.uint8)
    c = torch.nn.functional.pad(c, (0, n % 2))
    return c[0::2] | (c[1::2] << 4), (i + 1).to(torch.uint8)


E4M3_EXP = -11  # exponent the E4M3 weights are stored with: 6 sigma, and a norm gain's 1, fit under 448 * 2^e


def _e4m3_exp(role):
    return -8 if role == "norm" else E4M3_EXP


def prepare(case, seed):
    if case["entry"] == "toy":
        return _toy_prepare(case, seed)
    spec, fmts = shapes(case), formats(case)
    ns = [n for n, _ in spec]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    host = random.Random(seed)
    sd = [math.exp(host.uniform(math.log(1e-5), math.log(1e-2))) for _ in ns]  # of each tensor's gradients

    # binary32 draws, then each in its storage type and place
    wf, wv = _views(ns, _pad(case), torch.float32)
    wf.normal_(generator=gen).mul_(0.02)
    if case.get("zeros"):
        wf[torch.rand(wf.numel(), generator=gen, device="cuda") < case["zeros"]] = 0.0
    norms = [x for x, (_, role) in zip(wv, spec) if role == "norm"]
    if norms:
        torch._foreach_add_(norms, 1.0)
    md = TORCH[case["moments"]]
    x, xv = _views(ns, _pad(case), torch.float32)

    def place(draws, dtype):  # padding stays zero
        buf, views = _views(ns, _pad(case), dtype)
        torch._foreach_copy_(views, _split(draws, ns, _pad(case)))
        return buf, views

    x.normal_(generator=gen).mul_(0.3)
    torch._foreach_mul_(xv, sd)
    m, mv = place(x, md)
    x.uniform_(0.5, 1.5, generator=gen)
    torch._foreach_mul_(xv, sd)
    v, vv = place(x.square(), md)
    ve, vev = place(x.mul_(wf.abs().add_(1e-3)).mul_(math.log(2.0)).square_(), md)
    x.normal_(generator=gen)
    torch._foreach_mul_(xv, sd)
    grad, gv = _views(ns, _pad(case, grads=True), TORCH[case["grads"]])
    torch._foreach_copy_(gv, xv)
    del x, xv

    s = {"t": FIRST_STEP, "grads": gv, "m": mv, "v": vv, "ve": vev, "grad_buffer": grad}
    out = {"m": m, "v": v, "ve": ve}
    scales, glob, compute, low = [None] * len(ns), [0.0] * len(ns), [None] * len(ns), "e4m3_b32"
    if case["weights"] == "bf16":
        out["w"], w = place(wf, torch.bfloat16)
    elif case["weights"] == "e4m3":
        torch._foreach_mul_(wv, [2.0 ** -_e4m3_exp(role) for _, role in spec])
        out["w"], w = place(wf.clamp_(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8), torch.uint8)
    else:
        low = "e4m3_b32" if case["weights"] == "fp8_regime" else "nvfp4"
        coded = [(_block_codes(y) if low == "e4m3_b32" else _fp4_codes(y)) if f == low else (None, None)
                 for y, f in zip(wv, fmts)]
        sizes = [(n + 1) // 2 if low == "nvfp4" else n for n in ns]
        block = BLOCK if low == "e4m3_b32" else FP4_BLOCK
        bufs = []
        wl = _fill(bufs, [c for c, _ in coded], sizes, 256, torch.uint8)
        scales = _fill(bufs, [q for _, q in coded], [-(-n // block) for n in ns], 256,
                       torch.float16 if low == "e4m3_b32" else torch.uint8)
        wh = _fill(bufs, [None if f == low else y for y, f in zip(wv, fmts)], ns, 256, torch.bfloat16)
        w = [a if a is not None else b for a, b in zip(wl, wh)]
        out.update(w_low=bufs[0], scales=bufs[1], w=bufs[2])
        if low == "nvfp4":
            glob = [FP4_SCALE if f == low else 0.0 for f in fmts]
        if case.get("compute"):
            out["compute"], cv = _views([n if f == low else 0 for n, f in zip(ns, fmts)], 256, torch.bfloat16)
            compute = [c if f == low else None for c, f in zip(cv, fmts)]
    s.update(w=w, scales=scales, out=out)
    common = dict(grad_dtype=case["grads"], moment_dtype=case["moments"], rounding=case["rounding"], seed=seed)
    options = {k: case[k] for k in ("wd_add", "g_max", "w_max") if k in case}
    if case["entry"] == "noalloc":
        s["cfg"] = N.make_config(weight_dtype="bf16", **common, **options)
        s["tensors"] = [(a.data_ptr(), b.data_ptr(), c.data_ptr(), d.data_ptr(), n) for a, b, c, d, n in
                        zip(w, mv, vv, vev, ns)]
        return s
    mixed = case["weights"] in ("fp8_regime", "fp4_regime")
    s["opt"] = MPAdam(w, mv, vv, vev, weight_dtype=fmts if mixed else case["weights"], **common,
                      fp8_exp=[_e4m3_exp(role) for _, role in spec] if case["weights"] == "e4m3" else None,
                      first_step=FIRST_STEP, block_scales=scales if mixed else None,
                      compute=compute if mixed else None, global_scales=glob if mixed else None, **options)
    if case["weights"] == "e4m3":
        out["exp_ring"], out["amax_ring"] = s["opt"].fp8_exp_ring, s["opt"].fp8_amax_ring
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    if "toy" in state:
        toy, losses = state["toy"], state["losses"]
        toy.run(state["t"], losses.numel(), losses)
        state["t"] += losses.numel()
        return {"w": toy.w, "losses": losses}
    t = state["t"]
    state["t"] = t + 1
    if "opt" in state:
        state["opt"].step(state["grads"], t)
    else:
        N.mpadam_step_noalloc(state["tensors"], [g.data_ptr() for g in state["grads"]], state["cfg"], t,
                              stream=torch.cuda.current_stream().cuda_stream)
    return state["out"]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["entry"] == "toy":  # per sample: the weight read and written, the target read, the random lane
        samples = case["batch"] * case["steps"]
        return {"bytes": 8 * samples, "flops": 40 * samples}
    size = {"f32": 4, "bf16": 2}
    per = size[case["grads"]] + 6 * size[case["moments"]]
    total, flops = 0.0, 0
    for (n, _), f in zip(shapes(case), formats(case)):
        w = {"bf16": 2.0, "e4m3": 1.0, "e4m3_b32": 1.0 + 2.0 / BLOCK, "nvfp4": 0.5 + 1.0 / FP4_BLOCK}[f]
        total += n * (per + 2 * w + (2 if case.get("compute") and f != "bf16" else 0))
        flops += 30 * n
    return {"bytes": int(total), "flops": flops}


def tolerance(case):
    # Every stored bit is defined: each operation of the update is rounded on its own in binary32, in a stated order,
    # and random bits are keyed by seed, step and element.
    return "exact"


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _decoded(case, state):
    """The weights a step starts from, in 64 bits, tensor after tensor."""
    grid = torch.tensor([0, 0.5, 1, 1.5, 2, 3, 4, 6], dtype=torch.float64, device="cuda")
    for w, sc, f, (n, role) in zip(state["w"], state["scales"], formats(case), shapes(case)):
        if f == "bf16":
            yield w.double()
        elif f == "e4m3":
            yield w.view(torch.float8_e4m3fn).double().mul_(2.0 ** _e4m3_exp(role))
        elif f == "e4m3_b32":
            yield w.view(torch.float8_e4m3fn).double() * sc.double().repeat_interleave(BLOCK)[:n]
        else:
            c = torch.stack([w & 15, w >> 4], 1).reshape(-1)[:n].long()
            x = grid[c & 7] * (1 - 2 * (c >> 3))
            yield x * (sc.view(torch.float8_e4m3fn).double() * FP4_SCALE).repeat_interleave(FP4_BLOCK)[:n]


def exact(case, seed):
    """Moments and updated weights in 64 bits (weights before they are rounded into their format)."""
    if case["entry"] == "toy":
        return None  # hundreds of steps, each rounded to BF16: no value in 64 bits stays near them
    s = prepare(case, seed)
    b1, b2, lr, eps, tau, ln2 = 0.9, 0.999, 1e-3, 1e-8, 1e-8, math.log(2.0)
    c1, c2 = 1.0 - b1 ** FIRST_STEP, 1.0 - b2 ** FIRST_STEP
    fmts = formats(case)
    ns = [n for n, _ in shapes(case)]
    got = {k: None for k in s["out"]}  # codes, scales and rings are whole values
    views = {}
    for k in ("m", "v", "ve"):
        got[k], views[k] = _views(ns, _pad(case), torch.float64)
        got[k].copy_(s["out"][k])  # and their padding
    if "bf16" in fmts:
        pad = 256 if "w_low" in s["out"] else _pad(case)
        got["w"], views["w"] = _views([n if f == "bf16" else 0 for n, f in zip(ns, fmts)], pad, torch.float64)
        got["w"].copy_(s["out"]["w"])
    if case["weights"] == "fp8_regime" and case.get("compute"):  # an NVFP4 weight is too coarse to compare
        got["compute"], views["compute"] = _views([0 if f == "bf16" else n for n, f in zip(ns, fmts)], 256, torch.float64)
    inf = float("inf")
    for k, (w, g, f) in enumerate(zip(_decoded(case, s), s["grads"], fmts)):
        g, m, v, ve = g.double(), views["m"][k], views["v"][k], views["ve"][k]
        m.mul_(b1).add_(g, alpha=1 - b1)
        v.mul_(b2).add_(g * g, alpha=1 - b2)
        ge = g.mul_(w).mul_(ln2)
        ve.mul_(b2).add_(ge * ge, alpha=1 - b2)
        if f != "bf16" and "compute" not in views:
            continue
        ua = -lr * (m / c1) / ((v / c2).sqrt_() + eps) - lr * case.get("wd_add", 0.0) * w
        nn = (ge / ((ve / c2).sqrt_() + eps)).clamp(-case.get("g_max", inf), case.get("g_max", inf))
        um = (-lr * nn / w.abs().clamp(min=tau)).clamp(-0.75, 0.75)
        wn = (w + w * um + ua).clamp(-case.get("w_max", inf), case.get("w_max", inf))
        views["w" if f == "bf16" else "compute"][k].copy_(wn)
    return got
