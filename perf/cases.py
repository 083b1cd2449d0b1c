"""The work that users of the framework have it do, as cases that can be timed.

A case is one of six kinds of pass through the public entry points of `paper_2501_07139_b200`:

  gemv      one `fq_gemv` / `fq_gemv_batched` call on one layer
  calls     one token through a few decoder blocks, called as a serving loop has to call it when its own kernels
            (attention, norms) run in between: {q, k, v} and {gate, up} as small stacks, o and down as single calls
  decode    one token (or a batch of them) through a whole decoder stack in one `fq_gemv_stack` launch that
            honours the dependency order {q,k,v} -> o -> {gate,up} -> down -> next block
  switch    elastic hosting: a configuration is activated, some tokens are decoded, a smaller one is activated,
            some tokens are decoded; the layers are nested, so no weight moves
  prefill   a prompt (bf16 activations) through the matrices of one or more decoder blocks, one `fq_gemm` each
  quantize  preparing the stored variants of one matrix: `fq_quantize_layer` and `fq_pack_layer` at several widths

Layers have the shapes of Llama-2-7B (hidden 4096, FFN 11008) or 13B (5120, 13824) in the listed cases and other
multiples of 128 in the drawn ones.  Weights are N(0, 0.02) quantised with the library's own quantiser, activations
N(0, 1).  Mixed bit-widths are drawn per matrix, nested configurations per module (attention or MLP of a block).
"""
import random

import numpy as np
import torch

import paper_2501_07139_b200 as P

GROUP = 128
PACKED_CHOICES = (3, 4, 5, 6, 8)         # decode stacks: widths of the stored variants of a mixed configuration
PREFILL_CHOICES = (2, 3, 4, 6, 8)        # prefill: the same, down to two bits
QUANT_WIDTHS = (8, 5, 3)                 # an ensemble's stored precisions


def listed():
    return [
        # the smallest call there is in use: one attention matrix, one token; latency of a launch
        {"name": "gemv-1x4096x4096-4bit", "kind": "gemv", "fmt": "packed", "bits": 4, "n": 4096, "k": 4096, "batch": 1},
        # a small ragged projection for five sequences at once: no dimension is a multiple of a tile
        {"name": "gemv-5x1000x4224-nested5", "kind": "gemv", "fmt": "nested", "bits": 5, "n": 1000, "k": 4224, "batch": 5},
        # a serving loop that runs its own attention between the matrices
        {"name": "calls-7b-8blocks", "kind": "calls", "fmt": "packed", "hidden": 4096, "ffn": 11008, "blocks": 8, "batch": 1, "mix": 1},
        # the headline: one token through the whole mixed-bit 7B stack
        {"name": "decode-7b-packed", "kind": "decode", "fmt": "packed", "hidden": 4096, "ffn": 11008, "blocks": 32, "batch": 1, "mix": 1},
        # four sequences decoded together
        {"name": "decode-7b-packed-batch4", "kind": "decode", "fmt": "packed", "hidden": 4096, "ffn": 11008, "blocks": 16, "batch": 4, "mix": 2},
        # the largest decode batch on the larger model, nested layers at 4 bits on average
        {"name": "decode-13b-nested-batch8", "kind": "decode", "fmt": "nested", "hidden": 5120, "ffn": 13824, "blocks": 20, "batch": 8, "mix": 3},
        # memory gets short: the host goes from 7.0 to 3.5 bits on average and keeps decoding
        {"name": "switch-7b-nested", "kind": "switch", "fmt": "nested", "hidden": 4096, "ffn": 11008, "blocks": 32, "batch": 1, "tokens": 2, "mix": 4},
        # a short chat prompt
        {"name": "prefill-7b-77tokens", "kind": "prefill", "fmt": "packed", "hidden": 4096, "ffn": 11008, "blocks": 2, "tokens": 77, "mix": 5},
        # a longer one, ragged, on nested layers
        {"name": "prefill-7b-nested-600tokens", "kind": "prefill", "fmt": "nested", "hidden": 4096, "ffn": 11008, "blocks": 2, "tokens": 600, "mix": 6},
        # one calibration sequence through 13B layers at low bit-widths
        {"name": "prefill-13b-nested-2048tokens", "kind": "prefill", "fmt": "nested", "hidden": 5120, "ffn": 13824, "blocks": 1, "tokens": 2048, "mix": 7},
        # calibration-set evaluation: 4 x 2048 tokens
        {"name": "prefill-7b-8192tokens", "kind": "prefill", "fmt": "packed", "hidden": 4096, "ffn": 11008, "blocks": 1, "tokens": 8192, "mix": 8},
        # preparing an ensemble: one MLP matrix at the stored precisions 8, 5 and 3
        {"name": "quantize-11008x4096", "kind": "quantize", "fmt": "packed", "n": 11008, "k": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _width(rng, lo, hi):
    """A layer dimension: a multiple of 128, any of them."""
    return max(1, _log(rng, lo, hi) // GROUP) * GROUP


def draw(rng):
    kind = rng.choice(["gemv", "gemv", "calls", "decode", "decode", "switch", "prefill", "prefill", "prefill", "quantize"])
    fmt = rng.choice(["packed", "nested"])
    if kind == "gemv":
        return {"kind": kind, "fmt": fmt, "bits": rng.randint(2, 8), "n": _log(rng, 256, 16384), "k": _width(rng, 512, 14336),
                "batch": rng.choice([1, 1, 2, 3, 4, 5, 6, 7, 8])}
    if kind == "quantize":
        return {"kind": kind, "fmt": fmt, "n": _log(rng, 512, 11008), "k": _width(rng, 512, 4096)}
    hidden = _width(rng, 1024, 4096 if kind == "switch" else 5120)
    ffn = int(hidden * rng.uniform(2.0, 3.5)) // GROUP * GROUP
    c = {"kind": kind, "fmt": fmt, "hidden": hidden, "ffn": ffn, "mix": rng.randrange(1 << 30)}
    if kind == "calls":
        c.update(blocks=rng.randint(1, 8), batch=rng.choice([1, 1, 2, 4, 7]))
    elif kind == "decode":
        c.update(blocks=_log(rng, 1, 20), batch=rng.choice([1, 1, 1, 2, 3, 4, 6, 8]))
    elif kind == "switch":
        c.update(fmt="nested", blocks=_log(rng, 1, 16), batch=1, tokens=rng.randint(1, 3))
    else:
        c.update(blocks=1, tokens=_log(rng, 9, 4096))
    return c


# ------------------------------------------------------------------------------------------------ layers of a case
def _blocks(case):
    """(name, n_out, k_in, module, phase) of every matrix, in execution order."""
    h, f = case["hidden"], case["ffn"]
    out = []
    for b in range(case["blocks"]):
        for name, n, k, mod, ph in (("q", h, h, 0, 0), ("k", h, h, 0, 0), ("v", h, h, 0, 0), ("o", h, h, 0, 1),
                                    ("gate", f, h, 1, 2), ("up", f, h, 1, 2), ("down", h, f, 1, 3)):
            out.append((name, n, k, 2 * b + mod, 4 * b + ph))
    return out


def _module_bits(modules, average, lo, rng):
    """Widths per module: all at 8, then random modules go down one bit at a time until the mean is at most `average`."""
    bits = [8] * modules
    while sum(bits) / modules > average:
        m = rng.randrange(modules)
        if bits[m] > lo:
            bits[m] -= 1
    return bits


def _bits(case):
    """Bit-width per matrix; for "switch" a pair of such lists."""
    layers = _blocks(case)
    rng = random.Random(case["mix"])
    if case["kind"] == "switch":
        modules = 2 * case["blocks"]
        high = _module_bits(modules, 7.0, 3, rng)
        low = list(high)
        while sum(low) / modules > 3.5:                       # one-way: no module goes up
            m = rng.randrange(modules)
            if low[m] > 3:
                low[m] -= 1
        return [high[l[3]] for l in layers], [low[l[3]] for l in layers]
    if case["fmt"] == "nested":
        modules = _module_bits(2 * case["blocks"], 2.5 if case["kind"] == "prefill" else 4.0, 2, rng)
        return [modules[l[3]] for l in layers]
    choices = PREFILL_CHOICES if case["kind"] == "prefill" else PACKED_CHOICES
    return [rng.choice(choices) for _ in layers]


def _add_layer(fq, i, n, k, bits, fmt, gen):
    w = torch.randn((n, k), device="cuda", generator=gen).mul_(0.02)
    width, code = (8, P.FQ_FMT_PLANES) if fmt == "nested" else (bits, P.FQ_FMT_PACKED)
    codes, scales, zeros = P.fq_quantize_layer(w, width)
    fq.fq_pack_layer(i, codes, scales, zeros, width, code)


def _views(sizes, dtype):
    """One buffer, and a view of it per (rows, columns): the outputs of a pass lie side by side, 16-byte aligned."""
    offs, total = [], 0
    for r, c in sizes:
        offs.append(total)
        total += (r * c + 7) // 8 * 8
    buf = torch.zeros(total, dtype=dtype, device="cuda")
    return buf, [buf[o:o + r * c].view(r, c) for o, (r, c) in zip(offs, sizes)]


# ------------------------------------------------------------------------------------------------ state
def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "quantize":
        st["w"] = torch.randn((case["n"], case["k"]), device="cuda", generator=gen).mul_(0.02)
        st["fq"] = P.FlexQ(2)
        return st
    if kind == "gemv":
        st["fq"] = P.FlexQ(1)
        _add_layer(st["fq"], 0, case["n"], case["k"], case["bits"], case["fmt"], gen)
        st["fq"].fq_set_config([case["bits"]])
        st["x"] = torch.randn((case["batch"], case["k"]), device="cuda", generator=gen).half()
        st["y"] = torch.zeros((case["batch"], case["n"]), dtype=torch.float16, device="cuda")
        return st
    layers, bits = _blocks(case), _bits(case)
    fq = st["fq"] = P.FlexQ(len(layers))
    first = bits[0] if kind == "switch" else bits
    for i, (_, n, k, _, _) in enumerate(layers):
        _add_layer(fq, i, n, k, first[i], case["fmt"], gen)
    fq.fq_set_config(first)
    if kind == "prefill":
        m = case["tokens"]
        st["x"] = {k: torch.randn((m, k), device="cuda", generator=gen).bfloat16() for k in sorted({l[2] for l in layers})}
        st["y"] = [torch.zeros((m, l[1]), dtype=torch.bfloat16, device="cuda") for l in layers]
        return st
    b = case["batch"]
    xs = [torch.randn((b, l[2]), device="cuda", generator=gen).half() for l in layers]
    st["x"] = xs
    st["out"], ys = _views([(b, l[1]) for l in layers], torch.float16)
    st["y"] = ys
    index = list(range(len(layers)))
    if kind == "calls":
        # per block: stack (q, k, v), o, stack (gate, up), down
        st["stacks"] = []
        for i in range(0, len(layers), 7):
            st["stacks"].append((fq.stack_args(index[i:i + 3], xs[i:i + 3], ys[i:i + 3]),
                                 fq.stack_args(index[i + 4:i + 6], xs[i + 4:i + 6], ys[i + 4:i + 6])))
        return st
    phases = [l[4] for l in layers]
    st["args"] = fq.stack_args(index, xs, ys, phases)
    if kind == "switch":
        st["bits"] = bits
        st["out_low"], ys_low = _views([(b, l[1]) for l in layers], torch.float16)
        st["y_low"] = ys_low
        st["args_low"] = fq.stack_args(index, xs, ys_low, phases)
    return st


def run(st):
    case, fq = st["case"], st["fq"]
    kind = case["kind"]
    if kind == "gemv":
        if case["batch"] == 1:
            return fq.fq_gemv(0, st["x"], st["y"])
        return fq.fq_gemv_batched(0, st["x"], st["y"])
    if kind == "calls":
        b, x, y = case["batch"], st["x"], st["y"]
        for j, (qkv, gate_up) in enumerate(st["stacks"]):
            i = 7 * j
            fq.fq_gemv_stack_raw(qkv, b)
            fq.fq_gemv_batched(i + 3, x[i + 3], y[i + 3])
            fq.fq_gemv_stack_raw(gate_up, b)
            fq.fq_gemv_batched(i + 6, x[i + 6], y[i + 6])
        return st["out"]
    if kind == "decode":
        fq.fq_gemv_stack_raw(st["args"], case["batch"])
        return st["out"]
    if kind == "switch":
        high = fq.fq_set_config(st["bits"][0])
        for _ in range(case["tokens"]):
            fq.fq_gemv_stack_raw(st["args"], case["batch"])
        low = fq.fq_set_config(st["bits"][1])
        for _ in range(case["tokens"]):
            fq.fq_gemv_stack_raw(st["args_low"], case["batch"])
        return {"footprints": [high, low], "high": st["out"], "low": st["out_low"]}
    if kind == "prefill":
        for i, y in enumerate(st["y"]):
            fq.fq_gemm(i, st["x"][_k_of(case, i)], y)
        return st["y"]
    # quantize: a packed ensemble stores every width, a nested one the 8-bit parent
    out = []
    nested = case["fmt"] == "nested"
    for bits in (8,) if nested else QUANT_WIDTHS:
        codes, scales, zeros = P.fq_quantize_layer(st["w"], bits)
        store = fq.fq_pack_layer(int(nested), codes, scales, zeros, bits, P.FQ_FMT_PLANES if nested else P.FQ_FMT_PACKED)
        out += [codes, scales, zeros, store]
    return out


def _k_of(case, i):
    return case["ffn"] if i % 7 == 6 else case["hidden"]


# ------------------------------------------------------------------------------------------------ what a pass cannot do without
def _weight_bytes(n, k, bits):
    return n * k * bits / 8 + n * (k // GROUP) * 4           # codes, and a scale and a zero point per group


def work(case):
    kind = case["kind"]
    if kind == "quantize":
        n, k = case["n"], case["k"]
        widths = (8,) if case["fmt"] == "nested" else QUANT_WIDTHS
        meta = n * (k // GROUP) * 4
        return {"bytes": 4 * n * k + sum(n * k + meta + _weight_bytes(n, k, b) for b in widths), "flops": 0}
    if kind == "gemv":
        n, k, b = case["n"], case["k"], case["batch"]
        return {"bytes": _weight_bytes(n, k, case["bits"]) + 2 * b * (n + k), "flops": 2 * b * n * k}
    layers, bits = _blocks(case), _bits(case)
    if kind == "prefill":
        m = case["tokens"]
        x = sum(2 * m * k for k in {l[2] for l in layers})
        return {"bytes": x + sum(_weight_bytes(n, k, w) + 2 * m * n for (_, n, k, _, _), w in zip(layers, bits)),
                "flops": sum(2 * m * n * k for _, n, k, _, _ in layers)}
    b = case["batch"]
    passes = [(w, case["tokens"]) for w in bits] if kind == "switch" else [(bits, 1)]
    return {"bytes": sum(t * sum(_weight_bytes(n, k, w) + 2 * b * (n + k) for (_, n, k, _, _), w in zip(layers, ws)) for ws, t in passes),
            "flops": sum(t for _, t in passes) * sum(2 * b * n * k for _, n, k, _, _ in layers)}


def tolerance(case):
    """Quantising and packing is exact.  Against float64 sums decode shows 2.1e-4 with exact weights and up to 3.0e-4
    with weights rounded to fp16 (largest difference 1.1e-3), nearly all of it the one rounding of the sums to fp16;
    prefill, which rounds the weights and then the sums to bf16, shows 2.4e-3 (largest 1.3e-2)."""
    if case["kind"] == "quantize":
        return "exact"
    if case["kind"] == "prefill":
        return {"rel": 5e-3, "max": 0.05}
    return {"rel": 1e-3, "max": 5e-3}


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _weights64(n, k, bits, fmt, gen):
    """float64 [N][K]: the dequantised weights of a layer, from the real-valued ones that `_add_layer` draws."""
    w = torch.randn((n, k), device="cuda", generator=gen).mul_(0.02).double().view(n, k // GROUP, GROUP)
    width = 8 if fmt == "nested" else bits
    qmax = 2 ** width - 1
    low, high = w.amin(2, keepdim=True), w.amax(2, keepdim=True)
    s = ((high - low) / qmax).cpu().numpy().astype(np.float16)              # one rounding, to nearest
    s = torch.from_numpy(np.where(s == 0, np.float16(2.0 ** -14), s)).double().cuda()
    z = (-low / s).round().clamp(0, qmax)
    q = ((w / s).round() + z).clamp(0, qmax)
    if bits < width:                                                        # the child: high bits, mid-point fill
        step = 2 ** (width - bits)
        q = torch.floor(q / step) * step + step / 2
    return ((q - z) * s).view(n, k)


def exact(case, seed):
    """What `run` returns, in float64 with weights that are not rounded; quantising has whole numbers only."""
    kind = case["kind"]
    if kind == "quantize":
        return None
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if kind == "gemv":
        w = _weights64(case["n"], case["k"], case["bits"], case["fmt"], gen)
        return torch.randn((case["batch"], case["k"]), device="cuda", generator=gen).half().double() @ w.T
    layers, bits = _blocks(case), _bits(case)
    both = bits if kind == "switch" else (bits,)

    def products(inputs):
        """One list of outputs per configuration; the weights are drawn again from the seed, as often as they are needed."""
        out = []
        for widths in both:
            again = torch.Generator(device="cuda")
            again.manual_seed(seed)
            out.append([inputs[i] @ _weights64(n, k, widths[i], case["fmt"], again).T for i, (_, n, k, _, _) in enumerate(layers)])
        return out

    for _, n, k, _, _ in layers:                                            # `prepare` draws every weight before the activations
        torch.randn((n, k), device="cuda", generator=gen)
    if kind == "prefill":
        m = case["tokens"]
        x = {k: torch.randn((m, k), device="cuda", generator=gen).bfloat16().double() for k in sorted({l[2] for l in layers})}
        return products([x[l[2]] for l in layers])[0]
    b = case["batch"]
    got = products([torch.randn((b, l[2]), device="cuda", generator=gen).half().double() for l in layers])
    outs = []
    for ys in got:
        buf, views = _views([(b, l[1]) for l in layers], torch.float64)
        for v, y in zip(views, ys):
            v.copy_(y)
        outs.append(buf)
    return {"footprints": [None, None], "high": outs[0], "low": outs[1]} if kind == "switch" else outs[0]
