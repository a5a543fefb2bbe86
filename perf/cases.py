"""What this library is timed on: the calls a user of packed variable-width
weights makes, at the sizes of the decoder families this repository carries.

Three kinds of case:

  product  one packed matrix times 1..16 activation vectors (vbq_gemv,
           vbq_gemm_small): single calls, as a host program issues them;
  decode   the linear products of one decode step: `layers` decoder layers
           (Q, K, V, O, gate, up, down) and, with `vocab`, the LM head, for
           1..16 tokens, captured once in a CUDA graph and replayed per step,
           as a serving loop runs them. Activations are given per product (the
           library has no attention or norms); each product waits for the one
           before it, unless `issue` says otherwise;
  tensor   whole matrices: vbq_quantize, the export of a matrix
           (vbq_quantize, vbq_pack, and vbq_dequant as the check that reads
           the stored form back) and the training-time forward vbq_soft_quant.

`widths` of a matrix: "main", "mlp0" and "head" are the i.i.d. per-group mixes
of the searched allocation, "recipe" the fixed recipe (2-bit projections, a head
tiered by row), "all1" .. "all8" a single width.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_02893_gb300 import vbq

GROUP = 64
MIX = {
    "main": (0.69, 0.15, 0.11, 0.05),
    "mlp0": (0.40, 0.30, 0.22, 0.08),
    "head": (0.96, 0.025, 0.01, 0.005),
    "recipe": (0.0, 1.0, 0.0, 0.0),
    "all1": (1.0, 0.0, 0.0, 0.0),
    "all2": (0.0, 1.0, 0.0, 0.0),
    "all4": (0.0, 0.0, 1.0, 0.0),
    "all8": (0.0, 0.0, 0.0, 1.0),
}
# the recipe's head: cumulative share of rows, in frequency order, and width
HEAD_TIERS = ((0.005, 8), (0.02, 4), (0.12, 2), (1.0, 1))
# d_model, d_q, d_kv, d_ff of the decoder families
DIMS = {
    "131m": (768, 768, 768, 2048),
    "1b": (2048, 2048, 256, 5632),
    "9b": (4096, 4096, 1024, 14336),
}


def _decode(dims, layers, vocab, batch, widths, issue):
    d, q, kv, ff = dims
    return {"kind": "decode", "d": d, "q": q, "kv": kv, "ff": ff, "layers": layers, "vocab": vocab, "batch": batch,
            "widths": widths, "issue": issue}


def _product(n, k, widths, batch):
    return {"kind": "product", "n": n, "k": k, "widths": widths, "batch": batch}


def _tensor(kind, n, k, widths="main"):
    return {"kind": kind, "n": n, "k": k, "widths": widths}


def listed():
    return [
        # one small projection, one token: the smallest call, all latency
        dict(_product(768, 768, "main", 1), name="gemv_768"),
        # a whole decode step of the small decoder: 85 dependent products, logits last
        dict(_decode(DIMS["131m"], 12, 32000, 1, "main", "calls"), name="step_131m_b1"),
        # one layer of the middle and the large decoder at one token (the large
        # one also as an engine fuses it, and at the fixed recipe's widths)
        dict(_decode(DIMS["9b"], 1, 0, 1, "main", "calls"), name="layer_9b_b1"),
        dict(_decode(DIMS["9b"], 1, 0, 1, "main", "fused"), name="layer_9b_fused_b1"),
        dict(_decode(DIMS["9b"], 1, 0, 1, "recipe", "calls"), name="layer_9b_recipe_b1"),
        # a few concurrent sequences, or the tokens a speculative step verifies
        dict(_decode(DIMS["1b"], 1, 0, 4, "main", "calls"), name="layer_1b_b4"),
        dict(_decode(DIMS["9b"], 1, 0, 8, "main", "calls"), name="layer_9b_b8"),
        dict(_decode(DIMS["9b"], 1, 0, 16, "main", "calls"), name="layer_9b_b16"),
        # the largest matrix, one token
        dict(_product(128256, 4096, "head", 1), name="head_9b_b1"),
        # odd sizes: an odd number of rows, 33 group columns, 5 tokens
        dict(_product(32001, 2112, "head", 5), name="head_odd_b5"),
        # export of one MLP projection: quantise, pack, read back
        dict(_tensor("export", 14336, 4096), name="export_9b_mlp"),
        # the training-time soft forward of one MLP projection
        dict(_tensor("soft", 14336, 4096), name="soft_9b_mlp"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    r = rng.random()
    if r < 0.35:
        while True:
            n, k = int(_log(rng, 128, 131072)), GROUP * int(_log(rng, 4, 256))
            if 768 * 768 <= n * k <= 14336 * 8192:
                return _product(n, k, rng.choice(list(MIX)), rng.choice((1, 1, 2, 3, 4, 5, 8, 12, 16)))
    if r < 0.70:
        d = GROUP * int(_log(rng, 12, 65))
        dims = (d, d, GROUP * rng.randint(1, d // GROUP), GROUP * int(d / GROUP * rng.uniform(2.0, 3.5)))
        batch = rng.choice((1, 1, 1, 2, 4, 6, 8, 11, 16))
        issue = rng.choice(("calls", "calls", "fused", "group", "chain")) if batch == 1 else "calls"
        layers = 1 if d > 2048 else rng.randint(1, 4)
        vocab = rng.choice((0, 0, 4 * rng.randint(2000, 8000)))
        return _decode(dims, layers, vocab, batch, rng.choice(("main", "main", "recipe")), issue)
    kind = rng.choice(("quantize", "export", "soft"))
    n, k = int(_log(rng, 256, 14337)), GROUP * int(_log(rng, 8, 65))
    return _tensor(kind, n, k, "main" if kind == "soft" else rng.choice(("main", "main", "mlp0", "head", "all1", "all4")))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _rows_per_chunk(k):
    return max(1, (1 << 26) // k)


def _widths(n, k, widths, gen, head=False):
    g = k // GROUP
    if head and widths == "recipe":
        w = torch.empty(n, dtype=torch.uint8, device="cuda")
        start = 0
        for frac, b in HEAD_TIERS:
            end = n if frac >= 1.0 else int(round(frac * n))
            w[start:end] = b
            start = max(start, end)
        return w[:, None].repeat(1, g).contiguous()
    p = torch.tensor(MIX["head" if head else widths], dtype=torch.float64).cumsum(0).float().cuda()
    u = torch.rand((n, g), device="cuda", generator=gen) * 0.999999
    idx = torch.bucketize(u, p, right=True).clamp_(max=3)
    return torch.tensor([1, 2, 4, 8], dtype=torch.uint8, device="cuda")[idx]


def _matrix(n, k, widths, gen, head=False):
    """Widths, codes and FP16 scales of a matrix whose weights are normal with a
    magnitude of their own per group, as its quantiser leaves them: the largest
    weight (about 2.6 sigma) on the last level, symmetric codes; one bit keeps
    the sign and the mean magnitude."""
    w = _widths(n, k, widths, gen, head)
    wl = w.long()
    sigma = 0.02 * torch.exp(0.3 * torch.randn(w.shape, device="cuda", generator=gen))
    rel = torch.tensor([0.0, 0.8, 2.6, 0.0, 2.6 / 7, 0.0, 0.0, 0.0, 2.6 / 127], device="cuda")
    scales = (sigma * rel[wl]).half()
    qmax = torch.tensor([0.0, 0.0, 1.0, 0.0, 7.0, 0.0, 0.0, 0.0, 127.0], device="cuda")
    zero = torch.tensor([0.0, 0.0, 2.0, 0.0, 8.0, 0.0, 0.0, 0.0, 128.0], device="cuda")
    codes = torch.empty((n, k), dtype=torch.uint8, device="cuda")
    step = _rows_per_chunk(k)
    for r in range(0, n, step):
        wr = wl[r:r + step]
        v = torch.randn((wr.shape[0], k // GROUP, GROUP), device="cuda", generator=gen)
        q, z = qmax[wr][..., None], zero[wr][..., None]
        many = torch.minimum(torch.maximum((v * (q / 2.6)).round_(), -q), q) + z
        c = torch.where((wr == 1)[..., None], (v >= 0).float(), many)
        codes[r:r + step] = c.to(torch.uint8).view(wr.shape[0], k)
    return w, codes, scales


def _acts(batch, k, gen):
    """Activations: normal, with a few channels several times larger."""
    x = torch.randn((batch, k), device="cuda", generator=gen)
    x = x * torch.where(torch.rand(k, device="cuda", generator=gen) < 0.01, 8.0, 1.0)
    return x.to(torch.bfloat16)


def _dense(n, k, gen):
    """Dense weights: normal, a magnitude of its own per group, 1% outliers."""
    w = torch.randn((n, k // GROUP, GROUP), device="cuda", generator=gen)
    w *= 0.02 * torch.exp(0.5 * torch.randn((n, k // GROUP, 1), device="cuda", generator=gen))
    w *= torch.where(torch.rand(w.shape, device="cuda", generator=gen) < 0.01, 8.0, 1.0)
    return w.view(n, k)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _plan(case):
    """The products of a decode case in order: (output name, layer, n, k, widths, input)."""
    d, q, kv, ff = case["d"], case["q"], case["kv"], case["ff"]
    out = []
    for layer in range(case["layers"]):
        mlp = "mlp0" if case["widths"] == "main" and layer == 0 and case["layers"] > 1 else case["widths"]
        if case["issue"] == "fused":
            out += [("qkv", layer, q + 2 * kv, d, case["widths"], "attn_in"), ("o", layer, d, q, case["widths"], "o_in"),
                    ("gate_up", layer, 2 * ff, d, mlp, "mlp_in"), ("down", layer, d, ff, mlp, "gate_up")]
        else:
            out += [("q", layer, q, d, case["widths"], "attn_in"), ("k", layer, kv, d, case["widths"], "attn_in"),
                    ("v", layer, kv, d, case["widths"], "attn_in"), ("o", layer, d, q, case["widths"], "o_in"),
                    ("gate", layer, ff, d, mlp, "mlp_in"), ("up", layer, ff, d, mlp, "mlp_in"),
                    ("down", layer, d, ff, mlp, "down_in")]
    if case["vocab"]:
        out.append(("logits", 0, case["vocab"], d, case["widths"], "head_in"))
    return out


def _decode_data(case, seed, use):
    """Calls use(name, layer, widths, codes, scales, x) per product, in order
    (x is None where the input is the product before); one matrix at a time."""
    gen = _gen(seed)
    acts = {}
    for name, layer, n, k, widths, src in _plan(case):
        w, codes, scales = _matrix(n, k, widths, gen, head=name == "logits")
        if src != "gate_up" and (src, layer) not in acts:
            acts[src, layer] = _acts(case["batch"], k, gen)
        use(name, layer, w, codes, scales, acts.get((src, layer)))


def _capture(fn):
    fn()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fn()
    return graph


def _prepare_decode(case, seed):
    batch, prods = case["batch"], []
    outs = {}
    for name, layer, n, _, _, _ in _plan(case):
        if name not in outs:
            outs[name] = torch.zeros((1 if name == "logits" else case["layers"], batch, n), device="cuda")

    def use(name, layer, w, codes, scales, x):
        prods.append((name, vbq.vbq_pack(codes, w, scales), x, outs[name][layer]))

    _decode_data(case, seed, use)
    state = {"outs": outs, "prods": prods}
    issue = case["issue"]
    if issue == "chain":
        waits = [2 if name in ("k", "v", "up") else 1 for name, _, _, _ in prods]
        state["chain"] = vbq.vbq_chain_create([p[1] for p in prods], [p[2] for p in prods], [p[3] for p in prods], waits)

    def step():
        if issue == "chain":
            vbq.vbq_chain_run(state["chain"])
            return
        i = 0
        while i < len(prods):
            name, lay, x, y = prods[i]
            many = {"q": 3, "gate": 2}.get(name, 1) if issue == "group" else 1
            if many > 1:
                part = prods[i:i + many]
                vbq.vbq_gemv_group([p[1] for p in part], [p[2] for p in part], [p[3] for p in part])
            elif x is None:
                vbq.vbq_gemv_swiglu_in(lay, prods[i - 1][3], y)
            elif batch == 1:
                vbq.vbq_gemv(lay, x, y)
            else:
                vbq.vbq_gemm_small(lay, x, y)
            i += many

    state["graph"] = _capture(step)
    return state


def prepare(case, seed):
    kind = case["kind"]
    if kind == "decode":
        return dict(_prepare_decode(case, seed), kind=kind)
    gen = _gen(seed)
    n, k = case["n"], case["k"]
    if kind == "product":
        w, codes, scales = _matrix(n, k, case["widths"], gen)
        layout = vbq.vbq_pack(codes, w, scales)
        return {"kind": kind, "layout": layout, "x": _acts(case["batch"], k, gen),
                "y": torch.empty((case["batch"], n), device="cuda")}
    state = {"kind": kind, "w": _dense(n, k, gen)}
    g = k // GROUP
    if kind == "soft":
        state["logits"] = 2.0 * torch.randn((n, g, 4), device="cuda", generator=gen)
        u = torch.rand((n, g, 4), device="cuda", generator=gen).clamp_(1e-7, 1.0 - 1e-7)
        state["gumbel"] = -torch.log(-torch.log(u))
        state["out"] = (torch.empty((n, k), device="cuda"), torch.empty((n, g), device="cuda"),
                        torch.empty((n, g), dtype=torch.uint8, device="cuda"))
        return state
    state["widths"] = _widths(n, k, case["widths"], gen)
    state["codes"] = torch.empty((n, k), dtype=torch.uint8, device="cuda")
    state["scales"] = torch.empty((n, g), dtype=torch.int16, device="cuda")
    if kind == "export":
        state["back"] = {"codes": torch.empty_like(state["codes"]), "widths": torch.empty_like(state["widths"]),
                         "scales": torch.empty_like(state["scales"]), "w": torch.empty((n, k), device="cuda")}
    return state


TAU = 0.5


def run(state):
    kind = state["kind"]
    if kind == "decode":
        state["graph"].replay()
        return state["outs"]
    if kind == "product":
        if state["x"].shape[0] == 1:
            vbq.vbq_gemv(state["layout"], state["x"], state["y"])
        else:
            vbq.vbq_gemm_small(state["layout"], state["x"], state["y"])
        return state["y"]
    if kind == "soft":
        w_soft, bits, hard = state["out"]
        return vbq.vbq_soft_quant(state["w"], state["logits"], TAU, state["gumbel"], w_soft, bits, hard)
    vbq.vbq_quantize(state["w"], state["widths"], state["codes"], state["scales"])
    if kind == "quantize":
        return {"codes": state["codes"], "scales": state["scales"]}
    # the stored form stays until the next export of this matrix replaces it
    state["layout"] = vbq.vbq_pack(state["codes"], state["widths"], state["scales"])
    back = state["back"]
    vbq.vbq_dequant(state["layout"], back["codes"], back["widths"], back["scales"], back["w"])
    return dict(back, payload=vbq.vbq_packed_bytes(state["layout"])[0])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _mean_bits(widths, head=False):
    if head and widths == "recipe":
        return 0.005 * 8 + 0.015 * 4 + 0.10 * 2 + 0.88 * 1
    return sum(p * b for p, b in zip(MIX["head" if head else widths], (1, 2, 4, 8)))


def _product_work(n, k, widths, batch, head=False, x=True):
    weights = n * k * _mean_bits(widths, head) / 8 + 2 * n * (k // GROUP)
    return weights + (2 * k * batch if x else 0) + 4 * n * batch, 2.0 * n * k * batch


def work(case):
    kind = case["kind"]
    if kind == "decode":
        total, flops, seen = 0.0, 0.0, set()
        for name, layer, n, k, widths, src in _plan(case):
            first = src != "gate_up" and (src, layer) not in seen        # an input that several products read counts once
            seen.add((src, layer))
            b, f = _product_work(n, k, widths, case["batch"], name == "logits", first)
            total, flops = total + b, flops + f
        return {"bytes": total, "flops": flops}
    n, k = case["n"], case["k"]
    g = n * (k // GROUP)
    if kind == "product":
        b, f = _product_work(n, k, case["widths"], case["batch"])
        return {"bytes": b, "flops": f}
    if kind == "soft":
        return {"bytes": 8.0 * n * k + 37.0 * g, "flops": 30.0 * n * k}
    stored = n * k * _mean_bits(case["widths"]) / 8 + 2 * g
    if kind == "quantize":
        return {"bytes": 5.0 * n * k + 3.0 * g, "flops": 3.0 * n * k}
    # quantise (4 in, 1 out), pack (1 in, the stored form out), read back (the
    # stored form in, codes and float weights out)
    return {"bytes": (5.0 + 1.0 + 5.0) * n * k + 9.0 * g + 2 * stored, "flops": 4.0 * n * k}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _exact_product(w, codes, scales, x):
    """X W^T in float64: x (batch, k) float64."""
    n, k = codes.shape
    out = torch.empty((x.shape[0], n), dtype=torch.float64, device="cuda")
    step = max(1, _rows_per_chunk(k) // 2)
    for r in range(0, n, step):
        wr = w[r:r + step].long()[..., None]
        u = codes[r:r + step].view(wr.shape[0], k // GROUP, GROUP).double()
        level = torch.where(wr == 1, 2.0 * u - 1.0, u - (2 ** (wr - 1)).double())
        dense = (level * scales[r:r + step].double()[..., None]).view(wr.shape[0], k)
        out[:, r:r + step] = (dense @ x.t()).t()
    return out


def _exact_quantized(w, widths):
    """Codes and FP16 scale bits of §3.1's rules in float64."""
    n, k = w.shape
    codes = torch.empty((n, k), dtype=torch.uint8, device="cuda")
    scales = torch.empty(widths.shape, dtype=torch.float16, device="cuda")
    step = max(1, _rows_per_chunk(k) // 2)
    for r in range(0, n, step):
        wl = widths[r:r + step].long()
        v = w[r:r + step].view(wl.shape[0], k // GROUP, GROUP).double()
        qmax = torch.where(wl == 1, torch.ones_like(wl), 2 ** (wl - 1) - 1).double()
        s = torch.where(wl == 1, v.abs().mean(-1), v.abs().amax(-1) / qmax)
        # numpy rounds float64 to float16 in one step
        s16 = torch.from_numpy(np.minimum(s.cpu().numpy(), 65504.0).astype(np.float16)).cuda()
        sd, z = s16.double()[..., None], (2 ** (wl - 1)).double()[..., None]
        q = torch.where(sd > 0, torch.round(v / sd), torch.zeros_like(v))
        q = torch.minimum(torch.maximum(q, -qmax[..., None]), qmax[..., None])
        c = torch.where((wl == 1)[..., None], (v >= 0).double(), q + z)
        codes[r:r + step] = c.to(torch.uint8).view(wl.shape[0], k)
        scales[r:r + step] = s16
    return codes, scales


def _exact_soft(state):
    """§3.2's forward: the integer decisions in float32 (as specified), the rest in float64."""
    w, n, k = state["w"], state["w"].shape[0], state["w"].shape[1]
    z = (state["logits"].double() + state["gumbel"].double()) / TAU
    pi = torch.softmax(z, -1)
    bits = (pi * torch.tensor([1.0, 2.0, 4.0, 8.0], dtype=torch.float64, device="cuda")).sum(-1)
    out = torch.empty((n, k), dtype=torch.float64, device="cuda")
    step = max(1, _rows_per_chunk(k) // 4)
    for r in range(0, n, step):
        v = w[r:r + step].view(-1, k // GROUP, GROUP)
        p = pi[r:r + step]
        big = v.abs().amax(-1, keepdim=True)
        acc = p[..., 0:1] * torch.where(v >= 0, 1.0, -1.0).double() * v.double().abs().mean(-1, keepdim=True)
        for i, qmax in ((1, 1.0), (2, 7.0), (3, 127.0)):
            s = big / qmax
            q = torch.where(s > 0, torch.round(v / s), torch.zeros_like(v)).clamp_(-qmax, qmax)
            acc += p[..., i:i + 1] * q.double() * s.double()
        out[r:r + step] = acc.view(-1, k)
    return out, bits


def exact(case, seed):
    kind = case["kind"]
    if kind == "decode":
        outs = {}

        def use(name, layer, w, codes, scales, x):
            if x is None:
                gu = outs["gate_up"][layer]
                g, u = gu[:, 0::2], gu[:, 1::2]
                xd = g / (1.0 + torch.exp(-g)) * u
            else:
                xd = x.double()
            if name not in outs:
                outs[name] = torch.zeros((1 if name == "logits" else case["layers"], case["batch"], w.shape[0]),
                                         dtype=torch.float64, device="cuda")
            outs[name][layer] = _exact_product(w, codes, scales, xd)

        _decode_data(case, seed, use)
        return outs
    n, k = case["n"], case["k"]
    if kind == "product":
        gen = _gen(seed)
        w, codes, scales = _matrix(n, k, case["widths"], gen)
        return _exact_product(w, codes, scales, _acts(case["batch"], k, gen).double())
    if kind == "quantize":
        return {"codes": None, "scales": None}
    gen = _gen(seed)
    w = _dense(n, k, gen)
    if kind == "soft":
        state = {"w": w, "logits": 2.0 * torch.randn((n, k // GROUP, 4), device="cuda", generator=gen)}
        u = torch.rand((n, k // GROUP, 4), device="cuda", generator=gen).clamp_(1e-7, 1.0 - 1e-7)
        state["gumbel"] = -torch.log(-torch.log(u))
        w_soft, bits = _exact_soft(state)
        return w_soft, bits, None
    widths = _widths(n, k, case["widths"], gen)
    codes, scales = _exact_quantized(w, widths)
    wl = widths.long()[..., None]
    u = codes.view(n, k // GROUP, GROUP).double()
    level = torch.where(wl == 1, 2.0 * u - 1.0, u - (2 ** (wl - 1)).double())
    return {"codes": None, "widths": None, "scales": None, "w": (level * scales.double()[..., None]).view(n, k),
            "payload": None}
