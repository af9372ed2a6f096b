"""The work this library is used for, as cases that can be timed and compared.

A case is one of four kinds:

  layer : one routed quantized linear layer through the one-call entry point (sort, product and un-sort inside).
  block : the linear layers of one transformer block for a batch of sequences, as a serving loop runs them: route,
          sort once, then every layer on the sorted batch.  `decoding` sequences bring one row each, `prompts`
          sequences bring between `rows_min` and `rows_max` rows each.  Small batches use the entry points made for
          them (sibling layers in one launch; with `fused` also the gated pair and the residual adds).
  conv  : the four 1x1 convolutions of a residual CNN's bottlenecks for a batch of images.
  build : one expert built from full-precision weights and exported for storage.

Expert formats are written as in the workloads' tags: W<bits><s|a>-<pc|g<group>>, s / a = symmetric / asymmetric grid,
pc = one scale per output channel.
"""
import math
import random

import torch

import paper_2508_09204_b200 as moqe

LLAMA_EXPERTS = "W8s-pc W4a-g128 W3a-g128"
LLAMA_EXPERTS_W2 = "W8s-pc W4a-g128 W2a-g128"
QWEN_EXPERTS = "W8s-pc W4s-g128 W4a-g128 W3a-g64"
RESNET_EXPERTS = "W8s-pc W4a-pc W4a-g32"
TINY_EXPERTS = "W8s-pc W4a-g128"

# hidden size, width of q, width of k and v, width of the MLP
MODELS = {"llama7b": (4096, 4096, 4096, 11008), "qwen7b": (3584, 3584, 512, 18944)}
# N, K, rows per image
RESNET = ((64, 256, 56 * 56), (256, 64, 56 * 56), (256, 1024, 14 * 14), (1024, 256, 14 * 14))
# how the samples of a batch spread over the experts, most loaded first ("one": a batch that all goes to one expert)
MIXES = {"even": None, "skewed": (0.7, 0.2, 0.1), "one": (1.0,)}


def _block(name, model, experts, decoding=0, prompts=0, rows_min=0, rows_max=0, mix="even", router="logits", fused=False):
    case = {"name": name} if name else {}
    case.update(kind="block", model=model, experts=experts, decoding=decoding, prompts=prompts, rows_min=rows_min,
                rows_max=rows_max, mix=mix, router=router, fused=fused)
    return case


def listed():
    return [
        # the smallest call: one small layer, four short sequences
        {"name": "layer_1024_64rows", "kind": "layer", "N": 1024, "K": 1024, "samples": 4, "rows": 16, "experts": TINY_EXPERTS, "mix": "even"},
        # one user's generation, a token at a time
        _block("decode_llama_1", "llama7b", LLAMA_EXPERTS, decoding=1, fused=True),
        # a small server's decode step
        _block("decode_llama_16", "llama7b", LLAMA_EXPERTS, decoding=16),
        # a decode step with grouped-query attention and a narrow-group expert
        _block("decode_qwen_24", "qwen7b", QWEN_EXPERTS, decoding=24),
        # a busy server's decode step
        _block("decode_llama_96", "llama7b", LLAMA_EXPERTS, decoding=96),
        # continuous batching: decoding sequences beside a chunk of a prompt, 512 rows in all
        _block("chunk_llama_512", "llama7b", LLAMA_EXPERTS, decoding=45, prompts=1, rows_min=467, rows_max=467),
        # prompts of uneven length, with a 2-bit expert
        _block("prompts_llama_ragged", "llama7b", LLAMA_EXPERTS_W2, prompts=7, rows_min=30, rows_max=900),
        # full-length prompts, most of them easy ones
        _block("prefill_llama_8x2048", "llama7b", LLAMA_EXPERTS, prompts=8, rows_min=2048, rows_max=2048, mix="skewed"),
        # prompts and decoding sequences together, routed on the device by the router's own network
        _block("mixed_qwen_4160", "qwen7b", QWEN_EXPERTS, decoding=64, prompts=4, rows_min=1024, rows_max=1024, router="mlp"),
        # image classification: a large batch, and the few images of one request
        {"name": "conv_resnet_256", "kind": "conv", "images": 256, "experts": RESNET_EXPERTS, "mix": "even"},
        {"name": "conv_resnet_5", "kind": "conv", "images": 5, "experts": RESNET_EXPERTS, "mix": "even"},
        # building the experts of a model, one layer at a time
        {"name": "build_11008x4096_w4", "kind": "build", "N": 11008, "K": 4096, "format": "W4a-g128"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("layer", "decode", "decode", "serve", "prompts", "mixed", "conv", "build"))
    model = rng.choice(("llama7b", "qwen7b"))
    experts = rng.choice((LLAMA_EXPERTS, LLAMA_EXPERTS_W2, QWEN_EXPERTS))
    mix = rng.choice(("even", "even", "skewed", "one"))
    if kind == "layer":
        return {"kind": kind, "N": 8 * _log(rng, 16, 512), "K": 128 * _log(rng, 4, 48), "samples": _log(rng, 1, 40),
                "rows": _log(rng, 1, 300), "experts": rng.choice((TINY_EXPERTS, LLAMA_EXPERTS, QWEN_EXPERTS)), "mix": mix}
    if kind == "decode":
        return _block(None, model, experts, decoding=_log(rng, 1, 32), mix=mix, fused=rng.random() < 0.5)
    if kind == "serve":
        return _block(None, model, experts, decoding=_log(rng, 33, 300), mix=mix)
    if kind == "prompts":
        return _block(None, model, experts, prompts=rng.randint(1, 12), rows_min=_log(rng, 16, 200), rows_max=_log(rng, 201, 1000), mix=mix)
    if kind == "mixed":
        return _block(None, model, experts, decoding=_log(rng, 8, 128), prompts=rng.randint(1, 4), rows_min=_log(rng, 32, 300),
                      rows_max=_log(rng, 301, 1500), mix=mix, router=rng.choice(("logits", "mlp")))
    if kind == "conv":
        return {"kind": kind, "images": _log(rng, 2, 256), "experts": rng.choice((RESNET_EXPERTS, TINY_EXPERTS.replace("g128", "g64"))), "mix": mix}
    fmt = "W%d%s-%s" % (rng.choice((8, 4, 4, 3, 2)), rng.choice("sa"), rng.choice(("pc", "g32", "g64", "g128")))
    return {"kind": "build", "N": 8 * _log(rng, 16, 1376), "K": 128 * _log(rng, 4, 86), "format": fmt}


# ---- what a case consists of ---------------------------------------------------------------------------------------
def _format(tag):
    head, group = tag.split("-")
    return int(head[1:-1]), 0 if group == "pc" else int(group[1:]), head[-1] == "s"


def _formats(case):
    return [_format(t) for t in case["experts"].split()]


def _quota(n, case, E):
    """How many of n samples go to each expert."""
    p = list(MIXES[case["mix"]] or (1.0 / E,) * E)[:E]
    p += [0.0] * (E - len(p))
    counts = [int(n * x / sum(p) + 1e-9) for x in p]
    for i in range(n - sum(counts)):
        counts[i % E] += 1
    return counts


def _sample_rows(case):
    """Rows of every sample: single-row ones first."""
    if case["kind"] == "layer":
        return [case["rows"]] * case["samples"]
    r = random.Random("%(prompts)d %(rows_min)d %(rows_max)d" % case)
    return [1] * case["decoding"] + [r.randint(case["rows_min"], case["rows_max"]) for _ in range(case["prompts"])]


def _parts(case):
    """Sizes of the groups of samples that are spread over the experts separately."""
    if case["kind"] == "layer":
        return [case["samples"]]
    if case["kind"] == "conv":
        return [case["images"]]
    return [case["decoding"], case["prompts"]]


def _layers(case):
    """(name, N, K, which input it reads) of a block."""
    h, q, kv, f = MODELS[case["model"]]
    return [("q", q, h, "x"), ("k", kv, h, "x"), ("v", kv, h, "x"), ("o", h, q, "attn"), ("gate", f, h, "h"), ("up", f, h, "h"), ("down", h, f, "act")]


def _expert_bytes(fmt, N, K):
    bits, group, sym = fmt
    return N * K * bits / 8 + N * (K // group if group else 1) * (2 if sym else 4)


# ---- inputs --------------------------------------------------------------------------------------------------------
def _weights(g, N, K):
    return torch.randn((N, K), device="cuda", generator=g).mul_(0.02)


def _acts(g, M, K, relu=False):
    x = torch.randn((M, K), device="cuda", generator=g, dtype=torch.bfloat16)
    return x.relu_() if relu else x


def _experts(g, N, K, formats):
    W = _weights(g, N, K)
    return [moqe.moqe_quantize_rtn(W, *f) for f in formats]


def _sample_experts(case, seed, E):
    """The expert of every sample."""
    r, ids = random.Random("routing %d" % seed), []
    for n in _parts(case):
        part = [e for e, c in enumerate(_quota(n, case, E)) for _ in range(c)]
        r.shuffle(part)
        ids += part
    return torch.tensor(ids, dtype=torch.int64)


def _logits(g, ids, E):
    """Scores whose largest entry is the sample's expert."""
    S = ids.numel()
    lg = torch.rand((S, E), device="cuda", generator=g) - 1.0
    lg[torch.arange(S, device="cuda"), ids.cuda()] = 1.0
    return lg


def _row_offsets(rows):
    off = [0]
    for n in rows:
        off.append(off[-1] + n)
    return torch.tensor(off, dtype=torch.int32, device="cuda")


def _workspace(M, N, K, E):
    ws = moqe.alloc_workspace(moqe.moqe_routed_qgemm_workspace(M, N, K, E))
    moqe.moqe_routed_qgemm_workspace_clear(ws, M, N, K, E)
    return ws


def prepare(case, seed):
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "build":
        return {"kind": kind, "W": _weights(g, case["N"], case["K"]), "format": _format(case["format"])}
    formats = _formats(case)
    E = len(formats)
    ids = _sample_experts(case, seed, E)
    if kind == "layer":
        rows = torch.tensor(_sample_rows(case))
        return {"kind": kind, "X": _acts(g, int(rows.sum()), case["K"]), "experts": _experts(g, case["N"], case["K"], formats),
                "row_ids": torch.repeat_interleave(ids, rows).to(torch.int32).cuda()}
    if kind == "conv":
        s = {"kind": kind, "E": E, "logits": _logits(g, ids, E), "layers": [], "row_offsets": {}}
        for N, K, rows in RESNET:
            M = rows * case["images"]
            s["row_offsets"][rows] = _row_offsets([rows] * case["images"])
            s["layers"].append({"rows": rows, "X": _acts(g, M, K, relu=True), "experts": _experts(g, N, K, formats),
                                "Y": torch.empty((M, N), dtype=torch.bfloat16, device="cuda"), "ws": _workspace(M, N, K, E)})
        return s
    rows = _sample_rows(case)
    M = sum(rows)
    h, q, kv, f = MODELS[case["model"]]
    small = M <= 32 and all(group == 0 or group >= 128 for _, group, _ in formats)     # what the decode entry points take
    s = {"kind": kind, "M": M, "E": E, "S": len(rows), "small": small, "fused": small and case["fused"] and M <= 16,
         "row_offsets": _row_offsets(rows), "logits": None, "router": None,
         "in": {"x": _acts(g, M, h), "attn": _acts(g, M, q), "h": _acts(g, M, h), "act": _acts(g, M, f)},
         "experts": {}, "Y": {}, "ws": {}}
    if case["router"] == "mlp":
        s["router"] = (torch.randn((256, h), device="cuda", generator=g) / h ** 0.5, torch.randn((E, 256), device="cuda", generator=g) / 16.0)
        s["router_ws"] = moqe.alloc_workspace(moqe.lib().moqe_router_mlp_workspace(len(rows), h, 256))
    else:
        s["logits"] = _logits(g, ids, E)
    for name, N, K, _ in _layers(case):
        s["experts"][name] = _experts(g, N, K, formats)
        s["Y"][name] = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        s["ws"][name] = _workspace(M, N, K, E)
    s["layers"] = _layers(case)
    if s["fused"]:
        s["residual"] = {"o": _acts(g, M, h), "down": _acts(g, M, h)}
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------
def _sort(s):
    if s["router"] is None and s["M"] <= 1024 and s["S"] <= 1024:
        return moqe.moqe_route_permute(s["logits"], s["row_offsets"], s["M"])[2:]
    if s["router"] is None:
        ids = moqe.moqe_route(s["logits"])
    else:
        s["scores"], ids = moqe.moqe_router_mlp(s["in"]["x"], s["row_offsets"], *s["router"], workspace=s["router_ws"])
    row_ids = moqe.moqe_expand_ids(ids, s["row_offsets"], s["M"])
    return moqe.moqe_permute(None, row_ids, s["E"])[1:]


def _run_block(s):
    perm, offsets = _sort(s)
    X, ex, Y, ws = s["in"], s["experts"], s["Y"], s["ws"]
    if not s["small"]:
        for name, _, _, src in s["layers"]:
            moqe.moqe_routed_qgemm_sorted(X[src], perm, offsets, ex[name], Y[name], ws[name])
    else:
        for names in (("q", "k", "v"), ("o",), ("gate", "up"), ("down",)):
            src = {"q": "x", "o": "attn", "gate": "h", "down": "act"}[names[0]]
            first = names[0]
            if len(names) == 1 and s["fused"]:
                moqe.moqe_routed_qgemm_sorted_residual(X[src], perm, offsets, ex[first], s["residual"][first], Y[first], ws[first])
            elif len(names) == 1:
                moqe.moqe_routed_qgemm_sorted(X[src], perm, offsets, ex[first], Y[first], ws[first])
            elif names[0] == "gate" and s["fused"]:
                moqe.moqe_routed_qgemm_sorted_gated(X[src], perm, offsets, ex["gate"], ex["up"], Y["gate"], ws["gate"])
            else:
                moqe.moqe_routed_qgemm_sorted_multi([X[src]] * len(names), perm, offsets, [ex[n] for n in names],
                                                    [Y[n] for n in names], ws[first])
    out = {n: y for n, y in Y.items() if not (s["fused"] and n == "up")}
    if s["router"] is not None:
        out["scores"] = s["scores"]
    return out


def run(s):
    if s["kind"] == "build":
        return moqe.moqe_expert_export(moqe.moqe_quantize_rtn(s["W"], *s["format"]))
    if s["kind"] == "layer":
        return moqe.moqe_routed_qgemm(s["X"], s["row_ids"], s["experts"])
    if s["kind"] == "block":
        return _run_block(s)
    ids = moqe.moqe_route(s["logits"])
    order = {}
    for L in s["layers"]:
        if L["rows"] not in order:
            row_ids = moqe.moqe_expand_ids(ids, s["row_offsets"][L["rows"]], L["X"].shape[0])
            order[L["rows"]] = moqe.moqe_permute(None, row_ids, s["E"])[1:]
        moqe.moqe_routed_qgemm_sorted(L["X"], *order[L["rows"]], L["experts"], L["Y"], L["ws"])
    return [L["Y"] for L in s["layers"]]


# ---- what a pass cannot do without ---------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "build":
        N, K = case["N"], case["K"]
        bits, group, sym = _format(case["format"])
        exported = N * K + 4 * N * (K // group if group else 1)
        return {"bytes": N * K * 4 + _expert_bytes((bits, group, sym), N, K) + exported, "flops": 0}
    formats = _formats(case)
    E = len(formats)
    counts = [sum(c) for c in zip(*(_quota(n, case, E) for n in _parts(case)))]
    if case.get("router") == "mlp":
        counts = [1] * E
    if case["kind"] == "layer":
        layers = [(case["N"], case["K"], case["samples"] * case["rows"], 0)]
    elif case["kind"] == "conv":
        layers = [(N, K, rows * case["images"], i) for i, (N, K, rows) in enumerate(RESNET)]
    else:
        M = sum(_sample_rows(case))
        layers = [(N, K, M, src) for _, N, K, src in _layers(case)]
    weights = sum(_expert_bytes(f, N, K) for N, K, _, _ in layers for f, c in zip(formats, counts) if c)
    inputs = {src: M * K * 2 for N, K, M, src in layers}
    return {"bytes": weights + sum(inputs.values()) + sum(M * N * 2 for N, _, M, _ in layers),
            "flops": sum(2.0 * M * N * K for N, K, M, _ in layers)}


def tolerance(case):
    # An expert's codes, scales and zero-points are whole numbers fixed by the format's definition.
    if case["kind"] == "build":
        return "exact"
    # One rounding to bf16 of an fp32 sum.  Measured against the same product in 64 bits, every layer of every listed
    # case: relative error 1.66e-3 (2-norm), largest difference 3.9e-3 -- half a unit of the last place, which is what
    # the rounding alone gives.  Four times that.
    return {"rel": 6.6e-3, "max": 1.6e-2}
