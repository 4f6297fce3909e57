"""The work a program has this library do, as measurable cases.

A drafter decodes one token at a time (N = 1 activation row), for a handful of concurrent requests (N up to about
16), and runs prompts and verification windows as panels of rows (N up to a few hundred).  Every case below is one of
those calls through ``paper_2504_08838_b200.binding``, with the layer shapes, sparsities, masks and output types of the
repository's own configurations (``synth.py``, ``bench.py``, the tests), or with odd sizes of the same range.

Kinds of case:

* ``linear``   one ``sd2_spmm`` on a handle of the default format;
* ``panel``    one ``sd2_spmm`` on a handle of the format made for panels of rows;
* ``fused``    one ``sd2_spmm_fused``: q, k and v of a block from the same activations;
* ``block``    one ``sd2_block_step``: the seven linears of a block;
* ``drafter``  one ``sd2_drafter_step``: all linears of a stack of blocks;
* ``decode``   one whole decode step: embedding, blocks with norms, rotation and attention over a cache, final norm,
  dense LM head and greedy token.

Weights are N(0, 0.02), activations N(0, 1), masks Bernoulli, by magnitude with uneven rows, or 2:4, all drawn on the
GPU from the seed.
"""

import math

import torch

from paper_2504_08838_b200 import binding as sd2
from paper_2504_08838_b200 import synth

LLAMA_1B, QWEN, LLAMA_3B = synth.LLAMA_1B, synth.QWEN_1P5B, synth.LLAMA_3B
EPS, THETA = 1e-5, 500000.0


def _linear(kind, M, K, density, mask, N, f32):
    return {"kind": kind, "M": M, "K": K, "density": density, "mask": mask, "N": N, "f32": f32}


def _blocks(kind, hidden, kv, inter, blocks, density, mask, N, **more):
    return dict({"kind": kind, "hidden": hidden, "kv": kv, "inter": inter, "blocks": blocks, "density": density,
                 "mask": mask, "N": N}, **more)


def _shape(kind, s, blocks, density, mask, N, **more):
    return _blocks(kind, s.hidden, s.kv, s.inter, blocks, density, mask, N, **more)


def listed():
    cases = {
        # one small linear for one draft token: launch latency and the host path are most of it
        "linear_2048_n1": _linear("linear", 2048, 2048, 0.5, "bernoulli", 1, False),
        # a long reduction at high sparsity with rows of uneven density, fp32 out
        "linear_2048x11008_n1": _linear("linear", 2048, 11008, 0.3, "magnitude", 1, True),
        # odd sizes, a few concurrent requests; rows of X are not 16-byte aligned
        "linear_ragged_n5": _linear("linear", 1531, 3001, 0.5, "bernoulli", 5, False),
        # the default format under a wide panel: a verification window of 48 rows over a gate or up matrix
        "linear_8192x2048_n48": _linear("linear", 8192, 2048, 0.5, "bernoulli", 48, False),
        # q, k, v of a block from one input, two requests
        "fused_qkv_1b_n2": _shape("fused", LLAMA_1B, 1, 0.5, "2:4", 2),
        # the panel format at its smallest panel on a down projection
        "panel_3072x8192_n16": _linear("panel", 3072, 8192, 0.5, "bernoulli", 16, False),
        # ... and at a full panel on a gate or up projection, fp32 out
        "panel_8192x3072_n64": _linear("panel", 8192, 3072, 0.5, "bernoulli", 64, True),
        # the linears of a drafter for one token: the headline path
        "drafter_1b_n1": _shape("drafter", LLAMA_1B, 2, 0.5, "bernoulli", 1),
        # ... at higher sparsity with uneven rows
        "drafter_qwen_n1": _shape("drafter", QWEN, 2, 0.3, "magnitude", 1),
        # ... for eight concurrent requests
        "drafter_1b_n8": _shape("drafter", LLAMA_1B, 2, 0.5, "bernoulli", 8),
        # one large block in a caller's workspace, sixteen requests
        "block_3b_n16": _shape("block", LLAMA_3B, 1, 0.5, "bernoulli", 16),
        # a whole decode step with a realistic vocabulary (the head shares the embedding's table), 300 cached positions
        "decode_1b_n1": _shape("decode", LLAMA_1B, 2, 0.5, "bernoulli", 1, head_dim=64, vocab=128256, pos=300),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _density(rng, mask):
    return 0.5 if mask == "2:4" else round(rng.choice([0.1, 0.25, 0.3, 0.34, 0.4, 0.5, 0.5, 0.5, 0.6, 0.7]), 2)


def draw(rng):
    kind = rng.choice(["linear", "linear", "panel", "fused", "block", "drafter", "drafter", "decode"])
    mask = rng.choice(["bernoulli", "bernoulli", "magnitude", "2:4"])
    density = _density(rng, mask)
    if kind in ("linear", "panel"):
        M, K = _log(rng, 256, 8192), _log(rng, 256, 11008)
        if rng.random() < 0.6:                               # most layer widths are multiples of 64
            M, K = max(64, M // 64 * 64), max(64, K // 64 * 64)
        if mask == "2:4":
            K = (K + 3) // 4 * 4
        N = _log(rng, 1, 64) if kind == "linear" else _log(rng, 16, 192)
        while M * K * N > 8192 * 3072 * 96:
            N = max(1, N // 2)
        return _linear(kind, M, K, density, mask, N, rng.random() < 0.4)
    head_dim = rng.choice([64, 128])
    kv_heads = rng.randint(1, 8)
    heads = kv_heads * rng.randint(2, 4)
    hidden = min(heads * head_dim, 3072 // (kv_heads * head_dim) * kv_heads * head_dim)
    kv = kv_heads * head_dim
    if kind == "decode":
        hidden = min(hidden, 2048 // kv_heads // head_dim * kv_heads * head_dim)
    inter = min(8192, hidden * rng.randint(5, 12) // 2 // 32 * 32)
    blocks = 1 if kind in ("fused", "block") or hidden > 2048 else rng.randint(1, 2)
    N = _log(rng, 1, {"block": 16, "drafter": 8, "fused": 8, "decode": 4}[kind])
    more = {"head_dim": head_dim, "vocab": _log(rng, 8000, 128256) // 4 * 4, "pos": _log(rng, 8, 1000)} if kind == "decode" else {}
    return _blocks(kind, hidden, kv, inter, blocks, density, mask, N, **more)


# ---- inputs ----------------------------------------------------------------------------

def _weight(gen, M, K, density, mask_kind):
    w = torch.empty((M, K), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)
    if mask_kind == "bernoulli":
        mask = torch.rand((M, K), device="cuda", generator=gen) < density
    elif mask_kind == "2:4":
        rank = w.abs().view(M, K // 4, 4).argsort(dim=2, descending=True, stable=True).argsort(dim=2)
        mask = (rank < 2).view(M, K)
    else:                                                    # by magnitude, the rows' densities spread by Beta(2, 2)
        beta = torch.rand((M, 3), device="cuda", generator=gen).median(dim=1).values
        keep = ((density + 2.0 * min(density, 1.0 - density) * (beta - 0.5)) * K).round().long().clamp(0, K)
        rank = w.abs().argsort(dim=1, descending=True, stable=True).argsort(dim=1)
        mask = rank < keep[:, None]
    return w, mask.to(torch.uint8)


def _handle(gen, M, K, density, mask_kind, fmt=sd2.SD2_FORMAT_AUTO, f32=False):
    w, mask = _weight(gen, M, K, density, mask_kind)
    return sd2.sd2_compress(w, mask, fmt, sd2.SD2_DTYPE_F32 if f32 else sd2.SD2_DTYPE_BF16)


def _block_shape(case):
    return synth.DrafterShape("case", case["hidden"], case["kv"], case["inter"], case["blocks"])


def _block_handles(gen, case, last_f32):
    blocks = []
    for b in range(case["blocks"]):
        blocks.append([_handle(gen, M, K, case["density"], case["mask"], f32=last_f32 and b == case["blocks"] - 1 and i == 6)
                       for i, (_, M, K) in enumerate(_block_shape(case).linears())])
    return blocks


def _normal(gen, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, N = case["kind"], case["N"]
    s = {"kind": kind}
    if kind in ("linear", "panel"):
        fmt = sd2.SD2_FORMAT_AUTO if kind == "linear" else sd2.SD2_FORMAT_GAP4_MMA
        s["h"] = _handle(gen, case["M"], case["K"], case["density"], case["mask"], fmt, case["f32"])
        s["x"] = _normal(gen, N, case["K"])
        s["y"] = torch.zeros((N, case["M"]), dtype=torch.float32 if case["f32"] else torch.bfloat16, device="cuda")
        return s
    if kind == "fused":
        dims = _block_shape(case).linears()[:3]
        s["hs"] = [_handle(gen, M, K, case["density"], case["mask"]) for _, M, K in dims]
        s["x"] = _normal(gen, N, case["hidden"])
        s["ys"] = [torch.zeros((N, M), dtype=torch.bfloat16, device="cuda") for _, M, _ in dims]
        return s
    s["blocks"] = _block_handles(gen, case, last_f32=kind != "decode")
    if kind == "decode":
        H = case["hidden"]
        s["heads"] = (H // case["head_dim"], case["kv"] // case["head_dim"])
        s["pos"] = case["pos"]
        s["table"] = torch.empty((case["vocab"], H), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)
        s["token_in"] = torch.randint(0, case["vocab"], (N,), dtype=torch.int32, device="cuda", generator=gen)
        s["norms"] = [(1.0 + 0.1 * _normal(gen, 2, H).float()).to(torch.bfloat16) for _ in s["blocks"]]
        s["norm_out"] = (1.0 + 0.1 * _normal(gen, H).float()).to(torch.bfloat16)
        s["caches"] = [(_normal(gen, N, case["pos"] + 16, case["kv"]), _normal(gen, N, case["pos"] + 16, case["kv"]))
                       for _ in s["blocks"]]
        s["ws"] = torch.zeros(sd2.sd2_decoder_workspace_bytes(s["blocks"][0], N) // 2, dtype=torch.bfloat16, device="cuda")
        s["x"] = [torch.zeros((N, H), dtype=torch.bfloat16, device="cuda") for _ in range(len(s["blocks"]) + 2)]
        s["logits"] = torch.zeros((N, case["vocab"]), dtype=torch.float32, device="cuda")
        s["token_out"] = torch.zeros((N,), dtype=torch.int32, device="cuda")
        s["arrays"] = [sd2._handle_array(hs) for hs in s["blocks"]]
        return s
    s["x"] = _normal(gen, N, case["hidden"])
    s["y"] = torch.zeros((N, case["hidden"]), dtype=torch.float32, device="cuda")
    if kind == "drafter":
        s["drafter"] = sd2.sd2_drafter_create(s["blocks"], n_max=N)
    else:
        s["ws"] = torch.zeros(sd2.sd2_block_workspace_bytes(s["blocks"][0], N) // 2, dtype=torch.bfloat16, device="cuda")
    return s


# ---- one pass --------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind in ("linear", "panel"):
        sd2.sd2_spmm(s["h"], s["x"], s["y"])
        return s["y"]
    if kind == "fused":
        sd2.sd2_spmm_fused(s["hs"], s["x"], s["ys"])
        return s["ys"]
    if kind == "drafter":
        sd2.sd2_drafter_step(s["drafter"], s["x"], s["y"])
        return s["y"]
    if kind == "block":                                      # the workspace holds q, k, v, hdn, g, u, t afterwards
        sd2.sd2_block_step(s["blocks"][0], s["x"], s["y"], s["ws"])
        return {"y": s["y"], "intermediates": s["ws"]}
    x = s["x"]
    heads_q, heads_kv = s["heads"]
    sd2.sd2_embedding(s["token_in"], s["table"], x[0])
    for b, hs in enumerate(s["blocks"]):
        sd2.sd2_decoder_block_step(hs, s["norms"][b][0], s["norms"][b][1], x[b], x[b + 1], s["caches"][b][0], s["caches"][b][1],
                                   heads_q, heads_kv, s["pos"], EPS, THETA, s["ws"], handle_array=s["arrays"][b])
    n = len(s["blocks"])
    sd2.sd2_rmsnorm(x[n], s["norm_out"], x[n + 1], EPS)
    sd2.sd2_lm_head(x[n + 1], s["table"], s["logits"], s["token_out"])
    return {"logits": s["logits"], "tokens": s["token_out"], "caches": s["caches"], "hidden": x[n]}


# ---- what a pass cannot do without ------------------------------------------------------

def _linear_work(M, K, density, N):
    """Kept values once, one bit of position per dense slot, and the multiply-adds of the kept weights."""
    kept = density * M * K
    return 2.0 * kept + M * K / 8.0, 2.0 * kept * N


def work(case):
    N = case["N"]
    if case["kind"] in ("linear", "panel"):
        b, f = _linear_work(case["M"], case["K"], case["density"], N)
        return {"bytes": b + N * (2 * case["K"] + (4 if case["f32"] else 2) * case["M"]), "flops": f}
    linears = _block_shape(case).linears()
    linears = linears[:3] if case["kind"] == "fused" else linears
    bytes_, flops = 0.0, 0.0
    for _, M, K in linears:
        b, f = _linear_work(M, K, case["density"], N)
        bytes_ += b * case["blocks"]
        flops += f * case["blocks"]
    H, kv = case["hidden"], case["kv"]
    if case["kind"] == "fused":
        bytes_ += N * 2 * (H + H + 2 * kv)
    elif case["kind"] == "drafter":
        bytes_ += N * (2 + 4) * H
    elif case["kind"] == "block":
        bytes_ += N * ((2 + 4) * H + 2 * (2 * H + 2 * kv + 3 * case["inter"]))
    else:
        cached = 2 * N * (case["pos"] + 1) * kv * case["blocks"]
        bytes_ += 2.0 * cached + 2.0 * case["vocab"] * H + N * (4.0 * case["vocab"] + 4 * H)
        flops += 2.0 * N * case["vocab"] * H + 4.0 * N * (case["pos"] + 1) * H * case["blocks"]
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Four times what two formats of the library differ by, which form their sums in other orders: fp32 outputs of one
    linear by the order alone (8e-7 for sums of 1536 kept terms, so about 2.5e-6 for the longest rows), bf16 outputs by
    single roundings that fall the other way (7e-5, one step of the type at most), a chain of linears by such roundings
    carried on (block 3e-4, drafter 4e-3)."""
    if case["kind"] in ("linear", "panel", "fused"):
        return {"rel": 1e-5, "max": 1e-4} if case.get("f32") else {"rel": 5e-4, "max": 0.03}
    if case["kind"] == "drafter":
        return {"rel": 1.5e-2, "max": 0.1}
    return {"rel": 3e-3, "max": 0.05}
