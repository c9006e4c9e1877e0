"""The timed workloads of this library: what a prefill node and a decode node have it do.

A prefill node quantises the KV cache of finished requests; a decode node drafts tokens on the Anchor planes,
verifies windows of them on the recombined codes, appends a BF16 tail of its own tokens and, where the stock
attention of an engine has to read the cache, turns planes into BF16 pages.  Each case below is one pass of one of
these steps through the Python entry points.  Shapes are those of the repository's workloads: 8 KV heads of 128
channels with 32 or 64 query heads, contexts of 4096 to 131072 tokens, one launch per layer or several layers
flattened into the batch, blocks of 16 tokens (32 and 64 among the drawn cases), sequences of one length or a
ragged serving mix with a shuffled block table.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2607_01831_b200 as lynx

D = 128
PAGE = 256                 # tokens per page of Algorithm 1
MAX_TOKENS = 4_194_304     # tokens over all layers and sequences of a case: 16 layers x 2 sequences x 131072


def listed():
    cases = [
        # Prefill, large: the whole BF16 cache of one 32768-token request, 32 layers, K and V.
        dict(name="quantize_cache_32k", kind="quantize", layers=32, batch=1, ctx=32768, values="lognormal"),
        # Prefill, small: one layer of a 4096-token request that arrived in scattered blocks of a shared pool.
        dict(name="quantize_arrived_4k", kind="quantize_blocks", arrived=4096, pool=16384, values="student_t"),
        # Drafting, one call per layer: the shortest and the longest context of the workloads.
        dict(name="decode_layer_4k", kind="decode", batch=1, ctx=4096, values="outlier"),
        dict(name="decode_layer_128k", kind="decode", batch=1, ctx=131072, values="lognormal"),
        # Drafting, 70B class (8 query heads per KV head), 16 layers of two sequences flattened into one call.
        dict(name="decode_70b_16x128k", kind="decode", layers=16, batch=2, group=8, ctx=131072, values="outlier"),
        # Drafting in a serving mix: 16 ragged sequences in shuffled blocks, each with a BF16 tail of the tokens the
        # decode node generated itself, joined through the log-sum-exps.
        dict(name="decode_mix_tail", kind="decode_tail", batch=16, ctx_lo=8192, ctx=65536, tail_lo=1, tail=512,
             shuffled=True, values="student_t"),
        # Verification of a window of k drafted positions with the accept / reject decision: a short context, the
        # serving mix, and windows of 8 positions on long contexts (32 and 64 query columns per KV head).
        dict(name="verify_layer_4k", kind="verify", batch=1, n_q=4, ctx=4096, values="outlier"),
        dict(name="verify_mix_k4", kind="verify", batch=16, n_q=4, ctx_lo=8192, ctx=65536, shuffled=True,
             values="student_t"),
        dict(name="verify_layer_128k_k8", kind="verify", batch=1, n_q=8, ctx=131072, values="lognormal"),
        dict(name="verify_70b_128k_k8", kind="verify", batch=2, group=8, n_q=8, ctx=131072, values="outlier"),
        # The paper's own decode flow on one layer: planes to BF16 pages, then paged attention on the pages.
        dict(name="pages_32k", kind="pages", batch=1, ctx=32768, values="lognormal"),
        # The paper's own quantiser on one layer: K and V pages encoded on one node and decoded on the other.
        dict(name="algorithm1_32k", kind="algorithm1", batch=1, ctx=32768, values="outlier"),
    ]
    return [_full(c) for c in cases]


def _full(c):
    """Every option of a case spelt out; ctx_lo < ctx: ragged lengths, drawn from lens_seed."""
    base = dict(layers=1, batch=1, heads=8, group=4, n_q=1, causal=True, block=16, shuffled=False, lens_seed=1, values="lognormal")
    if c["kind"] in ("quantize_blocks", "algorithm1"):
        base = dict(heads=8, block=16, values="lognormal")
    out = {**base, **c}
    if "ctx" in out and "ctx_lo" not in out:
        out["ctx_lo"] = out["ctx"]
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: any of the kinds, sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(["quantize", "quantize_blocks", "decode", "decode", "decode_tail", "verify", "verify", "pages", "algorithm1"])
    values = rng.choice(["lognormal", "student_t", "outlier"])
    if kind == "quantize_blocks":
        pool = _log_int(rng, 512, 65536)
        return _full(dict(kind=kind, arrived=_log_int(rng, 16, pool), pool=pool, block=rng.choice([16, 16, 32, 64]),
                          values=values))
    if kind == "algorithm1":
        return _full(dict(kind=kind, batch=rng.choice([1, 1, 2]), ctx=_log_int(rng, 256, 131072), values=values))
    ctx = _log_int(rng, 64, 131072)
    ragged = rng.random() < 0.5
    batch = _log_int(rng, 1, 16)
    layers = _log_int(rng, 1, 32) if kind in ("quantize", "decode") and rng.random() < 0.5 else 1
    cap = {"quantize": 32 * 32768, "verify": 16 * 65536, "decode_tail": 16 * 65536, "pages": 4 * 65536}.get(kind, MAX_TOKENS)
    while layers * batch * ctx > cap:
        if layers > 1:
            layers //= 2
        elif batch > 1:
            batch //= 2
        else:
            ctx = cap
    group = rng.choice([4, 4, 8, 8, 1, 2])
    n_q = 1
    if kind == "verify":
        n_q = rng.choice([1, 2, 3, 4, 4, 5, 6, 7, 8, 8])
        if n_q * group > 32 and layers * batch * ctx > 2 * 131072:   # (64 columns: no more than the largest listed)
            batch, ctx = 1, min(ctx, 131072)
    elif kind == "decode" and rng.random() < 0.2:
        n_q = 2                                                      # two drafted positions in one call
    c = dict(kind=kind, layers=layers, batch=batch, group=group, n_q=n_q, ctx=ctx,
             ctx_lo=max(n_q, ctx // rng.randint(2, 8)) if ragged else ctx, block=rng.choice([16, 16, 32, 64]),
             shuffled=rng.random() < 0.5, lens_seed=rng.randint(1, 1000), values=values)
    if kind == "decode_tail":
        c.update(tail_lo=1, tail=_log_int(rng, 1, 1024))
    return _full(c)


# ------------------------------------------------------------------------------------------------ inputs
def _lens(c):
    r = random.Random(c["lens_seed"])
    return [r.randint(c["ctx_lo"], c["ctx"]) for _ in range(c["batch"])]


def _tail_lens(c):
    r = random.Random(c["lens_seed"] + 7919)
    return [r.randint(c["tail_lo"], c["tail"]) for _ in range(c["batch"])]


def _rows(c):
    """(token, KV head) pairs over all layers and sequences: rows of K, and as many of V."""
    return c["layers"] * c["heads"] * sum(_lens(c))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _channel_scale(c, g):
    """Per (head, channel) magnitudes, fixed over tokens: a spread of scales, or three channels of 128 ten times the rest."""
    h = c["heads"]
    if c["values"] == "lognormal":
        return torch.exp(0.5 * torch.randn(h, 1, D, generator=g, device="cuda"))
    s = torch.ones(h, 1, D, device="cuda")
    if c["values"] == "outlier":
        idx = torch.rand(h, D, generator=g, device="cuda").argsort(dim=1)[:, :3]
        s.scatter_(2, idx.unsqueeze(1), 10.0)
    return s


def _values(c, g, scale, n, tokens):
    """BF16 [n][heads][tokens][128] of K or V: Gaussian, or heavy-tailed (Student-t, 4 degrees of freedom)."""
    shape = (n, c["heads"], tokens, D)
    z = torch.randn(shape, generator=g, device="cuda")
    if c["values"] == "student_t":
        w = torch.zeros(shape, device="cuda")
        for _ in range(4):
            w.add_(torch.randn(shape, generator=g, device="cuda").square_())
        z /= (w * 0.25).sqrt_()
    return (z * scale).to(torch.bfloat16)


def _source(c, g, n_blocks):
    """BF16 [n_blocks][heads][block][128], drawn some 16 million values at a time."""
    out = torch.empty(n_blocks, c["heads"], c["block"], D, dtype=torch.bfloat16, device="cuda")
    scale = _channel_scale(c, g)
    step = max(1, (1 << 24) // (c["heads"] * c["block"] * D))
    for i in range(0, n_blocks, step):
        n = min(step, n_blocks - i)
        out[i:i + n] = _values(c, g, scale, n, c["block"])
    return out


def _planes(c, g, n_blocks):
    """The quantised planes of such a cache, without keeping its BF16 source."""
    out = lynx.alloc_planes((n_blocks, c["heads"], c["block"]), "cuda")
    scale = _channel_scale(c, g)
    step = max(1, (1 << 24) // (c["heads"] * c["block"] * D))
    for i in range(0, n_blocks, step):
        n = min(step, n_blocks - i)
        lynx.split_quantize(_values(c, g, scale, n, c["block"]),
                            out=lynx.Planes(out.anchor[i:i + n], out.residual[i:i + n], out.meta[i:i + n]))
    return out


def _table(lens, block, layers, shuffled, seed):
    """Block table int32 [layers * batch][blocks of the longest], and the number of blocks of the pool: every layer's
    blocks follow the previous layer's, in order or permuted within the layer."""
    need = [(n + block - 1) // block for n in lens]
    per_layer = sum(need)
    perm = torch.randperm(per_layer, generator=torch.Generator().manual_seed(seed)) if shuffled else torch.arange(per_layer)
    table = torch.zeros(len(lens), max(need), dtype=torch.int32)
    pos = 0
    for b, n in enumerate(need):
        table[b, :n] = perm[pos:pos + n].to(torch.int32)
        pos += n
    offs = (torch.arange(layers, dtype=torch.int32) * per_layer).view(layers, 1, 1)
    return (table.unsqueeze(0) + offs).reshape(layers * len(lens), -1).contiguous().cuda(), layers * per_layer


def _queries(c, g):
    return torch.randn(c["layers"] * c["batch"], c["n_q"], c["heads"] * c["group"], D, generator=g, device="cuda").to(torch.bfloat16)


def _geometry(c, n_blocks, table):
    return lynx.Geometry(c["heads"] * c["group"], c["heads"], c["block"], n_blocks, table.shape[1])


def prepare(case, seed):
    c, g = case, _gen(seed)
    s = {"case": c}
    if c["kind"] == "quantize_blocks":
        n_pool, n_new = (c["pool"] + c["block"] - 1) // c["block"], (c["arrived"] + c["block"] - 1) // c["block"]
        s["src"] = [_source(c, g, n_pool) for _ in range(2)]
        s["ids"] = torch.randperm(n_pool, generator=torch.Generator().manual_seed(seed))[:n_new].to(torch.int32).cuda()
        s["planes"] = [lynx.Planes(torch.zeros(n_pool, c["heads"], c["block"], 64, dtype=torch.uint8, device="cuda"),
                                   torch.zeros(n_pool, c["heads"], c["block"], 64, dtype=torch.uint8, device="cuda"),
                                   torch.zeros(n_pool, c["heads"], c["block"], 2, device="cuda")) for _ in range(2)]
        return s
    if c["kind"] == "algorithm1":
        n = c["batch"] * ((c["ctx"] + PAGE - 1) // PAGE)
        s["src"] = []
        for _ in range(2):
            scale = _channel_scale(c, g)
            s["src"].append(_values(c, g, scale, n, PAGE).reshape(n * c["heads"], PAGE, D))
        return s
    lens = _lens(c)
    table, n_blocks = _table(lens, c["block"], c["layers"], c["shuffled"], seed)
    if c["kind"] == "quantize":
        s["src"] = [_source(c, g, n_blocks) for _ in range(2)]
        s["planes"] = [lynx.alloc_planes((n_blocks, c["heads"], c["block"]), "cuda") for _ in range(2)]
        return s
    s["K"], s["V"] = _planes(c, g, n_blocks), _planes(c, g, n_blocks)
    s["table"] = table
    s["lens"] = torch.tensor(lens * c["layers"], dtype=torch.int32, device="cuda")
    s["geo"] = _geometry(c, n_blocks, table)
    s["q"] = _queries(c, g)
    B = s["q"].shape[0]
    if c["kind"] == "pages":
        n = int(lynx.load().lynx_bf16_workspace_bytes(s["geo"]._c(), B, c["n_q"]))
        s["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        return s
    s["ws"] = lynx.make_workspace(s["geo"], B, c["n_q"], "cuda")
    if c["kind"] == "decode_tail":
        tail = _tail_lens(c)
        s["tail_table"], n_tail = _table(tail, c["block"], 1, False, seed)
        s["tail_geo"] = _geometry(c, n_tail, s["tail_table"])
        s["tail_lens"] = torch.tensor(tail, dtype=torch.int32, device="cuda")
        s["tail_k"], s["tail_v"] = _source(c, g, n_tail), _source(c, g, n_tail)
        n = int(lynx.load().lynx_bf16_workspace_bytes(s["tail_geo"]._c(), B, c["n_q"]))
        s["tail_ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    if c["kind"] == "verify":   # the Anchor-state results of the same positions
        s["draft"] = lynx.anchor_attention(s["geo"], s["q"], s["K"], s["V"], s["table"], s["lens"], s["ws"], causal=c["causal"])
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "quantize":
        for src, out in zip(s["src"], s["planes"]):
            lynx.split_quantize(src, out=out)
        return [t for p in s["planes"] for t in (p.anchor, p.residual, p.meta)]
    if kind == "quantize_blocks":
        for src, out in zip(s["src"], s["planes"]):
            lynx.split_quantize(src, out=out, block_ids=s["ids"], rows_per_block=c["heads"] * c["block"])
        return [t for p in s["planes"] for t in (p.anchor, p.residual, p.meta)]
    if kind == "decode":
        return lynx.anchor_attention(s["geo"], s["q"], s["K"], s["V"], s["table"], s["lens"], s["ws"], causal=c["causal"])
    if kind == "decode_tail":
        B, n_q = s["q"].shape[:2]
        prefix = lynx.anchor_attention(s["geo"], s["q"], s["K"], s["V"], s["table"], s["lens"], s["ws"])
        tail = lynx.bf16_attention(s["tail_geo"], s["q"], s["tail_k"], s["tail_v"], s["tail_table"], s["tail_lens"],
                                   s["tail_ws"], causal=c["causal"])
        return lynx.lse_merge(prefix, lynx.workspace_lse(s["geo"], B, n_q, s["ws"]),
                              tail, lynx.bf16_workspace_lse(s["tail_geo"], B, n_q, s["tail_ws"]))
    if kind == "verify":
        return lynx.merge_verify_attention(s["geo"], s["q"], s["K"], s["V"], s["table"], s["lens"], s["ws"],
                                           draft_out=s["draft"], atol=0.5, rtol=0.1, causal=c["causal"])
    if kind == "pages":
        _, k = lynx.recombine(s["K"], want_codes=False, want_bf16=True)
        _, v = lynx.recombine(s["V"], want_codes=False, want_bf16=True)
        return k, v, lynx.bf16_attention(s["geo"], s["q"], k, v, s["table"], s["lens"], s["ws"], causal=c["causal"])
    out = []
    for src in s["src"]:
        h = lynx.hier_quantize(src)
        out += [h.q_anc, h.q_res, h.gamma_min, h.gamma_scale, h.mu, h.sigma, lynx.hier_dequantize(h)]
    return out


# ------------------------------------------------------------------------------------------------ accounting
def work(c):
    """Bytes of a row of 128 values: 256 BF16, 64 per nibble plane, 8 of scale and zero point; the operations of
    attention are those of its two contractions."""
    kind = c["kind"]
    if kind == "quantize_blocks":
        rows = 2 * ((c["arrived"] + c["block"] - 1) // c["block"]) * c["block"] * c["heads"]
        return {"bytes": rows * 392, "flops": 0}
    if kind == "algorithm1":
        pages = 2 * c["batch"] * ((c["ctx"] + PAGE - 1) // PAGE) * c["heads"]
        planes = PAGE * 128 + (2 + 16) * D * 4
        return {"bytes": pages * 2 * (PAGE * 256 + planes), "flops": 0}
    if kind == "quantize":
        blocks = sum((n + c["block"] - 1) // c["block"] for n in _lens(c))
        return {"bytes": 2 * c["layers"] * blocks * c["block"] * c["heads"] * 392, "flops": 0}
    cols = c["n_q"] * c["group"]
    rows = _rows(c)                          # of K, and as many of V
    io = c["layers"] * c["batch"] * c["heads"] * cols * D * (2 + 4)   # queries in, outputs out
    flops = 4 * rows * cols * D
    if kind == "decode":
        return {"bytes": 2 * rows * 72 + io, "flops": flops}
    if kind == "decode_tail":
        t = c["heads"] * sum(_tail_lens(c))
        return {"bytes": 2 * rows * 72 + 2 * t * 256 + io, "flops": flops + 4 * t * cols * D}
    if kind == "verify":
        return {"bytes": 2 * rows * 136 + io + io * 4 // 6, "flops": flops}
    # pages: planes in, pages out, pages in
    return {"bytes": 2 * rows * (136 + 256 + 256) + io, "flops": flops}


def tolerance(c):
    """About four times the largest difference from the same path in 64-bit arithmetic, over the cases above and drawn
    ones: attention 8e-6 (largest element 6e-5), 4e-4 (2e-3) where a window has more than 32 query columns per KV head
    (FP16 weights); Algorithm 1: 9e-6 of the packed codes fall on the other side of a rounding tie, and its pages
    are off by their BF16 rounding (2e-3) except at those codes (5e-2)."""
    kind = c["kind"]
    if kind in ("quantize", "quantize_blocks"):
        return "exact"
    if kind == "algorithm1":
        return {"rel": 6e-3, "max": 0.2, "differ": 4e-5}
    if kind == "verify" and c["n_q"] * c["group"] > 32:
        return {"rel": 1.5e-3, "max": 8e-3}
    return {"rel": 3.2e-5, "max": 2.5e-4}


# ------------------------------------------------------------------------------------------------ 64-bit results
def _dequantised(p, full):
    """Values float64 [blocks][heads][block][128] of quantised planes: the 8-bit code, or the middle of the Anchor's
    bucket of 16 codes."""
    def nibbles(t):
        return torch.stack((t & 15, t >> 4), dim=-1).reshape(*t.shape[:-1], D).double()
    level = nibbles(p.anchor) * 16 + (nibbles(p.residual) if full else 8)
    return p.meta[..., 1:2].double() + p.meta[..., 0:1].double() * level


def _pages(c, s, x_of, table, seq, n):
    """The first n tokens of a sequence, [heads][n][128], from the blocks of its table."""
    ids = table[seq, :(n + c["block"] - 1) // c["block"]].long()
    return x_of(ids).permute(1, 0, 2, 3).reshape(c["heads"], -1, D)[:, :n]


def _attend(c, s, parts):
    """Softmax attention over the concatenation of key sets; a part is (K of block ids, V of block ids, table, lengths,
    causal).  float64 [sequences][n_q][query heads][128]."""
    q = s["q"].double()
    B, n_q = q.shape[:2]
    out = torch.empty(q.shape, dtype=torch.float64, device=q.device)
    scale = float(torch.tensor(1.0 / math.sqrt(D), dtype=torch.float32))
    for b in range(B):
        qb = q[b].permute(1, 0, 2).reshape(c["heads"], c["group"] * n_q, D)     # rows: query head of the group, position
        scores, values = [], []
        for k_of, v_of, table, lens, causal in parts:
            n = lens[b]
            sc = qb @ _pages(c, s, k_of, table, b, n).transpose(1, 2) * scale
            if causal:
                last = n - n_q + torch.arange(n_q, device=q.device).repeat(c["group"])
                sc.masked_fill_(torch.arange(n, device=q.device) > last[:, None], -math.inf)
            scores.append(sc)
            values.append(_pages(c, s, v_of, table, b, n))
        o = torch.softmax(torch.cat(scores, 2), 2).nan_to_num_(0.0) @ torch.cat(values, 1)
        out[b] = o.reshape(c["heads"] * c["group"], n_q, D).permute(1, 0, 2)
    return out


def _algorithm1(x):
    """Algorithm 1 of pages [n][256][128] and its inverse: metadata and reconstruction (its packed codes left out)."""
    x = x.double()
    n, eps, log_a = x.shape[0], 1e-6, math.log(256.0)
    g_min = x.amin(1)
    g_scale = x.amax(1) - g_min
    xv = ((x - g_min[:, None]) / (g_scale[:, None] + eps)).view(n, 8, 32, D)
    mu = xv.mean(2)
    cent = xv - mu[:, :, None]
    sigma = cent.abs().amax(2)
    raw = torch.round(torch.log1p(255.0 * (cent / (sigma[:, :, None] + eps)).abs()) / log_a * 120.0)
    mag = torch.expm1(raw / 120.0 * log_a) / 255.0
    back = torch.where(cent < 0, -mag, mag) * (sigma[:, :, None] + eps) + mu[:, :, None]
    return [None, None, g_min, g_scale, mu, sigma, back.view(n, PAGE, D) * (g_scale[:, None] + eps) + g_min[:, None]]


def exact(case, seed):
    """What run() returns, in 64 bits; None for the integer planes of the quantiser, the codes of Algorithm 1 and the
    index of the first rejected position."""
    c = case
    kind = c["kind"]
    if kind in ("quantize", "quantize_blocks"):
        return None
    s = prepare(case, seed)
    if kind == "algorithm1":
        return [t for src in s["src"] for t in _algorithm1(src)]
    lens = _lens(c) * c["layers"]

    def rows(p, full):
        return lambda ids: _dequantised(lynx.Planes(p.anchor[ids], p.residual[ids], p.meta[ids]), full)
    if kind == "pages":
        k, v = _dequantised(s["K"], True), _dequantised(s["V"], True)
        kb, vb = k.float().to(torch.bfloat16), v.float().to(torch.bfloat16)
        return k, v, _attend(c, s, [(lambda i: kb[i].double(), lambda i: vb[i].double(), s["table"], lens, c["causal"])])
    full = kind == "verify"
    planes = (rows(s["K"], full), rows(s["V"], full), s["table"], lens, c["causal"] and kind != "decode_tail")
    if kind == "decode":
        return _attend(c, s, [planes])
    if kind == "decode_tail":
        return _attend(c, s, [planes, (lambda i: s["tail_k"][i].double(), lambda i: s["tail_v"][i].double(),
                                       s["tail_table"], _tail_lens(c), c["causal"])])
    out = _attend(c, s, [planes])
    dev = ((out - s["draft"].double()).abs() / (0.5 + 0.1 * out.abs())).amax((2, 3))
    return out, None, dev
