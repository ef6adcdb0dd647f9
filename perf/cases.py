"""The work that users of this library have it do, as cases to be timed and compared.

Three entry points carry it: fastmtp_draft (K recursive steps of the MTP head), fastmtp_target_step (the decoder
stack: decoding, scoring of drafts, prompt chunks) and fastmtp_verify_accept (acceptance on logits). A case is one
call. Sizes are those of the package's own shapes (inputs.QWEN7B, inputs.TINY) and of the configurations that
bench.py and the tests run: batch 1 to 64, contexts up to 8192 tokens, subsets of 8192 ids up to the full vocabulary,
1 to 5 draft steps, 1 to 28 target layers. Everything is drawn on the GPU: weights ~N(0, 0.02), norm gains
1 + N(0, 0.02), cached K/V and hidden states ~N(0, 1), a shuffled block table.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2509_18362_b200 import binding as Bd
from paper_2509_18362_b200 import inputs as I

SHAPES = {"7b": I.QWEN7B, "tiny": I.TINY}


def _draft(name, shape, B, K, ctx_min, ctx_max, subset, N, max_ext=1):
    return {"name": name, "op": "draft", "shape": shape, "B": B, "K": K, "ctx_min": ctx_min, "ctx_max": ctx_max,
            "subset": subset, "N": N, "max_ext": max_ext}


def _target(name, shape, layers, B, M, ctx_min, ctx_max):
    return {"name": name, "op": "target", "shape": shape, "layers": layers, "B": B, "M": M, "ctx_min": ctx_min,
            "ctx_max": ctx_max}


def _verify(name, B, K, V):
    return {"name": name, "op": "verify", "B": B, "K": K, "V": V}


def listed():
    return [
        # the smallest call: a small head at batch 1, where a draft is all latency
        _draft("draft_tiny", "tiny", 1, 3, 64, 64, "uniform", 1024),
        # the headline: a 7B-class head at batch 1, one request being decoded
        _draft("draft_b1", "7b", 1, 3, 2048, 2048, "uniform", 32768),
        # the same in a speculative loop: up to four positions were committed since the last draft and enter the cache
        _draft("draft_b1_extend", "7b", 1, 3, 1717, 1717, "zipf", 32768, max_ext=4),
        # a few requests at once, ragged contexts, a small vocabulary, a longer draft
        _draft("draft_b4_ragged", "7b", 4, 5, 500, 3000, "zipf", 16384),
        # ordinary serving: 16 requests, each with its committed positions to enter
        _draft("draft_b16_extend", "7b", 16, 3, 2048, 2048, "zipf", 32768, max_ext=4),
        # a full batch with ragged long contexts
        _draft("draft_b64_ragged", "7b", 64, 3, 512, 8192, "uniform", 32768),
        # a prompt enters the MTP cache, 64 pairs per call
        _draft("draft_prompt64", "7b", 1, 1, 448, 448, "uniform", 32768, max_ext=64),
        # acceptance on logits, one request and a full batch
        _verify("verify_b1", 1, 3, 152064),
        _verify("verify_b64", 64, 3, 152064),
        # the target: plain decoding of one request, scoring of its drafts, scoring for 16 requests
        _target("target_decode_b1", "7b", 28, 1, 1, 2048, 2048),
        _target("target_score_b1", "7b", 28, 1, 4, 2048, 2048),
        _target("target_score_b16", "7b", 28, 16, 4, 2048, 2048),
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], uniform over the logarithm."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    op = rng.choice(["draft", "draft", "draft", "target", "target", "verify"])
    if op == "verify":
        K = rng.randint(0, 7)
        V = rng.choice([152064, _log_int(rng, 1000, 152064)])
        B = _log_int(rng, 1, max(1, min(256, 256 * 152064 // ((K + 1) * V))))
        c = _verify("", B, K, V)
    elif op == "draft":
        shape = rng.choice(["7b"] * 6 + ["tiny"])
        V = SHAPES[shape].vocab
        B, K = _log_int(rng, 1, 64), rng.randint(1, 5)
        hi = _log_int(rng, 64, 8192)
        lo = rng.choice([hi, rng.randint(32, hi)])
        N = _log_int(rng, V // 18, V)
        kind = rng.choice(["uniform", "zipf", "full"])
        c = _draft("", shape, B, K, lo, hi, kind, V if kind == "full" else N, rng.choice([1, K + 1]))
    else:
        shape = rng.choice(["7b"] * 6 + ["tiny"])
        layers = _log_int(rng, 1, 28)
        B = _log_int(rng, 1, 64)
        M = rng.randint(1, min(8, max(1, (8 if B < 3 else 64) // B)))
        hi = _log_int(rng, 64, min(8192, max(64, 32768 // B)))
        lo = rng.choice([hi, rng.randint(32, hi)])
        c = _target("", shape, layers, B, M, lo, hi)
    del c["name"]
    return c


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _normal(g, shape, std, mean=0.0):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(mean, std, generator=g)


def _layer(g, s):
    return {"g_in": _normal(g, (s.d,), 0.02, 1.0), "wq": _normal(g, (s.q_dim, s.d), 0.02),
            "wk": _normal(g, (s.kv_dim, s.d), 0.02), "wv": _normal(g, (s.kv_dim, s.d), 0.02),
            "wo": _normal(g, (s.d, s.q_dim), 0.02), "g_post": _normal(g, (s.d,), 0.02, 1.0),
            "w_gate": _normal(g, (s.ffn, s.d), 0.02), "w_up": _normal(g, (s.ffn, s.d), 0.02),
            "w_down": _normal(g, (s.d, s.ffn), 0.02)}


def _caches(g, s, layers, ctx, longest, extra, seed):
    """Paged caches of `layers` layers in one pool with room for len(ctx) sequences of the longest context; all layers
    share lengths and block table."""
    need = [(int(L) + extra + s.page_size - 1) // s.page_size for L in ctx]
    pages = len(ctx) * ((longest + extra + s.page_size - 1) // s.page_size) + 1
    order = np.random.default_rng(seed).permutation(pages).astype(np.int32)
    table = np.full((len(ctx), max(need)), -1, dtype=np.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = order[at:at + n]
        at += n
    pool = (layers, pages, s.n_kv_heads, s.page_size, s.head_dim)
    k, v = _normal(g, pool, 1.0), _normal(g, pool, 1.0)
    table, lens = torch.from_numpy(table).cuda(), torch.from_numpy(ctx).cuda()
    per_layer = [Bd.kv({"k_pages": k[l], "v_pages": v[l], "block_table": table, "seq_lens": lens}) for l in range(layers)]
    return {"k": k, "v": v, "table": table, "lens": lens, "kv": per_layer}


def _context_lengths(c, seed):
    return I.context_lengths(c["B"], c["ctx_min"], c["ctx_max"], seed)


def _zeros(shape, dtype):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def prepare(case, seed):
    return {"draft": _prepare_draft, "target": _prepare_target, "verify": _prepare_verify}[case["op"]](case, seed)


def _prepare_draft(c, seed):
    s, B, K, E = SHAPES[c["shape"]], c["B"], c["K"], c["max_ext"]
    g = _generator(seed)
    w = {"embed": _normal(g, (s.vocab, s.d), 0.02), "lm_head": _normal(g, (s.vocab, s.d), 0.02),
         "g_hnorm": _normal(g, (s.d,), 0.02, 1.0), "g_enorm": _normal(g, (s.d,), 0.02, 1.0),
         "w_proj": _normal(g, (s.d, 2 * s.d), 0.02), "g_final": _normal(g, (s.d,), 0.02, 1.0), "layer": _layer(g, s)}
    ctx = _context_lengths(c, seed)
    subset = None
    if c["subset"] != "full":
        ids = (I.subset_zipf if c["subset"] == "zipf" else I.subset_uniform)(s.vocab, c["N"], seed)
        subset = torch.from_numpy(ids).cuda()
    n_ext = None
    if E > 1:
        # committed positions per sequence: all of a prompt chunk, else what the last round accepted plus one
        n_ext = np.full(B, E) if E > 8 else np.random.default_rng(seed + 1).integers(1, E + 1, size=B)
        n_ext = torch.from_numpy(n_ext.astype(np.int32)).cuda()
    return {"op": "draft", "B": B, "K": K, "E": E, "w": w, "cw": Bd.mtp_w(w), "subset": subset, "n_ext": n_ext,
            "cache": _caches(g, s, 1, ctx, c["ctx_max"], E + K, seed),
            "ctx": Bd.Context(s, max_rows=B * E, max_K=K, max_ctx=c["ctx_max"] + E + K),
            "h": _normal(g, (B, E, s.d), 1.0),
            "tok": torch.randint(0, s.vocab, (B, E), dtype=torch.int32, device="cuda", generator=g),
            "drafts": _zeros((B, K), torch.int32), "hidden": _zeros((B, K, s.d), torch.bfloat16),
            "status": _zeros(1, torch.int32)}


def _prepare_target(c, seed):
    s, B, M = SHAPES[c["shape"]].with_layers(c["layers"]), c["B"], c["M"]
    g = _generator(seed)
    w = {"embed": _normal(g, (s.vocab, s.d), 0.02), "lm_head": _normal(g, (s.vocab, s.d), 0.02),
         "g_final": _normal(g, (s.d,), 0.02, 1.0), "layers": [_layer(g, s) for _ in range(s.n_layers)]}
    cw, keep = Bd.target_w(w)
    ctx = _context_lengths(c, seed)
    return {"op": "target", "B": B, "M": M, "w": w, "cw": cw, "keep": keep,
            "cache": _caches(g, s, s.n_layers, ctx, c["ctx_max"], M, seed),
            "ctx": Bd.Context(s, max_rows=B * M, max_K=1, max_ctx=c["ctx_max"] + M),
            "tok": torch.randint(0, s.vocab, (B, M), dtype=torch.int32, device="cuda", generator=g),
            "hidden": _zeros((B, M, s.d), torch.bfloat16), "logits": _zeros((B, M, s.vocab), torch.bfloat16),
            "argmax": _zeros((B, M), torch.int32), "status": _zeros(1, torch.int32)}


def _prepare_verify(c, seed):
    """Logits ~N(0, 2) with one planted winner per row; drafts follow the winners for a geometric(0.3) prefix."""
    B, K, V = c["B"], c["K"], c["V"]
    g = _generator(seed)
    logits = _normal(g, (B, K + 1, V), 2.0)
    r = np.random.default_rng(seed)
    winner = r.integers(0, V, size=(B, K + 1))
    logits.scatter_(2, torch.from_numpy(winner).cuda().unsqueeze(2), 24.0)
    drafts = r.integers(0, V, size=(B, K)).astype(np.int32)
    for b, n in enumerate(np.minimum(r.geometric(0.3, size=B) - 1, K)):
        drafts[b, :n] = winner[b, :n]
    return {"op": "verify", "B": B, "K": K, "V": V, "logits": logits, "drafts": torch.from_numpy(drafts).cuda(),
            "ctx": Bd.Context(I.TINY, max_rows=8, max_K=8, max_ctx=64),
            "accept": _zeros(B, torch.int32), "bonus": _zeros(B, torch.int32), "argmax": _zeros((B, K + 1), torch.int32),
            "status": _zeros(1, torch.int32)}


def run(st):
    if st["op"] == "draft":
        st["ctx"].fastmtp_draft(st["cw"], st["h"], st["tok"], st["cache"]["kv"][0], st["B"], st["K"], st["subset"],
                                st["drafts"], out_h=st["hidden"], dev_status=st["status"], n_ext=st["n_ext"],
                                max_ext=st["E"])
        return {"drafts": st["drafts"], "hidden": st["hidden"], "k": st["cache"]["k"], "v": st["cache"]["v"],
                "status": st["status"]}
    if st["op"] == "target":
        st["ctx"].fastmtp_target_step(st["cw"], st["tok"], st["cache"]["kv"], st["B"], st["M"], out_h=st["hidden"],
                                      out_logits=st["logits"], out_argmax=st["argmax"], dev_status=st["status"])
        return {"argmax": st["argmax"], "hidden": st["hidden"], "logits": st["logits"], "k": st["cache"]["k"],
                "v": st["cache"]["v"], "status": st["status"]}
    st["ctx"].fastmtp_verify_accept(st["logits"], st["drafts"], st["B"], st["K"], st["V"], st["accept"], st["bonus"],
                                    st["argmax"], st["status"])
    return {"accept": st["accept"], "bonus": st["bonus"], "argmax": st["argmax"], "status": st["status"]}


def work(case):
    """Bytes and operations of one call. A draft reads its weights once per step: a step's input is the previous
    step's result, and the weights (518 MB and the subset's rows at the 7B shape) do not stay on the chip in between."""
    c = case
    if c["op"] == "verify":
        rows = c["B"] * (c["K"] + 1)
        return {"bytes": 2 * rows * c["V"] + 4 * (c["B"] * c["K"] + 2 * c["B"] + rows), "flops": 0}
    s = SHAPES[c["shape"]]
    layer = s.d * (s.q_dim + 2 * s.kv_dim) + s.q_dim * s.d + 3 * s.d * s.ffn
    ctx = c["B"] * (c["ctx_min"] + c["ctx_max"]) / 2
    tok_bytes, tok_flops = 4 * s.kv_dim, 4 * s.q_dim          # one cached position: K and V read; q.k and p.v
    if c["op"] == "target":
        rows = c["B"] * c["M"]
        params = c["layers"] * layer + s.vocab * s.d
        by = 2 * params + c["layers"] * tok_bytes * (ctx + rows) + 2 * rows * (s.vocab + 2 * s.d) + 8 * rows
        fl = 2 * params * rows + c["layers"] * tok_flops * c["M"] * ctx
        return {"bytes": by, "flops": fl}
    B, K, E = c["B"], c["K"], c["max_ext"]
    module, head = 2 * s.d * s.d + layer, c["N"] * s.d
    rows = B * (E if E == 1 or E > 8 else (E + 1) / 2)        # positions that enter in step 1
    by = K * (2 * (module + head) + tok_bytes * ctx) + tok_bytes * (rows + (K - 1) * B)
    by += 4 * s.d * (rows + (K - 1) * B) + 2 * K * B * s.d + 4 * c["N"]
    fl = 2 * module * (rows + (K - 1) * B) + 2 * head * K * B + tok_flops * (ctx * rows / B + (K - 1) * ctx)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Verification is exact. The others add in fp32, round hidden states, logits and cached K/V to bf16 and pick tokens
    by a maximum, so another order of the sums moves a few values by one bf16 step and seldom a token. The library's two
    kernel paths, which add in different orders, differ by rel 5e-4 and max 7.8e-3 (one bf16 step) at 28 layers."""
    if case["op"] == "verify":
        return "exact"
    return {"rel": 2e-3, "max": 3e-2, "differ": 1e-2}
