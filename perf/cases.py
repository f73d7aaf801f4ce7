"""Performance cases of the draft-tree verification library: the calls a speculative decoder makes around and inside
one forward of the target model, through the public Python binding.

Four kinds of pass:

    cycle    one verification cycle of the attention path: ancestor mask of the draft tree, then for every layer the
             tree attention (alone, after the rotary placement of the tree's rows, or with it folded in; on a
             contiguous cache or on a pool of blocks), then acceptance and commit of the accepted rows in all layers
    sampled  the end of a cycle at temperature > 0: sampled acceptance on the target's and the draft's probability
             rows, then the commit of the accepted rows in all layers
    draft    the hand-over from the drafter: rerank of the expansion's candidates, ancestor mask of the kept tree
    static   one layer's attention through the entry point for callers that cannot allocate device memory

Shapes are those of ``paper_2509_15235_b200.synth`` (the target models' heads, the prefix lengths, the tree sizes).
q, k, v are N(0,1) in bf16; trees, token ids and probability rows are drawn as ``synth`` draws them.
"""
import math

import numpy as np
import torch

from paper_2509_15235_b200 import binding, synth

DEV = "cuda"


# ------------------------------------------------------------------------------------------------ listed cases

def _cycle(name, B, N, heads, D, S, layers, vocab, p_match=0.7, depth=6, children=4, rope="none", page_rows=0,
           token_major=False, spare=0, lse=False, kind="cycle"):
    named = {"name": name} if name else {}
    return {**named, "kind": kind, "B": B, "N": N, "Hq": heads[0], "Hkv": heads[1], "D": D, "S_lo": S[0],
            "S_hi": S[1], "depth": depth, "children": children, "layers": layers, "vocab": vocab, "p_match": p_match,
            "rope": rope, "page_rows": page_rows, "token_major": token_major, "spare": spare, "lse": lse}


def listed():
    return [
        # the smallest call: a toy model's cycle, three launches of next to no work
        _cycle("tiny_cycle", 1, 8, (4, 4), 64, (256, 256), 1, 1000, depth=3, children=0),
        # LLaVA-1.6 7B (multi-head) on a long image prefix, a whole cycle of 32 layers: the benchmark's default
        _cycle("llava7b_cycle", 1, 60, (32, 32), 128, (3904, 3904), 32, 32000),
        # Qwen2.5-VL 7B (grouped heads), a whole cycle of 28 layers with the rotary embedding folded in
        _cycle("qwen7b_fused_rope", 1, 60, (28, 4), 128, (3344, 3344), 28, 152064, 0.6, rope="fused"),
        # LLaVA-1.6 13B, four sequences of different lengths, rotary placement and attention as two calls
        _cycle("llava13b_b4_rope", 4, 60, (40, 40), 128, (3000, 5000), 8, 32000, rope="rows"),
        # the same model served from a pool of 16-slot blocks in token-major order, as serving stacks keep it
        _cycle("llava13b_b4_paged16", 4, 60, (40, 40), 128, (3000, 5000), 8, 32000, rope="rows", page_rows=16,
               token_major=True),
        # Qwen2.5-VL 3B, short answer, small tree: 36 short attention calls, latency and launches
        _cycle("qwen3b_S2048_N16_B1", 1, 16, (16, 2), 128, (2048, 2048), 36, 151936, 0.6),
        # the same model batched at middle length, rotary embedding folded in
        _cycle("qwen3b_S8192_N60_B4", 4, 60, (16, 2), 128, (8192, 8192), 16, 151936, 0.6, rope="fused"),
        # one very long response: two kv heads to spread over the whole GPU
        _cycle("qwen3b_S32768_N16_B1", 1, 16, (16, 2), 128, (32768, 32768), 16, 151936, 0.6),
        # the largest: eight long sequences with full-size trees
        _cycle("qwen3b_S32768_N128_B8", 8, 128, (16, 2), 128, (32768, 32768), 16, 151936, 0.6),
        # the end of a cycle at temperature > 0 over the large vocabulary, commit of 28 layers
        _cycle("qwen7b_sampled", 1, 60, (28, 4), 128, (3344, 3344), 28, 152064, 0.6, kind="sampled"),
        # the drafter's hand-over at the paper's own sizes: 136 candidates, 30 kept
        {"name": "paper_draft", "kind": "draft", "B": 1, "width": 8, "levels": 3, "K": 30, "vocab": 32000},
        # one layer without any allocation, with the log-sum-exp that a caller merging caches asks for
        _cycle("llava7b_static", 1, 60, (32, 32), 128, (3904, 3904), 1, 32000, lse=True, kind="static"),
    ]


# ------------------------------------------------------------------------------------------------ drawn cases

_MODELS = [((32, 32), 128, 32000), ((28, 4), 128, 152064), ((40, 40), 128, 32000), ((16, 2), 128, 151936),
           ((4, 4), 64, 1000), ((16, 4), 64, 32000)]
_MOST_BYTES = 3.0e9      # of a case's caches
_MOST_FLOPS = 4.0e12     # of a pass (the largest listed case: 4.4e12)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: kind by use, lengths and counts spread over their ranges (odd values among them)."""
    kind = rng.choices(["cycle", "sampled", "draft", "static"], [7, 1, 1, 1])[0]
    if kind == "draft":
        # expansions of 4 to 12 children over 2 to 8 levels (20 to 1020 candidates), 8 to 127 kept
        while True:
            width, levels, K = rng.randint(4, 12), rng.randint(2, 8), _log_int(rng, 8, 127)
            if K <= width + (levels - 1) * width * width:
                return {"kind": "draft", "B": rng.randint(1, 8), "width": width, "levels": levels, "K": K,
                        "vocab": rng.choice([32000, 151936, 152064])}
    heads, D, vocab = rng.choice(_MODELS)
    B = rng.choice([1, 1, 1, 2, 3, 4, 6, 8])
    N = rng.choice([8, 16, 31, 60, 128, rng.randint(2, 127), rng.randint(2, 127)])
    if kind == "sampled":
        V = rng.choice([32000, 151936, 152064, _log_int(rng, 1000, 152064)])
        while B * N * V * 8 > 1.2e9:
            B = max(1, B // 2) if B > 1 else B
            N = N if B > 1 else max(2, N // 2)
        return _cycle(None, B, N, heads, D, (1000, 2000), rng.choice([4, 28, 32]) if heads[0] < 32 else 8, V,
                      rng.uniform(0.5, 0.8), kind=kind, spare=0)
    S_hi = _log_int(rng, 128, 32768 if heads[0] < 28 else 8192)
    if D == 64:
        S_hi = min(S_hi, 4096)
    S_lo = S_hi if rng.random() < 0.4 else max(1, int(S_hi * rng.uniform(0.4, 1.0)))     # ragged batches
    spare = rng.choice([0, 0, 512, 2048])                                # slots allocated for the rest of the response
    slots = S_hi + N + spare + 128
    if kind == "static":
        while B * heads[1] * ((heads[0] // heads[1] * N + 63) // 64) > 240:       # what the built-in scratch holds
            B, N = (B // 2, N) if B > 1 else (B, N // 2)
        return _cycle(None, B, N, heads, D, (S_lo, S_hi), 1, vocab, kind=kind, spare=spare, lse=rng.random() < 0.5)
    layer_bytes = 4.0 * B * heads[1] * slots * D
    layer_flops = 4.0 * D * heads[0] * N * B * (S_hi + N)
    most = int(min(36, _MOST_BYTES / layer_bytes, _MOST_FLOPS / layer_flops))
    while most < 1:
        B = B // 2
        layer_bytes, layer_flops = layer_bytes / 2, layer_flops / 2
        most = int(min(36, _MOST_BYTES / layer_bytes, _MOST_FLOPS / layer_flops))
    paged = D == 128 and rng.random() < 0.3
    rope = rng.choice(["none", "rows", "fused"]) if D == 128 and not paged else rng.choice(["none", "rows"])
    depth, children = rng.choice([(6, 4), (3, 8)]) if N <= 70 else (6, 4)
    return _cycle(None, B, N, heads, D, (S_lo, S_hi), _log_int(rng, 1, most), vocab, rng.choice([0.6, 0.7]), depth, children,
                  rope, rng.choice([16, 32, 64, 128]) if paged else 0, paged and rng.random() < 0.5, spare,
                  rng.random() < 0.2)


# ------------------------------------------------------------------------------------------------ inputs

def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)


def _normal(shape, gen):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)


def _trees(c, rng):
    B, N = c["B"], c["N"]
    parents = np.stack([synth.draw_tree(N, c["depth"], c["children"], rng) for _ in range(B)])
    ids = [synth.draw_ids(parents[b], c["vocab"], c["p_match"], rng) for b in range(B)]
    kv_len = rng.integers(c["S_lo"], c["S_hi"] + 1, size=B)
    return parents, np.stack([d for d, _ in ids]), np.stack([t for _, t in ids]), kv_len


def _slots(c):
    return (c["S_hi"] + c["N"] + c["spare"] + 127) // 128 * 128


def prepare(case, seed):
    c = dict(case)
    rng = np.random.Generator(np.random.SFC64(seed))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if c["kind"] == "draft":
        x = synth.make_rerank_candidates(c["B"], c["levels"], c["width"], c["vocab"], seed)
        N = c["K"] + 1
        s = {"c": c, "ctx": binding.VerifyContext(c["B"], N, 4, 4, 64, 256, 1)}
        s["cand"] = [_i32(x["cand_parent"]), _i32(x["cand_token"]), torch.from_numpy(x["cand_score"]).to(DEV)]
        s["parents"] = torch.zeros((c["B"], N), dtype=torch.int32, device=DEV)
        s["ids"] = torch.zeros_like(s["parents"])
        s["depth"] = torch.zeros_like(s["parents"])
        s["selected"] = torch.zeros((c["B"], c["K"]), dtype=torch.int32, device=DEV)
        s["mask"] = torch.zeros((c["B"], N, (N + 63) // 64), dtype=torch.int64, device=DEV)
        return s

    B, N, Hq, Hkv, D, L = (c[k] for k in ("B", "N", "Hq", "Hkv", "D", "layers"))
    S_max, pr = _slots(c), c["page_rows"]
    parents, draft, target, kv_len = _trees(c, rng)
    s = {"c": c, "scale": 1.0 / math.sqrt(D), "theta": 1e6 if Hq != Hkv else 1e4}
    s["parents"], s["draft"], s["target"], s["kv_len"] = _i32(parents), _i32(draft), _i32(target), _i32(kv_len)
    # the caches of all layers, every slot filled (the tree's own rows among them)
    if pr:
        per = S_max // pr
        shape = (B * per, pr, Hkv, D) if c["token_major"] else (B * per, Hkv, pr, D)
        s["table"] = _i32(rng.permutation(B * per).reshape(B, per))
    else:
        shape = (B, Hkv, S_max, D)
    s["cache"] = _normal((L, 2) + shape, gen)
    s["mask"] = torch.zeros((B, N, (N + 63) // 64), dtype=torch.int64, device=DEV)
    s["depth"] = torch.zeros((B, N), dtype=torch.int32, device=DEV)

    if c["kind"] == "static":
        s["q"] = _normal((B, N, Hq, D), gen)
        s["out"] = torch.zeros_like(s["q"])
        s["lse"] = torch.zeros((B, Hq, N), dtype=torch.float32, device=DEV) if c["lse"] else None
        ctx = binding.VerifyContext(B, N, Hq, Hkv, D, S_max, 1)
        ctx.tree_mask_build(s["parents"], s["mask"], s["depth"])
        torch.cuda.synchronize()
        ctx.close()
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        return s

    ctx = s["ctx"] = binding.VerifyContext(B, N, Hq, Hkv, D, S_max, L)
    for l in range(L):
        if pr:
            ctx.cache_register_paged(l, s["cache"][l, 0], s["cache"][l, 1], c["token_major"])
        else:
            ctx.cache_register(l, s["cache"][l, 0], s["cache"][l, 1])
    s["path"] = torch.zeros((B, N), dtype=torch.int32, device=DEV)
    s["alen"], s["bonus"], s["new_len"] = (torch.zeros(B, dtype=torch.int32, device=DEV) for _ in range(3))

    if c["kind"] == "sampled":
        V = c["vocab"]
        g = torch.randn((B, N, V), generator=gen, device=DEV)
        s["p"] = torch.softmax(6.0 * g, dim=-1)
        g += 0.3 * torch.randn((B, N, V), generator=gen, device=DEV)
        s["p_hat"] = torch.softmax(6.0 * g, dim=-1)
        del g
        # every node's token is a draw from its parent's draft row (siblings are i.i.d. draws, so they may repeat)
        pool = torch.multinomial(s["p_hat"].view(B * N, V), N, replacement=True, generator=gen).view(B, N, N)
        par = s["parents"].long().clamp(min=0)
        s["draft"] = torch.gather(pool, 1, par[:, :, None].expand(B, N, N)).diagonal(dim1=1, dim2=2).to(torch.int32).contiguous()
        s["u_accept"] = torch.rand((B, N), generator=gen, device=DEV)
        s["u_bonus"] = torch.rand(B, generator=gen, device=DEV)
        return s

    s["q"] = _normal((L, B, N, Hq, D), gen)
    s["out"] = torch.zeros_like(s["q"])
    s["lse"] = torch.zeros((L, B, Hq, N), dtype=torch.float32, device=DEV) if c["lse"] else None
    s["q_of"], s["out_of"] = list(s["q"]), list(s["out"])
    s["lse_of"] = list(s["lse"]) if c["lse"] else [None] * L
    if c["rope"] != "none":
        s["rows"] = _normal((L, 2, B, N, Hkv, D), gen)
        s["k_of"], s["v_of"] = [r[0] for r in s["rows"]], [r[1] for r in s["rows"]]
        depth = np.zeros((B, N), dtype=np.int32)                  # a node's position: committed length plus its depth
        for i in range(1, N):
            depth[:, i] = depth[np.arange(B), parents[:, i]] + 1
        s["positions"] = _i32(kv_len[:, None] + depth)
    if c["rope"] == "fused":
        s["angles"] = ctx.rope_table_build(s["positions"], s["theta"])
    return s


# ------------------------------------------------------------------------------------------------ the pass

def run(s):
    c = s["c"]
    if c["kind"] == "draft":
        s["ctx"].tree_rerank(*s["cand"], c["K"], s["parents"], s["ids"], s["selected"])
        s["ctx"].tree_mask_build(s["parents"], s["mask"], s["depth"])
        return {k: s[k] for k in ("parents", "ids", "selected", "mask", "depth")}
    if c["kind"] == "static":
        k, v = s["cache"][0, 0], s["cache"][0, 1]
        binding.tree_verify_attn_static(s["q"], k, v, s["kv_len"], s["mask"], s["scale"], s["out"], s["lse"], s["status"])
        return {k: s[k] for k in ("out", "lse", "status")}

    ctx, L, kv_len = s["ctx"], c["layers"], s["kv_len"]
    if c["kind"] == "sampled":
        ctx.accept_sampled(s["draft"], s["parents"], s["p"], s["p_hat"], s["u_accept"], s["u_bonus"], s["path"], s["alen"], s["bonus"])
        if c["page_rows"]:
            ctx.kv_compact_paged(0, L, s["path"], s["alen"], kv_len, s["table"], s["new_len"])
        else:
            ctx.kv_compact(0, L, s["path"], s["alen"], kv_len, s["new_len"])
        return {k: s[k] for k in ("path", "alen", "bonus", "new_len", "cache")}

    rope, paged, mask, scale = c["rope"], c["page_rows"] > 0, s["mask"], s["scale"]
    ctx.tree_mask_build(s["parents"], mask, s["depth"])
    if rope == "fused":
        ctx.rope_table_build(s["positions"], s["theta"], s["angles"])
    for l in range(L):
        q, out, lse = s["q_of"][l], s["out_of"][l], s["lse_of"][l]
        if rope == "fused":
            ctx.tree_verify_attn_rope(l, q, s["k_of"][l], s["v_of"][l], s["angles"], kv_len, mask, scale, out, lse)
            continue
        if rope == "rows" and paged:
            ctx.rope_tree_rows_paged(l, q, s["k_of"][l], s["v_of"][l], s["positions"], kv_len, s["table"], s["theta"])
        elif rope == "rows":
            ctx.rope_tree_rows(l, q, s["k_of"][l], s["v_of"][l], s["positions"], kv_len, s["theta"])
        if paged:
            ctx.tree_verify_attn_paged(l, q, kv_len, s["table"], mask, scale, out, lse)
        else:
            ctx.tree_verify_attn(l, q, kv_len, mask, scale, out, lse)
    if paged:
        ctx.accept_commit_paged(0, L, s["draft"], s["target"], s["parents"], kv_len, s["table"], s["path"], s["alen"],
                                s["bonus"], s["new_len"])
    else:
        ctx.accept_commit(0, L, s["draft"], s["target"], s["parents"], kv_len, s["path"], s["alen"], s["bonus"], s["new_len"])
    # lse, where asked for; q, which the rotary placement rotates in place
    more = (["lse"] if c["lse"] else []) + (["q"] if rope == "rows" else [])
    return {k: s[k] for k in ["out", "mask", "depth", "path", "alen", "bonus", "new_len", "cache"] + more}


# ------------------------------------------------------------------------------------------------ work and tolerance

def work(case):
    """Bytes read and written once, and the flops of the two contractions, of one pass.  Lengths drawn per sequence
    count at their mean; about three accepted rows per sequence move at the commit."""
    c = case
    if c["kind"] == "draft":
        M, N = c["width"] + (c["levels"] - 1) * c["width"] ** 2, c["K"] + 1
        return {"bytes": c["B"] * (12 * M + 4 * (3 * N - 1) + N * (4 + 8 * ((N + 63) // 64))), "flops": 0}
    B, N, Hq, Hkv, D, L = (c[k] for k in ("B", "N", "Hq", "Hkv", "D", "layers"))
    S = 0.5 * (c["S_lo"] + c["S_hi"])
    ints = B * N * (4 * 5 + 8 * ((N + 63) // 64))
    commit = L * B * Hkv * D * 2 * 2 * 3 * 2
    if c["kind"] == "sampled":
        # the last node's two rows have to be read for the bonus token, and two probabilities per decided node
        return {"bytes": B * c["vocab"] * 8 + ints + commit, "flops": 2.0 * B * c["vocab"]}
    kv = 4.0 * B * Hkv * D * (S + N)
    qo = 4.0 * B * N * Hq * D
    lse = 4.0 * B * N * Hq if c["lse"] else 0.0
    rows = 0.0
    if c["rope"] != "none":
        rows = 8.0 * B * N * Hkv * D + (2.0 * B * N * Hq * D if c["rope"] == "rows" else 0.0)
    flops = 4.0 * D * Hq * N * B * (S + N)
    if c["kind"] == "static":
        return {"bytes": kv + qo + lse, "flops": flops}
    return {"bytes": L * (kv + qo + lse + rows) + ints + commit, "flops": L * flops}


def tolerance(case):
    """Integers and committed rows are exact.  Attention: bf16 inputs, probabilities and outputs with fp32 sums (a few
    bf16 roundings of 2^-9 each); rotated rows may differ by one bf16 step."""
    if case["kind"] in ("draft", "sampled"):
        return "exact"
    return {"rel": 1e-2, "max": 0.05}
