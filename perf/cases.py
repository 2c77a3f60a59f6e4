"""The work that users of this framework have it do, as cases that can be timed and compared.

Every case is one pass through the public entry points of ``paper_2510_07535_b200``, on inputs that are resident
on the GPU as a serving loop keeps them:

  step      ``owl_verify_step``: attention of the drafted nodes over the paged cache, then acceptance from logits
  attn_f16  ``owl_verify_attn_f16``: the attention alone in fp16, for a verifier that runs in that type
  round     one round of the decoding loop around one attention layer: Prepare(d) on a routed batch, attention of the
            prepared trees, acceptance with the [SPEC] leaf, commit of the accepted rows to the cache
  accept    ``owl_tree_accept_spec``: acceptance of a batch from logits that the caller has
  lm_head   ``owl_lm_head_accept``: acceptance straight from the verifier's last hidden states
  cell      ``owl_lstm_cell``: one step of the drafter's cell

Shapes are those of the benchmark's workloads (8B: 32 query / 8 KV heads; 70B: 64 / 8; 128 channels; 128256 tokens),
of the drafts the loop makes (trees of up to 64 nodes and depth 8, chains of a few tokens) and generic sizes between.
The attention cases hold one layer's cache.
"""
import math
import random

import numpy as np
import torch

from paper_2510_07535_b200 import OwlContext, make_dims
from paper_2510_07535_b200 import workloads as W
from paper_2510_07535_b200.binding import owl_lstm_alpha

DEV = "cuda"
D = W.HEAD_DIM
HEADS = {"8b": (32, 8), "70b": (64, 8)}
SPEC_TOKEN = 128255


def _batch(path, model, seqs, ctx_lo, ctx_hi, tree, depth, chain, chains, **more):
    """A batch of ``seqs`` sequences with contexts in [ctx_lo, ctx_hi]: ``chains`` of them carry a chain of ``chain``
    drafted tokens, the others a tree of ``tree`` nodes of depth <= ``depth``."""
    c = {"path": path, "model": model, "seqs": seqs, "ctx_lo": ctx_lo, "ctx_hi": ctx_hi, "tree": tree, "depth": depth,
         "chain": chain, "chains": chains, "page": 16, "shuffled": True, "outliers": False, "vocab": W.VOCAB, "hit": 0.7}
    c.update(more)
    return c


def listed():
    return [
        # one user, short prompt, chain drafts: the smallest call, launch- and latency-bound
        dict(_batch("step", "8b", 1, 2048, 2048, 0, 0, 8, 1, shuffled=False), name="step_8b_1x2k_chain8"),
        # one user, long prompt, token tree
        dict(_batch("step", "8b", 1, 32768, 32768, 32, 6, 0, 0, shuffled=False), name="step_8b_1x32k_tree32"),
        # few users, longest prompts, largest trees, paged cache
        dict(_batch("step", "8b", 4, 131072, 131072, 64, 8, 0, 0, hit=0.6), name="step_8b_4x128k_tree64"),
        # the larger verifier: 8 query heads per KV head, keys with outlier channels
        dict(_batch("step", "70b", 8, 65536, 65536, 32, 6, 0, 0, shuffled=False, outliers=True), name="step_70b_8x64k_tree32"),
        # a serving batch of mixed lengths, chains and trees side by side
        dict(_batch("step", "8b", 16, 4096, 131072, 32, 6, 8, 8, hit=0.65), name="step_8b_16xmixed"),
        # a chat batch: many short ragged contexts, short chains
        dict(_batch("step", "8b", 48, 200, 6000, 0, 0, 5, 48), name="step_8b_48xshort_chain5"),
        # fp16 verifier on a tree of 30 drafted tokens with their 30 [SPEC] leaves, an odd context length
        dict(_batch("attn_f16", "8b", 1, 47003, 47003, 60, 8, 0, 0), name="attn_f16_8b_1x47k_tree60"),
        # the decoding loop's round for one user, a 30-node tree
        dict(_batch("round", "8b", 1, 8000, 8000, 30, 8, 0, 0), name="round_8b_1x8k_tree30"),
        # acceptance of a batch whose model hands over logits
        dict(_batch("accept", "8b", 16, 0, 0, 60, 8, 9, 4), name="accept_12x60_4x9"),
        # acceptance from hidden states: one user's tree; a batch of trees on the larger verifier
        dict(_batch("lm_head", "8b", 1, 0, 0, 30, 8, 0, 0, hidden=4096), name="lm_head_8b_1x30"),
        dict(_batch("lm_head", "70b", 8, 0, 0, 30, 8, 0, 0, hidden=8192), name="lm_head_70b_8x30"),
        # the drafter growing a tree: 10 open states at once
        {"path": "cell", "rows": 10, "d_in": 4096, "d": 12288, "name": "cell_10_4096_12288"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["step", "step", "step", "step", "step", "attn_f16", "round", "accept", "lm_head", "lm_head", "cell"])
    if path == "cell":
        return {"path": path, "rows": _log(rng, 1, 64), "d_in": rng.choice([2048, 4096, 5120, 8192]), "d": 4 * _log(rng, 1024, 3072)}
    model = rng.choice(["8b", "8b", "70b"])
    most = 64 if model == "8b" else 32
    if path == "lm_head":
        tree = rng.randint(2, most)
        seqs = _log(rng, 1, 384 // tree)
        chains = rng.randint(0, seqs)
        return _batch(path, model, seqs, 0, 0, tree, 8, min(tree, rng.randint(2, 9)), chains,
                      hidden=64 * rng.randint(32, 128), vocab=rng.choice([32000, 50257, W.VOCAB]), hit=0.7)
    if path == "accept":
        seqs = _log(rng, 1, 16)
        return _batch(path, model, seqs, 0, 0, rng.randint(8, 48), 8, rng.randint(2, 9), rng.randint(0, seqs),
                      vocab=rng.choice([32000, 50257, W.VOCAB]), hit=rng.uniform(0.4, 0.9))
    if path == "round":
        seqs = _log(rng, 1, 8)
        hi = _log(rng, 500, 65536 // seqs)
        return _batch(path, model, seqs, max(1, int(hi * rng.uniform(0.1, 1.0))), hi, rng.randint(4, most // 2), 8,
                      rng.randint(2, 9), rng.randint(0, seqs), hit=rng.uniform(0.4, 0.9))
    # step, attn_f16: contexts of 200 to 131072 tokens; 524288 keys and 320 nodes at most in a batch
    hi = _log(rng, 200, 131072)
    tree, chain = rng.randint(8, most), rng.randint(1, 9)
    seqs = _log(rng, 1, max(1, min(64, 524288 // hi)))
    kind = rng.random()
    chains = 0 if kind < 0.4 else seqs if kind < 0.6 else rng.randint(0, seqs)
    chains = max(chains, -(-(seqs * tree - 320) // (tree - chain)) if tree > chain else 0)
    if chains >= seqs:
        chains, chain = seqs, min(chain, max(1, 320 // seqs))
    lo = hi if rng.random() < 0.3 else max(1, int(hi * rng.uniform(0.03, 0.9)))
    return _batch(path, model, seqs, lo, hi, tree, 8, chain, chains, page=rng.choice([16, 16, 16, 32, 64]),
                  shuffled=rng.random() < 0.8, outliers=model == "70b" and rng.random() < 0.3,
                  vocab=rng.choice([32000, 50257, W.VOCAB, W.VOCAB]), hit=rng.uniform(0.4, 0.9))


def _shape(c):
    """(context length, is a chain, nodes) of every sequence: the case's alone, the same for every seed."""
    r = random.Random("%(seqs)d %(ctx_lo)d %(ctx_hi)d %(tree)d %(chain)d %(chains)d" % c)
    lens = [c["ctx_hi"]] + [r.randint(c["ctx_lo"], c["ctx_hi"]) for _ in range(c["seqs"] - 1)]
    chain = [True] * c["chains"] + [False] * (c["seqs"] - c["chains"])
    r.shuffle(lens)
    r.shuffle(chain)
    return [(n, k, c["chain"] if k else c["tree"]) for n, k in zip(lens, chain)]


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)


def _empty(*shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def _drafts(c, rng):
    """Packed offsets, parents and tokens of the batch's drafts (siblings distinct), and the children's planted matches:
    (row, token) pairs whose logit is raised so that the drafted token is the verifier's choice."""
    parents, tokens, plant, base = [], [], [], 0
    for _, is_chain, n in _shape(c):
        p = W.chain_parents(n) if is_chain else W.random_tree_parents(rng, n, c["depth"])
        t = rng.integers(0, c["vocab"] - n)
        tok = (t + rng.permutation(n)).astype(np.int32)
        hit = rng.random(n) < c["hit"]
        plant += [(base + int(p[i]), int(tok[i])) for i in range(1, n) if hit[i]]
        parents.append(p)
        tokens.append(tok)
        base += n
    offsets = np.concatenate([[0], np.cumsum([len(p) for p in parents])]).astype(np.int32)
    return offsets, np.concatenate(parents), np.concatenate(tokens), plant


def _logits(rows, vocab, plant, g):
    x = torch.randn(rows, vocab, generator=g, device=DEV)
    if plant:
        r, t = torch.tensor(plant, device=DEV).t()
        x.index_put_((r, t), torch.tensor(10.0, device=DEV), accumulate=True)
    return x


def _accept_out(seqs, rows):
    return {"accept_len": _empty(seqs), "accept_path": _empty(seqs, 64), "bonus": _empty(seqs), "argmax": _empty(rows)}


def _attention(c, nodes, dtype, rng, g):
    """Q, the paged cache with its table, lengths and outputs for sequences with ``nodes[b]`` draft slots."""
    hq, hkv = HEADS[c["model"]]
    lens = [s[0] for s in _shape(c)]
    pages = [-(-(n + m) // c["page"]) for n, m in zip(lens, nodes)]
    order = rng.permutation(sum(pages)) if c["shuffled"] else np.arange(sum(pages))
    table, at = np.zeros((len(lens), max(pages)), np.int32), 0
    for b, n in enumerate(pages):
        table[b, :n] = order[at:at + n]
        at += n
    rows = sum(nodes)
    k = torch.randn(sum(pages), hkv, c["page"], D, generator=g, device=DEV, dtype=dtype)
    v = torch.randn(sum(pages), hkv, c["page"], D, generator=g, device=DEV, dtype=dtype)
    if c["outliers"]:
        scale = torch.ones(hkv, 1, D, device=DEV, dtype=dtype)
        for h in range(hkv):
            scale[h, 0, torch.from_numpy(rng.choice(D, 2, replace=False)).to(DEV)] = 20.0
        k.mul_(scale)
    q = (torch.randn(rows, hq, D, generator=g, device=DEV) / math.sqrt(D)).to(dtype)
    return {"q": q, "k": k, "v": v, "table": _i32(table), "lens": _i32(lens), "out": _empty(rows, hq, D, dtype=dtype),
            "lse": _empty(rows, hq, dtype=torch.float32), "max_pages": max(pages), "num_pages": sum(pages)}


def _dims(c, nodes, a=None):
    hq, hkv = HEADS[c["model"]] if a else (0, 0)
    return make_dims(batch=len(nodes), total_nodes=sum(nodes), max_nodes=max(nodes), num_q_heads=hq, num_kv_heads=hkv,
                     page_size=c["page"], max_pages_per_seq=a["max_pages"] if a else 0, num_pages=a["num_pages"] if a else 0,
                     vocab=c["vocab"])


def prepare(case, seed):
    c = case
    rng = np.random.default_rng(seed)
    g = torch.Generator(device=DEV).manual_seed(seed)
    if c["path"] == "cell":
        rows, d_in, d = c["rows"], c["d_in"], c["d"]
        bf = torch.bfloat16
        return {"path": "cell", "ctx": OwlContext(make_dims(batch=1, total_nodes=64, max_nodes=64)), "alpha": owl_lstm_alpha(8, d),
                "h": torch.randn(rows, d_in, generator=g, device=DEV, dtype=bf), "emb": torch.randn(rows, d, generator=g, device=DEV, dtype=bf),
                "w": torch.randn(4 * d, d_in, generator=g, device=DEV, dtype=bf).mul_(d_in ** -0.5),
                "ln": [(1 + 0.1 * torch.randn(d, generator=g, device=DEV), 0.1 * torch.randn(d, generator=g, device=DEV)) for _ in range(2)],
                "z": torch.randn(rows, d, generator=g, device=DEV), "h_f32": _empty(rows, d, dtype=torch.float32),
                "h_bf16": _empty(rows, d, dtype=bf), "scratch": _empty(rows, 4 * d, dtype=torch.float32)}
    shape = _shape(c)
    nodes = [s[2] for s in shape]
    offsets, parents, tokens, plant = _drafts(c, rng)
    s = {"path": c["path"], "offsets": _i32(offsets), "parents": _i32(parents), "tokens": _i32(tokens)}
    if c["path"] in ("step", "attn_f16"):
        s.update(_attention(c, nodes, torch.bfloat16 if c["path"] == "step" else torch.float16, rng, g))
        s["dims"] = _dims(c, nodes, s)
        if c["path"] == "step":
            s["logits"] = _logits(sum(nodes), c["vocab"], plant, g)
            s.update(_accept_out(len(nodes), sum(nodes)))
    elif c["path"] == "round":
        # a tree's n nodes become 2n with their [SPEC] leaves, a chain (the linear route) stays as drafted
        full = [n if k else 2 * n for _, k, n in shape]
        first = np.concatenate([[0], np.cumsum(full)])
        moved = [int(first[b] + r - offsets[b]) for b, r in ((int(np.searchsorted(offsets, r, side="right")) - 1, r) for r, _ in plant)]
        s.update(_attention(c, full, torch.bfloat16, rng, g))
        s["drafted"], s["dims"] = _dims(c, nodes, s), _dims(c, full, s)
        s["route"] = _i32([0 if k else 2 for _, k, _ in shape])
        s["start_lens"] = s["lens"].clone()
        s["logits"] = _logits(sum(full), c["vocab"], [(r, t) for r, (_, t) in zip(moved, plant)], g)
        s["prep"] = [_empty(len(full) + 1)] + [_empty(2 * sum(nodes)) for _ in range(4)]
        s.update(_accept_out(len(full), sum(full)), leaf=_empty(len(full)))
    else:
        s["dims"] = _dims(c, nodes)
        s.update(_accept_out(len(nodes), sum(nodes)))
        if c["path"] == "accept":
            s["logits"] = _logits(sum(nodes), c["vocab"], plant, g)
            s["leaf"] = _empty(len(nodes))
        else:
            # a planted row's hidden state leans towards the weight row of the token it should choose
            s["weight"] = torch.randn(c["vocab"], c["hidden"], generator=g, device=DEV, dtype=torch.bfloat16).mul_(c["hidden"] ** -0.5)
            h = torch.randn(sum(nodes), c["hidden"], generator=g, device=DEV)
            last = dict(plant)
            if last:
                h[list(last)] += 8.0 * s["weight"][list(last.values())].float()
            s["hidden"] = h.to(torch.bfloat16)
    s["ctx"] = OwlContext(s["dims"])
    return s


def run(s):
    p, ctx = s["path"], s["ctx"]
    if p == "cell":
        ctx.owl_lstm_cell(s["h"], s["emb"], s["w"], s["alpha"], s["z"], s["h_f32"], s["h_bf16"], s["scratch"], ln_c=s["ln"][0], ln_z=s["ln"][1])
        return s["h_f32"], s["h_bf16"], s["z"]
    d = s["dims"]
    if p == "step":
        ctx.owl_verify_step(d, s["q"], s["k"], s["v"], s["table"], s["lens"], s["offsets"], s["parents"], s["out"], s["lse"], s["logits"],
                            s["tokens"], s["accept_len"], s["accept_path"], s["bonus"], s["argmax"])
        return s["out"], s["lse"], s["accept_len"], s["accept_path"], s["bonus"], s["argmax"]
    if p == "attn_f16":
        ctx.owl_verify_attn_f16(d, s["q"], s["k"], s["v"], s["table"], s["lens"], s["offsets"], s["parents"], s["out"], s["lse"])
        return s["out"], s["lse"]
    if p == "round":
        s["lens"].copy_(s["start_lens"])  # the commit below advances them: every pass is the same round again
        offsets, parents, tokens, _, _ = s["prep"]
        ctx.owl_prepare_hybrid(s["drafted"], s["offsets"], s["parents"], s["tokens"], s["lens"], s["route"], SPEC_TOKEN, *s["prep"])
        n = s["dims"].total_nodes
        parents, tokens = parents[:n], tokens[:n]
        ctx.owl_verify_attn(d, s["q"], s["k"], s["v"], s["table"], s["lens"], offsets, parents, s["out"], s["lse"])
        ctx.owl_tree_accept_spec(d, s["logits"], tokens, offsets, parents, s["accept_len"], s["accept_path"], s["bonus"], s["leaf"], s["argmax"])
        ctx.owl_kv_commit(d, s["k"], s["v"], s["table"], s["lens"], offsets, s["accept_len"], s["accept_path"])
        return {"out": s["out"], "lse": s["lse"], "accept": [s["accept_len"], s["accept_path"], s["bonus"], s["leaf"], s["argmax"]],
                "prepared": [t[:n] if i else t for i, t in enumerate(s["prep"])], "lens": s["lens"], "k": s["k"], "v": s["v"]}
    if p == "accept":
        ctx.owl_tree_accept_spec(d, s["logits"], s["tokens"], s["offsets"], s["parents"], s["accept_len"], s["accept_path"], s["bonus"],
                                 s["leaf"], s["argmax"])
        return s["accept_len"], s["accept_path"], s["bonus"], s["leaf"], s["argmax"]
    ctx.owl_lm_head_accept(d, s["hidden"], s["weight"], s["tokens"], s["offsets"], s["parents"], s["accept_len"], s["accept_path"],
                           s["bonus"], s["argmax"])
    return s["accept_len"], s["accept_path"], s["bonus"], s["argmax"]


def work(case):
    c = case
    if c["path"] == "cell":
        rows, d_in, d = c["rows"], c["d_in"], c["d"]
        return {"bytes": 2 * 4 * d * d_in + rows * (2 * d_in + 2 * d + 8 * d + 6 * d) + 16 * d, "flops": 2.0 * rows * 4 * d * d_in}
    shape = _shape(c)
    hq, hkv = HEADS[c["model"]]
    full = [2 * n if c["path"] == "round" and not k else n for _, k, n in shape]
    rows = sum(full)
    size = flops = 0.0
    if c["path"] in ("step", "attn_f16", "round"):
        keys = [s[0] + n for s, n in zip(shape, full)]
        size += sum(keys) * hkv * D * 4 + rows * hq * (4 * D + 4) + sum(-(-k // c["page"]) for k in keys) * 4
        flops += sum(k * n for k, n in zip(keys, full)) * hq * D * 4.0
    if c["path"] in ("step", "round", "accept"):
        size += rows * c["vocab"] * 4.0
    if c["path"] == "lm_head":
        size += 2.0 * c["hidden"] * (c["vocab"] + rows)
        flops += 2.0 * rows * c["vocab"] * c["hidden"]
    return {"bytes": size, "flops": flops}


def tolerance(case):
    # four times what the path is off from its own arithmetic in 64 bits; for the cell, whose state is fp32, the share of
    # bf16 roundings that another order of its sums can turn
    if case["path"] == "attn_f16":
        return {"rel": 1.2e-3, "max": 8e-3}
    if case["path"] in ("step", "round"):
        return {"rel": 8e-3, "max": 0.06}
    if case["path"] == "cell":
        return {"rel": 1e-3, "max": 0.02}
    if case["path"] == "lm_head":
        return {"differ": 0.005}  # two logits of an unplanted row closer than fp32 sums in another order can tell
    return "exact"
