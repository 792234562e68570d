"""The calls whose speed matters to a user of this library, with the sizes they come in.

A case is one pass through the public entry points as a decode loop makes it: the attention of a
forest of draft trees, the verification of its nodes, the draft stage, the cache update, or a whole
decode step of all of them.  Buffers, workspaces and launch facts are made in `prepare`, as a
serving program makes them once per shape; `run` only makes the calls.

The tensors have the distributions of the package's benchmark workloads (Gaussian queries, keys and
values; logits with a Zipf-shaped bias, the small model's logits near the large model's; draft tokens
sampled from the small model), so accept rates, widths and depths are theirs.
"""
import math

import numpy as np
import torch

import paper_2409_16560_b200 as dsbd
from paper_2409_16560_b200 import inputs

DEVICE = "cuda"


# ------------------------------------------------------------------------------------ cases
def listed():
    gqa = dict(Hq=32, Hkv=8, d=128)
    mha = dict(Hq=32, Hkv=32, d=128)
    plain = dict(temperature=1.0, top_k=0, top_p=1.0)
    return [
        # the smallest attention call: a toy model in fp32 (unit tests, debugging a port), two binary trees
        dict(name="attention-tiny-f32", kind="attention", R=1, W_lo=2, W_hi=2, tree="binary", depth=3, Hq=4, Hkv=4,
             d=64, dtype="f32", L_lo=64, L_hi=64, paged=False, layers=1),
        # one user in front of a 7B-shaped model: four beams, short caches; latency and launches count
        dict(name="attention-one-request", kind="attention", R=1, W_lo=4, W_hi=4, tree="chain", depth=4, **mha,
             dtype="bf16", L_lo=512, L_hi=512, paged=False, layers=1),
        # a batch of requests of different widths and context lengths, grouped heads, packed caches
        dict(name="attention-ragged", kind="attention", R=16, W_lo=1, W_hi=8, tree="chain", depth=5, **gqa,
             dtype="bf16", L_lo=1024, L_hi=4096, paged=False, layers=1),
        # a model with heads of 64 (small target models, draft models), ragged lengths
        dict(name="attention-heads-of-64", kind="attention", R=8, W_lo=4, W_hi=4, tree="chain", depth=5, Hq=32, Hkv=8,
             d=64, dtype="bf16", L_lo=512, L_hi=2047, paged=False, layers=1),
        # the large serving step: 64 requests x 8 beams over 4096-token caches in pages
        dict(name="attention-large-paged", kind="attention", R=64, W_lo=8, W_hi=8, tree="chain", depth=8, **gqa,
             dtype="bf16", L_lo=4096, L_hi=4096, paged=True, layers=1),
        # verification for one user: latency of the per-request part
        dict(name="verify-one-request", kind="verify", R=1, W_lo=4, W_hi=4, tree="chain", depth=4, V=32000, **plain),
        # a few requests over a vocabulary that is no multiple of anything, rows unpadded, wide trees
        dict(name="verify-odd-vocabulary", kind="verify", R=5, W_lo=3, W_hi=6, tree="wide", depth=6, V=50257, **plain),
        # a batch of requests of different widths
        dict(name="verify-ragged", kind="verify", R=16, W_lo=1, W_hi=8, tree="chain", depth=5, V=128256, **plain),
        # the large serving step, sampling at a temperature
        dict(name="verify-large", kind="verify", R=64, W_lo=8, W_hi=8, tree="chain", depth=8, V=128256,
             temperature=0.8, top_k=0, top_p=1.0),
        # the same with the joints warped by top-k / top-p, the sampling of the method's experiments
        dict(name="verify-large-warped", kind="verify", R=64, W_lo=8, W_hi=8, tree="chain", depth=8, V=128256,
             temperature=0.8, top_k=10, top_p=0.8),
        # the draft stage: five sampling steps of the small model, then the forest they trace
        dict(name="draft-stage", kind="draft", R=16, W_lo=8, W_hi=8, gamma=5, V=128256, temperature=1.0, top_k=10,
             top_p=0.8),
        # a whole decode step of a small batch (draft stage, forest, paged attention, verification, cache
        # update) on the forest that the draft stage samples; 13B-shaped heads and vocabulary
        dict(name="decode-step", kind="step", R=8, W_lo=4, W_hi=4, gamma=5, Hq=40, Hkv=40, d=128, dtype="bf16",
             L_lo=2048, L_hi=2048, V=32000, temperature=1.0, top_k=0, top_p=1.0),
    ]


# A drawn case moves at most the bytes of the largest listed one.  fp32 attention is the tool of tests and small
# models and heads of 64 belong to small models: their ranges end earlier, as their use does.
MAX_ATTENTION_BYTES = 8.6e9
MAX_D64_BYTES = 0.5e9
MAX_F32_BYTES = 64e6
MAX_VERIFY_BYTES = 4.7e9


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocabulary(rng):
    # half of the vocabularies are padded to a multiple of 128, the others come as they are
    v = _log_int(rng, 1000, 131072)
    return -(-v // 128) * 128 if rng.random() < 0.5 else v


def _draw_attention(rng):
    u = rng.random()
    dtype = "f32" if u < 0.12 else "bf16"
    d = 64 if (u < 0.3 or dtype == "f32" and rng.random() < 0.5) else 128
    Hq, Hkv = rng.choice([(32, 8), (32, 32), (40, 40), (16, 4), (28, 4), (12, 12)] if dtype == "bf16"
                         else [(4, 4), (8, 2), (12, 12)])
    paged = dtype == "bf16" and d == 128 and rng.random() < 0.5
    c = dict(kind="attention", R=_log_int(rng, 1, 64), W_lo=rng.randint(1, 4), W_hi=rng.randint(4, 8),
             tree=rng.choice(["chain", "chain", "wide", "binary"]), depth=rng.randint(1, 8), Hq=Hq, Hkv=Hkv, d=d,
             dtype=dtype, L_lo=_log_int(rng, 64, 2048), L_hi=0, paged=paged,
             layers=rng.choice([1, 1, 4]) if paged else 1)
    if c["tree"] != "chain":
        c["depth"] = 6 if c["tree"] == "wide" else rng.randint(2, 3)
    c["L_hi"] = c["L_lo"] if rng.random() < 0.3 else _log_int(rng, c["L_lo"], 8192)
    cap = MAX_F32_BYTES if dtype == "f32" else MAX_D64_BYTES if d == 64 else MAX_ATTENTION_BYTES
    while work(c)["bytes"] > cap:
        if c["R"] > 1:
            c["R"] = max(1, c["R"] * 3 // 4)
        elif c["L_hi"] > 64:
            c["L_hi"] = max(64, c["L_hi"] * 3 // 4)
            c["L_lo"] = min(c["L_lo"], c["L_hi"])
        else:
            c["W_hi"] = c["W_lo"] = max(1, c["W_lo"] - 1)
    return c


def _sampling(rng, V):
    # a top-k keeps a small share of the vocabulary; a model of a few thousand tokens is sampled plainly
    top_k = rng.choice([0, 0] + [k for k in (10, 10, 50) if V >= 1024 * k])
    return dict(temperature=rng.choice([1.0, 0.8, 0.6]), top_k=top_k,
                top_p=rng.choice([1.0, 0.8, 0.95]) if top_k else 1.0)


def _draw_verify(rng):
    c = dict(kind="verify", R=_log_int(rng, 1, 64), W_lo=rng.randint(1, 4), W_hi=rng.randint(4, 8),
             tree=rng.choice(["chain", "chain", "wide"]), depth=rng.randint(1, 8), V=_vocabulary(rng))
    c.update(_sampling(rng, c["V"]))
    if c["tree"] == "wide":
        c["depth"] = 6
    while work(c)["bytes"] > MAX_VERIFY_BYTES:
        c["R"] = max(1, c["R"] * 3 // 4)
    return c


def _draw_draft(rng):
    w, V = rng.randint(1, 8), _vocabulary(rng)
    return dict(kind="draft", R=_log_int(rng, 1, 64), W_lo=w, W_hi=w, gamma=rng.randint(2, 8), V=V,
                **_sampling(rng, V))


def _draw_step(rng):
    w = rng.randint(2, 8)
    lo, V = _log_int(rng, 128, 2048), _vocabulary(rng)
    Hq, Hkv = rng.choice([(32, 8), (32, 32), (40, 40)])
    return dict(kind="step", R=_log_int(rng, 1, 16), W_lo=w, W_hi=w, gamma=rng.randint(2, 5), Hq=Hq, Hkv=Hkv, d=128,
                dtype="bf16", L_lo=lo, L_hi=rng.choice([lo, 2 * lo + 1]), V=V, **_sampling(rng, V))


def _draw_commit(rng):
    lo = _log_int(rng, 64, 2048)
    Hq, Hkv = rng.choice([(32, 8), (32, 32), (16, 4)])
    paged = rng.random() < 0.7
    return dict(kind="commit", R=_log_int(rng, 1, 32), W_lo=rng.randint(1, 4), W_hi=rng.randint(4, 8), tree="chain",
                depth=rng.randint(1, 8), Hq=Hq, Hkv=Hkv, d=128, dtype="bf16", L_lo=lo, L_hi=2 * lo - 1, paged=paged,
                layers=rng.choice([1, 4]) if paged else 1)


def draw(rng):
    u = rng.random()
    if u < 0.36:
        return _draw_attention(rng)
    if u < 0.70:
        return _draw_verify(rng)
    if u < 0.82:
        return _draw_draft(rng)
    if u < 0.91:
        return _draw_commit(rng)
    return _draw_step(rng)


# ------------------------------------------------------------------------------------ inputs
def _tree(case):
    if case.get("tree") == "wide":
        return inputs.CONFIGS["C3"]["tree"]
    if case.get("tree") == "binary":
        return [-1] + [(i - 1) // 2 for i in range(1, 2 ** (case["depth"] + 1) - 1)]
    return [-1] + list(range(case["depth"]))


def _shape(case):
    """Forest arrays (numpy), widths and prefix offsets: widths and lengths belong to the case, not to the seed."""
    W = case["W_lo"] if case["W_lo"] == case["W_hi"] else (case["W_lo"], case["W_hi"])
    spec = dict(R=case["R"], W=W, tree=_tree(case), prefix=(case.get("L_lo", 1), case.get("L_hi", 1)))
    return inputs.build_forest(spec, np.random.default_rng(case["R"]))


def _dev(x, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype).to(DEVICE)


def _bytes_buffer(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device=DEVICE)


def _zero_status():
    return torch.zeros(1, dtype=torch.int32, device=DEVICE)


def _params(case, seed, extra=None):
    p = dict(V=case["V"], temperature=case["temperature"], thresh=0.7, W_min=1, W_max=case["W_hi"],
             W_nom=case["W_hi"], seed=int(seed), step=3, top_k=case["top_k"], top_p=case["top_p"])
    p.update(extra or {})
    return p


def _layers(gen, n, shape, dtype):
    """[n, *shape] (or shape for one layer) of N(0,1), filled a piece at a time."""
    t = torch.empty(*((n,) if n > 1 else ()), *shape, dtype=dtype, device=DEVICE)
    flat = t.view(-1)
    for s in range(0, flat.numel(), 1 << 26):
        e = min(s + (1 << 26), flat.numel())
        flat[s:e] = torch.randn(e - s, generator=gen, device=DEVICE)
    return t


def _pages(gen, case, prefix_off, extra):
    """Page pools with every page filled, page tables with shuffled ids, allocator state."""
    need = -(-np.diff(prefix_off) // inputs.PAGE_TOKENS)
    total = int(need.sum())
    n_pages = total + int(extra)
    ids = torch.randperm(n_pages, generator=gen, device=DEVICE).to(torch.int32)
    shape = (n_pages, case["Hkv"], inputs.PAGE_TOKENS, case["d"])
    n = case.get("layers", 1)
    free = torch.sort(ids[total:]).values
    stack = torch.zeros(n_pages, dtype=torch.int32, device=DEVICE)
    stack[:free.numel()] = free
    return dict(k_pool=_layers(gen, n, shape, torch.bfloat16), v_pool=_layers(gen, n, shape, torch.bfloat16),
                page_table=ids[:total].clone(), page_off=_dev(np.concatenate([[0], np.cumsum(need)]).astype(np.int64)),
                free0=stack.clone(), count0=torch.tensor([free.numel()], dtype=torch.int32, device=DEVICE),
                free_stack=stack, free_count=torch.tensor([free.numel()], dtype=torch.int32, device=DEVICE))


def _generator(seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed) + 1)
    return gen


def _attention_state(case, seed):
    forest, _, poff = _shape(case)
    gen, n, dtype = _generator(seed), case["layers"], torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    s = dict(case=case, scale=inputs.default_scale(case["d"]), status=_zero_status(),
             q=_layers(gen, n, (forest["N"], case["Hq"], case["d"]), dtype),
             k_new=_layers(gen, n, (forest["N"], case["Hkv"], case["d"]), dtype),
             v_new=_layers(gen, n, (forest["N"], case["Hkv"], case["d"]), dtype))
    if case["paged"]:
        s.update(_pages(gen, case, poff, 0))
    else:
        for name in ("k_prefix", "v_prefix"):
            s[name] = _layers(gen, 1, (int(poff[-1]) * case["Hkv"] * case["d"],), dtype)
    s["forest"] = dsbd.Forest(forest, DEVICE)
    s["poff"], s["poff_dev"] = poff, _dev(poff)
    s["out"] = torch.empty_like(s["q"])
    # partial results are kept per layer, the rest once: this many layers' worth is enough
    ws = dsbd.forest_attention_workspace(s["forest"], case["Hq"], case["Hkv"], case["d"], dtype, s["scale"], poff)
    s["workspace"] = _bytes_buffer(ws * n)
    return s


def _draft_tokens(gen, case, forest, logits_q):
    """Node n's token is drawn from the small model's next-token distribution at its parent (with the case's
    top-k / top-p, as a draft model samples)."""
    parent = _dev(forest["parent"]).long()
    token = torch.zeros(forest["N"], dtype=torch.int64, device=DEVICE)
    drafts = torch.nonzero(parent >= 0).squeeze(1)
    for rows in drafts.split(max(1, (1 << 25) // case["V"])):
        probs = torch.softmax(logits_q[parent[rows]] / case["temperature"], dim=1)
        if case["top_k"]:
            top, ids = torch.topk(probs, min(case["top_k"], case["V"]), dim=1)
            top /= top.sum(1, keepdim=True)
            top[torch.cumsum(top, 1) - top >= case["top_p"]] = 0.0
            token[rows] = ids.gather(1, torch.multinomial(top, 1, generator=gen)).squeeze(1)
        else:
            token[rows] = torch.multinomial(probs, 1, generator=gen).squeeze(1)
    return token.to(torch.int32)


def _verify_state(case, seed):
    forest, widths, _ = _shape(case)
    gen, N, V = _generator(seed), forest["N"], case["V"]
    bias = -torch.log1p(torch.randperm(V, generator=gen, device=DEVICE).to(torch.float32))
    s = dict(case=case, status=_zero_status(), logits_p=torch.empty(N, V, device=DEVICE),
             logits_q=torch.empty(N, V, device=DEVICE))
    for zp, zq in zip(s["logits_p"].split(256), s["logits_q"].split(256)):
        zp.normal_(generator=gen).mul_(3.0).add_(bias)
        zq.normal_(generator=gen).add_(zp)
    s["root_logp"] = torch.randn(forest["B"], generator=gen, device=DEVICE)
    s["root_logq"] = s["root_logp"] + 0.5 * torch.randn(forest["B"], generator=gen, device=DEVICE)
    s["forest"] = dsbd.Forest(forest, DEVICE)
    s["forest"].dev["token"] = _draft_tokens(gen, case, forest, s["logits_q"])
    s["params"] = _params(case, seed, dict(W_min_r=_dev(np.minimum(2, widths).astype(np.int32))))
    s["out"] = dsbd.alloc_verify_out(s["forest"], dsbd.default_out_off(forest, s["params"]), DEVICE)
    s["workspace"] = _bytes_buffer(dsbd.verify_workspace(s["forest"], s["params"]))
    return s


def _draft_state(case, seed):
    """The small model's logits of every sampling step: the roots' rows, then W rows per request and step."""
    gen = _generator(seed)
    R, W, gamma, V = case["R"], case["W_lo"], case["gamma"], case["V"]
    rows = R * W
    bias = -torch.log1p(torch.randperm(V, generator=gen, device=DEVICE).to(torch.float32))
    off = (W * np.arange(R + 1)).astype(np.int32)
    s = dict(case=case, off=off, off_dev=_dev(off), params=_params(case, seed), status=_zero_status(),
             logits=[torch.randn(rows, V, generator=gen, device=DEVICE) * 3.0 + bias for _ in range(gamma)],
             root_logq=torch.randn(rows, generator=gen, device=DEVICE), drafts=[None] * gamma)
    for l in range(gamma):
        s["drafts"][l] = dsbd.draft_layer(s["off_dev"], off, s["params"], l + 1, W, s["logits"][l], s["root_logq"],
                                          s["off_dev"], rows)
    return s


def _draft_stage(s):
    c, cur = s["case"], s["root_logq"]
    parents, tokens = [], []
    for l in range(c["gamma"]):
        d = dsbd.draft_layer(s["off_dev"], s["off"], s["params"], l + 1, c["W_lo"], s["logits"][l], cur, s["off_dev"],
                             c["R"] * c["W_lo"], workspace=s["drafts"][l]["workspace"], status=s["status"],
                             out=s["drafts"][l])
        parents.append(d["out_parent"])
        tokens.append(d["out_token"])
        cur = d["out_logq"]
    forest, node_of_draw, _ = dsbd.forest_build(s["off_dev"], s["off"], c["gamma"], c["W_lo"], torch.stack(parents),
                                                torch.stack(tokens), status=s["status"], exact=True)
    return forest, node_of_draw


def _commit_buffers(s, R, n_slots):
    s["n_slots"], s["table_capacity"] = n_slots, int(s["page_table"].numel()) + 2 * n_slots
    i32, i64 = torch.int32, torch.int64
    s["commit"] = dict(new_req_beam_off=torch.zeros(R + 1, dtype=i32, device=DEVICE),
                       new_prefix_off=torch.zeros(n_slots + 1, dtype=i64, device=DEVICE),
                       new_page_off=torch.zeros(n_slots + 1, dtype=i64, device=DEVICE),
                       new_page_table=torch.full((s["table_capacity"],), -1, dtype=i32, device=DEVICE),
                       new_beam_slot=torch.zeros(n_slots, dtype=i32, device=DEVICE))


def _commit_paged(s, forest, out):
    c = s["case"]
    # the next pass starts from the same allocator state
    s["free_stack"].copy_(s["free0"])
    s["free_count"].copy_(s["count0"])
    dsbd.kv_commit_paged(forest, c["Hkv"], c["d"], out["out_off"], out["out_width"], out["out_parent"],
                         out["out_root_beam"], out["out_logp"], s["k_new"], s["v_new"], s["k_pool"], s["v_pool"],
                         s["page_table"], s["page_off"], s["poff_dev"], s["poff"], s["free_stack"], s["free_count"],
                         n_slots=s["n_slots"], table_capacity=s["table_capacity"], workspace=s["commit_workspace"],
                         status=s["status"], out=s["commit"])
    res = {k: s["commit"][k] for k in ("new_req_beam_off", "new_prefix_off", "new_page_off", "new_page_table",
                                       "new_beam_slot")}
    res.update(free_stack=s["free_stack"], free_count=s["free_count"], k_pool=s["k_pool"], v_pool=s["v_pool"])
    return res


def _commit_state(case, seed):
    """The output beams of a verification: every request keeps its width of beams, at random nodes."""
    forest, widths, poff = _shape(case)
    rng = np.random.default_rng(int(seed))
    gen, n = _generator(seed), case["layers"]
    f = dsbd.Forest(forest, DEVICE)
    slots = int(widths.sum())
    nodes = np.array([rng.integers(forest["beam_node_off"][b], forest["beam_node_off"][b + 1])
                      for r in range(forest["R"])
                      for b in rng.integers(forest["req_beam_off"][r], forest["req_beam_off"][r + 1],
                                            int(widths[r]))], dtype=np.int32)
    beams = (np.searchsorted(forest["beam_node_off"], nodes, side="right") - 1).astype(np.int32)
    s = dict(case=case, forest=f, poff=poff, poff_dev=_dev(poff), status=_zero_status())
    s["out"] = dict(out_off=_dev(np.concatenate([[0], np.cumsum(widths)]).astype(np.int32)),
                    out_width=_dev(widths.astype(np.int32)), out_parent=_dev(nodes), out_root_beam=_dev(beams),
                    out_logp=torch.randn(slots, generator=gen, device=DEVICE))
    s["k_new"] = _layers(gen, n, (forest["N"], case["Hkv"], case["d"]), torch.bfloat16)
    s["v_new"] = _layers(gen, n, (forest["N"], case["Hkv"], case["d"]), torch.bfloat16)
    if case["paged"]:
        s.update(_pages(gen, case, poff, 2 * slots + 64))
        _commit_buffers(s, forest["R"], slots)
        s["commit_workspace"] = _first_commit_workspace(s, f, s["out"])
    else:
        total = int(poff[-1])
        s["k_prefix"] = _layers(gen, 1, (total * case["Hkv"] * case["d"],), torch.bfloat16)
        s["v_prefix"] = _layers(gen, 1, (total * case["Hkv"] * case["d"],), torch.bfloat16)
        L = np.diff(poff)[forest["req_beam_off"][:-1]]                # the beams of a request have one length
        s["capacity"] = int((widths * (L + case["depth"] + 1)).sum())
        s["k_dst"], s["v_dst"] = (torch.zeros(s["capacity"] * case["Hkv"] * case["d"], dtype=torch.bfloat16,
                                              device=DEVICE) for _ in range(2))
        s["commit"] = _commit_packed(s, None)
    return s


def _first_commit_workspace(s, forest, out):
    # the call makes its workspace when it is given none (on copies: it updates its pools and stack)
    c = s["case"]
    got = dsbd.kv_commit_paged(forest, c["Hkv"], c["d"], out["out_off"], out["out_width"], out["out_parent"],
                               out["out_root_beam"], out["out_logp"], s["k_new"], s["v_new"], s["k_pool"].clone(),
                               s["v_pool"].clone(), s["page_table"], s["page_off"], s["poff_dev"], s["poff"],
                               s["free_stack"].clone(), s["free_count"].clone(), n_slots=s["n_slots"],
                               table_capacity=s["table_capacity"], status=s["status"])
    return got["workspace"]


def _commit_packed(s, prev):
    c, out = s["case"], s["out"]
    return dsbd.kv_commit(s["forest"], c["Hkv"], c["d"], out["out_off"], out["out_width"], out["out_parent"],
                          out["out_root_beam"], out["out_logp"], s["k_new"], s["v_new"], s["k_prefix"], s["v_prefix"],
                          s["poff_dev"], s["poff"], n_slots=int(out["out_parent"].numel()),
                          dst_capacity=s["capacity"], k_dst=s["k_dst"], v_dst=s["v_dst"],
                          workspace=prev["workspace"] if prev else None, status=s["status"], out=prev)


def _step_state(case, seed):
    """A decode step: the state of the draft stage, and the large model's tensors on the forest that the
    draft stage samples (so that the small model's rows of the verification are those it drafted from)."""
    s = _draft_state(case, seed)
    gen = _generator(seed + (1 << 20))
    R, W, gamma, V = case["R"], case["W_lo"], case["gamma"], case["V"]
    B = R * W
    N = B + gamma * B
    forest, node_of_draw = _draft_stage(s)
    L = np.random.default_rng(R).integers(case["L_lo"], case["L_hi"] + 1, size=R)
    s["poff"] = np.concatenate([[0], np.cumsum(np.repeat(L, W))]).astype(np.int64)
    s["poff_dev"] = _dev(s["poff"])
    zq = torch.empty(N, V, device=DEVICE)
    zq[forest.dev["beam_node_off"][:-1].long()] = s["logits"][0]
    for l in range(gamma):
        rows = node_of_draw[l].long()
        # the last layer's nodes have rows of their own: the small model has looked at them as well
        zq[rows] = s["logits"][l + 1] if l + 1 < gamma else torch.randn(B, V, generator=gen, device=DEVICE) * 3.0
    s["logits_q"] = zq
    s["logits_p"] = zq + torch.randn(N, V, generator=gen, device=DEVICE)
    s["root_logp"] = s["root_logq"] + 0.5 * torch.randn(B, generator=gen, device=DEVICE)
    s["q"] = _layers(gen, 1, (N, case["Hq"], case["d"]), torch.bfloat16)
    s["k_new"] = _layers(gen, 1, (N, case["Hkv"], case["d"]), torch.bfloat16)
    s["v_new"] = _layers(gen, 1, (N, case["Hkv"], case["d"]), torch.bfloat16)
    s["attention_out"] = torch.empty_like(s["q"])
    s["scale"] = inputs.default_scale(case["d"])
    slots = R * W
    s.update(_pages(gen, case, s["poff"], 2 * slots + 64))
    # any forest that the draft stage can sample fits these
    bound = dsbd.Forest.from_device(R, B, N, gamma, forest.dev, max_tree_nodes=min(1 + gamma * W, 128),
                                    max_req_beams=W, max_layer_nodes=W)
    s["workspace"] = _bytes_buffer(max(dsbd.forest_attention_workspace(
        f, case["Hq"], case["Hkv"], case["d"], torch.bfloat16, s["scale"], s["poff"]) for f in (bound, forest)))
    off = (W * np.arange(R + 1)).astype(np.int32)
    s["out"] = dsbd.alloc_verify_out(forest, off, DEVICE)
    s["verify_workspace"] = _bytes_buffer(dsbd.verify_workspace(bound, s["params"]))
    _commit_buffers(s, R, slots)
    _verify_call(s, forest)
    s["commit_workspace"] = _first_commit_workspace(s, forest, s["out"])
    return s


def _verify_call(s, forest):
    dsbd.verify_step(forest, s["params"], s["logits_p"], s["logits_q"], s["root_logp"], s["root_logq"], s["out"],
                     workspace=s["verify_workspace"] if "verify_workspace" in s else s["workspace"],
                     status=s["status"])


def prepare(case, seed):
    return dict(attention=_attention_state, verify=_verify_state, draft=_draft_state, commit=_commit_state,
                step=_step_state)[case["kind"]](case, seed)


# ------------------------------------------------------------------------------------ one pass
def _run_attention(s):
    c = s["case"]
    if c["paged"]:
        dsbd.forest_attention_paged(s["forest"], c["Hq"], c["Hkv"], c["d"], s["scale"], s["q"], s["k_new"], s["v_new"],
                                    s["k_pool"], s["v_pool"], s["page_table"], s["page_off"], s["poff_dev"], s["poff"],
                                    out=s["out"], workspace=s["workspace"], status=s["status"])
    else:
        dsbd.forest_attention(s["forest"], c["Hq"], c["Hkv"], c["d"], s["scale"], s["q"], s["k_new"], s["v_new"],
                              s["k_prefix"], s["v_prefix"], s["poff_dev"], s["poff"], out=s["out"],
                              workspace=s["workspace"], status=s["status"])
    return [s["out"], s["status"]]


def _results(out):
    # all of them but the counters of the library's own passes, which no program computes with
    return {k: v for k, v in out.items() if k != "req_stats"}


def _run_verify(s):
    _verify_call(s, s["forest"])
    return [_results(s["out"]), s["status"]]


def _run_draft(s):
    forest, node_of_draw = _draft_stage(s)
    draws = [{k: d[k] for k in ("out_parent", "out_token", "out_logq", "req_error")} for d in s["drafts"]]
    arrays = {k: forest.dev[k] for k in ("beam_node_off", "parent", "token", "draft_rank")}
    return [draws, arrays, node_of_draw, forest.max_tree_nodes, s["status"]]


def _run_commit(s):
    if s["case"]["paged"]:
        return [_commit_paged(s, s["forest"], s["out"]), s["status"]]
    s["commit"] = _commit_packed(s, s["commit"])
    return [{k: s["commit"][k] for k in ("k_dst", "v_dst", "new_req_beam_off", "new_prefix_off", "new_beam_slot")},
            s["status"]]


def _run_step(s):
    c = s["case"]
    forest, node_of_draw = _draft_stage(s)
    dsbd.forest_attention_paged(forest, c["Hq"], c["Hkv"], c["d"], s["scale"], s["q"], s["k_new"], s["v_new"],
                                s["k_pool"], s["v_pool"], s["page_table"], s["page_off"], s["poff_dev"], s["poff"],
                                out=s["attention_out"], workspace=s["workspace"], status=s["status"])
    _verify_call(s, forest)
    return [node_of_draw, s["attention_out"], _results(s["out"]), _commit_paged(s, forest, s["out"]), s["status"]]


def run(state):
    return dict(attention=_run_attention, verify=_run_verify, draft=_run_draft, commit=_run_commit,
                step=_run_step)[state["case"]["kind"]](state)


# ------------------------------------------------------------------------------------ work and tolerance
def _means(case):
    return 0.5 * (case["W_lo"] + case["W_hi"]), 0.5 * (case.get("L_lo", 0) + case.get("L_hi", 0))


def _attention_work(beams, nodes_per_tree, L, case):
    esz = 4 if case["dtype"] == "f32" else 2
    n = beams * nodes_per_tree
    b = beams * L * case["Hkv"] * case["d"] * 2 * esz + n * (2 * case["Hq"] + 2 * case["Hkv"]) * case["d"] * esz
    return dict(bytes=b, flops=4.0 * n * case["Hq"] * case["d"] * (L + 0.5 * nodes_per_tree))


def work(case):
    W, L = _means(case)
    beams = case["R"] * W
    if case["kind"] == "attention":
        w = _attention_work(beams, len(_tree(case)), L, case)
        return {k: v * case["layers"] for k, v in w.items()}
    if case["kind"] == "verify":
        # every row of both models once (their log-sum-exps are outputs)
        return dict(bytes=8.0 * beams * len(_tree(case)) * case["V"], flops=0.0)
    if case["kind"] == "draft":
        return dict(bytes=4.0 * beams * case["gamma"] * case["V"], flops=0.0)
    if case["kind"] == "commit":
        # kept beams: the path and the partly filled last page (paged), or the whole caches, read and written
        tokens = 0.5 * case["depth"] + 1 + (32 if case["paged"] else L)
        return dict(bytes=beams * tokens * case["Hkv"] * case["d"] * 2 * 2 * 2 * case["layers"], flops=0.0)
    a = _attention_work(beams, 1 + case["gamma"], L, case)
    v = 8.0 * beams * (1 + case["gamma"]) * case["V"] + 4.0 * beams * case["gamma"] * case["V"]
    return dict(bytes=a["bytes"] + v, flops=a["flops"])


def tolerance(case):
    # Attention in bf16: products of bf16 values, probabilities and outputs rounded to 8 bits: 0.0023 from a 64-bit
    # evaluation (2-norm; one value by 0.009).  fp32: 2.5e-7 from it.
    if case["kind"] == "attention":
        return dict(rel=1e-2, max=0.04) if case["dtype"] == "bf16" else dict(rel=2e-6)
    if case["kind"] == "commit":
        return "exact"
    # verification and drafting: log-probabilities in fp32 (2.4e-8 from a 64-bit evaluation); tokens, parents and
    # widths are whole numbers, of which a uniform within a rounding error of a cell's boundary may move one
    if case["kind"] == "step":
        return dict(rel=1e-2, max=0.04, differ=2e-3)
    return dict(rel=1e-6, differ=2e-3)
