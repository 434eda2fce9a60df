"""The work that a decoding loop has this library do, as cases that can be timed.

Each case is one call (or the calls of one decode step) through the public binding, on
arguments, outputs and workspaces that the loop keeps between steps. Kinds:

  step    the fused verify step: attention of one layer beside the acceptance
  attn    the verify attention alone (the layers below the last one)
  accept  the lossless acceptance alone, filtered (top-k / top-p) where top_k > 0
  draft   drawing the block from the drafter's rows, filtered where top_k > 0
  build   the tree sampler: a candidate tree from the drafter's rows
  tree    verification of a candidate tree: masked attention, then tree acceptance
  head    the LM head with the row statistics fused

Contexts are ragged (uniform on ctx_lo..ctx_hi), pages a random permutation of the cache.
Logits are normal with a spread of 3, the drafter's rows the target's plus noise, and
drafts are drawn from the drafter, so that a usual share of them is accepted.
"""

import math

import torch

from paper_2609_04010_gb300 import binding


def listed():
    return [
        # one request on a small model: launches and latency are the whole step
        dict(name="step_one_request", kind="step", batch=1, gamma=4, vocab=32000, dtype="f32",
             greedy=0.0, T=1.0, noise=0.5, hq=8, hkv=8, dim=64, page=16, ctx_lo=512, ctx_hi=512),
        # a few requests on an 8B-shaped model
        dict(name="step_batch8", kind="step", batch=8, gamma=8, vocab=128256, dtype="bf16",
             greedy=0.0, T=1.0, noise=1.0, hq=32, hkv=8, dim=128, page=16, ctx_lo=4096, ctx_hi=4096),
        # high-batch serving, ragged contexts, half of the requests greedy
        dict(name="step_serving", kind="step", batch=64, gamma=16, vocab=128256, dtype="bf16",
             greedy=0.5, T=1.0, noise=0.5, hq=32, hkv=8, dim=128, page=16, ctx_lo=512, ctx_hi=4096),
        # the smallest block (plain decoding), ragged long contexts: the cache read once
        dict(name="attn_decode", kind="attn", batch=32, gamma=1, hq=32, hkv=8, dim=128, page=16,
             ctx_lo=256, ctx_hi=16384),
        # a 70B-shaped model at long context: the most arithmetic per byte of cache
        dict(name="attn_long", kind="attn", batch=4, gamma=32, hq=64, hkv=8, dim=128, page=64,
             ctx_lo=32768, ctx_hi=32768),
        # acceptance alone: fp32 logits of an odd vocabulary (unaligned rows)
        dict(name="accept_f32_odd", kind="accept", batch=16, gamma=5, vocab=50257, dtype="f32",
             greedy=0.25, T=0.7, noise=1.0, top_k=0, top_p=1.0),
        # the evaluation sampling (top-k 50, top-p 0.95) at serving batch
        dict(name="accept_topk_serving", kind="accept", batch=64, gamma=16, vocab=128256,
             dtype="bf16", greedy=0.0, T=1.0, noise=0.5, top_k=50, top_p=0.95),
        # the draft side of a serving step
        dict(name="draft_serving", kind="draft", batch=64, gamma=16, vocab=128256, dtype="bf16",
             greedy=0.5, T=1.0, top_k=0, top_p=1.0),
        # the tree sampler for one request
        dict(name="tree_build_one", kind="build", batch=1, gamma=16, vocab=128256, dtype="bf16",
             top_k=32, nodes=33),
        # tree verification of one request, sampled
        dict(name="tree_verify_one", kind="tree", batch=1, nodes=33, vocab=128256, dtype="bf16",
             greedy=0.0, T=1.0, hq=32, hkv=8, dim=128, page=16, ctx_lo=4096, ctx_hi=4096),
        # the LM head of a small batch's block rows: the weight streams once
        dict(name="head_64_rows", kind="head", rows=64, rows_per_seq=8, hidden=4096, vocab=128256),
        # the LM head of a serving step's rows: a contraction
        dict(name="head_1024_rows", kind="head", rows=1024, rows_per_seq=16, hidden=4096, vocab=128256),
    ]


# ---------------------------------------------------------------------------------------
# Cases drawn from the ranges that the listed ones stand for
# ---------------------------------------------------------------------------------------
MAX_BYTES, MAX_FLOPS = 1.0e9, 1.0e12


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_attn(rng, gamma_hi):
    hkv = rng.choice([2, 4, 8, 8])
    ctx = _log_int(rng, 64, 32768)
    return dict(batch=_log_int(rng, 1, 128), gamma=_log_int(rng, 1, gamma_hi),
                hq=hkv * rng.choice([1, 2, 4, 4, 5, 8]), hkv=hkv, dim=rng.choice([64, 128, 128]),
                page=rng.choice([16, 16, 32, 64]), ctx_lo=max(1, int(ctx * rng.choice([0.1, 0.5, 1.0]))),
                ctx_hi=ctx)


def _draw_logits(rng):
    return dict(vocab=rng.choice([32000, 128256, 151936, _log_int(rng, 30000, 152000)]),
                dtype=rng.choice(["bf16", "bf16", "f32"]), greedy=rng.choice([0.0, 0.0, 0.5, 1.0]),
                T=rng.choice([0.7, 1.0]))


def draw(rng):
    kind = rng.choice(["step", "step", "attn", "attn", "attn", "accept", "accept", "draft", "build",
                       "tree", "head"])
    topk = dict(top_k=rng.choice([20, 50, 50, 200]), top_p=rng.choice([0.9, 0.95, 1.0]))
    if rng.random() < 0.5:
        topk = dict(top_k=0, top_p=1.0)
    case = dict(kind=kind)
    if kind == "step":
        case.update(_draw_attn(rng, 32), **_draw_logits(rng), noise=rng.choice([0.1, 0.5, 1.0, 3.0]))
    elif kind == "attn":
        case.update(_draw_attn(rng, 32))
    elif kind == "accept":
        case.update(batch=_log_int(rng, 1, 128), gamma=_log_int(rng, 1, 32), **_draw_logits(rng),
                    noise=rng.choice([0.1, 0.5, 1.0, 3.0]), **topk)
    elif kind == "draft":
        case.update(batch=_log_int(rng, 1, 128), gamma=_log_int(rng, 1, 32), **_draw_logits(rng), **topk)
    elif kind == "build":
        case.update(batch=_log_int(rng, 1, 16), gamma=_log_int(rng, 4, 16), top_k=rng.choice([8, 32]),
                    nodes=rng.randint(9, 64), **_draw_logits(rng))
        del case["greedy"], case["T"]
    elif kind == "tree":
        case.update(_draw_attn(rng, 1), **_draw_logits(rng))
        del case["gamma"]
        case.update(batch=_log_int(rng, 1, 16), nodes=rng.randint(5, 64))
    else:
        case.update(rows=_log_int(rng, 1, 1024), rows_per_seq=rng.choice([1, 4, 8, 16]),
                    hidden=rng.choice([2048, 4096, 8192, 5120]), vocab=_log_int(rng, 30000, 152000))
    while work(case)["bytes"] > MAX_BYTES or work(case)["flops"] > MAX_FLOPS:
        if kind == "head":
            case["rows"] = (case["rows"] * 2 + 2) // 3
            case["vocab"] = max(30000, case["vocab"] * 5 // 6)
            case["hidden"] = max(2048, case["hidden"] // 2 // 64 * 64)
        elif case["batch"] > 1:
            case["batch"] = (case["batch"] * 2) // 3
        else:
            case["ctx_hi"] = case["ctx_hi"] * 2 // 3
            case["ctx_lo"] = min(case["ctx_lo"], case["ctx_hi"])
    return case


# ---------------------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------------------
def _esize(case):
    return 2 if case["dtype"] == "bf16" else 4


def _greedy_count(case):
    return int(round(case["batch"] * case["greedy"]))


def _attn_work(case, gamma):
    keys = case["batch"] * ((case["ctx_lo"] + case["ctx_hi"]) / 2 + gamma)
    kv = keys * case["hkv"] * case["dim"] * 2 * 2
    q = case["batch"] * gamma * case["hq"] * case["dim"] * 2
    return kv + 2 * q + q / case["dim"] * 2, 4.0 * case["dim"] * case["hq"] * gamma * keys


def work(case):
    """Bytes and floating-point operations of one pass that the path cannot do without:
    the cache's visible keys and values, every logits row that the rule reads, weights and
    outputs once; two operations a multiply-add of the contractions, four a logit."""
    kind = case["kind"]
    nbytes = flops = 0.0
    if kind in ("step", "attn", "tree"):
        gamma = case["nodes"] if kind == "tree" else case["gamma"]
        nbytes, flops = _attn_work(case, gamma)
    if kind in ("step", "accept"):
        rows = case["batch"] * case["gamma"]
        rows += (case["batch"] - _greedy_count(case)) * (case["gamma"] - 1)
    elif kind == "draft":
        rows = case["batch"] * case["gamma"]
    elif kind == "build":
        rows = case["batch"] * min(case["gamma"] - 1, case["nodes"] - 1)
    elif kind == "tree":
        rows = case["batch"] * case["nodes"]
    else:
        rows = 0
    if rows:
        nbytes += float(rows) * case["vocab"] * _esize(case)
        flops += 4.0 * rows * case["vocab"]
    if kind == "head":
        nbytes = 2.0 * case["hidden"] * (case["vocab"] + case["rows"]) + 20.0 * case["rows"]
        flops = 2.0 * case["rows"] * case["hidden"] * case["vocab"]
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------
DEV = "cuda"


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + stream)
    return g


def _temperatures(case):
    T = torch.full((case["batch"],), float(case["T"]))
    n = _greedy_count(case)
    if n:  # greedy requests spread over the batch
        T[torch.linspace(0, case["batch"] - 1, n).round().long()] = 0.0
    return T.to(DEV)


def _uniforms(g, *shape):
    """(0, 1], multiples of 2^-24."""
    return 1.0 - torch.rand(*shape, generator=g, device=DEV)


def _attn_inputs(case, gamma, seed):
    g, host = _gen(seed, 1), torch.Generator().manual_seed(int(seed) * 1009 + 2)
    B, P = case["batch"], case["page"]
    ctx = torch.randint(case["ctx_lo"], case["ctx_hi"] + 1, (B,), generator=host)
    kv_len = ctx + gamma
    pages = (kv_len + P - 1) // P
    total = int(pages.sum())
    perm = torch.randperm(total, generator=host).to(torch.int32)
    table = torch.full((B, int(pages.max())), -1, dtype=torch.int32)
    at = 0
    for b in range(B):
        n = int(pages[b])
        table[b, :n] = perm[at:at + n]
        at += n

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32).to(torch.bfloat16)

    return dict(q=normal(B, gamma, case["hq"], case["dim"]),
                k=normal(total, case["hkv"], P, case["dim"]), v=normal(total, case["hkv"], P, case["dim"]),
                table=table.to(DEV), kv_len=kv_len.to(torch.int32).to(DEV))


def _pick(rows, T, g, case):
    """One token of each row [n, gamma, vocab] at its sequence's temperature [n], among the
    row's top_k only where the proposal is filtered."""
    greedy = rows.argmax(-1)
    t = torch.where(T > 0, T, torch.ones_like(T)).view(-1, 1, 1)
    if case.get("top_k", 0) > 0:
        rows, ids = rows.topk(case["top_k"], dim=-1)
    e = torch.empty_like(rows).exponential_(generator=g).clamp_min_(1e-30)
    at = (rows / t - e.log_()).argmax(-1, keepdim=True)
    if case.get("top_k", 0) > 0:
        at = ids.gather(-1, at)
    return torch.where(T.view(-1, 1) > 0, at.squeeze(-1), greedy).to(torch.int32)


def _logit_inputs(case, seed):
    g = _gen(seed, 3)
    B, G, V = case["batch"], case["gamma"], case["vocab"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    T = _temperatures(case)
    draft = torch.empty(B, G, V, dtype=dt, device=DEV)
    verify = case["kind"] != "draft"
    target = torch.empty_like(draft) if verify else None
    tokens = torch.empty(B, G, dtype=torch.int32, device=DEV)
    for b in range(0, B, 8):
        n = min(8, B - b)
        t = torch.randn(n, G, V, generator=g, device=DEV).mul_(3.0)
        if verify:
            target[b:b + n] = t
            d = torch.empty_like(t)
            d[:, 0].normal_(0.0, 3.0, generator=g)
            if G > 1:
                d[:, 1:].normal_(0.0, case["noise"], generator=g).add_(t[:, :-1])
            draft[b:b + n] = d
            tokens[b:b + n] = _pick(draft[b:b + n].float(), T[b:b + n], g, case)
        else:
            draft[b:b + n] = t
    return dict(target=target, draft=draft, tokens=tokens, T=T, u=_uniforms(g, B, G))


def _build_inputs(case, seed):
    g = _gen(seed, 5)
    B, G, V = case["batch"], case["gamma"], case["vocab"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    draft = torch.randn(B, G, V, generator=g, device=DEV).mul_(3.0).to(dt)
    root = torch.randint(0, V, (B,), generator=g, device=DEV, dtype=torch.int32)
    return dict(draft=draft, T=torch.ones(B, device=DEV), root=root)


def _tree_inputs(case, seed):
    """Target rows and a tree over them: each node hangs below a random earlier one, its
    token one of its parent row's eight likeliest, no two siblings with the same."""
    g, host = _gen(seed, 6), torch.Generator().manual_seed(int(seed) * 1009 + 7)
    B, N, V = case["batch"], case["nodes"], case["vocab"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    target = torch.randn(B, N, V, generator=g, device=DEV).mul_(3.0).to(dt)
    top = target.float().topk(8, dim=-1).indices.cpu()
    roots = torch.randint(0, V, (B,), generator=host)
    tokens = torch.zeros(B, N, dtype=torch.int32)
    parents = torch.full((B, N), -1, dtype=torch.int32)
    mask = torch.ones(B, N, dtype=torch.int64)
    tokens[:, 0] = roots.to(torch.int32)
    for b in range(B):
        used, seen = [0] * N, [1] * N
        for c in range(1, N):
            tries = torch.randint(0, c, (64,), generator=host).tolist()
            p = next((x for x in tries if used[x] < 8), next(x for x in range(c) if used[x] < 8))
            parents[b, c] = p
            tokens[b, c] = top[b, p, used[p]]
            used[p] += 1
            seen[c] = seen[p] | (1 << c)
            mask[b, c] = seen[c] - (1 << 64) if seen[c] >> 63 else seen[c]
    return dict(target=target, tokens=tokens.to(DEV), parents=parents.to(DEV), mask=mask.to(DEV),
                T=_temperatures(case), u=_uniforms(g, B, N))


def _head_inputs(case, seed):
    g = _gen(seed, 8)
    R, H, V = case["rows"], case["hidden"], case["vocab"]
    h = torch.randn(R, H, generator=g, device=DEV).to(torch.bfloat16)
    w = torch.empty(V, H, dtype=torch.bfloat16, device=DEV).normal_(0.0, 3.0 / math.sqrt(H), generator=g)
    T = torch.ones((R + case["rows_per_seq"] - 1) // case["rows_per_seq"], device=DEV)
    tok = torch.randint(0, V, (R,), generator=g, device=DEV, dtype=torch.int32)
    return dict(h=h, w=w, T=T, tok=tok)


# ---------------------------------------------------------------------------------------
# What a decoding loop keeps, and one pass
# ---------------------------------------------------------------------------------------
def _attn_state(x, mask=None):
    out = torch.empty_like(x["q"])
    lse = torch.empty(x["q"].shape[:3], dtype=torch.float32, device=DEV)
    a = binding.attn_args(x["q"], x["k"], x["v"], x["table"], x["kv_len"], out, lse, tree_mask=mask)
    return a, dict(out=out, lse=lse)


def _ints(*shape):
    return torch.empty(*shape, dtype=torch.int32, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, keep=[], outputs={})
    if kind in ("step", "attn", "tree"):
        gamma = case["nodes"] if kind == "tree" else case["gamma"]
        x = _attn_inputs(case, gamma, seed)
        t = _tree_inputs(case, seed) if kind == "tree" else None
        s["attn"], outs = _attn_state(x, None if t is None else t["mask"])
        s["keep"] += [x, t]
        s["outputs"].update(outs)
        if kind != "step":
            s["attn_ws"] = binding.new_workspace(binding.workspace_size(attn=s["attn"]))
    if kind in ("step", "accept"):
        x = _logit_inputs(case, seed)
        B, G, _ = x["target"].shape
        o = dict(num_accepted=_ints(B), out_tokens=_ints(B, G + 1), num_emitted=_ints(B),
                 diag=torch.empty(B, G, 2, dtype=torch.float32, device=DEV))
        s["accept"] = binding.accept_args(x["target"], x["draft"], x["tokens"], x["T"], x["u"],
                                          o["num_accepted"], o["out_tokens"], o["num_emitted"], o["diag"])
        s["keep"].append(x)
        s["outputs"].update(o)
        s["filter"] = None
        if case.get("top_k", 0) > 0:
            f = (torch.full((B,), case["top_k"], dtype=torch.int32, device=DEV),
                 torch.full((B,), case["top_p"], dtype=torch.float32, device=DEV))
            s["keep"].append(f)
            s["filter"] = binding.filter_args(*f, B, max_top_k=case["top_k"])
            n = binding.filtered_workspace_size(s["accept"], s["filter"])
        else:
            n = binding.workspace_size(attn=s.get("attn"), accept=s["accept"])
        s["ws"] = binding.new_workspace(n)
    elif kind == "draft":
        x = _logit_inputs(case, seed)
        B, G, _ = x["draft"].shape
        o = dict(block_tokens=_ints(B, G), q_tok=torch.empty(B, G, dtype=torch.float32, device=DEV))
        s["draft"] = binding.draft_args(x["draft"], x["T"], x["u"], o["block_tokens"], o["q_tok"])
        s["filter"] = None
        if case["top_k"] > 0:
            f = (torch.full((B,), case["top_k"], dtype=torch.int32, device=DEV),
                 torch.full((B,), case["top_p"], dtype=torch.float32, device=DEV))
            s["keep"].append(f)
            s["filter"] = binding.filter_args(*f, B, max_top_k=case["top_k"])
        s["ws"] = binding.new_workspace(binding.draft_workspace_size(s["draft"], s["filter"]))
        s["keep"].append(x)
        s["outputs"].update(o)
    elif kind == "build":
        x = _build_inputs(case, seed)
        B, N = case["batch"], case["nodes"]
        o = dict(tokens=_ints(B, N), parents=_ints(B, N), depth=_ints(B, N),
                 mask=torch.empty(B, N, dtype=torch.int64, device=DEV))
        s["build"] = binding.tree_build_args(x["draft"], x["T"], x["root"], case["top_k"], o["tokens"],
                                             o["parents"], o["depth"], o["mask"])
        s["ws"] = binding.new_workspace(binding.tree_build_workspace_size(s["build"]))
        s["keep"].append(x)
        s["outputs"].update(o)
    elif kind == "tree":
        B, N = case["batch"], case["nodes"]
        o = dict(path=_ints(B, N), num_accepted=_ints(B), out_tokens=_ints(B, N + 1), num_emitted=_ints(B))
        s["tree"] = binding.tree_accept_args(t["target"], t["tokens"], t["parents"], o["path"],
                                             o["num_accepted"], o["out_tokens"], o["num_emitted"],
                                             t["T"], t["u"])
        s["ws"] = binding.new_workspace(binding.tree_workspace_size(s["tree"]))
        s["outputs"].update(o)
    elif kind == "head":
        x = _head_inputs(case, seed)
        R = case["rows"]
        o = dict(row_max=torch.empty(R, device=DEV), row_sum=torch.empty(R, device=DEV),
                 row_argmax=_ints(R), token_logit=torch.empty(R, device=DEV))
        s["head"] = binding.lm_head_args(x["h"], x["w"], x["T"], case["rows_per_seq"], o, x["tok"])
        s["ws"] = binding.new_workspace(binding.lm_head_workspace_size(s["head"]))
        s["keep"].append(x)
        s["outputs"].update(o)
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        binding.verify_step_args(s["attn"], s["accept"], s["ws"])
    elif kind == "attn":
        binding.verify_attention_args(s["attn"], s["attn_ws"])
    elif kind == "accept" and s["filter"] is None:
        binding.accept_block_args(s["accept"], s["ws"])
    elif kind == "accept":
        binding.accept_block_filtered_args(s["accept"], s["filter"], s["ws"])
    elif kind == "draft":
        binding.sample_block_args(s["draft"], s["filter"], s["ws"])
    elif kind == "build":
        binding.build_tree_args(s["build"], s["ws"])
    elif kind == "tree":
        binding.verify_attention_args(s["attn"], s["attn_ws"])
        binding.accept_tree_args(s["tree"], s["ws"])
    else:
        binding.lm_head_stats_args(s["head"], s["ws"])
    return s["outputs"]


# ---------------------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------------------
def _exact_attn(case, gamma, seed, mask=None):
    x = _attn_inputs(case, gamma, seed)
    B, G, Hq, D = x["q"].shape
    Hkv, P = case["hkv"], case["page"]
    out = torch.empty(B, G, Hq, D, dtype=torch.float64, device=DEV)
    lse = torch.empty(B, G, Hq, dtype=torch.float64, device=DEV)
    lens = x["kv_len"].tolist()
    for b in range(B):
        n = lens[b]
        pages = x["table"][b, :(n + P - 1) // P].long()
        rows = x["q"][b].double().view(G, Hkv, Hq // Hkv, D).permute(1, 0, 2, 3).reshape(Hkv, -1, D)
        at = torch.arange(n, device=DEV)
        if mask is None:
            seen = at.view(1, n) <= (n - G + torch.arange(G, device=DEV)).view(G, 1)
        else:
            bit = (at - (n - G)).clamp_min(0)
            seen = (at < n - G).view(1, n) | ((mask[b].view(G, 1) >> bit.view(1, n)) & 1).bool()
        seen = seen.repeat_interleave(Hq // Hkv, 0)
        for h in range(Hkv):
            k = x["k"][pages, h].reshape(-1, D)[:n].double()
            v = x["v"][pages, h].reshape(-1, D)[:n].double()
            sc = (rows[h] @ k.T / math.sqrt(D)).masked_fill_(~seen, -math.inf)
            l = sc.logsumexp(-1)
            o = (sc - l.view(-1, 1)).exp_() @ v
            at_h = slice(h * (Hq // Hkv), (h + 1) * (Hq // Hkv))
            out[b, :, at_h] = o.view(G, -1, D)
            lse[b, :, at_h] = l.view(G, -1)
    return dict(out=out, lse=lse)


def _exact_probs(rows, T, tok, top_k, top_p):
    """The probability of tok [n] under each of rows [n, vocab] at T, filtered where top_k > 0."""
    z = rows.double() / T
    if top_k <= 0:
        return (z.gather(-1, tok.view(-1, 1)).squeeze(-1) - z.logsumexp(-1)).exp()
    vals, ids = z.sort(dim=-1, descending=True, stable=True)
    vals, ids = vals[:, :top_k], ids[:, :top_k]
    p = vals.softmax(-1)
    p = p * ((p.cumsum(-1) - p) < top_p)
    p = p / p.sum(-1, keepdim=True)
    return (p * (ids == tok.view(-1, 1))).sum(-1)


def _exact_diag(case, seed):
    x = _logit_inputs(case, seed)
    B, G, _ = x["target"].shape
    diag = torch.full((B, G, 2), math.nan, dtype=torch.float64)
    diag[:, 0] = 0.0
    if G == 1:
        return diag
    temps, u, tok = x["T"].tolist(), x["u"].double().cpu(), x["tokens"].long()
    for b in range(B):
        drafts = tok[b, 1:]
        if temps[b] > 0:
            T = float(torch.tensor(temps[b], dtype=torch.float32))
            p = _exact_probs(x["target"][b, :-1], T, drafts, case.get("top_k", 0), case.get("top_p", 1.0)).cpu()
            q = _exact_probs(x["draft"][b, 1:], T, drafts, case.get("top_k", 0), case.get("top_p", 1.0)).cpu()
        else:
            p, q = (x["target"][b, :-1].float().argmax(-1) == drafts).double().cpu(), torch.ones(G - 1)
        for i in range(1, G):
            pi, qi = float(p[i - 1]), float(q[i - 1])
            diag[b, i, 0], diag[b, i, 1] = pi, qi
            reject = pi < 1 if temps[b] <= 0 else (pi <= 0 if qi <= 0 else float(u[b, i - 1]) > min(1.0, pi / qi))
            if reject:
                break
    return diag


def exact(case, seed):
    kind = case["kind"]
    r = {}
    if kind in ("step", "attn"):
        r.update(_exact_attn(case, case["gamma"], seed))
    elif kind == "tree":
        r.update(_exact_attn(case, case["nodes"], seed, _tree_inputs(case, seed)["mask"]))
    if kind in ("step", "accept"):
        r["diag"] = _exact_diag(case, seed)
    if kind == "head":
        x = _head_inputs(case, seed)
        h = x["h"].double()
        T = x["T"].double().repeat_interleave(case["rows_per_seq"])[:case["rows"], None]
        best = torch.full((case["rows"],), -math.inf, dtype=torch.float64, device=DEV)
        total = torch.zeros(case["rows"], dtype=torch.float64, device=DEV)
        tok = torch.empty_like(best)
        for v in range(0, case["vocab"], 16384):
            l = h @ x["w"][v:v + 16384].double().T
            new = torch.maximum(best, l.amax(-1))
            total = total * ((best - new) / T[:, 0]).exp() + ((l - new[:, None]) / T).exp_().sum(-1)
            best = new
            at = x["tok"].long() - v
            here = (at >= 0) & (at < l.shape[1])
            tok = torch.where(here, l.gather(1, at.clamp(0, l.shape[1] - 1)[:, None])[:, 0], tok)
        r.update(row_max=best, row_sum=total, token_logit=tok)
    if not r:
        return None
    names = {"step": ("num_accepted", "num_emitted", "out_tokens"), "accept": ("num_accepted", "num_emitted", "out_tokens"),
             "tree": ("path", "num_accepted", "num_emitted", "out_tokens"), "head": ("row_argmax",)}.get(kind, ())
    r.update({k: None for k in names})
    return r
