"""Performance cases of the verification step: what a decode loop asks of this
library, through the Python binding, over the sizes it is built for.

Kinds of case (field "kind"):
  step    one fused verification step (ppd_verify_step, or with typical=True
          ppd_verify_step_typical): the attention of every layer, top-1 tokens,
          acceptance and compaction in one call
  layers  the attention as a model's forward pass runs it, one
          ppd_tree_attention call per layer over that layer's own cache
  after   what follows a forward pass run that way: top-1 tokens (or softmax
          statistics), acceptance, compaction of every layer, the next tree
  next    the next step's candidate tree alone, from ensemble prompt tokens

Sizes: L layers, B sequences, H heads of D, cache prefix P (B > 1: ragged, P the
longest), cache capacity S, trees of T tokens, vocabulary V.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_18628_gb300 import ppd
from paper_2405_18628_gb300 import workloads as W

N_STATES, TOP_K, T_NEXT = 4, 10, 64           # next tree: states 0..3, guesses per depth, nodes
TEMPERATURE, EPSILON, DELTA = 0.7, 0.09, 0.3  # typical acceptance
MATCH_RATE = 0.6                              # share of guesses that copy the top-1 token


def case(name, kind, L, B, H, D, P, T, V, S=None, dtype="bf16", typical=False, n_ept=1, ept_mean="logits"):
    c = dict(kind=kind, L=L, B=B, H=H, D=D, P=P, T=T, V=V, S=S if S is not None else P + T,
             dtype=dtype, typical=typical, n_ept=n_ept, ept_mean=ept_mean)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call, a test-sized model: latency and launches are all there is
        case("tiny_step", "step", 1, 1, 4, 64, 128, 48, 1024),
        # a small draft-sized model's layers kept in fp32, an odd tree and prefix
        case("small_f32_layers", "layers", 2, 1, 16, 64, 1003, 37, 1024, S=1280, dtype="f32"),
        # one step of a 1.4B model, short context
        case("mobilellama_step", "step", 24, 1, 16, 128, 512, 64, 32000),
        # one step of a 7B model, the headline size
        case("vicuna7b_step", "step", 32, 1, 32, 128, 2048, 64, 32000),
        # the same model sampling at a temperature: an odd tree, a ragged last key tile
        case("vicuna7b_typical", "step", 32, 1, 32, 128, 1777, 53, 32000, S=4096, typical=True),
        # one step of a 13B model with a tree beyond 64 tokens
        case("vicuna13b_step", "step", 40, 1, 40, 128, 4096, 96, 32000),
        # the largest tree input length of the paper's tables on the 7B model
        case("vicuna7b_tree285", "step", 32, 1, 32, 128, 1500, 285, 32000, S=2048),
        # the 7B model's forward pass: 32 attention calls, one per layer
        case("vicuna7b_layers", "layers", 32, 1, 32, 128, 2048, 64, 32000),
        # what follows that forward pass
        case("vicuna7b_after", "after", 32, 1, 32, 128, 2048, 64, 32000),
        # four sequences whose candidates carry four ensemble chains of three prompt tokens
        case("next_tree_ept4", "next", 1, 4, 1, 64, 64, 208, 32000, n_ept=4),
        # a large batch of short chats on a narrow model: more sequences than one fused grid takes
        case("batch80_step", "step", 4, 80, 16, 64, 700, 32, 32000),
        # long contexts, eight ragged sequences, four of the 32 layers (the caches of all
        # would take 70 GB): the largest
        case("long_batch8_step", "step", 4, 8, 32, 128, 16384, 128, 32000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "layers", "layers", "after", "next"])
    typical = rng.random() < 0.3
    n_ept = 1
    D = rng.choice([64, 128, 128])
    H = rng.choice([4, 8, 16, 32, 40])
    V = rng.choice([1024, 32000, 32000, 32003, 50257, 128256])
    B = 1 if rng.random() < 0.6 else _log_int(rng, 2, 96)
    P = _log_int(rng, 16, 16384)
    T = _log_int(rng, 4, 512)
    dtype = "f32" if kind != "next" and rng.random() < 0.15 else "bf16"
    if kind == "next":
        # every candidate carries n_ept chains of N_STATES - 1 prompt tokens
        n_ept = rng.choice([1, 1, 2, 4, 8])
        per = 1 + n_ept * (N_STATES - 1)
        T = per * max(2, min(500 // per, T // per))
        B, P, H, D, L = min(B, 32), 64, 1, 64, 1
    if B * T > 4096:   # the logits of one step stay below 2.1 GB
        B = max(1, 4096 // T)
    if kind != "next":
        # time grows with the cache bytes and, past 128 tokens, with the blocks of queries
        eb = 2 if dtype == "bf16" else 6
        blocks = 1 if T <= 64 else 1.2 * ((T + 127) // 128)
        budget = 7.0e9 / (2.0 * eb * D * blocks)   # (layer, sequence, head, key) rows
        while B > 1 and B * H * (P + T) > budget:
            B //= 2
        L = _log_int(rng, 1, 40)
        L = max(1, min(L, int(budget / (B * H * (P + T)))))
    return case(None, kind, L, B, H, D, P, T, V, S=P + T + rng.choice([0, 0, 1, 63, 250]), dtype=dtype,
                typical=typical if kind in ("step", "after") else False, n_ept=n_ept,
                ept_mean=rng.choice(["logits", "probs"]) if n_ept > 1 else "logits")


def _lens(c):
    """Cached tokens of each sequence: P, or ragged between P / 2 and P."""
    return [c["P"] - (b * 7919) % (c["P"] // 2 + 1) for b in range(c["B"])]


def _trees(c, seed):
    """Parents and prompt-token flags [B][T] of trees shaped like the paper's."""
    T, n_ept = c["T"], c["n_ept"]
    if c["kind"] == "next":
        n_cand, chains = T // (1 + n_ept * (N_STATES - 1)), f"ept{n_ept}x{N_STATES - 1}"
    else:
        n_cand, chains = max(1, (T + 3) // 4), "fill3"
    w = W.Workload("case", L=1, B=1, H=1, D=64, P=0, T=T, V=1, n_cand=n_cand, max_depth=6,
                   chains=chains, match_rate=MATCH_RATE)
    rng = np.random.Generator(np.random.PCG64(seed))
    got = [W.make_tree(rng, w) for _ in range(c["B"])]
    return np.stack([p for p, _ in got]), np.stack([i for _, i in got]), rng


def prepare(case, seed):
    c, dev = case, torch.device("cuda")
    L, B, H, D, T, V, S = (c[k] for k in ("L", "B", "H", "D", "T", "V", "S"))
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 1000003 + 17)
    parent, is_prompt, rng = _trees(c, seed)
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.int32)).to(dev)  # noqa: E731
    s = dict(case=c, parent=i32(parent), prefix_len=i32(_lens(c)))
    new = lambda *shape: torch.empty(shape, dtype=torch.int32, device=dev)  # noqa: E731
    if c["kind"] != "next":
        dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
        n = lambda *shape: torch.randn(shape, dtype=dt, device=dev, generator=g)  # noqa: E731
        s.update(q=n(L, B, H, T, D), k_cache=n(L, B, H, S, D), v_cache=n(L, B, H, S, D),
                 k_tree=n(L, B, H, T, D), v_tree=n(L, B, H, T, D))
        ws_L = 1 if c["kind"] == "layers" else L
        s["workspace"] = ppd.workspace(ws_L, B, H, T, D, V, S, ppd.PPD_BF16 if c["dtype"] == "bf16" else ppd.PPD_F32)
    if c["kind"] in ("step", "layers"):
        s["out"] = torch.empty(L, B, H, T, D, dtype=torch.float32, device=dev)
        s["status"] = new(B)
    if c["kind"] == "layers":
        # one tensor per layer, as a model holds its caches
        s["lse"] = torch.empty(L, B, H, T, dtype=torch.float32, device=dev)
        s["status"] = new(L, B)
        s["calls"] = [tuple(s[k][l:l + 1] for k in ("q", "k_cache", "v_cache", "k_tree", "v_tree", "out", "lse")) +
                      (s["status"][l],) for l in range(L)]
        return s
    # logits as sharp as a language model's, guesses that copy the parent's top-1 token
    # or are drawn, prompt tokens marked by -1
    s["logits"] = torch.randn(B, T, V, device=dev, generator=g) * 2.5
    top = s["logits"].argmax(-1).cpu().numpy()
    cand = rng.integers(V, size=(B, T))
    hit = rng.random((B, T)) < MATCH_RATE
    hit[:, 0] = False
    cand = np.where(hit, np.take_along_axis(top, np.maximum(parent, 0), 1), cand)
    s["cand"] = i32(np.where(is_prompt, -1, cand))
    s.update(argmax=new(B, T), accept_len=new(B), path=new(B, T), next_token=new(B), new_len=new(B))
    if c["kind"] == "step":
        return s
    s["status"] = new(B)
    tp, tr = W.make_tree_templates(N_STATES, T_NEXT, TOP_K, rng, n_ept=c["n_ept"])
    s.update(tmpl_parent=i32(tp), tmpl_rank=i32(tr), next_parent=new(B, T_NEXT), next_cand=new(B, T_NEXT),
             next_state=new(B), next_status=new(B))
    s["next_ws"] = torch.empty(max(int(ppd.load().ppd_next_tree_workspace_bytes(B, N_STATES, TOP_K)), 256),
                               dtype=torch.uint8, device=dev)
    s["lse"], s["entropy"] = (torch.empty(B, T, dtype=torch.float32, device=dev) for _ in range(2))
    if c["kind"] == "next":
        # the accepted path of the step before, from plain torch
        acc = [_accept(parent[b], np.where(is_prompt[b], -1, cand[b]), top[b]) for b in range(B)]
        path = np.full((B, T), -1)
        for b, p in enumerate(acc):
            path[b, :len(p)] = p
        s["path"] = i32(path)
        s["accept_len"] = i32([len(p) for p in acc])
        s["next_token"] = i32([top[b, p[-1]] for b, p in enumerate(acc)])
    return s


def _next(s):
    ppd.ppd_next_tree(s["logits"], s["parent"], s["cand"], s["path"], s["accept_len"], s["next_token"],
                      s["tmpl_parent"], s["tmpl_rank"], TOP_K, s["next_parent"], s["next_cand"],
                      s["next_state"], s["next_status"], workspace=s["next_ws"], n_ept=s["case"]["n_ept"],
                      ept_mean=s["case"]["ept_mean"])


def run(state):
    s, kind, typical = state, state["case"]["kind"], state["case"]["typical"]
    if kind == "layers":
        for q, kc, vc, kt, vt, out, lse, status in s["calls"]:
            ppd.ppd_tree_attention(q, kc, vc, kt, vt, s["prefix_len"], s["parent"], out, status, lse=lse,
                                   workspace=s["workspace"])
        return {k: s[k] for k in ("out", "lse", "status")}
    if kind == "next":
        _next(s)
        return {k: s[k] for k in ("next_parent", "next_cand", "next_state", "next_status")}
    accepted = ("argmax", "accept_len", "path", "next_token", "new_len", "status", "k_cache", "v_cache")
    if kind == "step":
        head = (s["q"], s["k_cache"], s["v_cache"], s["k_tree"], s["v_tree"], s["prefix_len"], s["parent"],
                s["cand"], s["logits"])
        tail = (s["out"], s["argmax"], s["accept_len"], s["path"], s["next_token"], s["new_len"], s["status"],
                s["workspace"])
        if typical:
            ppd.ppd_verify_step_typical(*head, TEMPERATURE, EPSILON, DELTA, *tail)
        else:
            ppd.ppd_verify_step(*head, *tail)
        return {k: s[k] for k in ("out",) + accepted}
    res = (s["accept_len"], s["path"], s["next_token"], s["new_len"], s["status"])
    V, S = s["case"]["V"], s["case"]["S"]
    if typical:
        ppd.ppd_node_stats(s["logits"], TEMPERATURE, s["argmax"], s["lse"], s["entropy"], s["workspace"])
        ppd.ppd_typical_accept(s["logits"], s["lse"], s["entropy"], s["argmax"], s["cand"], s["parent"],
                               s["prefix_len"], S, TEMPERATURE, EPSILON, DELTA, *res)
    else:
        ppd.ppd_node_argmax(s["logits"], s["argmax"], s["workspace"])
        ppd.ppd_accept_path(s["argmax"], s["cand"], s["parent"], s["prefix_len"], V, S, *res)
    ppd.ppd_kv_compact(s["k_cache"], s["v_cache"], s["k_tree"], s["v_tree"], s["path"], s["accept_len"],
                       s["prefix_len"])
    _next(s)
    stats = ("lse", "entropy") if typical else ()
    return {k: s[k] for k in accepted + stats + ("next_parent", "next_cand", "next_state", "next_status")}


def work(case):
    """Each input read once, each output written once; of the cache the prefix
    rows, of the logits every row (next tree: the ranked rows alone)."""
    c = case
    L, B, H, D, T, V = (c[k] for k in ("L", "B", "H", "D", "T", "V"))
    eb = 2 if c["dtype"] == "bf16" else 4
    keys = L * H * sum(_lens(c))
    attn = 2 * keys * D * eb + L * B * H * T * D * (3 * eb + 4)
    # every query against its sequence's prefix and about six ancestors
    attn_flops = 4 * D * T * (keys + 6 * L * B * H)
    rows = 2 * 2 * L * B * H * D * eb * 2   # about two accepted rows of K and V, read and written
    if c["kind"] == "layers":
        return {"bytes": attn + 4 * L * B * H * T, "flops": attn_flops}
    if c["kind"] == "step":
        return {"bytes": attn + rows + 4 * B * T * V, "flops": attn_flops + B * T * V}
    ranked = B * (N_STATES - 1) * c["n_ept"]
    if c["kind"] == "next":
        return {"bytes": 4 * ranked * V + 16 * B * (T + T_NEXT), "flops": ranked * V}
    return {"bytes": 4 * B * T * V + rows + 16 * B * (T + T_NEXT), "flops": B * T * V}


def tolerance(case):
    # Attention outputs against 64 bits, measured: 4e-6 to 6e-6 up to 2048 keys (bf16
    # products, probabilities kept to about 2^-17), 1.1e-5 at 4096 and 2.4e-5 at 16384
    # (the rounding of the fp32 accumulation over the keys); four times that is stated.
    # Copied rows and whole numbers are exact, but a typical acceptance or a mean of
    # probabilities may fall the other way on a tie.
    t = {"rel": 2e-5 + 5e-9 * case["P"]}
    if case["typical"] or case["ept_mean"] == "probs":
        t["differ"] = 2e-3
    return t


# ------------------------------------------------------------------ 64-bit results

def _accept(parent, cand, top, passes=None):
    """The deepest root-to-node path of accepted candidates (lowest index on ties)."""
    depth = np.full(len(parent), -1)
    depth[0] = 0
    for i in range(1, len(parent)):
        p = parent[i]
        good = cand[i] == top[p] if passes is None else passes(i)
        if cand[i] >= 0 and depth[p] >= 0 and good:
            depth[i] = depth[p] + 1
    n, path = int(np.argmax(depth)), []
    while n >= 0:
        path.append(n)
        n = parent[n]
    return path[::-1]


def _attention(c, s, parent, lens):
    T, D = c["T"], c["D"]
    # fp32 operands are rounded to bf16 by contract
    f = lambda x: x.to(torch.bfloat16).double()  # noqa: E731
    out = torch.empty(s["q"].shape, dtype=torch.float64, device="cuda")
    lse = torch.empty(s["q"].shape[:-1], dtype=torch.float64, device="cuda")
    for b in range(c["B"]):
        see = np.eye(T, dtype=bool)
        for i in range(1, T):
            see[i] |= see[parent[b, i]]
        hide = torch.from_numpy(~see).to("cuda")
        for l in range(c["L"]):
            k = torch.cat([f(s["k_cache"][l, b, :, :lens[b]]), f(s["k_tree"][l, b])], 1)
            v = torch.cat([f(s["v_cache"][l, b, :, :lens[b]]), f(s["v_tree"][l, b])], 1)
            x = f(s["q"][l, b]) @ k.transpose(1, 2) / math.sqrt(D)
            x[:, :, lens[b]:].masked_fill_(hide, -math.inf)
            lse[l, b] = torch.logsumexp(x, -1)
            out[l, b] = torch.softmax(x, -1) @ v
    return out, lse


def exact(case, seed):
    c = case
    if c["kind"] == "next":
        return None   # whole numbers alone
    s, lens = prepare(c, seed), _lens(c)
    parent = s["parent"].cpu().numpy()
    r = {}
    if c["kind"] in ("step", "layers"):
        out, lse = _attention(c, s, parent, lens)
        r["out"] = out
        r["status"] = torch.zeros_like(s["status"])
        if c["kind"] == "layers":
            r["lse"] = lse
            return r
    cand = s["cand"].cpu().numpy()
    top = s["logits"].argmax(-1).cpu().numpy()
    B, T = cand.shape
    if c["typical"]:
        x = s["logits"].double() / TEMPERATURE
        logz = torch.logsumexp(x, -1)
        ent = torch.stack([-(torch.exp(x[b] - logz[b, :, None]) * (x[b] - logz[b, :, None])).sum(-1) for b in range(B)])
        if c["kind"] == "after":
            r["lse"], r["entropy"] = logz, ent
    r["path"] = torch.full((B, T), -1, dtype=torch.int32)
    r["accept_len"], r["next_token"], r["new_len"] = (torch.zeros(B, dtype=torch.int32) for _ in range(3))
    for b in range(B):
        passes = None
        if c["typical"]:
            at = torch.arange(1, T, device="cuda")
            pa, tk = s["parent"][b, at].long(), s["cand"][b, at].long().clamp(min=0)
            p = torch.exp(x[b, pa, tk] - logz[b, pa])
            fine = [False] + (p > torch.clamp(DELTA * torch.exp(-ent[b, pa]), max=EPSILON)).cpu().tolist()
            passes = fine.__getitem__
        path = _accept(parent[b], cand[b], top[b], passes)
        n, P = len(path), lens[b]
        r["path"][b, :n] = torch.tensor(path, dtype=torch.int32)
        r["accept_len"][b], r["next_token"][b], r["new_len"][b] = n, int(top[b, path[-1]]), P + n
        for cache, tree in (("k_cache", "k_tree"), ("v_cache", "v_tree")):
            s[cache][:, b, :, P:P + n] = s[tree][:, b][:, :, torch.tensor(path, device="cuda")]
    r["argmax"] = torch.from_numpy(top.astype(np.int32))
    r.update(k_cache=s["k_cache"], v_cache=s["v_cache"], status=torch.zeros_like(s["status"]))
    if c["kind"] == "after":
        r.update(next_parent=None, next_cand=None, next_state=None, next_status=None)
    return r
