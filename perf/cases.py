"""What a user of this library has it do, as measurable cases.

Three kinds of call, each through the Python binding:

``round``     one drafting round (``Drafter.draft``; ``Drafter.draft_from_host``
              where the serving loop keeps its inputs and outputs in pinned
              host memory; ``pctree_draft_noalloc`` where it may not hold a
              workspace).  One round is ``B`` dependent stages that each
              stream the whole head projection.
``attention`` one layer of the target's tree verification
              (``pctree_tree_attention``).
``verified``  what follows the target's forward: greedy acceptance
              (``pctree_accept``) and the accepted-row compaction of the KV
              caches and hidden states (``pctree_compact``).

The listed cases are the repository's own workloads; ``draw`` spreads over the
sizes around them: one request to a full serving batch, toy vocabularies to
Qwen3's, both head types and layouts, both child scorings, short and long
prefixes, ragged sizes.  Inputs are drawn on the GPU from the seed, with the
distributions of the repository's generators (peaked and flat Zipf-shaped
base logits, small-scale heads, normal Q/K/V, random breadth-first trees).
"""
import math
import random

import numpy as np
import torch

from paper_2608_02123_gb300 import pctree as P

V_QWEN3 = 151936
L2_BYTES = 126 << 20      # a head smaller than this stays in L2 between stages


def _round(name, V, H, B, k, N, batch, dtype="bf16", mode="parent",
           layout="tiled", temp="one", via="draft"):
    return {"name": name, "kind": "round", "V": V, "H": H, "B": B, "k": k, "N": N,
            "batch": batch, "dtype": dtype, "mode": mode, "layout": layout,
            "temp": temp, "via": via}


def _attention(name, batch, N, Hq, Hkv, B, prefix_max):
    return {"name": name, "kind": "attention", "batch": batch, "N": N, "Hq": Hq,
            "Hkv": Hkv, "B": B, "prefix_max": prefix_max}


def _verified(name, batch, N, B, layers, row_bytes, hidden_bytes, prefix_max):
    return {"name": name, "kind": "verified", "batch": batch, "N": N, "B": B,
            "layers": layers, "row_bytes": row_bytes, "hidden_bytes": hidden_bytes,
            "prefix_max": prefix_max}


def listed():
    return [
        # the smallest round: a toy f32 head, all launches and latency
        _round("round_tiny_f32", 1024, 64, 4, 4, 8, 1, dtype="f32", layout="rowmajor"),
        # an f32 head of a small model, a few requests at once
        _round("round_f32_bs4", 32000, 256, 7, 8, 32, 4, dtype="f32", layout="rowmajor"),
        # Qwen3-4B-shaped interactive decoding, short block, serving loop on
        # the host: pinned inputs in, tree back on the host
        _round("round_4b_b7_host", V_QWEN3, 2560, 7, 8, 32, 1, via="host"),
        # Qwen3-4B-shaped interactive decoding, long block (the headline)
        _round("round_4b_b16", V_QWEN3, 2560, 16, 8, 64, 1),
        # the same as a single chain (k = 1)
        _round("round_4b_b16_chain", V_QWEN3, 2560, 16, 1, 16, 1),
        # Qwen3-8B-shaped serving, 16 requests
        _round("round_8b_b7_bs16", V_QWEN3, 4096, 7, 8, 64, 16),
        # Qwen3-14B-shaped serving, 32 requests, wide trees: the largest
        _round("round_14b_b16_bs32", V_QWEN3, 5120, 16, 16, 128, 32, temp="mixed"),
        # one verification layer of the same three targets
        _attention("attention_4b_bs1", 1, 64, 32, 8, 16, 2048),
        _attention("attention_8b_bs16", 16, 64, 32, 8, 7, 1024),
        _attention("attention_14b_bs32", 32, 128, 40, 8, 16, 1024),
        # after verification: one request, and a full serving batch
        _verified("verified_4b_bs1", 1, 64, 16, 36, 2048, 5120, 2048),
        _verified("verified_14b_bs32", 32, 128, 16, 40, 2048, 10240, 1024),
    ]


def _log(rng, lo, hi):
    """An integer, uniform in the logarithm over [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["interactive", "interactive", "serving", "serving", "f32",
                       "attention", "attention", "verified"])
    if kind in ("interactive", "serving"):
        if kind == "interactive":           # at most 16 Markov rows a stage
            k = rng.randint(1, 16)
            batch = rng.randint(1, 16 // k)
        else:
            k = rng.randint(1, 16)
            batch = rng.randint(16 // k + 1, 32)
            if rng.random() < 0.1:
                k, batch = rng.randint(17, 32), rng.randint(1, 2)
        c = _round("", V=_log(rng, 1000, V_QWEN3), H=8 * _log(rng, 8, 640),
                   B=rng.randint(1, 16), k=k, N=_log(rng, 4, 256), batch=batch,
                   mode="shared" if rng.random() < 0.15 else "parent",
                   layout=rng.choice(["tiled", "tiled", "rowmajor"]),
                   temp=rng.choice(["one", "mixed"]))
        if kind == "interactive":
            c["via"] = rng.choice(["draft", "draft", "host", "noalloc"])
    elif kind == "f32":
        k = rng.randint(1, 8)
        c = _round("", V=_log(rng, 500, 65536), H=_log(rng, 32, 512),
                   B=rng.randint(1, 8), k=k, N=_log(rng, 4, 64), batch=rng.randint(1, 8),
                   dtype="f32", layout="rowmajor",
                   mode="shared" if rng.random() < 0.15 else "parent")
    elif kind == "attention":
        Hq, Hkv = rng.choice([(32, 8), (32, 8), (40, 8), (16, 8), (64, 8), (10, 2)])
        c = _attention("", batch=_log(rng, 1, 32), N=_log(rng, 4, 256), Hq=Hq, Hkv=Hkv,
                       B=rng.randint(2, 16), prefix_max=_log(rng, 32, 8192))
    else:
        c = _verified("", batch=_log(rng, 1, 32), N=_log(rng, 4, 256), B=rng.randint(2, 16),
                      layers=rng.randint(2, 40), row_bytes=16 * _log(rng, 4, 128),
                      hidden_bytes=16 * _log(rng, 16, 640), prefix_max=_log(rng, 32, 1024))
    del c["name"]
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFF)
    return g


def _round_inputs(c, seed):
    """Base logits [batch][B][V], head matrices [V][H] and root tokens."""
    V, H, B, R = c["V"], c["H"], c["B"], c["batch"]
    f32 = dict(dtype=torch.float32, device="cuda")
    g = _gen(seed, 1)
    L = torch.randn(R, B, V, generator=g, **f32).mul_(4.0)
    rank = torch.rand(R, B, V, generator=g, **f32).mul_(V).floor_().add_(1.0)
    L.sub_(rank.log_().mul_(1.1))               # Zipf(1.1) log-rank boost
    del rank
    if c["temp"] == "mixed":                    # flat and peaked depths
        flat = torch.rand(R, B, 1, generator=g, **f32) < 0.5
        L.div_(torch.where(flat, 2.0, 0.3))
    root = torch.randint(0, V, (R,), generator=g, device="cuda", dtype=torch.int32)
    g = _gen(seed, 2)
    if c["dtype"] == "f32":
        E = torch.randn(V, H, generator=g, **f32)
        W = torch.randn(V, H, generator=g, **f32).mul_(2.0 / math.sqrt(H))
    else:
        bf = dict(dtype=torch.bfloat16, device="cuda")
        E = torch.randn(V, H, generator=g, **bf).mul_(0.02)
        W = torch.randn(V, H, generator=g, **bf).mul_(0.02)
    return L, E, W, root


def _trees(batch, N, B, rng):
    """Random trees in breadth-first packed order, depth at most B: node
    counts [batch] and parents [batch][N] (-1: root and padding).  Request 0
    fills the budget."""
    n_nodes = np.zeros(batch, np.int32)
    parents = np.full((batch, N), -1, np.int32)
    for r in range(batch):
        n = N if r == 0 else rng.randint(max(1, N // 2), N)
        par, depth = [-1], [0]
        for i in range(1, n):
            while True:                          # shallow nodes are likelier
                p = int(i * rng.random() ** 2)
                if depth[p] < B:
                    break
            par.append(p)
            depth.append(depth[p] + 1)
        order = sorted(range(n), key=lambda i: (depth[i], i))
        pos = {old: new for new, old in enumerate(order)}
        n_nodes[r] = n
        for old in order[1:]:
            parents[r, pos[old]] = pos[par[old]]
    return n_nodes, parents


def _prefixes(batch, prefix_max, rng):
    pre = [rng.randint(0, prefix_max) for _ in range(batch)]
    pre[0] = prefix_max
    return np.asarray(pre, np.int32)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _prepare_round(c, seed):
    L, E, W, root = _round_inputs(c, seed)
    cfg = P.make_config(c["V"], c["H"], c["B"], c["k"], c["N"], c["batch"],
                        weight_dtype=c["dtype"], mode=c["mode"], head_layout=c["layout"])
    if c["layout"] == "tiled":                  # a serving process packs at load
        W = P.pack_head(cfg, W)
    if c["via"] == "host":
        L, root = L.cpu().pin_memory(), root.cpu().pin_memory()
    return {"cfg": cfg, "drafter": P.Drafter(cfg), "L": L, "E": E, "W": W, "root": root}


def _attention_inputs(c, seed):
    rng = random.Random(seed)
    R, N, Hq, Hkv = c["batch"], c["N"], c["Hq"], c["Hkv"]
    slots = c["prefix_max"] + N
    n_nodes, parent = _trees(R, N, c["B"], rng)
    prefix = _prefixes(R, c["prefix_max"], rng)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    g = _gen(seed, 3)
    q = torch.randn(R, N, Hq, 128, generator=g, **bf).mul_(1.5)
    k = torch.randn(R, slots, Hkv, 128, generator=g, **bf).mul_(1.5)
    v = torch.randn(R, slots, Hkv, 128, generator=g, **bf)
    return q, k, v, prefix, n_nodes, parent


def _prepare_attention(c, seed):
    q, k, v, prefix, n_nodes, parent = _attention_inputs(c, seed)
    cfg = P.attn_config(c["batch"], c["N"], c["Hq"], c["Hkv"], c["prefix_max"] + c["N"])
    nb = P.pctree_tree_attention_workspace_bytes(cfg)
    return {"cfg": cfg, "q": q, "k": k, "v": v, "prefix": _dev(prefix),
            "n_nodes": _dev(n_nodes), "parent": _dev(parent), "out": torch.empty_like(q),
            "ws": torch.empty(nb, dtype=torch.uint8, device="cuda") if nb else None,
            "status": torch.zeros(1, dtype=torch.int32, device="cuda")}


def _prepare_verified(c, seed):
    rng = random.Random(seed)
    R, N, B = c["batch"], c["N"], c["B"]
    n_nodes, parent = _trees(R, N, B, rng)
    prefix = _prefixes(R, c["prefix_max"], rng)
    # distinct tokens; after each node the target wants one of its children's
    # tokens with probability 0.85, else a token no child has
    tokens = np.stack([np.asarray(rng.sample(range(V_QWEN3), N), np.int32) for _ in range(R)])
    target = np.full((R, N), V_QWEN3, np.int32)
    for r in range(R):
        for i in range(int(n_nodes[r])):
            kids = np.flatnonzero(parent[r] == i)
            if len(kids) and rng.random() < 0.85:
                target[r, i] = tokens[r, rng.choice(kids.tolist())]
    slots = c["prefix_max"] + N
    u8 = dict(dtype=torch.uint8, device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")
    g = _gen(seed, 4)
    cache = torch.randint(0, 256, (c["layers"], 2, R, slots, c["row_bytes"]), generator=g, **u8)
    hidden = torch.randint(0, 256, (R, N, c["hidden_bytes"]), generator=g, **u8)
    cfg = P.make_config(V_QWEN3, 64, B, 1, N, R)
    tree = P.alloc_tree(cfg, "cuda")
    tree.n_nodes.copy_(_dev(n_nodes))
    tree.tokens.copy_(_dev(tokens))
    tree.parent.copy_(_dev(parent))
    return {"cfg": cfg, "tree": tree, "target": _dev(target), "prefix": _dev(prefix),
            "layout": P.compact_layout(R, B, N, c["layers"], 2, slots, c["row_bytes"],
                                       c["hidden_bytes"]),
            "idx": torch.empty(R, B + 1, **i32), "len": torch.empty(R, **i32),
            "bonus": torch.empty(R, **i32), "cache": cache, "hidden": hidden,
            "hidden_out": torch.zeros(R, B + 1, c["hidden_bytes"], **u8),
            "status": torch.zeros(1, **i32)}


def prepare(case, seed):
    s = {"round": _prepare_round, "attention": _prepare_attention,
         "verified": _prepare_verified}[case["kind"]](case, seed)
    s["kind"], s["via"] = case["kind"], case.get("via")
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

TREE = ("n_nodes", "tokens", "parent", "depth", "logp", "position_ids", "mask",
        "retrieve", "n_leaves", "status")


def run(s):
    if s["kind"] == "round":
        d = s["drafter"]
        if s["via"] == "host":
            return d.draft_from_host(s["L"], s["root"], s["E"], s["W"])
        if s["via"] == "noalloc":
            P.pctree_draft_noalloc(s["cfg"], s["L"], s["E"], s["W"], s["root"], d.tree)
            tree = d.tree
        else:
            tree = d.draft(s["L"], s["E"], s["W"], s["root"])
        return {f: getattr(tree, f) for f in TREE}
    if s["kind"] == "attention":
        P.pctree_tree_attention(s["cfg"], s["q"], s["k"], s["v"], s["prefix"], s["n_nodes"],
                                s["parent"], s["out"], s["ws"], s["status"])
        return {"out": s["out"], "status": s["status"]}
    P.pctree_accept(s["cfg"], s["tree"], s["target"], s["idx"], s["len"], s["bonus"])
    P.pctree_compact(s["layout"], s["idx"], s["len"], s["prefix"], s["cache"], s["hidden"],
                     s["hidden_out"], s["status"])
    return {"idx": s["idx"], "len": s["len"], "bonus": s["bonus"], "cache": s["cache"],
            "hidden": s["hidden_out"], "status": s["status"]}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _rows(c, d):
    return c["batch"] * (1 if d == 0 or c["mode"] == "shared" else c["k"])


def work(case):
    c = case
    R, N, B = c["batch"], c["N"], c["B"]
    if c["kind"] == "round":
        el = 2 if c["dtype"] == "bf16" else 4
        head = c["V"] * c["H"] * el
        rows = sum(_rows(c, d) for d in range(B))
        # the stages depend on one another, so a head larger than L2 comes
        # from HBM once a stage
        byts = (head * (B if head > L2_BYTES else 1) + R * B * c["V"] * 4 +
                rows * c["H"] * el + R * (N * 20 + N * N + N * (B + 1) * 4))
        return {"bytes": byts, "flops": 2.0 * c["V"] * c["H"] * rows}
    # request sizes vary with the seed: their expectations
    nodes = N + (R - 1) * (max(1, N // 2) + N) / 2.0
    prefix = c["prefix_max"] * (1 + (R - 1) / 2.0)
    if c["kind"] == "attention":
        n_mean, p_mean, depth = nodes / R, prefix / R, min(B, N) / 2.0
        return {"bytes": 4.0 * 128 * c["Hkv"] * (prefix + nodes) + 2 * 2.0 * 128 * c["Hq"] * R * N,
                "flops": 4.0 * 128 * c["Hq"] * R * n_mean * (p_mean + depth + 1)}
    moved = R * 3.0                              # accepted nodes, about
    return {"bytes": 2 * moved * (2.0 * c["layers"] * c["row_bytes"] + c["hidden_bytes"]) +
            R * N * 12, "flops": 0}


def tolerance(case):
    if case["kind"] == "round":
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.005}
    if case["kind"] == "attention":
        return {"rel": 1e-2, "max": 0.1}
    return "exact"


# --------------------------------------------------------------------------
# the same results in 64 bits
# --------------------------------------------------------------------------

def _project(W, X, V):
    """X W^T in 64 bits, a slice of W at a time."""
    out = torch.empty(X.shape[0], V, dtype=torch.float64, device="cuda")
    Xt = X.double().t().contiguous()
    for v in range(0, V, 16384):
        out[:, v:v + 16384] = (W[v:v + 16384].double() @ Xt).t()
    return out


def _exact_round(c, seed):
    if 2.0 * c["V"] * c["H"] * sum(_rows(c, d) for d in range(c["B"])) > 1.4e13:
        return None
    L, E, W, root = _round_inputs(c, seed)
    R, B, k, N, V = c["batch"], c["B"], c["k"], c["N"], c["V"]
    pool = [[(int(t), -1, 0.0, 0)] for t in root.tolist()]      # token, parent, score, level
    front = [[0] for _ in range(R)]
    chain = root.tolist()
    for d in range(B):
        if c["mode"] == "shared":
            par = [[chain[r]] for r in range(R)]
        else:
            par = [[pool[r][i][0] for i in front[r]] for r in range(R)]
        per = len(par[0])
        X = E[torch.tensor([t for p in par for t in p], device="cuda")]
        z = _project(W, X, V).view(R, per, V)
        z += L[:, d].double().unsqueeze(1)
        best, tok = z.topk(k, dim=2)
        lp = (best - torch.logsumexp(z, 2, keepdim=True)).cpu().numpy()
        tok = tok.cpu().numpy()
        del z
        for r in range(R):
            base = len(pool[r])
            for j, i in enumerate(front[r]):
                jj = 0 if c["mode"] == "shared" else j
                s = pool[r][i][2]
                pool[r] += [(int(tok[r, jj, m]), i, s + float(lp[r, jj, m]), d + 1)
                            for m in range(k)]
            chain[r] = int(tok[r, 0, 0])
            layer = sorted(range(base, len(pool[r])), key=lambda i: (-pool[r][i][2], i))
            front[r] = layer[:k]
    logp = np.full((R, N), -np.inf)
    for r in range(R):
        p = pool[r]
        keep = sorted(range(len(p)), key=lambda i: (-p[i][2], i))[:N]
        place, at = {}, 0
        for lvl in range(B + 1):                 # breadth first
            ids = [i for i in keep if p[i][3] == lvl]
            ids.sort(key=lambda i: (place.get(p[i][1], -1), p[i][0]))
            for i in ids:
                place[i] = at
                logp[r, at] = p[i][2]
                at += 1
    return {f: (torch.from_numpy(logp) if f == "logp" else None) for f in TREE}


def _exact_attention(c, seed):
    q, k, v, prefix, n_nodes, parent = _attention_inputs(c, seed)
    G = c["Hq"] // c["Hkv"]
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    for r in range(c["batch"]):
        T, n = int(prefix[r]), int(n_nodes[r])
        see = np.zeros((n, T + n), bool)
        see[:, :T] = True
        for i in range(n):
            x = i
            while x >= 0:
                see[i, T + x] = True
                x = int(parent[r, x])
        hide = _dev(~see)
        for h in range(c["Hkv"]):
            qh = q[r, :n, h * G:(h + 1) * G].double().transpose(0, 1)       # [G][n][128]
            sc = (qh @ k[r, :T + n, h].double().t()) * 128 ** -0.5
            p = sc.masked_fill(hide, -math.inf).softmax(-1)
            out[r, :n, h * G:(h + 1) * G] = (p @ v[r, :T + n, h].double()).transpose(0, 1)
    return {"out": out, "status": None}


def exact(case, seed):
    if case["kind"] == "round":
        return _exact_round(case, seed)
    if case["kind"] == "attention":
        return _exact_attention(case, seed)
    return None
