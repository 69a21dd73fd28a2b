"""The cases that this library's speed is measured on.

Every case is one call of a program that decodes (or trains a draft) with the
library: a draft step's cross-attention, the target's verification of the tree,
the acceptance, the sampled acceptance, the training-time block mask, and whole
speculative rounds.  Shapes are those of the evaluation workloads and of the
bench (Vicuna-7B/13B/33B and Mistral-7B layers, vocabulary 32000); ``draw``
spreads over the same ranges.  Inputs are random numbers made on the GPU from
the seed; the K/V caches, the workspaces and the output buffers are kept by the
program between calls, as a decoding loop keeps them.
"""
import math
import random

import torch

from paper_2402_02082_gb300 import binding as g

CAPE_CAP = 32   # tokens a CaPE round verifies at most (the tree then has 33 node slots)
KV_BYTES_MOST = 4 * 52 * 16384 * 128 * 2 * 2
PAIRS_MOST = 4 * 32 * 2048 * 2048 * 128


def listed():
    attn = dict(D=128, dtype="bf16", len_seed=0)
    return [
        # one draft step of a single user's Vicuna-7B decode: the smallest call, all launch and latency
        dict(attn, name="cross-7b-b1", kind="cross", B=1, H=32, H_kv=32, kv_min=2048, kv_max=2048),
        # the same step with Vicuna-33B heads, four long contexts: the largest, all HBM
        dict(attn, name="cross-33b-long", kind="cross", B=4, H=52, H_kv=52, kv_min=16384, kv_max=16384),
        # a draft step over a grouped-query target (Mistral-7B: 32 query over 8 cached heads)
        dict(attn, name="cross-mistral-gqa", kind="cross", B=4, H=32, H_kv=8, kv_min=16384, kv_max=16384),
        # verification of a plain gamma = 5 proposal, single user
        dict(attn, name="verify-7b-chain", kind="verify", B=1, H=32, H_kv=32, kv_min=2048, kv_max=2048, n=6,
             depth=5, branch=1),
        # verification in a served batch of ragged contexts, odd lengths
        dict(attn, name="verify-13b-ragged", kind="verify", B=8, H=40, H_kv=40, kv_min=512, kv_max=4096, n=26,
             depth=5, branch=4, len_seed=3),
        # verification of 64-node trees over long contexts
        dict(attn, name="verify-33b-long", kind="verify", B=4, H=52, H_kv=52, kv_min=16384, kv_max=16384, n=64,
             depth=6, branch=6),
        # verification of CaPE-sized trees (32 tokens and the root) on a grouped-query target
        dict(attn, name="verify-mistral-cape", kind="verify", B=4, H=32, H_kv=8, kv_min=16384, kv_max=16384, n=33,
             depth=5, branch=4),
        # greedy acceptance of those trees: the target's logits of every node are read once
        dict(name="accept-33b", kind="accept", B=4, n=64, V=32000, depth=6, branch=6, std=1.0, p_accept=0.6),
        # speculative-sampling acceptance of a gamma = 5 proposal
        dict(name="sample-b4", kind="sample", B=4, gamma=5, V=32000),
        # the draft's training-time cross-attention under the block mask (Vicuna-7B, 2048 positions)
        dict(name="block-7b-train", kind="block", B=4, T=2048, H=32, H_kv=32, D=128, L=5, len_min=2048, len_seed=0),
        # a whole GliDe-with-CaPE round of a single user on one Vicuna-7B layer: the draft steps, the
        # expansion, the verification of its tree, the acceptance and the cache update
        dict(attn, name="round-7b-cape", kind="round", B=1, H=32, H_kv=32, kv_min=2048, kv_max=2048, gamma=5,
             V=32000),
        # the tiny fp32 workload's round: one draft step, a five-node chain, its acceptance
        dict(name="round-tiny-f32", kind="tiny", B=1, H=4, H_kv=4, D=64, dtype="f32", kv_min=128, kv_max=128,
             len_seed=0, n=5, depth=4, branch=1, V=1000, std=2.0, p_accept=0.7),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["cross", "cross", "verify", "verify", "verify", "accept", "sample", "block", "round", "tiny"])
    if kind == "accept":
        n = _log_int(rng, 1, 64)
        return dict(kind=kind, B=_log_int(rng, 1, 256 // n if n > 16 else 16), n=n,
                    V=rng.choice([32000, 32000, 32001, _log_int(rng, 1000, 50257)]), depth=6, branch=6, std=1.0,
                    p_accept=round(rng.uniform(0.3, 0.9), 2))
    if kind == "sample":
        return dict(kind=kind, B=_log_int(rng, 1, 16), gamma=rng.randint(1, 8),
                    V=rng.choice([32000, 32000, 32001, _log_int(rng, 1000, 50257)]))
    if kind == "block":
        H, H_kv = rng.choice([(32, 32), (40, 40), (32, 8)])
        c = dict(kind=kind, B=_log_int(rng, 1, 8), T=_log_int(rng, 100, 4096), H=H, H_kv=H_kv,
                 D=rng.choice([128, 128, 64]), L=rng.randint(1, 8), len_seed=rng.randrange(1000))
        while c["B"] > 1 and c["B"] * H * c["T"] ** 2 * c["D"] > PAIRS_MOST:
            c["B"] -= 1
        while H * c["T"] ** 2 * c["D"] > PAIRS_MOST:
            c["T"] = c["T"] * 3 // 4
        c["len_min"] = rng.choice([c["T"], max(1, c["T"] // 2)])
        return c
    H, H_kv = rng.choice([(32, 32), (40, 40), (52, 52), (32, 32), (32, 8), (32, 8), (8, 8), (24, 8)])
    kv = _log_int(rng, 128, 16384)
    c = dict(kind=kind, B=_log_int(rng, 1, 8), H=H, H_kv=H_kv, D=rng.choice([128, 128, 128, 64]), dtype="bf16",
             kv_max=kv, kv_min=rng.choice([kv, max(1, kv // 8)]), len_seed=rng.randrange(1000))
    if kind == "tiny":  # fp32 is what small checks and comparisons run in
        c.update(B=rng.randint(1, 2), H=4, H_kv=rng.choice([4, 4, 2]), D=rng.choice([64, 128]), dtype="f32",
                 kv_max=_log_int(rng, 64, 1024), V=rng.choice([1000, 4097]), std=2.0, p_accept=0.7)
        c["kv_min"] = c["kv_max"]
    while c["B"] > 1 and c["B"] * H_kv * kv * c["D"] * 4 > KV_BYTES_MOST:
        c["B"] -= 1
    if kind in ("verify", "tiny"):
        n = min(_log_int(rng, 1, 64), 256 * H_kv // H, 16 if kind == "tiny" else 64)
        c.update(n=n, **(dict(depth=64, branch=1) if n <= 8 else dict(depth=6, branch=6)))
    if kind == "round":
        c.update(B=min(c["B"], 4), gamma=rng.randint(2, 6), V=32000)
        while c["B"] * H_kv * c["kv_max"] * c["D"] * 4 * (c["gamma"] + 1) > KV_BYTES_MOST:
            c["kv_max"] = c["kv_max"] * 3 // 4
        c["kv_min"] = min(c["kv_min"], c["kv_max"])
    return c


# ------------------------------------------------------------------ inputs
def _lengths(c, lo="kv_min", hi="kv_max"):
    """Lengths of the batch's sequences: part of the case, so that its work is known without the inputs."""
    r = random.Random(c["len_seed"])
    return [r.randint(c[lo], c[hi]) for _ in range(c["B"])]


def _tree(r, n, depth, branch):
    """Parents of a random tree of n nodes: each node a child of an earlier one with room."""
    parent, level, kids = [-1], [0], [0] * n
    for i in range(1, n):
        p = r.choice([j for j in range(i) if level[j] < depth and kids[j] < branch])
        kids[p] += 1
        parent.append(p)
        level.append(level[p] + 1)
    return parent


def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(seed * 1009 + k)


def _normal(seed, k, shape, dtype):
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    return torch.randn(shape, generator=_gen(seed, k), device="cuda", dtype=t)


def _i32(v):
    return torch.tensor(v, dtype=torch.int32, device="cuda")


def _kv_inputs(c, seed, extra):
    lens = _lengths(c)
    cap = (c["kv_max"] + extra + 15) // 16 * 16
    shape = (c["B"], c["H_kv"], cap, c["D"])
    return dict(K=_normal(seed, 1, shape, c["dtype"]), V=_normal(seed, 2, shape, c["dtype"]), kv_len=_i32(lens),
                lens=lens, kv_max=c["kv_max"])


def _cross_inputs(c, seed):
    s = _kv_inputs(c, seed, 64)
    s["q"] = _normal(seed, 3, (c["B"], 1, c["H"], c["D"]), c["dtype"])
    return s


def _trees(c, seed):
    r = random.Random(seed * 31 + 7)
    return [_tree(r, c["n"], c["depth"], c["branch"]) for _ in range(c["B"])]


def _verify_inputs(c, seed):
    s = _kv_inputs(c, seed, 64)
    s["q"] = _normal(seed, 3, (c["B"], c["n"], c["H"], c["D"]), c["dtype"])
    s["parents"] = _trees(c, seed)
    s["parent"] = _i32(s["parents"])
    return s


def _accept_inputs(c, seed):
    """Logits N(0, std); at each node with children the row's maximum is one child's token with
    probability p_accept, another token otherwise."""
    r = random.Random(seed * 37 + 5)
    parents, tokens, where = _trees(c, seed), [], []
    for b, parent in enumerate(parents):
        tok = r.sample(range(c["V"]), c["n"])
        tokens.append(tok)
        for p in range(c["n"]):
            kids = [k for k in range(c["n"]) if parent[k] == p]
            if kids:
                top = tok[r.choice(kids)] if r.random() < c["p_accept"] else r.randrange(c["V"])
                where.append((b, p, top))
    logits = _normal(seed, 4, (c["B"], c["n"], c["V"]), "f32").mul_(c["std"])
    if where:
        b, p, t = (torch.tensor(x, device="cuda") for x in zip(*where))
        logits[b, p, t] = logits.amax(-1)[b, p] + 1.0
    return dict(tokens=_i32(tokens), parent=_i32(parents), logits=logits)


def _distributions(seed, k, B, rows, V):
    """fp32 distributions [B, rows, V] as a language model gives them: a most probable token whose
    probability is uniform on [0.05, 0.98], and a tail of a few runners-up and many small values."""
    gen = _gen(seed, k)
    p = torch.softmax(torch.randn((B, rows, V), generator=gen, device="cuda") * 2.5, -1)
    top = torch.randint(V, (B, rows, 1), generator=gen, device="cuda")
    conf = torch.rand((B, rows, 1), generator=gen, device="cuda") * 0.93 + 0.05
    p.scatter_(2, top, 0.0)
    p = torch.minimum(p * ((1.0 - conf) / p.sum(-1, keepdim=True)), conf * 0.99)
    return p.scatter_(2, top, conf).contiguous()


def _sample_inputs(c, seed):
    """A draft's distributions, its own samples of them, and target logits whose distributions
    lie between the draft's and independent ones."""
    B, n, V = c["B"], c["gamma"], c["V"]
    probs = _distributions(seed, 5, B, n, V)
    other = _distributions(seed, 6, B, n + 1, V)
    tokens = torch.multinomial(probs.view(B * n, V), 1, generator=_gen(seed, 7)).view(B, n).to(torch.int32)
    mixed = torch.cat([0.6 * probs + 0.4 * other[:, :n], other[:, n:]], 1)
    u = torch.rand((B, n + 1), generator=_gen(seed, 8), device="cuda")
    return dict(tokens=tokens, probs=probs, logits=mixed.clamp_min(1e-30).log_().contiguous(), u=u)


def _block_inputs(c, seed):
    shape = (c["B"], c["H_kv"], c["T"], c["D"])
    lens = _lengths(c, "len_min", "T")
    return dict(K=_normal(seed, 1, shape, "bf16"), V=_normal(seed, 2, shape, "bf16"), lens=lens, seq_len=_i32(lens),
                q=_normal(seed, 3, (c["B"], c["T"], c["H"], c["D"]), "bf16"))


def _round_inputs(c, seed):
    """The target agrees with the draft up to the last proposal token and takes a sibling there."""
    B, n = c["B"], 1 + CAPE_CAP
    s = _kv_inputs(c, seed, n)
    s["q_draft"] = [_normal(seed, 20 + i, (B, 1, c["H"], c["D"]), c["dtype"]) for i in range(c["gamma"])]
    s["q"] = _normal(seed, 3, (B, n, c["H"], c["D"]), c["dtype"])
    s["probs"] = _distributions(seed, 5, B, c["gamma"], c["V"])
    s["root"] = torch.randint(c["V"], (B,), generator=_gen(seed, 9), device="cuda").to(torch.int32)
    best = torch.topk(s["probs"], 2, dim=-1).indices  # [B, gamma, 2]
    logits = _normal(seed, 4, (B, n, c["V"]), "f32")
    top = logits.amax(-1) + 1.0
    for i in range(c["gamma"]):
        token = best[:, i, 1 if i == c["gamma"] - 1 else 0]
        logits[:, i].scatter_(1, token[:, None], top[:, i:i + 1])
    s["logits"] = logits
    return s


_INPUTS = dict(cross=_cross_inputs, verify=_verify_inputs, accept=_accept_inputs, sample=_sample_inputs,
               block=_block_inputs, round=_round_inputs)


def _inputs(c, seed):
    if c["kind"] == "tiny":
        s = _verify_inputs(c, seed)
        s.update(_accept_inputs(c, seed))
        s["q_draft"] = _normal(seed, 20, (c["B"], 1, c["H"], c["D"]), c["dtype"])
        return s
    return _INPUTS[c["kind"]](c, seed)


# ----------------------------------------------------------- state and pass
def _attn_workspace(s, H, n):
    B, H_kv, cap, D = s["K"].shape
    code = g.GLIDE_BF16 if s["K"].dtype == torch.bfloat16 else g.GLIDE_F32
    size = g.glide_attn_workspace_bytes(g.make_desc(B, H, D, cap, code, H_kv=H_kv), n)
    return torch.zeros(size, dtype=torch.uint8, device="cuda")


def _out(like):
    return torch.empty(like.shape, dtype=torch.float32, device="cuda")


def _accept_buffers(B, n):
    i32 = dict(dtype=torch.int32, device="cuda")
    return dict(path=torch.empty((B, n), **i32), length=torch.empty(B, **i32), bonus=torch.empty(B, **i32),
                ws_accept=torch.zeros(g.glide_accept_workspace_bytes(B, n), dtype=torch.uint8, device="cuda"))


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = _inputs(c, seed)
    s["kind"] = kind
    B = c["B"]
    i32 = dict(dtype=torch.int32, device="cuda")
    if kind in ("cross", "verify", "tiny"):
        s["ws"] = _attn_workspace(s, c["H"], c.get("n", 1))
        s["out"] = _out(s["q"])
    if kind == "tiny":
        s["out_draft"] = _out(s["q_draft"])
    if kind in ("accept", "tiny"):
        s.update(_accept_buffers(B, c["n"]))
    if kind == "sample":
        s["ws"] = torch.zeros(g.glide_sample_workspace_bytes(B, c["gamma"]), dtype=torch.uint8, device="cuda")
        s["n_acc"], s["next"] = torch.empty(B, **i32), torch.empty(B, **i32)
    if kind == "block":
        desc = g.make_desc(B, c["H"], c["D"], c["T"], g.GLIDE_BF16, H_kv=c["H_kv"])
        s["ws"] = torch.zeros(g.glide_block_attn_workspace_bytes(desc, c["T"]), dtype=torch.uint8, device="cuda")
        s["out"], s["L"] = _out(s["q"]), c["L"]
    if kind == "round":
        n = 1 + CAPE_CAP
        s.update(_accept_buffers(B, n))
        s["ws"] = _attn_workspace(s, c["H"], n)
        s["ws_cape"] = torch.zeros(g.glide_cape_workspace_bytes(B, c["gamma"], c["V"]), dtype=torch.uint8,
                                   device="cuda")
        s["out"], s["out_draft"] = _out(s["q"]), [_out(q) for q in s["q_draft"]]
        s["tokens"], s["parent"] = torch.empty((B, n), **i32), torch.empty((B, n), **i32)
        s["n_nodes"], s["new_len"] = torch.empty(B, **i32), torch.empty(B, **i32)
        s["conf"] = torch.empty((B, c["gamma"]), dtype=torch.float32, device="cuda")
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "cross":
        return g.glide_cross_attn(s["q"], s["K"], s["V"], s["kv_len"], s["kv_max"], s["out"], s["ws"])
    if kind == "verify":
        return g.tree_verify_attn(s["q"], s["parent"], s["K"], s["V"], s["kv_len"], s["kv_max"], s["out"], s["ws"])
    if kind == "accept":
        return g.tree_accept(s["tokens"], s["parent"], s["logits"], s["path"], s["length"], s["bonus"],
                             s["ws_accept"])
    if kind == "sample":
        return g.spec_sample_accept(s["tokens"], s["probs"], s["logits"], s["u"], s["n_acc"], s["next"], s["ws"])
    if kind == "block":
        return g.glide_block_cross_attn(s["q"], s["K"], s["V"], s["seq_len"], s["L"], s["out"], s["ws"])
    if kind == "tiny":
        g.glide_cross_attn(s["q_draft"], s["K"], s["V"], s["kv_len"], s["kv_max"], s["out_draft"], s["ws"])
        g.tree_verify_attn(s["q"], s["parent"], s["K"], s["V"], s["kv_len"], s["kv_max"], s["out"], s["ws"])
        g.tree_accept(s["tokens"], s["parent"], s["logits"], s["path"], s["length"], s["bonus"], s["ws_accept"])
        return dict(draft=s["out_draft"], tree=s["out"], path=s["path"], length=s["length"], bonus=s["bonus"])
    # a whole round; the cache update of a CaPE tree moves one row over the last proposal token's,
    # so passes after the first start from the same cache as one another
    for q, out in zip(s["q_draft"], s["out_draft"]):
        g.glide_cross_attn(q, s["K"], s["V"], s["kv_len"], s["kv_max"], out, s["ws"])
    g.cape_expand(s["probs"], s["root"], CAPE_CAP, s["tokens"], s["parent"], s["n_nodes"], s["ws_cape"],
                  conf=s["conf"])
    g.tree_verify_attn(s["q"], s["parent"], s["K"], s["V"], s["kv_len"], s["kv_max"], s["out"], s["ws"])
    g.tree_accept(s["tokens"], s["parent"], s["logits"], s["path"], s["length"], s["bonus"], s["ws_accept"])
    g.glide_kv_compact(s["K"], s["V"], s["kv_len"], s["path"], s["length"], s["new_len"])
    return dict(draft=s["out_draft"], tree=s["out"], tokens=s["tokens"], parent=s["parent"], n_nodes=s["n_nodes"],
                conf=s["conf"], path=s["path"], length=s["length"], bonus=s["bonus"], new_len=s["new_len"],
                K=s["K"], V=s["V"])


# -------------------------------------------------------------------- work
def _attn_work(c, n, tree):
    e = 2 if c["dtype"] == "bf16" else 4
    lens = _lengths(c)
    keys = sum(l + (n if tree else 0) for l in lens)
    return dict(bytes=c["H_kv"] * keys * c["D"] * 2 * e + c["B"] * n * c["H"] * c["D"] * (e + 4) + 4 * c["B"] * (n + 1),
                flops=4.0 * c["D"] * c["H"] * n * keys)


def _accept_work(B, n, V):
    return dict(bytes=B * n * V * 4 + 12 * B * n + 8 * B, flops=float(B * n * V))


def work(case):
    c, kind = case, case["kind"]
    B = c["B"]
    if kind == "cross":
        return _attn_work(c, 1, False)
    if kind == "verify":
        return _attn_work(c, c["n"], True)
    if kind == "accept":
        return _accept_work(B, c["n"], c["V"])
    if kind == "sample":
        # the target's logits, and one row of the draft's distributions for the residual draw
        rows = B * (c["gamma"] + 1) + B
        return dict(bytes=rows * c["V"] * 4 + 8 * B * c["gamma"] + 4 * B * (c["gamma"] + 1) + 8 * B,
                    flops=3.0 * rows * c["V"])
    if kind == "block":
        lens = _lengths(c, "len_min", "T")
        pairs = sum(c["L"] * (j // c["L"]) for l in lens for j in range(l))
        rows = sum(lens)
        return dict(bytes=rows * c["H_kv"] * c["D"] * 4 + rows * c["H"] * c["D"] * 2 + B * c["T"] * c["H"] * c["D"] * 4,
                    flops=4.0 * c["D"] * c["H"] * pairs)
    parts = [_attn_work(c, 1, False)] * c.get("gamma", 1)
    n = c["n"] if kind == "tiny" else 1 + CAPE_CAP
    parts = parts + [_attn_work(c, n, True), _accept_work(B, n, c["V"])]
    if kind == "round":
        parts.append(dict(bytes=B * c["gamma"] * c["V"] * 4, flops=float(B * c["gamma"] * c["V"])))
    return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))


# ------------------------------------------------------- results in 64 bits
def _softmax_attention(q, K, V, allowed=None):
    """q [rows, D], K/V [keys, D] in 64 bits."""
    x = q @ K.T / math.sqrt(q.shape[-1])
    if allowed is not None:
        x = x.masked_fill(~allowed, -math.inf)
    return torch.softmax(x, -1) @ V


def _exact_attn(s, q, parents=None):
    B, n, H, D = q.shape
    H_kv = s["K"].shape[1]
    group = H // H_kv
    out = torch.zeros((B, n, H, D), dtype=torch.float64, device="cuda")
    for b, length in enumerate(s["lens"]):
        allowed = None
        keys = length
        if parents is not None:
            keys = length + n
            own = torch.zeros((n, n), dtype=torch.bool)
            for i in range(n):
                j = i
                while j >= 0:
                    own[i, j] = True
                    j = parents[b][j]
            allowed = torch.cat([torch.ones((n, length), dtype=torch.bool), own], 1).cuda()
            allowed = allowed.repeat_interleave(group, 0)
        for h in range(H_kv):
            rows = q[b, :, h * group:(h + 1) * group].double().reshape(n * group, D)
            o = _softmax_attention(rows, s["K"][b, h, :keys].double(), s["V"][b, h, :keys].double(), allowed)
            out[b, :, h * group:(h + 1) * group] = o.view(n, group, D)
    return out


def _exact_block(s, L):
    B, T, H, D = s["q"].shape
    group = H // s["K"].shape[1]
    out = torch.zeros((B, T, H, D), dtype=torch.float64, device="cuda")
    j = torch.arange(T, device="cuda")
    allowed = j[None, :] < (j // L * L)[:, None]
    for b, length in enumerate(s["lens"]):
        first = min(L, length)
        for h in range(H):
            K, V = (s[x][b, h // group, :length].double() for x in "KV")
            out[b, first:length, h] = _softmax_attention(s["q"][b, first:length, h].double(), K, V,
                                                         allowed[first:length, :length])
    return out


def _cape_parents(probs):
    """The parents of CaPE's expanded tree of one sequence (Section 3.2): the proposal as a chain, then
    every position's expansion set, its size from the confidence; past the cap the least probable go."""
    gamma, V = probs.shape
    p, _ = torch.sort(probs, dim=-1, descending=True, stable=True)
    p = p[:, :8].double().tolist()
    sets = []
    for i in range(gamma):
        conf = p[i][0]
        k = 7 if conf <= 0.3 else 5 if conf <= 0.6 else 3 if conf <= 0.8 else 1
        sets += [(-p[i][r], i, r) for r in range(1, min(k, V - 1) + 1)]
    kept = sorted(sorted(sets)[:CAPE_CAP - gamma], key=lambda x: (x[1], x[2]))
    parent = [-1] + list(range(gamma)) + [i for _, i, _ in kept]
    return parent + [0] * (1 + CAPE_CAP - len(parent))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("accept", "sample"):
        return None  # tokens, indices and counts only
    s = _inputs(c, seed)
    if kind == "cross":
        return _exact_attn(s, s["q"])
    if kind == "verify":
        return _exact_attn(s, s["q"], s["parents"])
    if kind == "block":
        return _exact_block(s, c["L"])
    if kind == "tiny":
        return dict(draft=_exact_attn(s, s["q_draft"]), tree=_exact_attn(s, s["q"], s["parents"]), path=None,
                    length=None, bonus=None)
    parents = [_cape_parents(s["probs"][b]) for b in range(c["B"])]
    return dict(draft=[_exact_attn(s, q) for q in s["q_draft"]], tree=_exact_attn(s, s["q"], parents), tokens=None,
                parent=None, n_nodes=None, conf=s["probs"].amax(-1).double(), path=None, length=None, bonus=None,
                new_len=None, K=None, V=None)
