"""Performance cases of the batched Traversal Verification library: what a
serving program calls, through ``paper_2505_12398_gb300.Verifier``.

One decoding cycle of speculative decoding with trees is: draft the children
of every node from the drafter's rows (``draft_children``), run the target
model's last layer on every node's hidden state (``lm_head``), verify the
trees (``verify``, or ``verify_stats`` with the normalisers the LM head
computed).  The cases time these calls one by one, from a single request
(B = 1) to the largest batches, on tree shapes, vocabularies, temperatures
and drafter qualities of the repository's own workloads.

Inputs are synthetic: Zipf-biased Gaussian target logits (a rank prior shared
by all rows), draft rows softmax((logits + sigma noise) / T), children drawn
without replacement from the draft rows, uniforms in [0, 1).  Draft rows of
leaves are never read and stay zero.
"""

import math

import torch

# Tree shapes: nodes per level and most children per node of a level.
SHAPES = {
    # a chain of 8 draft tokens (plain speculative decoding)
    "chain8": ((1,) * 8, (1,) * 8),
    # a binary tree of depth 4
    "binary4": ((2, 4, 8, 16), (2, 2, 2, 2)),
    # 26, 60 and 120 nodes: sparse trees, wide near the root
    "tree26": ((2, 4, 8, 8, 4), (2, 2, 2, 1, 1)),
    "tree60": ((4, 10, 16, 16, 8, 6), (4, 3, 2, 2, 1, 1)),
    "tree120": ((4, 12, 24, 24, 20, 16, 12, 8), (4, 3, 2, 1, 1, 1, 1, 1)),
}

# Rows a tree's traversal needs, averages over synthetic batches at sigma = 2:
# target rows normalised, nodes with at least one rejection pass.
NEEDED = {"chain8": (8.0, 5.0), "binary4": (4.5, 3.5), "tree26": (5.8, 4.9),
          "tree60": (7.2, 6.2), "tree120": (10.3, 9.4)}
# Share of those passes' nodes at other drafter qualities.
PASS_SHARE = {0.5: 0.43, 1.0: 0.75, 2.0: 1.0}


def _parents(shape):
    levels, most = SHAPES[shape]
    parents, prev = [-1], [0]
    for size, k in zip(levels, most):
        cur = []
        for j in range(size):
            parents.append(prev[j // k])
            cur.append(len(parents) - 1)
        prev = cur
    return parents


def _kids(parents):
    kids = [[] for _ in parents]
    for c in range(1, len(parents)):
        kids[parents[c]].append(c)
    return kids


def _verify(name, tree, batch, vocab, dtype="bf16", T=1.0, sigma=1.0):
    return {"name": name, "call": "verify", "tree": tree, "batch": batch, "vocab": vocab,
            "dtype": dtype, "T": T, "sigma": sigma}


def _draft(name, tree, batch, vocab, T=1.0):
    return {"name": name, "call": "draft", "tree": tree, "batch": batch, "vocab": vocab, "T": T,
            "sigma": 1.0, "dtype": "bf16"}


def _lm_head(name, tree, batch, vocab, hidden, T=1.0):
    return {"name": name, "call": "lm_head", "tree": tree, "batch": batch, "vocab": vocab,
            "hidden": hidden, "T": T}


def listed():
    return [
        # plain chain drafting for a few requests, fp32 logits: launch and
        # latency count
        _verify("verify_chain8_b16_v32k_fp32", "chain8", 16, 32000, dtype="fp32"),
        # one interactive request at a large vocabulary: the serial chain of
        # vocabulary jobs of one tree
        _verify("verify_tree60_b1_v128k", "tree60", 1, 128256, T=0.7),
        # a serving batch at a small vocabulary
        _verify("verify_tree60_b64_v32k", "tree60", 64, 32000),
        # a serving batch at a large vocabulary
        _verify("verify_tree60_b128_v128k", "tree60", 128, 128256, T=0.7),
        # the largest batch (offline generation), weak drafter: most re-reads
        _verify("verify_tree60_b1024_v152k", "tree60", 1024, 151936, sigma=2.0),
        # a vocabulary with a few added tokens: rows not 16-byte aligned
        _verify("verify_tree60_b32_v32003", "tree60", 32, 32003),
        # verification after the LM head, with its normalisers
        {"name": "verify_stats_tree60_b32_v128k", "call": "stats", "tree": "tree60", "batch": 32,
         "vocab": 128256, "dtype": "bf16", "T": 0.7, "sigma": 1.0},
        # drafting for one interactive request, and for a serving batch
        _draft("draft_tree60_b1_v128k", "tree60", 1, 128256, T=0.7),
        _draft("draft_tree60_b128_v128k", "tree60", 128, 128256, T=0.7),
        # the LM head on the rows of one request (the weight's bytes count),
        # of a batch at a small vocabulary, and of a batch at a large one
        _lm_head("lm_head_b1_v128k", "tree60", 1, 128256, 4096, T=0.7),
        _lm_head("lm_head_b64_v32k", "tree60", 64, 32000, 4096),
        _lm_head("lm_head_b128_v128k", "tree60", 128, 128256, 4096, T=0.7),
    ]


# No drawn case is larger than the largest listed ones: elements of
# [B][N+1][V] for verification, of the rows read for drafting, and
# multiply-adds for the LM head.
MOST_VERIFY = 1024 * 61 * 151936
MOST_DRAFT = 128 * 61 * 128256
MOST_LM_HEAD = 128 * 61 * 128256 * 4096


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["verify", "verify", "verify", "stats", "draft", "lm_head"])
    tree = rng.choice(sorted(SHAPES))
    rows = len(_parents(tree))
    T = rng.choice([0.6, 0.7, 0.8, 1.0])
    vocab = rng.choice([32000, 128256, 151936, _log_int(rng, 1000, 151936)])
    if call in ("stats", "lm_head") or rng.random() < 0.5:
        vocab = vocab // 8 * 8
    elif rng.random() < 0.5:
        vocab = vocab - rng.randrange(1, 8)
    if call == "lm_head":
        hidden = 64 * _log_int(rng, 8, 64)
        batch = _log_int(rng, 1, max(1, min(256, MOST_LM_HEAD // (rows * vocab * hidden))))
        return {"call": call, "tree": tree, "batch": batch, "vocab": vocab, "hidden": hidden,
                "T": T}
    most = (MOST_DRAFT if call == "draft" else MOST_VERIFY) // (rows * vocab)
    dtype = rng.choice(["bf16", "bf16", "fp32"])
    if dtype == "fp32":
        most = most * 3 // 4
    batch = _log_int(rng, 1, max(1, min(1024, most)))
    return {"call": call, "tree": tree, "batch": batch, "vocab": vocab, "dtype": dtype, "T": T,
            "sigma": rng.choice([0.5, 1.0, 2.0])}


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rank_prior(vocab, g):
    return -1.1 * torch.log1p(torch.randperm(vocab, generator=g, device="cuda").float())


def _tree_inputs(case, seed):
    parents = _parents(case["tree"])
    kids = _kids(parents)
    B, R, V, T = case["batch"], len(parents), case["vocab"], case["T"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    g = _generator(seed)
    prior = _rank_prior(V, g)
    need_logits = case["call"] != "draft"
    logits = torch.empty(B, R, V, dtype=dtype, device="cuda") if need_logits else None
    drafts = torch.zeros(B, R, V, dtype=torch.float32, device="cuda")
    tokens = torch.zeros(B, R, dtype=torch.int32, device="cuda")
    for i in range(R):
        if not need_logits and not kids[i]:
            continue
        l = torch.randn(B, V, generator=g, device="cuda").mul_(3.0).add_(prior).to(dtype)
        if need_logits:
            logits[:, i] = l
        if kids[i]:
            z = torch.randn(B, V, generator=g, device="cuda").mul_(case["sigma"]).add_(l)
            q = torch.softmax(z.div_(T), dim=-1)
            drafts[:, i] = q
            # the largest q / Exp(1): draws without replacement, in order
            e = torch.empty(B, V, device="cuda").exponential_(generator=g).clamp_(min=1e-30)
            top = torch.topk(q.div_(e), len(kids[i]), dim=-1, sorted=True).indices
            tokens[:, kids[i]] = top.to(torch.int32)
    par = torch.tensor(parents, dtype=torch.int32, device="cuda").expand(B, R).contiguous()
    u = torch.rand(B, R + 1, generator=g, device="cuda")
    return par, tokens, logits, drafts, u


def _outputs(B, N):
    """The three outputs side by side in one buffer, read back in one copy."""
    buf = torch.empty(B * N + 2 * B, dtype=torch.int32, device="cuda")
    path = buf[:B * N].view(B, N)
    return buf, (path, buf[B * N:B * N + B], buf[B * N + B:])


def _row_stats(logits, T):
    """(max, sum of 2^((l - max) log2(e) / T)) of every row, as the LM head
    writes them."""
    B, R, V = logits.shape
    out = torch.empty(B, R, 2, dtype=torch.float32, device="cuda")
    for b in range(B):
        l = logits[b].double()
        m = l.max(dim=-1).values
        out[b, :, 0] = m.float()
        out[b, :, 1] = torch.exp((l - m[:, None]) / T).sum(dim=-1).float()
    return out


def _lm_head_inputs(case, seed):
    M, K, V = case["batch"] * len(_parents(case["tree"])), case["hidden"], case["vocab"]
    g = _generator(seed)
    H = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    H[:, 0] = 1.0
    W = torch.randn(V, K, generator=g, device="cuda").mul_(3.0 / math.sqrt(K - 1))
    W = W.to(torch.bfloat16)
    W[:, 0] = _rank_prior(V, g).to(torch.bfloat16)
    return H, W


def prepare(case, seed):
    from paper_2505_12398_gb300 import Verifier

    N = len(_parents(case["tree"])) - 1
    B, V = case["batch"], case["vocab"]
    v = Verifier(V, N, B, case.get("dtype", "bf16"))
    s = {"call": case["call"], "v": v, "T": case["T"]}
    if case["call"] == "lm_head":
        H, W = _lm_head_inputs(case, seed)
        M = B * (N + 1)
        s.update(H=H, W=W, out=(torch.empty(M, V, dtype=torch.bfloat16, device="cuda"),
                                torch.empty(M, 2, dtype=torch.float32, device="cuda")))
        return s
    par, tok, logits, drafts, u = _tree_inputs(case, seed)
    s.update(par=par, tok=tok, logits=logits, drafts=drafts, u=u)
    if case["call"] == "draft":
        s["u"] = u[:, :N + 1].contiguous()
        s["out"] = torch.empty(B, N + 1, dtype=torch.int32, device="cuda")
        return s
    if case["call"] == "stats":
        s["row_stats"] = _row_stats(logits, case["T"])
    s["buf"], s["out"] = _outputs(B, N)
    return s


def run(s):
    v = s["v"]
    if s["call"] == "verify":
        v.verify(s["par"], s["tok"], s["logits"], s["drafts"], s["T"], s["u"], out=s["out"])
        return s["buf"]
    if s["call"] == "stats":
        v.verify_stats(s["par"], s["tok"], s["logits"], s["drafts"], s["T"], s["u"],
                       s["row_stats"], out=s["out"])
        return s["buf"]
    if s["call"] == "draft":
        return v.draft_children(s["par"], s["drafts"], s["u"], out=s["out"])
    return v.lm_head(s["H"], s["W"], s["T"], out=s["out"])


def work(case):
    parents = _parents(case["tree"])
    B, R, V = case["batch"], len(parents), case["vocab"]
    if case["call"] == "lm_head":
        M, K = B * R, case["hidden"]
        return {"bytes": 2 * M * K + 2 * V * K + 2 * M * V + 8 * M, "flops": 2 * M * K * V}
    small = B * R * 4 * 4
    if case["call"] == "draft":
        internal = sum(1 for k in _kids(parents) if k)
        return {"bytes": B * internal * V * 4 + small, "flops": B * internal * V}
    size = 2 if case["dtype"] == "bf16" else 4
    rows, nodes = NEEDED[case["tree"]]
    nodes *= PASS_SHARE[case["sigma"]]
    if case["call"] == "stats":   # the normalisers are given: rows with a pass only
        return {"bytes": int(B * nodes * V * (size + 4)) + small,
                "flops": int(B * nodes * V * 12)}
    return {"bytes": int(B * V * (rows * size + nodes * 4)) + small,
            "flops": int(B * V * (rows * 8 + nodes * 12))}


def tolerance(case):
    if case["call"] == "lm_head":
        # bf16 logits: a value near a rounding boundary may take the other of
        # two neighbours (2^-8 apart, relative)
        return {"rel": 5e-3, "max": 2e-2}
    # whole numbers: a draw within float32 summation error of a step of the
    # CDF may fall on the neighbouring token
    return {"rel": 1e-5, "differ": 5e-3}


# ------------------------------------------------------------ 64-bit results


def _traverse(parents, kids, tok, logits, drafts, T, u):
    """One tree, literally: (path, tau, bonus), every distribution in 64 bits."""
    R = len(parents)
    mb, ms, p = {}, {}, [0.0] * R
    gone = [False] * R
    p[0], node = 1.0, 0

    def rows(i):
        if i not in mb:
            mb[i] = torch.softmax(logits[i].double() / T, dim=-1)
            ms[i] = drafts[i].double()

    def reject(i, c):
        gone[c] = True
        d = (p[i] * mb[i] - ms[i]).clamp_(min=0.0)
        S = float(d.sum())
        left = 1.0 - float(ms[i][tok[c]])
        ms[i][tok[c]] = 0.0
        ms[i] = ms[i] / left if left > 0.0 else ms[i] * 0.0
        if S > 0.0:
            mb[i] = d / S
            p[i] = S / (S + (1.0 - p[i]))
        else:
            p[i] = 1.0 if p[i] == 1.0 else 0.0

    for c in range(1, R):
        if float(drafts[parents[c]][tok[c]]) <= 0.0:
            return [-1] * (R - 1), -1, -1
    while True:
        c = next((k for k in kids[node] if not gone[k]), None)
        if c is None:
            if node == 0 or u[node] < p[node]:
                break
            reject(parents[node], node)
            node = parents[node]
        else:
            rows(node)
            at = torch.stack([mb[node][tok[c]], ms[node][tok[c]]]).tolist()
            if at[1] <= 0.0:
                return [-1] * (R - 1), -1, -1
            p[c] = min(p[node] * at[0] / at[1], 1.0)
            if p[c] > 0.0:
                node = c
                continue
            reject(node, c)
        while node != 0 and p[node] == 0.0:
            up = parents[node]
            reject(up, node)
            node = up
    if node not in mb:
        mb[node] = torch.softmax(logits[node].double() / T, dim=-1)
    cdf = torch.cumsum(mb[node], 0)
    y = int(torch.searchsorted(cdf, cdf[-1:] * u[R], right=True))
    path, i = [], node
    while i != 0:
        path.append(i)
        i = parents[i]
    path.reverse()
    return path + [-1] * (R - 1 - len(path)), len(path), min(y, cdf.numel() - 1)


def _exact_draft(par, drafts, u, kids):
    B, R, _ = drafts.shape
    out = torch.zeros(B, R, dtype=torch.int32, device="cuda")
    at = torch.arange(B, device="cuda")
    for i, ks in enumerate(kids):
        if not ks:
            continue
        q = drafts[:, i].double()
        for c in ks:
            cdf = torch.cumsum(q, dim=-1)
            y = torch.searchsorted(cdf, cdf[:, -1:] * u[:, c:c + 1].double(), right=True)[:, 0]
            y = y.clamp_(max=q.shape[1] - 1)
            out[:, c] = y.to(torch.int32)
            q[at, y] = 0.0
    return out


def exact(case, seed):
    if case["call"] == "lm_head":
        H, W = _lm_head_inputs(case, seed)
        if H.shape[0] * W.shape[0] * W.shape[1] > 5e12:
            return None
        logits = H.double() @ W.double().T
        stored = logits.to(torch.bfloat16).double()
        m = stored.max(dim=-1).values
        s = torch.empty_like(m)
        for r in range(0, H.shape[0], 256):
            s[r:r + 256] = torch.exp((stored[r:r + 256] - m[r:r + 256, None]) /
                                     case["T"]).sum(dim=-1)
        return logits, torch.stack([m, s], dim=-1)
    par, tok, logits, drafts, u = _tree_inputs(case, seed)
    parents = _parents(case["tree"])
    kids = _kids(parents)
    if case["call"] == "draft":
        return _exact_draft(par, drafts, u[:, :len(parents)], kids)
    B, N = case["batch"], len(parents) - 1
    toks, us = tok.tolist(), u.double().tolist()
    trees = [_traverse(parents, kids, toks[b], logits[b], drafts[b], case["T"], us[b])
             for b in range(B)]
    flat = [x for t in trees for x in t[0]] + [t[1] for t in trees] + [t[2] for t in trees]
    return torch.tensor(flat, dtype=torch.int32, device="cuda")
