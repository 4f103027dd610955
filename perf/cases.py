"""Performance cases of the repair-verify step: the calls that a serving engine makes, at the sizes
of the repository's workloads (``paper_2608_00531_gb300/workload.py``) and between and around them.

A case names a ``stage``:

``score``    draft logits -> ranked candidates, margin, log-prob (once per decoding step)
``attn``     tree attention of one layer (once per layer and step: most of a step's time); contiguous or
             paged cache, the tree's rows in tensors of their own or already in the cache (in place)
``accept``   verification of the target's logits: greedy (argmax and walk) or at a temperature
             (sampling and walk)
``lm_head``  the target's greedy tokens straight from its final hidden states
``step``     a whole step, score to resync, through ``RepairVerifyStep``

Inputs are drawn on the GPU from the seed: N(0,1) logits with a planted draft token and a rival an
exponential gap below it, trees built from those, Gaussian Q/K/V, shuffled pages.
"""
import math

import numpy as np
import torch

from paper_2608_00531_gb300 import cure
from paper_2608_00531_gb300.step import RepairVerifyStep, StepInputs

D = 128
SCALE = 1.0 / math.sqrt(D)


# ---------------------------------------------------------------- the cases
def _score(name, rows, block, vocab, topk):
    return dict(name=name, stage="score", batch=rows, block=block, vocab=vocab, topk=topk)


def _attn(name, batch, block, budget, branches, depth, tau, heads_q, heads_kv, lo, hi, page, inplace):
    return dict(name=name, stage="attn", batch=batch, block=block, budget=budget, branches=branches, depth=depth,
                tau=tau, heads_q=heads_q, heads_kv=heads_kv, len_lo=lo, len_hi=hi, page=page, inplace=inplace)


def listed():
    return [
        # one user waiting for a code completion: a single sequence, 8B-class model; latency counts
        _score("score_single", 1, 16, 128256, 2),
        # a full serving batch: 32 sequences of 16 draft positions, three candidates each
        _score("score_serve", 32, 16, 151936, 3),
        # the single sequence's tree attention (32 query heads on 8 kv heads, contiguous cache)
        _attn("attn_single", 1, 16, 8, 2, 1, 1.0, 32, 8, 4096, 4096, 0, False),
        # the serving batch: ragged lengths, 16-token pages, groups of 7 query heads
        _attn("attn_serve", 32, 16, 16, 3, 1, 0.8, 28, 4, 1024, 8192, 16, False),
        # long blocks with wide repairs, the tree's rows written into the paged cache by the target
        _attn("attn_wide_inplace", 16, 32, 32, 3, 1, 1.0, 28, 4, 5001, 8191, 16, True),
        # long documents: 64 sequences of 32 K tokens, 70B-class heads, depth-2 repairs
        _attn("attn_long", 64, 16, 32, 2, 2, 1.0, 64, 8, 32768, 32768, 0, False),
        # greedy verification of the serving batch's target logits
        dict(name="accept_serve", stage="accept", batch=32, block=16, budget=16, branches=3, depth=1, tau=0.8,
             vocab=151936, temperature=0.0),
        # the same at a sampling temperature
        dict(name="sample_serve", stage="accept", batch=32, block=16, budget=16, branches=3, depth=1, tau=0.8,
             vocab=151936, temperature=0.8),
        # LM head of one sequence's tree: the weight's bytes are the work
        dict(name="lm_head_single", stage="lm_head", rows=21, d_model=4096, vocab=128256),
        # LM head of the serving batch's tree nodes: a large contraction
        dict(name="lm_head_serve", stage="lm_head", rows=817, d_model=4096, vocab=151936),
        # a whole step of the single sequence, 32 layers: launch after launch
        dict(name="step_single", stage="step", batch=1, block=16, budget=8, branches=2, depth=1, tau=1.0, vocab=128256,
             layers=32, heads_q=32, heads_kv=8, len_lo=4096, len_hi=4096, page=0),
        # a whole step of the serving batch, 28 layers, paged
        dict(name="step_serve", stage="step", batch=32, block=16, budget=16, branches=3, depth=1, tau=0.8,
             vocab=151936, layers=28, heads_q=28, heads_kv=4, len_lo=1024, len_hi=8192, page=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _tree_shape(rng):
    return dict(block=rng.randint(4, 32), budget=rng.randint(0, 32), branches=rng.choice([2, 2, 3, 4]),
                depth=rng.choice([1, 1, 2]), tau=round(rng.uniform(0.25, 2.0), 2))


def draw(rng):
    stage = rng.choice(["score", "attn", "attn", "accept", "lm_head", "step"])
    heads_q, heads_kv = rng.choice([(28, 4), (32, 8), (64, 8), (8, 2), (16, 16), (40, 8)])
    vocab = _log_int(rng, 32000, 160000)
    page = rng.choice([0, 0, 8, 16, 16, 32, 64])
    if stage == "score":
        return dict(stage=stage, batch=_log_int(rng, 1, 64), block=rng.randint(4, 32), vocab=vocab,
                    topk=rng.choice([2, 3, 4, 6]))
    if stage == "attn":
        # at most the cached tokens of the largest listed case
        batch = _log_int(rng, 1, 64)
        hi = _log_int(rng, 256, min(65536, 64 * 32768 * 8 // (batch * heads_kv) // 2))
        return dict(stage=stage, batch=batch, heads_q=heads_q, heads_kv=heads_kv, len_lo=max(1, int(hi * rng.random())),
                    len_hi=hi, page=page, inplace=rng.random() < 0.3, **_tree_shape(rng))
    if stage == "accept":
        return dict(stage=stage, batch=_log_int(rng, 1, 64), vocab=vocab,
                    temperature=rng.choice([0.0, 0.0, 0.5, 1.0]), **_tree_shape(rng))
    if stage == "lm_head":
        return dict(stage=stage, rows=_log_int(rng, 9, 1600), d_model=64 * _log_int(rng, 16, 128), vocab=vocab)
    batch = _log_int(rng, 1, 32)
    hi = _log_int(rng, 256, min(16384, 32 * 8192 * 4 // (batch * heads_kv) // 2))
    return dict(stage=stage, batch=batch, vocab=vocab, layers=rng.randint(1, 16), heads_q=heads_q, heads_kv=heads_kv,
                len_lo=max(1, int(hi * rng.random())), len_hi=hi, page=page, **_tree_shape(rng))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed * 1000003 + 17)


def _randn(g, *shape, std=1.0):
    x = torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=g)
    return x


def _randint(g, hi, *shape):
    return torch.randint(0, hi, shape, device="cuda", generator=g)


def _draft(g, B, K, V):
    """Logits bf16 [B][K][V]: noise, the draft token at +16, a rival an Exp(2.5) gap below it."""
    x = _randn(g, B, K, V)
    y = _randint(g, V, B, K)
    r = (y + 1 + _randint(g, V - 1, B, K)) % V
    gap = torch.empty(B, K, device="cuda").exponential_(1 / 2.5, generator=g)
    x.scatter_(2, y[..., None], 16.0)
    x.scatter_(2, r[..., None], (16.0 - gap).to(torch.bfloat16)[..., None])
    return x, y, r


def _tree(g, c, V, cache_len, logits=None):
    """The tree that the framework builds for a draft block, the draft's tokens and rivals."""
    B, K = c["batch"], c["block"]
    k = max(2, c["branches"])
    logits, y, r = _draft(g, B, K, V) if logits is None else logits
    ids, _, margin, _ = cure.cure_score_draft(logits, k)
    root = _randint(g, V, B).to(torch.int32)
    redraft = None
    if c["depth"] == 2:  # the successor of a substituted token: the draft's own next token
        nxt = torch.cat([y[:, 1:], torch.full((B, 1), -1, device="cuda")], 1).to(torch.int32)
        redraft = nxt[..., None].expand(B, K, c["branches"] - 1).contiguous()
    tree = cure.cure_build_tree(ids, margin, root, cache_len, c["tau"], c["budget"], c["branches"], c["depth"], redraft)
    return dict(tree=tree, y=y, r=r, root=root, redraft=redraft)


def _lengths(g, c):
    return torch.randint(c["len_lo"], c["len_hi"] + 1, (c["batch"],), device="cuda", generator=g).to(torch.int32)


def _cache(g, c, layers, room):
    """Per-layer caches (one tensor for K, one for V), their geometry, lengths.  `room`: slots past the length."""
    B, Hkv, ps = c["batch"], c["heads_kv"], c["page"]
    L = _lengths(g, c)
    if ps == 0:
        max_len = c["len_hi"] + room
        shape, table = (layers, B, max_len, Hkv, D), None
        kv = cure.kv_desc(Hkv, D, max_len)
    else:
        # a pool of fixed size, as a server keeps one: pages for every sequence at its largest
        need = (L.cpu().numpy().astype(np.int64) + room + ps - 1) // ps
        most = (c["len_hi"] + room + ps - 1) // ps
        total = B * most
        perm = torch.randperm(total, device="cuda", generator=g).to(torch.int32).cpu().numpy()
        t = np.full((B, most), -1, dtype=np.int32)
        o = 0
        for b, n in enumerate(need):
            t[b, :n] = perm[o:o + n]
            o += n
        table = torch.from_numpy(t).cuda()
        shape = (layers, total, ps, Hkv, D)
        kv = cure.kv_desc(Hkv, D, t.shape[1], block_table=table, page_size=ps, num_pages=total)
    return _randn(g, *shape), _randn(g, *shape), kv, L, table


def _target_logits(g, c, V, t):
    """bf16 [B][n_max][V]: noise with the target's token planted at +14.  The target follows the draft up to a random
    first error, where it takes the rival in half of the sequences; after that it agrees again."""
    B, K = c["batch"], c["block"]
    e = _randint(g, K + 1, B)
    other = _randint(g, V, B)
    truth = torch.cat([t["y"], _randint(g, V, B, 1)], 1)
    rival = torch.cat([t["r"], truth[:, -1:]], 1).gather(1, e[:, None])[:, 0]
    at = torch.where(_randint(g, 2, B) > 0, rival, other)
    truth.scatter_(1, e[:, None], at[:, None])
    ids = truth.gather(1, t["tree"]["depth"].clamp(min=0).long())
    x = _randn(g, B, ids.shape[1], V)
    x.scatter_(2, ids[..., None], 14.0)
    return x


def prepare(case, seed):
    c, g = case, _gen(seed)
    if c["stage"] == "score":
        x, _, _ = _draft(g, c["batch"], c["block"], c["vocab"])
        lead = (c["batch"], c["block"])
        out = (torch.empty(*lead, c["topk"], dtype=torch.int32, device="cuda"),
               torch.empty(*lead, c["topk"], device="cuda"), torch.empty(lead, device="cuda"),
               torch.empty(lead, device="cuda"))
        return dict(c=c, logits=x, out=out)
    if c["stage"] == "lm_head":
        V, d, rows = c["vocab"], c["d_model"], c["rows"]
        w = _randn(g, V, d, std=d ** -0.5)
        h = _randn(g, rows, d)
        planted = _randint(g, V, rows)
        # a tenth of the rows stays noise: their argmax is decided by small gaps
        h += ((torch.arange(rows, device="cuda") % 10 != 9).to(torch.bfloat16) * 12)[:, None] * w[planted]
        return dict(c=c, h=h, w=w, out=torch.empty(rows, dtype=torch.int32, device="cuda"),
                    ws=torch.empty(max(256, cure.cure_lm_head_workspace_size(rows, V)), dtype=torch.uint8, device="cuda"))
    B, K = c["batch"], c["block"]
    N = 1 + K + c["budget"]
    if c["stage"] == "accept":
        V = c["vocab"]
        t = _tree(g, c, V, torch.zeros(B, dtype=torch.int32, device="cuda"))
        i32 = dict(dtype=torch.int32, device="cuda")
        out = dict(accept_len=torch.empty(B, **i32), best_node=torch.empty(B, **i32),
                   path_nodes=torch.empty(B, K + 2, **i32), out_tokens=torch.empty(B, K + 2, **i32),
                   diverge_depth=torch.empty(B, **i32))
        return dict(c=c, tree=t["tree"], logits=_target_logits(g, c, V, t), out=out, targ=torch.empty(B, N, **i32),
                    u=torch.rand(B, N, device="cuda", generator=g))
    if c["stage"] == "attn":
        k, v, kv, L, table = _cache(g, c, 1, N + 1)
        t = _tree(g, c, 32000, L)["tree"]
        q = _randn(g, B, N, c["heads_q"], D, std=1.5)
        tk, tv = _randn(g, B, N, c["heads_kv"], D), _randn(g, B, N, c["heads_kv"], D)
        ws = torch.empty(max(256, cure.cure_tree_attn_workspace_size(B, N, c["heads_q"], kv)), dtype=torch.uint8,
                         device="cuda")
        s = dict(c=c, q=q, tk=tk, tv=tv, k=k[0], v=v[0], kv=kv, L=L, tree=t, table=table, ws=ws,
                 out=torch.zeros_like(q))
        if c["inplace"]:  # the target has written the tree's rows at slots L + j
            for b in range(B):
                n = int(t["n_nodes"][b])
                at = _slots(s, b, int(L[b]), n)
                s["k"].view(-1, c["heads_kv"], D)[at] = tk[b, :n]
                s["v"].view(-1, c["heads_kv"], D)[at] = tv[b, :n]
        return s
    V, layers = c["vocab"], c["layers"]
    k, v, kv, L, table = _cache(g, c, layers, N + 1)
    draft = _draft(g, B, K, V)
    t = _tree(g, c, V, L, logits=draft)
    step = RepairVerifyStep(B, K, V, max(2, c["branches"]), c["tau"], c["budget"], c["branches"], c["depth"], layers,
                            c["heads_q"], kv, torch.device("cuda", torch.cuda.current_device()))
    step.attn_out.zero_()
    x = StepInputs(draft[0], t["root"], L, t["redraft"], _randn(g, layers, B, N, c["heads_q"], D, std=1.5),
                   _randn(g, layers, B, N, c["heads_kv"], D), _randn(g, layers, B, N, c["heads_kv"], D),
                   _target_logits(g, c, V, t))
    return dict(c=c, step=step, x=x, k=k, v=v, kl=list(k), vl=list(v), kv=kv, table=table)


# ---------------------------------------------------------------- one pass
def run(state):
    s, c = state, state["c"]
    if c["stage"] == "score":
        return cure.cure_score_draft(s["logits"], c["topk"], out=s["out"])
    if c["stage"] == "lm_head":
        return cure.cure_lm_head_argmax(s["h"], s["w"], out=s["out"], workspace=s["ws"])
    if c["stage"] == "attn":
        tk, tv = (None, None) if c["inplace"] else (s["tk"], s["tv"])
        return cure.cure_tree_attn(s["q"], tk, tv, s["k"], s["v"], s["kv"], s["L"], s["tree"]["n_nodes"],
                                   s["tree"]["anc"], SCALE, out=s["out"], workspace=s["ws"])
    if c["stage"] == "accept":
        if c["temperature"] > 0:
            targ = cure.cure_sample_target(s["logits"], s["tree"]["n_nodes"], s["u"], c["temperature"], out=s["targ"])
            return cure.cure_accept(s["tree"], c["block"], targ=targ, out=s["out"])
        return cure.cure_accept(s["tree"], c["block"], target_logits=s["logits"], targ=s["targ"], out=s["out"])
    r = s["step"].run(s["x"], s["kl"], s["vl"])
    return dict(score=r["score"], tree=r["tree"], attn=r["attn"], acc=r["acc"], resync=r["resync"], k=s["k"], v=s["v"])


# ---------------------------------------------------------------- what a pass cannot do without
def _nodes(c):
    """Expected tree nodes of one sequence."""
    p = 1.0 - math.exp(-c["tau"] / 2.5)
    return 1 + c["block"] + min(c["budget"], c["block"] * p * (c["branches"] - 1) * c["depth"])


def _attn_work(c):
    n, L, Hq, Hkv = _nodes(c), (c["len_lo"] + c["len_hi"]) / 2, c["heads_q"], c["heads_kv"]
    return (c["batch"] * (L * Hkv * D * 4 + n * (2 * Hq + 2 * Hkv) * D * 2),
            4.0 * Hq * D * c["batch"] * n * (L + c["block"] / 2 + 1))


def work(case):
    c = case
    if c["stage"] == "score":
        rows = c["batch"] * c["block"]
        return dict(bytes=rows * (2.0 * c["vocab"] + 8 * c["topk"] + 8), flops=3.0 * rows * c["vocab"])
    if c["stage"] == "lm_head":
        return dict(bytes=2.0 * c["d_model"] * (c["vocab"] + c["rows"]) + 4 * c["rows"],
                    flops=2.0 * c["rows"] * c["d_model"] * c["vocab"])
    if c["stage"] == "attn":
        b, f = _attn_work(c)
        return dict(bytes=b, flops=f)
    targ = c["batch"] * _nodes(c) * c["vocab"]
    if c["stage"] == "accept":
        return dict(bytes=2.0 * targ, flops=targ * (3.0 if c["temperature"] > 0 else 1.0))
    b, f = _attn_work(c)
    draft = c["batch"] * c["block"] * c["vocab"]
    kept = c["layers"] * c["batch"] * (c["block"] / 2 + 1) * c["heads_kv"] * D * 8.0
    return dict(bytes=c["layers"] * b + 2.0 * (targ + draft) + kept, flops=c["layers"] * f + 3.0 * draft + targ)


def tolerance(case):
    c = case
    if c["stage"] == "score":
        # exact ids, values and margins; logp1 is the difference of two numbers near 16 that leaves a few hundredths
        return dict(rel=1e-5, differ=0.0)
    if c["stage"] == "lm_head":
        return dict(rel=0.0, max=0.0, differ=0.002)  # rows whose top two logits lie within float32 accumulation
    if c["stage"] == "accept":
        # sampling: ids whose cumulative probability lies within float32 sums of u
        return dict(rel=0.0, max=0.0, differ=0.002) if c["temperature"] > 0 else "exact"
    return dict(rel=1e-2, max=0.1, differ=0.0)  # probabilities and outputs are rounded to bf16


# ---------------------------------------------------------------- the same in 64 bits
def _slots(s, b, first, count):
    """Row numbers of cache slots first .. first + count - 1 of sequence b in the flattened cache."""
    at = torch.arange(first, first + count, device="cuda")
    if s["table"] is None:
        return b * s["kv"].max_len + at
    ps = s["kv"].page_size
    return s["table"][b].long()[at // ps] * ps + at % ps


def _exact_attn(s, q, tk, tv, k, v, L, n_nodes, anc, inplace):
    B, N, Hq, _ = q.shape
    Hkv = k.shape[-2]
    G = Hq // Hkv
    out = torch.zeros(B, N, Hq, D, dtype=torch.float64, device="cuda")
    words = anc.cpu().numpy().view(np.uint64).reshape(B, N, -1)
    for b in range(B):
        n, l = int(n_nodes[b]), int(L[b])
        at = _slots(s, b, 0, l + (n if inplace else 0))
        kb, vb = k.view(-1, Hkv, D)[at], v.view(-1, Hkv, D)[at]
        if not inplace:
            kb, vb = torch.cat([kb, tk[b, :n]]), torch.cat([vb, tv[b, :n]])
        mask = np.array([[(int(words[b, j, a >> 6]) >> (a & 63)) & 1 for a in range(n)] for j in range(n)], dtype=bool)
        hide = ~torch.from_numpy(mask).cuda().repeat_interleave(G, 0)
        for h in range(Hkv):
            qh = q[b, :n, h * G:(h + 1) * G].double().reshape(n * G, D)
            sc = (qh @ kb[:, h].double().T) * SCALE
            sc[:, l:].masked_fill_(hide, -math.inf)
            out[b, :n, h * G:(h + 1) * G] = (torch.softmax(sc, 1) @ vb[:, h].double()).view(n, G, D)
    return out


def _exact_score(x, k):
    x = x.reshape(-1, x.shape[-1])
    ids, vals, lp = [], [], []
    for i in range(0, x.shape[0], 64):
        y = x[i:i + 64].double()
        v, j = torch.sort(y, dim=1, descending=True, stable=True)
        ids.append(j[:, :k].to(torch.int32))
        vals.append(v[:, :k])
        lp.append(v[:, 0] - torch.logsumexp(y, 1))
    return torch.cat(ids), torch.cat(vals), torch.cat(lp)


def _first_max(x):
    """Lowest index of each row's maximum."""
    m = x.amax(-1, keepdim=True)
    idx = torch.arange(x.shape[-1], device=x.device)
    return torch.where(x == m, idx, x.shape[-1]).amin(-1).to(torch.int32)


def _exact_walk(tree, targ, block):
    """Longest accepted path (deepest node, lowest index on ties)."""
    tok, par, dep, n = (tree[k].cpu().numpy() for k in ("tok", "parent", "depth", "n_nodes"))
    t = targ.cpu().numpy()
    B, P = tok.shape[0], block + 2
    o = dict(accept_len=np.zeros(B, np.int32), best_node=np.zeros(B, np.int32), path_nodes=np.full((B, P), -1, np.int32),
             out_tokens=np.full((B, P), -1, np.int32), diverge_depth=np.full(B, -1, np.int32))
    for b in range(B):
        ok = [True]
        for j in range(1, int(n[b])):
            ok.append(ok[par[b, j]] and tok[b, j] == t[b, par[b, j]])
        best = max((j for j in range(int(n[b])) if ok[j]), key=lambda j: (dep[b, j], -j))
        a, j = int(dep[b, best]), best
        o["accept_len"][b], o["best_node"][b], o["out_tokens"][b, a] = a, best, t[b, best]
        while j >= 0:
            o["path_nodes"][b, dep[b, j]] = j
            if j > 0:
                o["out_tokens"][b, dep[b, j] - 1] = tok[b, j]
            if j > block:
                o["diverge_depth"][b] = dep[b, j]
            j = int(par[b, j])
    return o


def _exact_targ(s, c):
    x, tree = s["logits"], s["tree"]
    B, N, _ = x.shape
    n = tree["n_nodes"]
    targ = torch.full((B, N), -1, dtype=torch.int32, device="cuda")
    for b in range(B):
        y = x[b, :int(n[b])].double()
        if c["temperature"] > 0:
            p = torch.cumsum(torch.softmax(y / c["temperature"], 1), 1)
            u = s["u"][b, :int(n[b]), None].double()
            targ[b, :int(n[b])] = (p <= u).sum(1).clamp(max=y.shape[1] - 1).to(torch.int32)
        else:
            targ[b, :int(n[b])] = _first_max(y)
    return targ


def exact(case, seed):
    c, s = case, prepare(case, seed)
    if c["stage"] == "score":
        ids, vals, lp = _exact_score(s["logits"], c["topk"])
        lead = (c["batch"], c["block"])
        return (ids.view(*lead, -1), vals.view(*lead, -1), (vals[:, 0] - vals[:, 1]).view(lead), lp.view(lead))
    if c["stage"] == "lm_head":
        h = s["h"].double()
        best = torch.full((c["rows"],), -math.inf, dtype=torch.float64, device="cuda")
        ids = torch.zeros(c["rows"], dtype=torch.int32, device="cuda")
        for v0 in range(0, c["vocab"], 8192):
            x = h @ s["w"][v0:v0 + 8192].double().T
            m = x.amax(1)
            ids = torch.where(m > best, _first_max(x) + v0, ids)
            best = torch.maximum(best, m)
        return ids
    if c["stage"] == "attn":
        return _exact_attn(s, s["q"], s["tk"], s["tv"], s["k"], s["v"], s["L"], s["tree"]["n_nodes"], s["tree"]["anc"],
                           c["inplace"])
    if c["stage"] == "accept":
        targ = _exact_targ(s, c)
        return dict(_exact_walk(s["tree"], targ, c["block"]), targ=targ)
    x, step = s["x"], s["step"]
    ids, vals, lp = _exact_score(x.draft_logits, step.k)
    lead = (c["batch"], c["block"])
    margin = (vals[:, 0] - vals[:, 1]).view(lead)
    # the tree is whole numbers; it is taken as the framework builds it for these candidates
    tree = cure.cure_build_tree(ids.view(*lead, -1).contiguous(), margin.float(), x.root_tok, x.cache_len, c["tau"],
                                c["budget"], c["branches"], c["depth"], x.redraft)
    attn = torch.stack([_exact_attn(s, x.q[l], x.tree_k[l], x.tree_v[l], s["k"][l], s["v"][l], x.cache_len,
                                    tree["n_nodes"], tree["anc"], False).float() for l in range(c["layers"])])
    return dict(score=(ids.view(*lead, -1), vals.view(*lead, -1), margin, lp.view(lead)),
                tree={k: None for k in tree}, attn=attn, acc=None, resync=None, k=None, v=None)
