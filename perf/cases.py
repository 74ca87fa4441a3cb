"""The work this library is used for, as cases that can be timed.

One case is one call of a verification step (or the whole step) through the public entry points,
with the tensors a serving program has in hand: `listed()` names twelve of them, `draw()` gives
more of the same ranges.  Kinds:

  step     gsd_build_mask, gsd_verify_attn, gsd_accept, gsd_commit_kv: one iteration for one layer
  attn     gsd_verify_attn alone: what every further layer of the model adds to an iteration
  accept   gsd_accept alone (greedy verification)
  sampled  gsd_accept_sampled with the draft model's logits (non-deterministic verification)
  draft    gsd_draft_expand: one level of growth of the draft graph

The step from host buffers is left out: it copies the whole KV cache over the host link on every
call, which only a measurement of that link does.
"""
import math

import numpy as np
import torch

import paper_2407_16207_b200 as gsd

_DEV = "cuda"


def listed():
    return [
        # the smallest call there is: a tiny model's layer, one short sequence, all four entry
        # points of an iteration; launches and host work are all of it
        dict(name="step_tiny", kind="step", B=1, Hq=4, Hkv=4, D=64, Lmin=128, Lmax=128, rows=160, N=16, depth=5, V=1000),
        # LLaMA-2-7B layer shape (one kv head per query head), one user, moderate context
        dict(name="attn_llama7b", kind="attn", B=1, Hq=32, Hkv=32, D=128, Lmin=2048, Lmax=2048, rows=2048, N=64, depth=8),
        # LLaMA-2-13B layer shape, four users with contexts of different lengths in a padded cache
        dict(name="attn_llama13b", kind="attn", B=4, Hq=40, Hkv=40, D=128, Lmin=1024, Lmax=4096, rows=4096, N=128, depth=12),
        # LLaMA-2-70B layer shape, eight users, large draft graphs: the whole iteration
        dict(name="step_llama70b", kind="step", B=8, Hq=64, Hkv=8, D=128, Lmin=4096, Lmax=4096, rows=4352, N=256, depth=16, V=32000),
        # one user with a long document and a small draft graph
        dict(name="attn_long_context", kind="attn", B=1, Hq=64, Hkv=8, D=128, Lmin=32768, Lmax=32768, rows=32768, N=32, depth=10),
        # a busy server: many users, short and ragged contexts, graphs of an odd size
        dict(name="attn_busy_ragged", kind="attn", B=32, Hq=64, Hkv=8, D=128, Lmin=200, Lmax=2100, rows=2304, N=57, depth=9),
        # the largest batch: many users, long contexts, the largest graphs
        dict(name="attn_largest", kind="attn", B=32, Hq=64, Hkv=8, D=128, Lmin=8192, Lmax=8192, rows=8192, N=512, depth=18),
        # three query heads per kv head (a group size that is no power of two), odd sizes throughout
        dict(name="attn_group3", kind="attn", B=5, Hq=24, Hkv=8, D=128, Lmin=300, Lmax=1999, rows=2001, N=77, depth=10),
        # the small head dimension, ragged contexts
        dict(name="attn_head64", kind="attn", B=4, Hq=32, Hkv=8, D=64, Lmin=1000, Lmax=4000, rows=4096, N=128, depth=12),
        # greedy verification for a few users over an odd vocabulary (rows that start anywhere)
        dict(name="accept_odd_vocab", kind="accept", B=3, N=61, depth=8, V=50257),
        # non-deterministic verification of large graphs, residual resampling
        dict(name="sampled_llama70b", kind="sampled", B=8, N=256, depth=16, V=32000),
        # one level of draft growth for eight users with 64 open nodes each
        dict(name="draft_level", kind="draft", B=8, F=64, V=32000, Ncap=512, k=4, tau=2),
    ]


_HEADS = [(32, 32, 128), (40, 40, 128), (64, 8, 128), (32, 8, 128), (24, 8, 128), (28, 4, 128), (8, 1, 128), (32, 8, 64), (12, 12, 64)]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _depth(n):
    return max(1, min(n - 1, int(round(2 * math.log2(n)))))


def draw(rng):
    kind = rng.choice(["attn", "attn", "attn", "step", "accept", "sampled", "draft"])
    vocab = rng.choice([32000, 32000, 50257, 50272, 128256, _log_int(rng, 1000, 130000)])
    if kind in ("attn", "step"):
        while True:
            Hq, Hkv, D = rng.choice(_HEADS)
            B, N, L = _log_int(rng, 1, 32), _log_int(rng, 8, 512), _log_int(rng, 64, 32768)
            Lmin = L if rng.random() < 0.4 else max(1, int(L * rng.uniform(0.1, 0.9)))
            c = dict(kind=kind, B=B, Hq=Hq, Hkv=Hkv, D=D, Lmin=Lmin, Lmax=L, rows=L + rng.choice([0, 1, 17, 128, L // 4]),
                     N=N, depth=_depth(N))
            if kind == "step":
                c["V"] = vocab
                c["rows"] = L + N
                if B * N * vocab > 1 << 28:
                    continue
            w = work(c)
            # no more work than the largest listed case (head dimension 64 and odd group sizes count
            # for more: they cannot be expected to run at the same rate) and 6 GB of cache at most
            plain = D == 128 and 128 % (Hq // Hkv) == 0
            if w["flops"] < (1.6e12 if plain else 5e11) and B * c["rows"] * Hkv * D * 4 < 6e9:
                return c
    if kind == "draft":
        k = rng.choice([2, 4, 4, 8])
        B, F = _log_int(rng, 1, 32), _log_int(rng, 1, min(64, 512 // (k + 1)))
        return dict(kind=kind, B=B, F=F, V=vocab, Ncap=512, k=k, tau=rng.choice([1, 2, 3]))
    while True:
        B, N = _log_int(rng, 1, 32), _log_int(rng, 8, 512)
        if B * N * vocab <= 1 << 28:
            return dict(kind=kind, B=B, N=N, depth=_depth(N), V=vocab)


# ------------------------------------------------------------------------------ inputs
def _graph(rng, N, depth, kmax=4, pmax=3):
    """Parents per node of a level-structured graph: node 0 is the root, every other node has 1 to
    pmax parents in the level above, no node more than kmax children."""
    sizes, left = [1], N - 1
    for lvl in range(depth):
        sizes.append(min(-(-left // (depth - lvl)), kmax * sizes[-1]))
        left -= sizes[-1]
    while left > 0:                     # (a graph too wide for its depth grows deeper)
        sizes.append(min(left, kmax * sizes[-1]))
        left -= sizes[-1]
    parents, start, prev = [[]], 1, [0]
    for n in sizes[1:]:
        slots = rng.permutation(np.tile(np.array(prev), kmax))
        mine = [{int(p)} for p in slots[:n]]
        want = rng.integers(1, pmax + 1, n)
        spare = iter(slots[n:])
        for v in range(n):
            for _ in range(int(want[v]) - 1):
                p = next(spare, None)
                if p is not None:
                    mine[v].add(int(p))
        parents += [sorted(m) for m in mine]
        prev = list(range(start, start + n))
        start += n
    return parents


def _graphs(c, rng):
    B, N, V = c["B"], c["N"], c.get("V", 32000)
    gs = [_graph(rng, N, c["depth"]) for _ in range(B)]
    ecap = max(1, max(sum(len(p) for p in g) for g in gs))
    ptr, idx = np.zeros((B, N + 1), np.int32), np.full((B, ecap), -1, np.int32)
    for b, g in enumerate(gs):
        ptr[b, 1:] = np.cumsum([len(p) for p in g])
        flat = [p for ps in g for p in ps]
        idx[b, :len(flat)] = flat
    tok = rng.integers(0, V, (B, N), dtype=np.int32)
    return gs, dict(draft_tokens=torch.from_numpy(tok).to(_DEV), parent_ptr=torch.from_numpy(ptr).to(_DEV),
                    parent_idx=torch.from_numpy(idx).to(_DEV))


def _logits(c, rng, gen, gs, tok):
    """N(0,1) rows; with probability 0.7 a node's row has its peak on the token of one of its children."""
    B, N, V = c["B"], c["N"], c["V"]
    x = torch.randn((B, N, V), generator=gen, device=_DEV)
    at = []
    for b, g in enumerate(gs):
        child = {}
        for v, ps in enumerate(g):
            for p in ps:
                child.setdefault(p, []).append(v)
        at += [(b, p, vs[int(rng.integers(len(vs)))]) for p, vs in child.items() if rng.random() < 0.7]
    if at:
        b, p, v = (torch.tensor(a, device=_DEV) for a in zip(*at))
        x[b, p, tok[b, v].long()] = 12.0
    return x


def _attn_inputs(c, rng, gen, s):
    B, Hq, Hkv, D, N, rows = (c[k] for k in ("B", "Hq", "Hkv", "D", "N", "rows"))

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=_DEV, dtype=torch.bfloat16)
    s["q"], s["k_cache"], s["v_cache"] = normal(B, N, Hq, D), normal(B, rows, Hkv, D), normal(B, rows, Hkv, D)
    s["draft_k"], s["draft_v"] = normal(B, N, Hkv, D), normal(B, N, Hkv, D)
    lens = rng.integers(c["Lmin"], c["Lmax"] + 1, B, dtype=np.int32)
    s["seq_lens"] = torch.from_numpy(lens).to(_DEV)
    s["mask"] = gsd.gsd_build_mask(s["parent_ptr"], s["parent_idx"])


def prepare(case, seed):
    c, kind = case, case["kind"]
    rng = np.random.default_rng([seed, 1])
    gen = torch.Generator(device=_DEV).manual_seed(seed)
    if kind == "draft":
        B, F, V, Ncap, k = (c[n] for n in ("B", "F", "V", "Ncap", "k"))
        n0 = min(F + F // 2 + 1, Ncap - F * k)      # the graph so far; its last F nodes are open
        n0 = max(n0, F)
        s = dict(kind=kind, k=k, tau=c["tau"], logits=torch.randn((B, F, V), generator=gen, device=_DEV))
        # the draft model is fairly sure of itself: four peaked entries per row
        at = torch.randint(0, V, (B, F, 4), generator=gen, device=_DEV)
        s["logits"].scatter_(2, at, torch.tensor([12.5, 11.5, 11.0, 9.5], device=_DEV).expand(B, F, 4))
        s["frontier"] = torch.arange(n0 - F, n0, device=_DEV, dtype=torch.int32).expand(B, F).contiguous()
        s["frontier_len"] = torch.full((B,), F, dtype=torch.int32, device=_DEV)
        tok = np.zeros((B, Ncap), np.int32)
        tok[:, :n0] = rng.integers(0, V, (B, n0))
        par = np.full((B, Ncap), -1, np.int32)
        for v in range(1, n0):
            par[:, v] = rng.integers(max(0, (v - 1) // k - 1), v, B)
        s["graph"] = dict(tokens=torch.from_numpy(tok).to(_DEV), tree_parent=torch.from_numpy(par).to(_DEV),
                          merge_to=torch.full((B, Ncap), -1, dtype=torch.int32, device=_DEV),
                          leaf=torch.zeros((B, Ncap), dtype=torch.uint8, device=_DEV),
                          prob=torch.zeros((B, Ncap), device=_DEV),
                          num_nodes=torch.full((B,), n0, dtype=torch.int32, device=_DEV))
        s["n0"] = s["graph"]["num_nodes"].clone()
        return s
    gs, s = _graphs(c, rng)
    s["kind"] = kind
    if kind in ("attn", "step"):
        _attn_inputs(c, rng, gen, s)
    if kind != "attn":
        s["logits"] = _logits(c, rng, gen, gs, s["draft_tokens"])
    if kind == "step":
        s["lens0"] = s["seq_lens"].clone()
    if kind == "sampled":
        B, N, V = c["B"], c["N"], c["V"]
        # the draft model: close to the target, but sure of every token it drafted, of which the
        # target agrees with some
        s["draft_logits"] = s["logits"] + 0.3 * torch.randn((B, N, V), generator=gen, device=_DEV)
        eb, ep, ev = (torch.tensor(a, device=_DEV) for a in zip(*((b, p, v) for b, g in enumerate(gs) for v, ps in enumerate(g) for p in ps)))
        s["draft_logits"][eb, ep, s["draft_tokens"][eb, ev].long()] = 11.0
        first = np.array([[ps[0] if ps else 0 for ps in g] for g in gs])
        rows = torch.from_numpy(first).to(_DEV)
        lse = torch.logsumexp(s["draft_logits"], 2)
        b = torch.arange(B, device=_DEV)[:, None]
        s["draft_q"] = torch.exp(s["draft_logits"][b, rows, s["draft_tokens"].long()] - lse.gather(1, rows)).contiguous()
        s["u_accept"] = torch.rand((B, N), generator=gen, device=_DEV)
        s["u_sample"] = torch.rand((B,), generator=gen, device=_DEV)
    return s


# -------------------------------------------------------------------------------- calls
def run(state):
    s, kind = state, state["kind"]
    if kind == "attn":
        return gsd.gsd_verify_attn(s["q"], s["k_cache"], s["v_cache"], s["draft_k"], s["draft_v"], s["mask"], s["seq_lens"])
    if kind == "accept":
        return gsd.gsd_accept(s["logits"], s["draft_tokens"], s["parent_ptr"], s["parent_idx"])
    if kind == "sampled":
        return gsd.gsd_accept_sampled(s["logits"], s["draft_tokens"], s["parent_ptr"], s["parent_idx"], s["draft_q"],
                                      s["u_accept"], s["u_sample"], draft_logits=s["draft_logits"])
    if kind == "draft":
        g = s["graph"]
        g["num_nodes"].copy_(s["n0"])           # a pass starts from the same graph again
        nf, nfl = gsd.gsd_draft_expand(s["logits"], s["frontier"], s["frontier_len"], g["tokens"], g["tree_parent"],
                                       g["merge_to"], g["leaf"], g["prob"], g["num_nodes"], k=s["k"], tau=s["tau"],
                                       theta_prob=0.05, theta_sib=0.3)
        return dict(g, new_frontier=nf, new_frontier_len=nfl)
    s["seq_lens"].copy_(s["lens0"])             # a pass starts from the same committed lengths again
    mask = gsd.gsd_build_mask(s["parent_ptr"], s["parent_idx"])
    out = gsd.gsd_verify_attn(s["q"], s["k_cache"], s["v_cache"], s["draft_k"], s["draft_v"], mask, s["seq_lens"])
    toks, lens, nodes = gsd.gsd_accept(s["logits"], s["draft_tokens"], s["parent_ptr"], s["parent_idx"])
    gsd.gsd_commit_kv(s["k_cache"], s["v_cache"], s["draft_k"], s["draft_v"], nodes, lens, s["seq_lens"])
    return dict(mask=mask, out=out, tokens=toks, lens=lens, nodes=nodes, k_cache=s["k_cache"], v_cache=s["v_cache"],
                seq_lens=s["seq_lens"])


# ------------------------------------------------------------------------- 64-bit answer
def _exact_attn(s):
    """The attention of `s` in 64 bits: visible keys are the committed prefix and, among the draft
    nodes, the node itself and all its ancestors."""
    q, B, N = s["q"], s["q"].shape[0], s["q"].shape[1]
    Hq, D, Hkv = q.shape[2], q.shape[3], s["draft_k"].shape[2]
    G = Hq // Hkv
    ptr, idx, lens = s["parent_ptr"].cpu().numpy(), s["parent_idx"].cpu().numpy(), s["seq_lens"].cpu().numpy()
    out = torch.empty(q.shape, dtype=torch.float64, device=_DEV)
    for b in range(B):
        L = int(lens[b])
        see = np.eye(N, dtype=bool)
        for v in range(N):              # (parents come before their children)
            for p in idx[b, ptr[b, v]:ptr[b, v + 1]]:
                see[v] |= see[p]
        hide = ~torch.from_numpy(see).to(_DEV).repeat_interleave(G, 0)
        for c in range(Hkv):
            k = torch.cat((s["k_cache"][b, :L, c], s["draft_k"][b, :, c])).double()
            v = torch.cat((s["v_cache"][b, :L, c], s["draft_v"][b, :, c])).double()
            x = q[b, :, c * G:(c + 1) * G].reshape(N * G, D).double() @ k.T
            x *= D ** -0.5
            x[:, L:].masked_fill_(hide, -math.inf)
            out[b, :, c * G:(c + 1) * G] = (torch.softmax(x, 1) @ v).view(N, G, D)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("accept", "sampled"):
        return None                     # whole numbers only
    s = prepare(case, seed)
    if kind == "attn":
        return _exact_attn(s)
    if kind == "step":
        return dict(mask=None, out=_exact_attn(s), tokens=None, lens=None, nodes=None, k_cache=None, v_cache=None,
                    seq_lens=None)
    B, F, V, k = (case[n] for n in ("B", "F", "V", "k"))
    n0, Ncap = int(s["n0"][0]), case["Ncap"]
    prob = torch.zeros((B, Ncap), dtype=torch.float64, device=_DEV)
    new = torch.softmax(s["logits"].double(), 2).topk(k, 2).values.reshape(B, F * k)
    prob[:, n0:n0 + F * k] = new[:, :Ncap - n0]
    return dict(tokens=None, tree_parent=None, merge_to=None, leaf=None, prob=prob, num_nodes=None, new_frontier=None,
                new_frontier_len=None)


def work(case):
    c, kind = case, case["kind"]
    if kind == "draft":
        rows = c["B"] * c["F"]
        return {"bytes": rows * c["V"] * 4 + rows * c["k"] * 17, "flops": 4.0 * rows * c["V"]}
    B, N = c["B"], c["N"]
    nbytes, flops = B * N * 12.0, 0.0
    if kind in ("attn", "step"):
        L = (c["Lmin"] + c["Lmax"]) / 2
        nbytes += 2 * B * N * c["Hq"] * c["D"] * 2 + 2 * B * (L + N) * c["Hkv"] * c["D"] * 2 + B * N * ((N + 31) // 32) * 4
        # every node sees the prefix and its ancestors (about one to two per level above it)
        flops += 4.0 * B * N * c["Hq"] * c["D"] * (L + c["depth"])
    if kind != "attn":
        nbytes += B * N * c["V"] * 4.0
        flops += (4.0 if kind == "sampled" else 1.0) * B * N * c["V"]
    if kind == "sampled":
        nbytes += B * c["V"] * 4.0          # of the draft logits only the end node's row is needed
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "accept":
        return "exact"
    if case["kind"] in ("attn", "step"):
        # bf16 weights of the second product and a bf16 result; whole values (mask, tokens, lengths) exact
        return {"rel": 1e-2, "max": 5e-2}
    # fp32 softmax sums in another order; a random number or a threshold within that error of a
    # decision may fall to either side
    return {"rel": 1e-5, "max": 1e-4, "differ": 2e-3}
