"""The calls of an iteration start beside the end of whatever precedes them on the stream: none may read an input
before that is written, or write an output that is still being read - behind copies and kernels and behind
one another, eagerly and in a captured graph."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
from gpu_util import accept_tensors, attn_tensors

pytestmark = pytest.mark.gpu


def inputs(seed, B, N, V, L, Hq, Hkv, D):
    cfg = gi.VerifyConfig("c", 3, B, Hq, Hkv, D, L, N, 6, 3, 2, V, 7, 0.7)
    inp = gi.make_inputs(cfg, seed)
    rng = np.random.default_rng(seed)
    inp["seq_lens"][:] = rng.integers(L // 4, L + 1, B)
    t = {**attn_tensors(inp), **accept_tensors(inp)}
    pad = 8 * (N + 1)                                  # the graphs of the three sets have different numbers of edges
    idx = torch.full((B, pad), -1, dtype=torch.int32, device="cuda")
    idx[:, :t["parent_idx"].shape[1]] = t["parent_idx"]
    t["parent_idx"] = idx
    gen = torch.Generator(device="cuda").manual_seed(seed)
    t["draft_logits"] = t["logits"] + 0.3 * torch.randn(t["logits"].shape, generator=gen, device="cuda")
    t["draft_q"] = torch.rand((B, N), generator=gen, device="cuda") * 0.2
    t["u_accept"], t["u_sample"] = torch.rand((B, N), generator=gen, device="cuda"), torch.rand((B,), generator=gen, device="cuda")
    k, F, n0 = 3, 5, 9
    t["d_logits"] = torch.randn((B, F, V), generator=gen, device="cuda")
    t["frontier"] = torch.arange(n0 - F, n0, device="cuda", dtype=torch.int32).expand(B, F).contiguous()
    t["frontier_len"] = torch.randint(1, F + 1, (B,), generator=gen, device="cuda", dtype=torch.int32)
    t["tokens"] = torch.randint(0, V, (B, 64), generator=gen, device="cuda", dtype=torch.int32)
    t["tree_parent"] = torch.tensor([[-1] + [(v - 1) // 2 for v in range(1, 64)]] * B, device="cuda", dtype=torch.int32)
    t["merge_to"] = torch.full((B, 64), -1, device="cuda", dtype=torch.int32)
    t["leaf"], t["prob"] = torch.zeros((B, 64), device="cuda", dtype=torch.uint8), torch.zeros((B, 64), device="cuda")
    t["num_nodes"] = torch.full((B,), n0, device="cuda", dtype=torch.int32)
    return t


def iteration(t):
    """Every call of an iteration, in the order of a serving loop."""
    import paper_2407_16207_b200 as gsd
    mask = gsd.gsd_build_mask(t["parent_ptr"], t["parent_idx"])
    out = gsd.gsd_verify_attn(t["q"], t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], mask, t["seq_lens"])
    a = gsd.gsd_accept(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"])
    gsd.gsd_commit_kv(t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], a[2], a[1], t["seq_lens"])
    again = gsd.gsd_verify_attn(t["q"], t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], mask, t["seq_lens"])
    s = gsd.gsd_accept_sampled(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"], t["draft_q"], t["u_accept"],
                               t["u_sample"], draft_logits=t["draft_logits"])
    d = gsd.gsd_draft_expand(t["d_logits"], t["frontier"], t["frontier_len"], t["tokens"], t["tree_parent"], t["merge_to"], t["leaf"],
                             t["prob"], t["num_nodes"], k=3, tau=2, theta_prob=0.0, theta_sib=0.0)
    e = gsd.gsd_draft_expand(t["d_logits"], d[0][:, :5].contiguous(), d[1].clamp(max=5), t["tokens"], t["tree_parent"], t["merge_to"],
                             t["leaf"], t["prob"], t["num_nodes"], k=3, tau=2, theta_prob=0.0, theta_sib=0.0)
    return [mask, out, *a, again, *s, *d, *e] + [t[n].clone() for n in ("k_cache", "v_cache", "seq_lens", "tokens", "tree_parent", "merge_to",
                                                                       "leaf", "prob", "num_nodes")]


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("shape", [dict(B=2, N=20, V=3000, L=150, Hq=4, Hkv=4, D=64), dict(B=3, N=70, V=40000, L=700, Hq=16, Hkv=2, D=128)])
def test_inputs_written_just_before(shape, captured):
    src = [inputs(seed, **shape) for seed in (1, 2, 3)]
    want = []
    for t in src:
        fresh = {n: v.clone() for n, v in t.items()}
        torch.cuda.synchronize()
        want.append(iteration(fresh))
        torch.cuda.synchronize()
    live = {n: torch.zeros_like(v) for n, v in src[0].items()}
    main = torch.cuda.Stream()

    def work(pieces):
        for t in src:
            for n in live:
                live[n].copy_(t[n])
            pieces.append(iteration(live))
            for n in live:                             # and overwritten right behind the calls
                live[n].zero_()

    with torch.cuda.stream(main):
        got = []
        if captured:
            work([])
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=main):
                work(got)
            for _ in range(3):
                g.replay()
        else:
            for _ in range(3):
                got = []
                work(got)
    torch.cuda.synchronize()
    for k, (g, w) in enumerate(zip(got, want)):
        for i, (x, y) in enumerate(zip(g, w)):
            assert torch.equal(x, y), (k, i)


CALLS = {
    "mask": (("parent_ptr", "parent_idx"), lambda g, t: g.gsd_build_mask(t["parent_ptr"], t["parent_idx"])),
    "accept": (("logits", "draft_tokens", "parent_ptr", "parent_idx"),
               lambda g, t: g.gsd_accept(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"])),
    "sampled": (("logits", "draft_tokens", "parent_ptr", "parent_idx", "draft_q", "u_accept", "u_sample", "draft_logits"),
                lambda g, t: g.gsd_accept_sampled(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"], t["draft_q"],
                                                  t["u_accept"], t["u_sample"], draft_logits=t["draft_logits"])),
    "grow": (("d_logits", "frontier", "frontier_len", "tokens", "tree_parent", "num_nodes"),
             lambda g, t: grow(g, t, t["d_logits"], t["frontier"], t["frontier_len"])),
    "commit": (("draft_k", "draft_v", "nodes", "lens", "seq_lens"),
               lambda g, t: g.gsd_commit_kv(t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], t["nodes"], t["lens"], t["seq_lens"])),
}
CHANGED = {"grow": ("tokens", "tree_parent", "merge_to", "leaf", "prob", "num_nodes"), "commit": ("k_cache", "v_cache", "seq_lens")}


def grow(g, t, logits, frontier, frontier_len):
    return g.gsd_draft_expand(logits, frontier, frontier_len, t["tokens"], t["tree_parent"], t["merge_to"], t["leaf"], t["prob"],
                              t["num_nodes"], k=3, tau=2, theta_prob=0.0, theta_sib=0.0)


def more(seed, B, N, V, L, Hq, Hkv, D):
    t = inputs(seed, B, N, V, L, Hq, Hkv, D)
    rng = np.random.default_rng(seed + 100)
    gen = torch.Generator(device="cuda").manual_seed(seed + 100)
    t["lens"] = torch.from_numpy(rng.integers(1, 6, B).astype(np.int32)).cuda()
    t["nodes"] = torch.full((B, N), -1, dtype=torch.int32, device="cuda")
    for b in range(B):
        t["nodes"][b, :5] = torch.from_numpy(np.sort(rng.choice(N, 5, replace=False)).astype(np.int32))
    # what the calls of a chain read beside each other's outputs: logits of the next two levels of growth and of the
    # grown graph, a chain of parents for its nodes, and lists that make the last node the child of a whole accepted path
    for n, rows in (("d2_logits", 15), ("d3_logits", 45)):
        t[n] = torch.randn((B, rows, V), generator=gen, device="cuda")
    t["g_logits"], t["g_draft"] = (torch.randn((B, 64, V), generator=gen, device="cuda") for _ in range(2))
    t["g_ptr"] = torch.tensor([[0] + list(range(64))] * B, dtype=torch.int32, device="cuda")
    t["g_idx"] = torch.tensor([[max(0, (v - 1) // 2) for v in range(1, 64)]] * B, dtype=torch.int32, device="cuda")
    t["g_q"], t["g_u"] = torch.full((B, 64), 1e-6, device="cuda"), torch.rand((B, 64), generator=gen, device="cuda")
    t["last_ptr"] = torch.tensor([[0] * N + [N]] * B, dtype=torch.int32, device="cuda")
    return t


def agreeing(t, tokens):
    """`g_logits` with its peaks on the tokens of every second node: paths of some length are accepted."""
    x = t["g_logits"].clone()
    for v in range(1, 64, 2):
        x[:, (v - 1) // 2].scatter_(1, tokens[:, v:v + 1].long(), 20.0)
    t["g_logits"] = x


SHAPES = [dict(B=2, N=20, V=3000, L=150, Hq=4, Hkv=4, D=64), dict(B=37, N=70, V=4000, L=100, Hq=2, Hkv=2, D=128)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("call", sorted(CALLS))
def test_each_input_written_by_a_kernel_right_before(call, shape):
    import paper_2407_16207_b200 as gsd
    names, fn = CALLS[call]
    src = [more(seed, **shape) for seed in (1, 2)]
    changed = CHANGED.get(call, ())
    want = []
    for t in src:
        fresh = {n: v.clone() for n, v in t.items()}
        torch.cuda.synchronize()
        got = fn(gsd, fresh)
        want.append([x for x in (got if isinstance(got, tuple) else (got,)) if x is not None] + [fresh[n] for n in changed])
        torch.cuda.synchronize()
    live = {n: torch.zeros_like(v) for n, v in src[0].items()}
    for last in names:
        for k in (0, 1, 0):
            for n in live:
                if n != last:
                    live[n].copy_(src[k][n])
            live[last].zero_()
            live[last].add_(src[k][last])              # a kernel, and nothing between it and the call
            got = fn(gsd, live)
            got = [x for x in (got if isinstance(got, tuple) else (got,)) if x is not None]
            live[last].zero_()                         # a kernel that overwrites it right behind the call
            if last in changed:
                live[last].copy_(want[k][len(got) + changed.index(last)])
            for x, y in zip(got + [live[n] for n in changed], want[k]):
                assert torch.equal(x, y), (last, k)


def chain(t, between):
    """Calls whose inputs are what the call right before them writes last, while that one lets them start early."""
    import paper_2407_16207_b200 as gsd
    outs = []

    def then(got):
        outs.extend(x for x in (got if isinstance(got, tuple) else (got,)) if x is not None)
        between()
        return got
    # growth: the second level's frontier and graph come from the first, the third's from the second
    d = then(grow(gsd, t, t["d_logits"], t["frontier"], t["frontier_len"]))
    d = then(grow(gsd, t, t["d2_logits"], d[0], d[1]))
    then(grow(gsd, t, t["d3_logits"], d[0], d[1]))
    # acceptance of the graph that has just been grown (its second launch reads the tokens before it waits)
    a = then(gsd.gsd_accept(t["g_logits"], t["tokens"], t["g_ptr"], t["g_idx"]))
    # growth from the path that has just been accepted
    d = then(grow(gsd, t, t["g_logits"], a[2], a[1]))
    # sampling over the tokens that this one has just written
    then(gsd.gsd_accept_sampled(t["g_logits"], t["tokens"], t["g_ptr"], t["g_idx"], t["g_q"], t["g_u"], t["u_sample"],
                                draft_logits=t["g_draft"]))
    # a mask whose lists are the path that has just been accepted (entries that are no earlier node are skipped)
    a = then(gsd.gsd_accept(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"]))
    m = then(gsd.gsd_build_mask(t["last_ptr"], a[2]))
    then(gsd.gsd_verify_attn(t["q"], t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], m, t["seq_lens"]))
    s = then(gsd.gsd_accept_sampled(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"], t["draft_q"], t["u_accept"],
                                    t["u_sample"]))
    then(gsd.gsd_commit_kv(t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], s[2], s[1], t["seq_lens"]))
    then(gsd.gsd_verify_attn(t["q"], t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], m, t["seq_lens"]))
    return outs + [t[n].clone() for n in ("k_cache", "v_cache", "seq_lens", "tokens", "tree_parent", "merge_to", "leaf", "prob", "num_nodes")]


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_calls_fed_by_the_one_right_before(shape, captured):
    src = []
    for seed in (1, 2, 3):
        t = more(seed, **shape)
        # (the tokens of the grown graph are known after a run of the growth: peaks go there)
        trial = {n: v.clone() for n, v in t.items()}
        chain(trial, torch.cuda.synchronize)
        agreeing(t, trial["tokens"].clamp(0, shape["V"] - 1))
        src.append(t)
    want = [chain({n: v.clone() for n, v in t.items()}, torch.cuda.synchronize) for t in src]
    assert all(int(w[7].max()) > 3 for w in want)      # (accepted paths of the grown graph are more than the root)
    live = {n: torch.zeros_like(v) for n, v in src[0].items()}
    main = torch.cuda.Stream()

    def work(pieces):
        for t in src:
            for n in live:
                live[n].copy_(t[n])
            pieces.append(chain(live, lambda: None))

    with torch.cuda.stream(main):
        got = []
        if captured:
            work([])
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=main):
                work(got)
            for _ in range(3):
                g.replay()
        else:
            for _ in range(3):
                got = []
                work(got)
    torch.cuda.synchronize()
    for k, (g, w) in enumerate(zip(got, want)):
        assert len(g) == len(w)
        for i, (x, y) in enumerate(zip(g, w)):
            assert torch.equal(x, y), (k, i)
