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
    """Every call of an iteration, each fed by the one before it where it can be."""
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
