"""The entries of new_frontier behind the new frontier: -1 from the Python call, untouched by the C ABI's."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def graph(B, F, V, Ncap, n0):
    i32 = dict(dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(F)
    return dict(logits=torch.randn((B, F, V), generator=gen, device="cuda"), frontier=torch.arange(F, **i32).expand(B, F).contiguous(),
                frontier_len=torch.full((B,), F, **i32), tokens=torch.randint(0, V, (B, Ncap), generator=gen, **i32),
                tree_parent=torch.tensor([[-1] + list(range(Ncap - 1))] * B, **i32), merge_to=torch.full((B, Ncap), -1, **i32),
                leaf=torch.zeros((B, Ncap), dtype=torch.uint8, device="cuda"), prob=torch.zeros((B, Ncap), device="cuda"),
                num_nodes=torch.full((B,), n0, **i32))


# (sequence 1 has a frontier that is too long, sequence 2 none, sequence 3 no room for all of its children)
@pytest.mark.parametrize("F,k,theta", [(1, 1, 0.0), (7, 4, 0.0), (7, 4, 2.0), (60, 8, 0.0)])
def test_rest_of_the_new_frontier(F, k, theta):
    import paper_2407_16207_b200 as gsd
    B, V, Ncap = 4, 700, 512
    n0 = max(F, 5)
    g = graph(B, F, V, Ncap, n0)
    g["frontier_len"][1] = F + 1
    g["frontier_len"][2] = 0
    g["num_nodes"][3] = Ncap - 1
    h = {n: t.clone() for n, t in g.items()}
    for _ in range(3):                                  # memory the allocator hands out again holds something else
        torch.full((B, F * k), 77, dtype=torch.int32, device="cuda")
    nf, n = gsd.gsd_draft_expand(*g.values(), k=k, tau=1, theta_prob=theta, theta_sib=0.0)
    n = n.tolist()
    assert n[1] == n[2] == 0 and n[3] <= 1
    for b in range(B):
        assert (nf[b, :n[b]] >= 0).all() and (nf[b, n[b]:] == -1).all()
    # the C ABI writes the first entries only
    L = gsd.binding.lib()
    own = torch.full((B, F * k), 77, dtype=torch.int32, device="cuda")
    n2 = torch.zeros((B,), dtype=torch.int32, device="cuda")
    p = gsd.binding.DraftParams(B, F, V, Ncap, k, 1, theta, 0.0)
    ws = torch.empty(max(8, int(L.gsd_draft_expand_workspace_bytes(ctypes.byref(p)))), dtype=torch.uint8, device="cuda")
    rc = L.gsd_draft_expand(*(h[x].data_ptr() for x in h), own.data_ptr(), n2.data_ptr(), ctypes.byref(p), ws.data_ptr(), ws.numel(), None,
                            torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and n2.tolist() == n
    for b in range(B):
        assert torch.equal(own[b, :n[b]], nf[b, :n[b]]) and (own[b, n[b]:] == 77).all()
