"""The token drawn from the residual, entry by entry: a handful of entries carry equal weights, all others
none, and one sequence per entry draws the middle of its share; two more draw 0 and the very end."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# (8 CTAs keep up to 32768 entries of a row in registers, fewer CTAs fewer; many sequences leave one each)
@pytest.mark.parametrize("V,by", [(5, 0), (7, 3), (130, 1), (4096, 0), (4097, 2), (8195, 1), (16384, 3), (32000, 0), (32768, 0),
                                  (32770, 1), (50257, 2), (128256, 0)])
def test_every_entry_can_be_drawn(V, by):
    import paper_2407_16207_b200 as gsd
    rng = np.random.default_rng(V)
    at = np.unique(np.concatenate([np.arange(min(V, 4)), np.arange(max(0, V - 5), V), rng.integers(0, V, 6)]))
    x = np.full((1, 2, V), -6.0, np.float32)
    y = np.full((1, 2, V), 4.0, np.float32)          # the draft model believes in the others
    x[0, 0, at] = 12.0
    y[0, 0, at] = -6.0
    n = len(at)
    us = np.concatenate([(np.arange(n) + 0.5) / n, [0.0, 1.0]]).astype(np.float32)    # (1: where rounding can leave no crossing)
    want = np.concatenate([at, [at[0], at[-1]]])
    if n == V:                                        # nothing is left for the others to carry
        y[0, 0, :] = 0.0
        y[0, 0, at[0]] = 8.0                          # and the first entry has no weight
        us, want = us[1:], np.concatenate([at[1:], [at[1], at[-1]]])
        us[:n - 1] = (np.arange(n - 1) + 0.5) / (n - 1)

    def row_start(a):                                 # the same values, starting `by` floats behind a 16-byte boundary
        buf = torch.empty(a.size + 8, dtype=torch.float32, device="cuda")
        buf[by:by + a.size] = torch.from_numpy(a).cuda().flatten()
        return buf[by:by + a.size].view(a.shape)

    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    for group in ([[i] for i in range(len(us))], [list(range(len(us)))] if len(us) * V < 1 << 21 else []):
        for seqs in group:                            # one sequence (a cluster of CTAs), then all of them in one call
            B = len(seqs)
            lx, ly = row_start(np.repeat(x, B, 0)), row_start(np.repeat(y, B, 0))
            ones = torch.ones((B, 2), device="cuda")  # a child that is never accepted
            toks, lens, nodes = gsd.gsd_accept_sampled(lx, i32([[0, int(at[-1])]] * B), i32([[0, 0, 1]] * B), i32([[0]] * B), ones, ones,
                                                       torch.from_numpy(us[seqs]).cuda(), draft_logits=ly)
            assert lens.tolist() == [1] * B
            assert toks[:, 0].tolist() == want[seqs].tolist()


@pytest.mark.parametrize("B,N,V", [(1, 3, 131072), (1, 11, 70000), (2, 255, 9000), (2, 256, 4100), (1, 257, 8200), (1, 512, 33000)])
def test_statistics_of_every_node(B, N, V):
    """Steps from the root to every node: the probability of each is decided by the pairs of the first launch, shared by
    one to many threads or two nodes a thread."""
    import paper_2407_16207_b200 as gsd
    gen = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn((B, N, V), generator=gen, device="cuda")
    tok = torch.randint(0, V, (B, N), generator=gen, device="cuda", dtype=torch.int32)
    ptr = torch.arange(-1, N, device="cuda", dtype=torch.int32).clamp(min=0).expand(B, N + 1).contiguous()
    idx = torch.arange(N - 1, device="cuda", dtype=torch.int32).expand(B, N - 1).contiguous()      # a chain
    b = torch.arange(B, device="cuda")[:, None]
    p = torch.softmax(x.double(), 2)[b, torch.arange(N - 1, device="cuda"), tok[:, 1:].long()]     # of node v under v - 1
    q = torch.ones((B, N), device="cuda")
    us = torch.full((B,), 0.5, device="cuda")
    stop = torch.randint(1, N, (B,), generator=gen, device="cuda")
    for end in [1, N - 1] + stop.tolist():
        # every step passes by 1e-4 (the statistics are good to 1e-6), the one into node `end` fails by as much
        u = torch.zeros((B, N), device="cuda")
        u[:, 1:] = (p * (1 - 1e-4)).float()
        u[:, end] = (p[:, end - 1] * (1 + 1e-4)).float()
        toks, lens, nodes = gsd.gsd_accept_sampled(x, tok, ptr, idx, q, u, us)
        assert lens.tolist() == [end] * B
        assert torch.equal(nodes[:, :end], torch.arange(end, device="cuda", dtype=torch.int32).expand(B, end))
