"""gsd_accept at the edges of its cut of the rows into slices, with full and with the least scratch, and
the path pass at the edges of its on-chip lists, bit by bit against the oracle."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
import oracle
from gpu_util import accept_tensors

pytestmark = pytest.mark.gpu


def random_graph(rng, N, pmax):
    return [[]] + [sorted(rng.choice(v, size=min(v, int(rng.integers(1, pmax + 1))), replace=False).tolist()) for v in range(1, N)]


def check(B, N, V, parents, agree=0.7):
    import paper_2407_16207_b200 as gsd
    rng = np.random.default_rng([B, N, V])
    ptr, idx = gi.parents_to_csr(parents)
    x = rng.standard_normal((B, N, V)).astype(np.float32)
    tok = rng.integers(0, V, (B, N)).astype(np.int32)
    for b in range(B):
        for v in range(1, N):
            if rng.random() < agree:
                p = parents[b][v][0]
                x[b, p, :] = np.minimum(x[b, p, :], 5.0)
                x[b, p, tok[b, v]] = 9.0                 # (the last child that agrees wins; equal logits: the lowest token)
    inp = dict(logits=x, draft_tokens=tok, parent_ptr=ptr, parent_idx=idx)
    want = oracle.accept(x, tok, ptr, idx, visit_cap=5_000_000)
    t = accept_tensors(inp)
    least = (B * N * 8 + B * 4 + 255) // 256 * 256
    assert gsd.gsd_accept_workspace_bytes(B, N) >= least
    for ws in (None, torch.full((least,), 0xA5, dtype=torch.uint8, device="cuda")):
        got = gsd.gsd_accept(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"], workspace=ws)
        for g, w in zip(got, want[:3]):
            assert np.array_equal(g.cpu().numpy(), w)


@pytest.mark.parametrize("B,N,V", [(1, 1, 8191), (1, 2, 8192), (1, 3, 131075), (2, 5, 16385), (3, 61, 50257), (5, 33, 12289),
                                   (1, 512, 8200), (2, 257, 4096),
                                   # more slices than a thread reads keys of at a time: shared by 2 to 32 threads a node, N
                                   # on both sides of the half and the quarter of the threads, more than 32 slices
                                   (1, 2, 1048576), (2, 1, 524289), (1, 20, 262147), (3, 63, 65536), (1, 64, 262144), (1, 65, 131072),
                                   (1, 128, 131075), (1, 129, 131072)])
def test_slices(B, N, V):
    rng = np.random.default_rng(N)
    check(B, N, V, [random_graph(rng, N, 2) for _ in range(B)], agree=0.4)


@pytest.mark.parametrize("N,pmax", [(2, 1), (33, 9), (255, 2), (256, 6), (257, 7), (512, 5)])
def test_many_parents(N, pmax):
    """More parents than a thread looks at in one go, nodes on both sides of the thread count, and (N 512) more
    steps than the list on chip holds."""
    rng = np.random.default_rng(N + pmax)
    parents = [random_graph(rng, N, pmax), random_graph(rng, N, 1)]
    check(2, N, 64, parents, agree=0.3 if N > 100 else 0.7)
