"""Masks of many words (above 1024 a unit the warps share a unit's rows): draft tiles that no row sees, rows without any
bit, bits past the last node, mask tensors that start anywhere, one to many units a CTA; against the oracle."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
import oracle
from gpu_util import attn_tensors, out_to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,D,N,L", [(1, 2, 2, 128, 129, 100), (2, 3, 3, 128, 161, 300), (1, 24, 8, 128, 512, 130), (2, 2, 2, 64, 346, 700),
                                            (3, 60, 60, 128, 289, 40), (7, 64, 64, 128, 257, 20), (1, 1, 1, 128, 512, 0),
                                            # one word fewer than the shared form needs and one more, groups of one to three
                                            (2, 3, 3, 128, 170, 100), (2, 3, 3, 128, 171, 100), (1, 4, 2, 128, 256, 100),
                                            (1, 4, 2, 128, 257, 100), (1, 6, 2, 64, 384, 60), (1, 6, 2, 64, 385, 60)])
@pytest.mark.parametrize("shift", [0, 1])
def test_live_tiles_of_long_masks(B, Hq, Hkv, D, N, L, shift):
    import paper_2407_16207_b200 as gsd
    cfg = gi.VerifyConfig("w", 6, B, Hq, Hkv, D, max(L, 1), N, 8, 3, 2, 8, 8, 0.5)
    inp = gi.make_inputs(cfg, N, accept=False)
    rng = np.random.default_rng(N + shift)
    inp["seq_lens"][:] = rng.integers(0, L + 1, B)
    mask = np.zeros_like(inp["ancestor_mask"])
    W = mask.shape[2]
    for b in range(B):
        # bits in one or two words of a few rows: most draft tiles of most units are dead
        for n in rng.choice(N, size=max(1, N // 40), replace=False):
            for w in rng.integers(0, W, 2):
                mask[b, n, w] = np.uint32(1) << np.uint32(rng.integers(0, 32))
    mask[:, 0, W - 1] |= np.uint32(1 << 31)            # past the last node unless N is a multiple of 32
    inp["ancestor_mask"] = mask
    t = attn_tensors(inp)
    buf = torch.zeros(mask.size + 4, dtype=torch.int32, device="cuda")
    m = buf[shift:shift + mask.size].view(mask.shape)
    m.copy_(t["ancestor_mask"].view(torch.int32))
    got = out_to_f64(gsd.gsd_verify_attn(t["q"], t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], m, t["seq_lens"]))
    want = oracle.attn(inp["q"], inp["k_cache"], inp["v_cache"], inp["draft_k"], inp["draft_v"], mask, inp["seq_lens"])
    # rows with a single visible key are that key's value; the bounds are those of every attention test
    err = np.abs(got - want)
    assert err.max() <= 1e-2 * max(1.0, np.abs(want).max()) and err.mean() <= 1e-3
    seen = np.zeros((B, N), bool)
    for n in range(N):
        bits = mask[:, n].copy()
        if N % 32:
            bits[:, W - 1] &= np.uint32((1 << (N % 32)) - 1)
        seen[:, n] = bits.any(1) | (inp["seq_lens"] > 0)
    assert (got[~seen] == 0).all()
