"""gsd_verify_attn sets itself up beside the end of whatever precedes it on the stream and must not
read anything before that has finished: behind kernels, copies, fills, joins of two streams, and
behind itself, eagerly and in a captured graph."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
from gpu_util import attn_tensors

pytestmark = pytest.mark.gpu

NAMES = ("q", "k_cache", "v_cache", "draft_k", "draft_v", "ancestor_mask", "seq_lens")


@pytest.mark.parametrize("shape", [dict(Hq=32, Hkv=32, D=128, L=600, N=64),        # cut items, merge pass
                                   dict(Hq=64, Hkv=8, D=128, L=900, N=300), # several units per CTA
                                   dict(Hq=8, Hkv=2, D=64, L=500, N=40), dict(Hq=4, Hkv=4, D=64, L=100, N=16)])
@pytest.mark.parametrize("captured", [False, True])
def test_inputs_written_just_before_the_call(shape, captured):
    import paper_2407_16207_b200 as gsd
    cfg = gi.VerifyConfig("g", 7, 4, shape["Hq"], shape["Hkv"], shape["D"], shape["L"], shape["N"], 8, 3, 2, 8, 8, 0.5)
    src = []
    for seed in (1, 2, 3):
        inp = gi.make_inputs(cfg, seed, accept=False)
        inp["seq_lens"][:] = np.random.default_rng(seed).integers(shape["L"] // 8, shape["L"] + 1, cfg.B)
        src.append(attn_tensors(inp))
    want = [gsd.gsd_verify_attn(*(t[n] for n in NAMES)) for t in src]
    live = {n: torch.zeros_like(src[0][n]) for n in NAMES}
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    args = [live[n] for n in NAMES]

    def work(pieces):
        cur = torch.cuda.current_stream()
        for t in src:
            for n in NAMES:                       # copies, the lengths last
                live[n].copy_(t[n])
            pieces.append(gsd.gsd_verify_attn(*args))
            live["q"].zero_()                     # a kernel that overwrites an input right behind it
            live["q"].add_(t["q"])                # a kernel that writes it right before
            pieces.append(gsd.gsd_verify_attn(*args))
            side.wait_stream(cur)
            with torch.cuda.stream(side):
                live["v_cache"].zero_()
                live["v_cache"].add_(t["v_cache"])
            live["seq_lens"].fill_(1)
            live["seq_lens"].copy_(t["seq_lens"])
            cur.wait_stream(side)                 # a join of two streams
            pieces.append(gsd.gsd_verify_attn(*args))
            pieces.append(gsd.gsd_verify_attn(*args))
        live["k_cache"].zero_()

    with torch.cuda.stream(main):
        got = []
        if captured:
            work([])                              # (allocations and attributes first)
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
    for k, o in enumerate(got):
        assert torch.equal(o, want[k // 4]), k
