"""mma.sync attention with at most 16, 32 and more rows an item (the warps share the keys of a tile between four, two or
one): edges of rows and of keys, empty key sets, cut key ranges; against the oracle."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
import oracle
from gpu_util import attn_tensors, out_to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("N,G", [(2, 1), (15, 1), (16, 1), (4, 4), (17, 1), (11, 3), (8, 4), (31, 1), (33, 1), (16, 3)])
def test_rows_and_keys(D, N, G):
    import paper_2407_16207_b200 as gsd
    lens = [0, 1, 15, 16, 17, 47, 48, 63, 64, 65, 127, 200]
    cfg = gi.VerifyConfig("f", 4, len(lens), 2 * G, 2, D, max(lens), N, min(4, N - 1), 3, 2, 8, 8, 0.5)
    inp = gi.make_inputs(cfg, 100 * N + G, accept=False)
    inp["seq_lens"][:] = lens
    rng = np.random.default_rng(N)
    inp["ancestor_mask"][3] = 0                        # no draft key at all
    inp["ancestor_mask"][5] = rng.integers(0, 1 << 32, inp["ancestor_mask"][5].shape, dtype=np.uint32)
    inp["ancestor_mask"][0, : N // 2] = 0              # and, with an empty prefix, rows without any key
    t = attn_tensors(inp)
    for b, L in enumerate(lens):                       # nothing behind a sequence's end may reach the result
        t["k_cache"][b, L:] = float("nan")
        t["v_cache"][b, L:] = float("nan")
    want = oracle.attn(inp["q"], inp["k_cache"], inp["v_cache"], inp["draft_k"], inp["draft_v"], inp["ancestor_mask"], inp["seq_lens"])
    for splits in (1, 0, 3):
        got = out_to_f64(gsd.gsd_verify_attn(*(t[n] for n in ("q", "k_cache", "v_cache", "draft_k", "draft_v", "ancestor_mask", "seq_lens")),
                                             kernel=gsd.GSD_ATTN_MMA, num_splits=splits))
        err = np.abs(got - want)
        # few keys, so outputs of the size of single values: the weights and the result are rounded to 8 bits, which is
        # 2^-9 of max |v| each, and 2^-9 of E |v| = 0.8 on average
        assert err.max() <= 2 * 2.0 ** -9 * max(1.0, np.abs(want).max()) * 2 and err.mean() <= 2.0 ** -9, (splits, err.max(), err.mean())
        assert (got[0, : N // 2] == 0).all()
