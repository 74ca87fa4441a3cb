"""The merge pass at the edges of its batches of parts, with few and with many blocks, parts without a key among
them: the same call with one key range."""
import pytest
import torch

import gsd_inputs as gi
from gpu_util import attn_tensors, out_to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,D,N,kernel", [(1, 8, 2, 128, 40, "tc"), (9, 32, 8, 128, 70, "tc"),       # few blocks, many
                                                 # 448, 512 and 592 of them: blocks of eight warps, 64 columns and 128
                                                 (28, 4, 1, 128, 25, "tc"), (4, 32, 8, 128, 30, "tc"), (37, 4, 1, 128, 32, "tc"),
                                                 (8, 32, 8, 64, 32, "auto"),
                                                 (1, 6, 6, 64, 21, "mma"), (3, 8, 2, 128, 30, "mma"), (40, 12, 12, 64, 33, "mma")])
def test_number_of_parts(B, Hq, Hkv, D, N, kernel):
    import paper_2407_16207_b200 as gsd
    L = 700
    cfg = gi.VerifyConfig("m", 5, B, Hq, Hkv, D, L, N, 6, 3, 2, 8, 8, 0.5)
    t = attn_tensors(gi.make_inputs(cfg, 3, accept=False))
    t["seq_lens"][0] = 5                               # nearly all of its parts are empty
    args = [t[n] for n in ("q", "k_cache", "v_cache", "draft_k", "draft_v", "ancestor_mask", "seq_lens")]
    kern = {"tc": gsd.GSD_ATTN_TCGEN05, "mma": gsd.GSD_ATTN_MMA, "auto": gsd.GSD_ATTN_AUTO}[kernel]
    whole = out_to_f64(gsd.gsd_verify_attn(*args, kernel=kern, num_splits=1))
    for parts in (2, 3, 4, 5, 7, 8, 9, 12, 16, 17, 33, 64):
        got = out_to_f64(gsd.gsd_verify_attn(*args, kernel=kern, num_splits=parts))
        # Every part rounds its weights to bf16 against a maximum of its own: two results differ by at most
        # 2 * 2^-9 sum w |v| and two roundings of the result, together 4 * 2^-9 * max |v| < 2^-5 for |v| < 4;
        # on average the signs cancel: 2 * 2^-9 / sqrt 3 * sqrt(sum w^2 v^2), at most half of it here (few keys
        # in one sequence only), and half a bf16 step of the result, below 2^-10 together.
        assert abs(got - whole).max() <= 2.0 ** -5 and abs(got - whole).mean() <= 2.0 ** -10, parts
