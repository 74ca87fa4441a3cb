"""The two plans the attention kernel makes from the sequence lengths - one wave of units when the
items do not fill the device, longest sequences first when they do - against the fp64 oracle and
the plan without the lengths.  Tolerance as in tests/test_gpu_attn.py; against the other plan one
bf16 step of the largest output (both round fp32 results that differ by reassociation)."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
import oracle
from gpu_util import attn_tensors, out_to_f64
from test_gpu_attn import assert_close_scaled, cpu_attn, sampled_rows_check

pytestmark = pytest.mark.gpu

NAMES = ("q", "k_cache", "v_cache", "draft_k", "draft_v", "ancestor_mask", "seq_lens")


def inputs(B, Hq, Hkv, D, N, lens, seed=1):
    cfg = gi.VerifyConfig("l", 7, B, Hq, Hkv, D, int(max(lens)) or 1, N, min(N - 1, 9), 4, 3, 8, 8, 0.5)
    inp = gi.make_inputs(cfg, seed, accept=False)
    inp["seq_lens"][:] = lens
    for b, n in enumerate(lens):
        inp["k_cache"][b, int(n):] = 0x7FC0
        inp["v_cache"][b, int(n):] = 0x7FC0
    return inp


def call(inp, **kw):
    import paper_2407_16207_b200 as gsd
    t = attn_tensors(inp)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = gsd.gsd_verify_attn(*(t[n] for n in NAMES), status=status, **kw)
    assert int(status.item()) == 0
    return out


@pytest.mark.parametrize("Hq,Hkv,D,N", [(8, 2, 128, 40), (4, 4, 128, 100), (32, 2, 128, 40), (8, 2, 64, 70), (6, 2, 128, 90)])
@pytest.mark.parametrize("lens", [(0, 3000), (0, 0, 0), (1, 1, 1, 1), (2600, 0, 130, 127, 1281), (900, 901, 899, 900, 1025, 1024, 1023), tuple(range(40, 1640, 50))])
def test_one_wave(Hq, Hkv, D, N, lens):
    inp = inputs(len(lens), Hq, Hkv, D, N, lens)
    got = call(inp)
    assert torch.equal(got, call(inp))
    assert_close_scaled(out_to_f64(got), cpu_attn(inp))


@pytest.mark.parametrize("Hq,Hkv,D,N", [(32, 8, 128, 40), (32, 8, 64, 100), (24, 8, 128, 50)])
@pytest.mark.parametrize("long,short,n_long,B", [(1700, 100, 1, 10), (1700, 100, 2, 12), (1100, 1100, 0, 11), (1500, 0, 1, 17), (1700, 100, 1, 18)])
def test_one_wave_that_can_cut_few(Hq, Hkv, D, N, long, short, n_long, B):
    # more items than half the device: only some sequences can be cut (with 18 none), the others are
    # stored by the attention kernel itself; the long one first, last and in between
    for at in {0, B // 2, B - n_long}:
        lens = [long if at <= b < at + n_long else short for b in range(B)]
        inp = inputs(B, Hq, Hkv, D, N, lens)
        got = call(inp)
        assert torch.equal(got, call(inp))
        assert_close_scaled(out_to_f64(got), cpu_attn(inp))


def test_scratch_sized_without_the_lengths_is_enough():
    # the size that three forced key ranges need lies between that of the two automatic plans
    import paper_2407_16207_b200 as gsd
    inp = inputs(3, 8, 2, 128, 40, (2000, 300, 1100))
    size = (3, 40, 8, 2, 128, inp["Lmax"])
    need, nominal = gsd.gsd_verify_attn_workspace_bytes(*size), gsd.gsd_verify_attn_num_splits(*size)
    without = gsd.gsd_verify_attn_workspace_bytes(*size, num_splits=nominal)
    assert 0 < without < need
    want = cpu_attn(inp)
    for n in (need, without):
        assert_close_scaled(out_to_f64(call(inp, workspace=torch.empty(n, dtype=torch.uint8, device="cuda"))), want)
    with pytest.raises(gsd.GsdError) as e:
        call(inp, workspace=torch.empty(without - 256, dtype=torch.uint8, device="cuda"))
    assert e.value.code == -4


@pytest.mark.parametrize("B,Hq,Hkv,N,Lmax", [(24, 64, 8, 57, 1500), (5, 40, 40, 128, 1700), (75, 16, 2, 33, 700), (384, 4, 1, 20, 300), (400, 4, 1, 20, 300)])
def test_longest_first(B, Hq, Hkv, N, Lmax):
    rng = np.random.default_rng(B)
    lens = rng.integers(0, Lmax + 1, B)
    lens[rng.integers(0, B, max(2, B // 4))] = Lmax          # ties
    lens[0], lens[B - 1] = 0, Lmax
    inp = inputs(B, Hq, Hkv, 128, N, lens)
    got = call(inp)
    assert torch.equal(got, call(inp))
    assert (got.float() - call(inp, num_splits=1).float()).abs().max().item() <= 2.0 ** -8 * max(1.0, got.float().abs().max().item())
    sampled_rows_check(inp, got, rng, n_random=600, units=[(1, 0), (B // 2, Hkv - 1)])


@pytest.mark.parametrize("Hq,Hkv,N", [(4, 4, 1), (8, 2, 3), (3, 3, 31), (6, 2, 21)])
@pytest.mark.parametrize("lens", [(511,), (512,), (0, 1, 600), (1300, 128, 129, 700)])
def test_few_rows(Hq, Hkv, N, lens):
    # fewer than 64 stacked rows, on either side of the cache length from which the automatic choice changes
    inp = inputs(len(lens), Hq, Hkv, 128, N, lens)
    want = cpu_attn(inp)
    for splits in (0, 2):
        assert_close_scaled(out_to_f64(call(inp, num_splits=splits)), want)


@pytest.mark.parametrize("D,G,N", [(128, 1, 1), (128, 1, 15), (128, 4, 4), (128, 1, 17), (128, 2, 16), (128, 3, 11), (128, 1, 48), (128, 7, 9),
                                   (64, 1, 16), (64, 3, 6), (64, 1, 49)])
def test_few_rows_of_many_items(D, G, N):
    # more (sequence, kv head) pairs than SMs: the mma.sync kernel whatever the cache length, whose warps
    # without a row (16 rows each) only help to load; cut items are merged by eight rows
    import paper_2407_16207_b200 as gsd
    B, Hkv = 40, 4
    assert B * Hkv > torch.cuda.get_device_properties(0).multi_processor_count
    lens = np.random.default_rng(N).integers(0, 600, B)
    lens[:3] = 0, 600, 64
    inp = inputs(B, G * Hkv, Hkv, D, N, lens)
    want = cpu_attn(inp)
    got = call(inp)
    assert torch.equal(got, call(inp, kernel=gsd.GSD_ATTN_MMA))
    assert_close_scaled(out_to_f64(got), want)
    for splits in (1, 3):
        assert_close_scaled(out_to_f64(call(inp, num_splits=splits, kernel=gsd.GSD_ATTN_MMA)), want)


@pytest.mark.parametrize("B,Hkv,splits", [(384, 52, 0), (400, 48, 0), (25, 12, 64)])
def test_more_units_than_one_launch_takes(B, Hkv, splits):
    # more than 128 units a CTA go out in several launches: longest first (up to 384 sequences), in
    # order, and cut (most of the 64 parts are empty), where each launch is a dependent of the one before
    N, D = 64, 64
    rng = np.random.default_rng(B)
    inp = inputs(B, Hkv, Hkv, D, N, rng.integers(0, 40 if splits == 0 else 900, B))
    assert B * Hkv * max(splits, 1) > 128 * torch.cuda.get_device_properties(0).multi_processor_count
    got = call(inp, num_splits=splits)
    assert torch.equal(got, call(inp, num_splits=splits))
    sampled_rows_check(inp, got, rng, n_random=2000, units=[(0, 0), (B // 2, Hkv - 1), (B - 1, Hkv - 1)])
