"""The calls that stream rows of logits - greedy and sampled acceptance, draft growth - over
vocabularies and base addresses that make rows start anywhere inside a 16-byte group, and over rows
that are cut into slices, against the CPU oracle (bit by bit, random numbers and thresholds kept
away from every decision as in tests/test_gpu_accept_sampled.py and tests/test_gpu_draft.py)."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
import oracle
import test_gpu_accept_sampled as sampled_cases
import test_gpu_draft as draft_cases
from gpu_util import accept_tensors

pytestmark = pytest.mark.gpu


def shifted(x, by):
    """The same values at an address `by` floats past a 16-byte boundary."""
    flat = torch.empty(x.numel() + 4, dtype=torch.float32, device="cuda")
    out = flat[by:by + x.numel()].view(x.shape)
    out.copy_(x)
    assert out.data_ptr() % 16 == 4 * by
    return out


def graph_inputs(B, N, V, seed):
    depth = 0 if N == 1 else int(np.ceil(np.log(2 * N + 1) / np.log(3))) + 1
    cfg = gi.VerifyConfig("v", 7, B, 1, 1, 64, 8, N, min(depth, N - 1), 3, 2, V, min(V, 64), 0.7)
    return gi.make_inputs(cfg, seed, attn=False)


@pytest.mark.parametrize("by", [0, 1, 2, 3])
@pytest.mark.parametrize("V", [1, 2, 3, 4, 5, 7, 1023, 1025, 4099, 16387, 50257])
def test_accept_rows_that_start_anywhere(V, by):
    import paper_2407_16207_b200 as gsd
    inp = graph_inputs(2, 11, V, 40 + V)
    t = accept_tensors(inp)
    lg = inp["logits"].copy()
    # the best entry of a row at its first, last and second-last position; a row of -inf but its end
    lg[0, 0, 0] = lg[0, 1, V - 1] = lg[0, 2, max(0, V - 2)] = 50.0
    lg[0, 3] = -np.inf
    lg[0, 4, :] = np.nan
    lg[0, 4, V - 1] = -np.inf
    want = oracle.accept(lg, inp["draft_tokens"], inp["parent_ptr"], inp["parent_idx"])
    got = gsd.gsd_accept(shifted(torch.from_numpy(lg), by), t["draft_tokens"], t["parent_ptr"], t["parent_idx"])
    for g, w in zip(got, want[:3]):
        assert np.array_equal(g.cpu().numpy(), w)


@pytest.mark.parametrize("V,by,dby", [(5, 0, 0), (1003, 1, 1), (1004, 2, 0), (4097, 0, 3), (8195, 3, 2), (16385, 0, 0),
                                      (16388, 1, 1), (50257, 0, 0), (128256, 0, 0), (131071, 2, 1)])
def test_sampled_rows_that_start_anywhere(V, by, dby):
    # target and draft rows with equal and with different alignment, clusters of one to eight CTAs
    import paper_2407_16207_b200 as gsd
    inp = graph_inputs(3, 9, V, 60 + by)
    dl = sampled_cases.draft_logits_for(inp["logits"], 5)
    for residual in (False, True):
        q, u, us, want = sampled_cases.decisive_inputs(inp, 9 + V, q_lo=2.0, q_hi=20.0, dl=dl if residual else None)
        t = accept_tensors(inp)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        got = gsd.gsd_accept_sampled(shifted(t["logits"], by), t["draft_tokens"], t["parent_ptr"], t["parent_idx"],
                                     *(torch.from_numpy(a).cuda() for a in (q, u, us)), status=status,
                                     draft_logits=shifted(torch.from_numpy(dl), dby) if residual else None)
        for g, w in zip(got, want[:3]):
            assert np.array_equal(g.cpu().numpy(), w)
        assert int(status.item()) == 0


@pytest.mark.parametrize("B,F,V,k,by", [(1, 1, 8, 8, 1), (1, 1, 4099, 1, 0), (1, 1, 131071, 8, 3), (2, 3, 50257, 4, 0),
                                        (1, 2, 65536, 4, 2), (3, 40, 8193, 2, 0), (5, 60, 1003, 4, 1), (8, 64, 8192, 4, 0)])
def test_draft_rows_in_slices(B, F, V, k, by):
    # one to eight CTAs per row; ties across slices, slices without a finite entry, NaN flagged
    import paper_2407_16207_b200 as gsd
    rng = np.random.default_rng(V + k)
    lg = (3 * rng.normal(size=(B, F, V))).astype(np.float32)
    hot = rng.integers(0, V, size=(B, F, 2 * k))
    np.put_along_axis(lg, hot, rng.integers(14, 18, size=hot.shape).astype(np.float32), axis=-1)
    if V > 4096:
        lg[0, 0, V // 3:] = -np.inf             # most slices of this row are empty
    fr, fl = np.zeros((B, F), np.int32), np.full((B,), F, np.int32)
    fl[-1] = max(1, F - 1)
    state = draft_cases.fresh(B, 512)
    tp, ts = draft_cases.decisive_thresholds(lg, fl, k, rng, (0.001, 0.9), (0.001, 0.9))
    out = oracle.draft_expand(lg, fr, fl, *state, k=k, tau=2, theta_prob=tp, theta_sib=ts)
    t = [torch.from_numpy(a.copy()).cuda() for a in state]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    nf, nfl = gsd.gsd_draft_expand(shifted(torch.from_numpy(lg), by), torch.from_numpy(fr).cuda(), torch.from_numpy(fl).cuda(), *t,
                                   k=k, tau=2, theta_prob=tp, theta_sib=ts, status=status)
    draft_cases.compare([a.cpu().numpy() for a in t], list(out[:6]), nf.cpu().numpy(), nfl.cpu().numpy(), out[6], out[7])
    assert int(status.item()) == (0x80 if out[8] else 0)
    bad = lg.copy()
    bad[0, 0] = -np.inf
    bad[0, 0, :k - 1] = 1.0                     # one entry short of k
    bad[-1, 0, V - 1] = np.nan
    for b, x in ((0, bad[:1]), (B - 1, bad[-1:])):
        t = [torch.from_numpy(a[b:b + 1].copy()).cuda() for a in state]
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        gsd.gsd_draft_expand(shifted(torch.from_numpy(x), by), torch.from_numpy(fr[b:b + 1]).cuda(), torch.from_numpy(fl[b:b + 1]).cuda(), *t,
                             k=k, tau=2, theta_prob=tp, theta_sib=ts, status=status)
        assert int(status.item()) & 0x40


@pytest.mark.parametrize("by", [0, 1, 2, 3])
@pytest.mark.parametrize("V", [1, 3, 6, 1003, 16389])
def test_nan_anywhere_in_a_row_is_flagged(V, by):
    # target rows and the end node's draft row; the first and last entries of a row are not part of
    # its 16-byte groups, and an entry may be the first its thread meets or follow entries of -inf
    import paper_2407_16207_b200 as gsd
    rng = np.random.default_rng(V)
    B, N = 1, 4
    lg, dl = (rng.normal(size=(B, N, V)).astype(np.float32) for _ in range(2))
    g = [torch.tensor(x, dtype=torch.int32, device="cuda") for x in ([[0, 0, 0, 0]], [[0, 0, 1, 2, 3]], [[0, 1, 2]])]
    q, u, us = torch.ones(B, N, device="cuda"), torch.ones(B, N, device="cuda"), torch.full((B,), 0.5, device="cuda")   # nothing is accepted

    def flags(lg, dl):
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        gsd.gsd_accept_sampled(shifted(torch.from_numpy(lg), by), *g, q, u, us, draft_logits=shifted(torch.from_numpy(dl), by), status=status)
        return int(status.item())
    assert flags(lg, dl) == 0
    at = sorted({0, 1, 2, 3, 4, V // 2, V - 4, V - 3, V - 2, V - 1} & set(range(V)))
    for e in at:
        for rest in (1.0, -np.inf):
            bad = lg.copy()
            bad[0, 2] += 0.0 if rest == 1.0 else rest
            bad[0, 2, (e + 1) % V] = 1.0
            bad[0, 2, e] = np.nan
            assert flags(bad, dl) == 0x40, (e, rest)
            bad = dl.copy()
            bad[0, 0] += 0.0 if rest == 1.0 else rest
            bad[0, 0, (e + 1) % V] = 1.0
            bad[0, 0, e] = np.nan
            assert flags(lg, bad) == 0x40, (e, rest)


MASKS = [-1e9, -1e10, -3e30, float(np.finfo(np.float32).min)]


@pytest.mark.parametrize("mask", MASKS)
@pytest.mark.parametrize("V", [1003, 4099, 32000])
def test_entries_masked_with_a_large_negative_number(V, mask):
    # a filtered distribution whose entries are finite: whole runs of a row, of a thread's share
    # and of its first loads hold nothing else
    import paper_2407_16207_b200 as gsd
    rng = np.random.default_rng(V)
    inp = graph_inputs(2, 9, V, 70)
    keep = np.zeros(inp["logits"].shape, bool)
    keep[:, :, rng.integers(0, V, 40)] = True
    keep[:, :, inp["draft_tokens"].ravel()] = True
    inp["logits"] = np.where(keep, inp["logits"], np.float32(mask))
    dl = np.where(keep, sampled_cases.draft_logits_for(inp["logits"], 5), np.float32(mask))
    t = accept_tensors(inp)
    for residual in (False, True):
        q, u, us, want = sampled_cases.decisive_inputs(inp, 9 + V, q_lo=2.0, q_hi=20.0, dl=dl if residual else None)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        got = gsd.gsd_accept_sampled(t["logits"], t["draft_tokens"], t["parent_ptr"], t["parent_idx"],
                                     *(torch.from_numpy(a).cuda() for a in (q, u, us)), status=status,
                                     draft_logits=torch.from_numpy(dl).cuda() if residual else None)
        assert int(status.item()) == 0
        for g, w in zip(got, want[:3]):
            assert np.array_equal(g.cpu().numpy(), w)
    B, F, k = 2, 9, 4
    fr, fl = np.zeros((B, F), np.int32), np.full((B,), F, np.int32)
    state = draft_cases.fresh(B, 64)
    tp, ts = draft_cases.decisive_thresholds(inp["logits"], fl, k, rng, (0.001, 0.9), (0.001, 0.9))
    out = oracle.draft_expand(inp["logits"], fr, fl, *state, k=k, tau=2, theta_prob=tp, theta_sib=ts)
    g = [torch.from_numpy(a.copy()).cuda() for a in state]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    nf, nfl = gsd.gsd_draft_expand(t["logits"], torch.from_numpy(fr).cuda(), torch.from_numpy(fl).cuda(), *g, k=k, tau=2,
                                   theta_prob=tp, theta_sib=ts, status=status)
    assert int(status.item()) == 0
    draft_cases.compare([a.cpu().numpy() for a in g], list(out[:6]), nf.cpu().numpy(), nfl.cpu().numpy(), out[6], out[7])
