"""The CPython extension that marshals the calls: what is not the plain case is left to the Python
path (same refusals, same results), and the two paths give the same outputs."""
import threading

import numpy as np
import pytest
import torch

import gsd_inputs as gi
from gpu_util import accept_tensors, attn_tensors


def test_cpu_tensors_are_left_to_the_python_path_and_refused_there():
    import paper_2407_16207_b200 as gsd
    native = gsd.binding.native()
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32)
    assert native.build_mask(i32(1, 5), i32(1, 4), None, None) is None
    assert native.accept(torch.zeros(1, 4, 8), i32(1, 4), i32(1, 5), i32(1, 4), 0, True, None, None) is None
    assert native.accept(None, "x", 3, [], 0, True, None, None) is None
    with pytest.raises(ValueError, match="parent_ptr: expected a CUDA tensor"):
        gsd.gsd_build_mask(i32(1, 5), i32(1, 4))
    with pytest.raises(ValueError, match="logits: expected contiguous torch.float32"):
        gsd.gsd_accept(torch.zeros(1, 4, 8).double(), i32(1, 4), i32(1, 5), i32(1, 4))
    with pytest.raises(TypeError):
        native.accept(1, 2)


def test_the_table_names_the_calls_in_order():
    # the order of the addresses handed to bind() is the order of struct Table
    import os
    import re
    import paper_2407_16207_b200 as gsd
    src = open(os.path.join(os.path.dirname(gsd.__file__), "csrc", "gsd_native.cpp")).read()
    table = src[src.index("struct Table {"):src.index("constexpr Py_ssize_t kTable")]
    assert tuple(re.findall(r"decltype\(&(gsd_\w+)\)", table)) == gsd.binding._NATIVE_CALLS


@pytest.mark.parametrize("why", ["missing", "another torch"])
def test_without_the_extension_the_calls_go_through_ctypes(why, monkeypatch):
    import sys
    import types
    import warnings
    import paper_2407_16207_b200 as gsd
    b = gsd.binding
    for name in ("_native", "_native_lib", "_declines"):
        monkeypatch.setattr(b, name, None)
    other = None if why == "missing" else types.SimpleNamespace(torch_version="0.0")
    monkeypatch.setitem(sys.modules, b.__package__ + "._native", other)
    monkeypatch.delattr(sys.modules[b.__package__], "_native", raising=False)
    if other is not None:
        monkeypatch.setattr(sys.modules[b.__package__], "_native", other, raising=False)
    with pytest.raises(gsd.GsdError, match="_native.so"):
        b.native()
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32)
    with pytest.warns(RuntimeWarning, match="ctypes"), pytest.raises(ValueError, match="parent_ptr: expected a CUDA tensor"):
        gsd.gsd_build_mask(i32(1, 5), i32(1, 4))
    with warnings.catch_warnings(), pytest.raises(ValueError, match="logits: expected contiguous torch.float32"):
        warnings.simplefilter("error")              # said once
        gsd.gsd_accept(torch.zeros(1, 4, 8).double(), i32(1, 4), i32(1, 5), i32(1, 4))


def inputs(seed, Hkv=2, D=128, N=70):
    cfg = gi.VerifyConfig("n", 7, 3, 4 * Hkv, Hkv, D, (50, 700), N, 9, 3, 2, 1003, 64, 0.6)
    inp = gi.make_inputs(cfg, seed)
    return {**attn_tensors(inp), **accept_tensors(inp)}


def all_calls(t, plain):
    """Every call once; plain=False makes an argument something only the Python path takes."""
    import paper_2407_16207_b200 as gsd
    num = 0 if plain else np.int64(0)
    B, N, V = t["logits"].shape
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = dict(status=status)
    g = (t["draft_tokens"], t["parent_ptr"], t["parent_idx"])
    mask = gsd.gsd_build_mask(*g[1:], **st)
    if not plain:
        mask = gsd.gsd_build_mask(*g[1:], out=mask.zero_(), **st)
    out = gsd.gsd_verify_attn(t["q"], t["k_cache"], t["v_cache"], t["draft_k"], t["draft_v"], mask, t["seq_lens"], num_splits=num, **st)
    rng = torch.Generator().manual_seed(5)
    u = [torch.rand(s, generator=rng).cuda() for s in ((B, N), (B, N), (B,))]
    res = [mask, out]
    for want_nodes in (True, False) if plain else (1, 0):
        acc = gsd.gsd_accept(t["logits"], *g, want_nodes=want_nodes, **st)
        smp = gsd.gsd_accept_sampled(t["logits"], *g, *u, draft_logits=t["logits"].roll(3, 2), Tcap=N - 1 if plain else np.int32(N - 1), want_nodes=want_nodes, **st)
        assert (acc[2] is None) == (not want_nodes) and (smp[2] is None) == (not want_nodes)
        res += [x for x in acc + smp if x is not None]
        if want_nodes:
            nodes, lens = acc[2], acc[1]
    kc, vc, sl = t["k_cache"].clone(), t["v_cache"].clone(), t["seq_lens"].clone()
    gsd.gsd_commit_kv(kc, vc, t["draft_k"], t["draft_v"], nodes, lens, sl, **st)
    graph = [torch.full((B, 64), -1, dtype=torch.int32, device="cuda") for _ in range(3)]
    graph += [torch.zeros(B, 64, dtype=torch.uint8, device="cuda"), torch.zeros(B, 64, device="cuda"), torch.ones(B, dtype=torch.int32, device="cuda")]
    graph[0][:, 0] = 1
    nf = gsd.gsd_draft_expand(t["logits"][:, :1].contiguous(), torch.zeros(B, 1, dtype=torch.int32, device="cuda"),
                              torch.ones(B, dtype=torch.int32, device="cuda"), *graph, k=4 if plain else np.int32(4), tau=2,
                              theta_prob=0.0, theta_sib=0.0, **st)
    return res + [kc, vc, sl, *graph, *nf, status]


@pytest.mark.gpu
def test_both_paths_give_the_same():
    t = inputs(3)
    for a, b in zip(all_calls(t, True), all_calls(t, False)):
        assert a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b)


@pytest.mark.gpu
def test_given_outputs_and_scratch_and_errors():
    import paper_2407_16207_b200 as gsd
    t = inputs(4)
    args = [t[n] for n in ("q", "k_cache", "v_cache", "draft_k", "draft_v", "ancestor_mask", "seq_lens")]
    want = gsd.gsd_verify_attn(*args)
    out = torch.empty_like(want)
    assert gsd.gsd_verify_attn(*args, out=out) is out and torch.equal(out, want)
    need = gsd.gsd_verify_attn_workspace_bytes(*t["q"].shape[:3], t["k_cache"].shape[2], 128, t["k_cache"].shape[1], 3)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    gsd.gsd_verify_attn(*args, num_splits=3, workspace=ws)
    with pytest.raises(gsd.GsdError) as e:
        gsd.gsd_verify_attn(*args, num_splits=3, workspace=ws[:need - 256])
    assert e.value.code == -4
    with pytest.raises(gsd.GsdError) as e:
        gsd.gsd_verify_attn(*args, num_splits=65)
    assert e.value.code == -2
    with pytest.raises(ValueError, match="seq_lens"):
        gsd.gsd_verify_attn(*args[:-1], args[-1].long())
    with pytest.raises(ValueError, match="k_cache"):
        gsd.gsd_verify_attn(args[0], args[1].transpose(0, 1), *args[2:])


@pytest.mark.gpu
def test_threads_on_streams_of_their_own():
    ts = [inputs(10 + k) for k in range(4)]
    want = [all_calls(t, True) for t in ts]
    torch.cuda.synchronize()
    got, errors = [None] * 4, []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(5):
                    got[k] = all_calls(ts[k], True)
            torch.cuda.synchronize()
        except Exception as e:          # noqa: BLE001
            errors.append(e)
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    [x.start() for x in threads]
    [x.join() for x in threads]
    assert not errors
    for a, b in zip(want, got):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
