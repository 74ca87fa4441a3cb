"""gsd_build_mask on the GPU against the oracle's upward search: bit-exact."""
import numpy as np
import pytest
import torch

import gsd_inputs as gi
import oracle
from gpu_util import i32_tensor

pytestmark = pytest.mark.gpu


def gpu_mask(ptr, idx, status=None):
    import paper_2407_16207_b200 as gsd
    out = gsd.gsd_build_mask(i32_tensor(ptr, "cuda"), i32_tensor(idx, "cuda"), status=status)
    torch.cuda.synchronize()
    return out.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("name", ["tiny", "llama7b", "llama13b", "llama70b", "sweep512"])
def test_configs_bit_exact_and_equal_to_the_generated_mask(name):
    cfg = gi.sweep_config(4, 512, 512) if name == "sweep512" else gi.CONFIGS[name]
    inp = gi.make_inputs(cfg, attn=False, accept=False)
    got = gpu_mask(inp["parent_ptr"], inp["parent_idx"])
    assert np.array_equal(got, oracle.build_mask(inp["parent_ptr"], inp["parent_idx"]))
    assert np.array_equal(got, inp["ancestor_mask"])


def test_chain_of_maximum_length_and_odd_sizes():
    for N in (1, 31, 33, 100, 512):
        ptr, idx = gi.parents_to_csr([[[]] + [[i - 1] for i in range(1, N)]])
        got = gpu_mask(ptr, idx)
        assert np.array_equal(got, oracle.build_mask(ptr, idx))


def test_bad_edges_are_ignored_and_flagged():
    ptr = np.array([[0, 0, 2, 3]], dtype=np.int32)
    idx = np.array([[0, 5, 2]], dtype=np.int32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = gpu_mask(ptr, idx, status)
    assert np.array_equal(got, oracle.build_mask(ptr, idx))
    assert int(status.item()) == 0x1


@pytest.mark.parametrize("N,deg", [(33, 6), (100, 3), (512, 9), (512, 1)])
def test_mask_with_many_parents(N, deg):
    # more parents per node than sit in registers, more edges than the on-chip copy holds, repeated
    # and invalid parents
    rng = np.random.default_rng(N + deg)
    ptr = np.zeros((2, N + 1), np.int32)
    idx = np.zeros((2, N * deg), np.int32)
    for b in range(2):
        n = 0
        for v in range(N):
            d = int(rng.integers(0, deg + 1)) if v else 0
            idx[b, n:n + d] = rng.integers(max(0, v - 40), v, size=d) if d else 0
            n += d
            ptr[b, v + 1] = n
    for flagged in (False, True):
        if flagged:
            idx[1, ptr[1, N] - 1] = N + 3
            idx[1, ptr[1, N // 2]] = -2
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert np.array_equal(gpu_mask(ptr, idx, status), oracle.build_mask(ptr, idx))
        assert int(status.item()) == (1 if flagged else 0)
