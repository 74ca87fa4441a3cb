"""A kernel that may be resident before its predecessor has finished must not promise the compiler that nobody
writes its inputs meanwhile (`const __restrict__` lets loads go ahead of the wait, whatever the source says)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_16207_b200", "csrc")


def sources():
    return {os.path.basename(f): open(f).read() for f in glob.glob(os.path.join(CSRC, "*.cu*"))}


def dependents():
    """All kernels but those launched with <<<>>>, which start when everything before them is over."""
    text = "\n".join(sources().values())
    names = set(re.findall(r"__global__ void[^;{]*?\b(\w+_kernel)\(", text))
    return sorted(names - set(re.findall(r"\b(\w+_kernel)(?:<[^;<>]*>)?<<<", text)))


def test_the_dependent_kernels_are_found():
    must = {"build_mask_kernel", "commit_kernel", "accept_kernel", "accept_tail_kernel", "accept_sampled_kernel",
            "accept_sampled_tail_kernel", "draft_expand_kernel", "draft_grow_kernel", "attn_mma_kernel", "attn_tc_kernel",
            "attn_merge_kernel"}
    assert must <= set(dependents())


@pytest.mark.parametrize("name", dependents())
def test_no_promise_about_the_inputs(name):
    found = [m for text in sources().values()
             for m in re.findall(r"__global__ void[^;{]*?\b" + name + r"\(([^{;]*?)\)\s*\{", text)]
    assert len(found) == 1, name
    assert "__restrict__" not in found[0], name
