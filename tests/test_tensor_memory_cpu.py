"""The allocation of tensor memory waits without a limit.  What keeps it from waiting for ever is the order of a few
instructions, read here from the sources: a GPU that such a wait holds up is lost to its other users, so no run shows it."""
import os
import re

import pytest

from paper_2604_07853_b200 import build

FILES = sorted(f for f in os.listdir(build.CSRC) if f.endswith((".cu", ".cuh")))


def source(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", FILES)
def test_no_kernel_allocates_for_a_pair_of_ctas(name):
    """`cta_group::2` allocates for two CTAs at once and waits for both: with one of them not begun, or gone, nothing ends it."""
    assert not re.search(r"cta_group::2|tmem_alloc_pair|umma_\w+_pair", source(name))


@pytest.mark.parametrize("name", [f for f in FILES if "tmem_alloc(" in source(f) and "pdl_" in source(f) and f != "ptx_sm100.cuh"])
def test_dependents_may_start_once_the_tensor_memory_is_held(name):
    """A kernel that lets its successor start first may find that the successor holds the columns and waits for its end."""
    text = source(name)
    held = re.findall(r"tmem_alloc\([^;]*;\s*pdl_trigger\(\);", text)
    assert len(held) == len(re.findall(r"tmem_alloc\(", text)) == len(re.findall(r"pdl_trigger\(\)", text)) > 0
