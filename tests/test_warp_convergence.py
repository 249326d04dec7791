"""Warp-wide (.aligned) instructions that stand behind code which lanes leave one by one, read from the source: a warp
that is still split executes them more than once, which for a TMEM release is a trap on the device."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_3751_gb300", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("wrapper", ["tmem_alloc", "tmem_dealloc", "tmem_alloc_pair", "tmem_dealloc_pair",
                                     "tmem_ld_32x32b_x32", "cluster_sync"])
def test_wrapper_reconverges_its_warp_first(wrapper):
    body = re.search(r"void %s\([^{]*\{(.*?)\n\}" % wrapper, _source("ptx_sm100.cuh"), flags=re.S).group(1)
    assert ".aligned" in body and body.lstrip().startswith("__syncwarp();")


@pytest.mark.parametrize("instruction", ["tcgen05.alloc", "tcgen05.dealloc", "tcgen05.ld", "barrier.cluster"])
def test_kernels_use_the_wrappers(instruction):
    for name in sorted(os.listdir(CSRC)):
        assert name == "ptx_sm100.cuh" or instruction not in _source(name), name
