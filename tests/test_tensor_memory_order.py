"""Order of tensor-memory allocation and programmatic launch in the pre-LLM chain, read
from the kernels' source (CPU only).

A kernel of the chain lets the next one start while it runs, and that one may take
tensor memory and keep it while it waits for this grid to complete. A CTA that has let
it start and still wants tensor memory could then wait for ever (neither wait has a
limit), so every kernel of the chain must hold its tensor memory, block-wide, before it
lets the next one start. (The head-score kernels are followed by kernels that hold no
tensor memory and that pass the start on only after their own wait.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_25332_gb300", "csrc")
KERNELS = [("similarity_tc.cu", "crit_gram_tc"), ("similarity_tc.cu", "relevance_fused_tc"),
           ("similarity_tc.cu", "merge_argmax_tc"), ("merge_pair_tc.cu", "merge_argmax_pair_tc")]


def _body(file, kernel):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    m = re.search(r"__global__[^{;]*\b" + kernel + r"\(", src)
    assert m, kernel
    i = src.index("{", m.end())
    depth = 0
    for j in range(i, len(src)):
        depth += (src[j] == "{") - (src[j] == "}")
        if depth == 0:
            return src[i:j]
    raise AssertionError(kernel)


@pytest.mark.parametrize("file,kernel", KERNELS)
def test_tensor_memory_is_held_before_the_next_kernel_may_start(file, kernel):
    body = _body(file, kernel)
    alloc = re.search(r"\btmem_alloc\w*\(", body).end()
    held = re.search(r"__syncthreads\(\)|\bpair_cluster_sync\(\)", body[alloc:])
    assert held, "a barrier must publish the allocation"
    for m in re.finditer(r"\bpdl_allow_next\(\)|launch_dependents", body):
        assert m.start() > alloc + held.end(), f"{kernel} lets the next kernel start before it holds its tensor memory"


def test_every_kernel_with_tensor_memory_is_known():
    """A new kernel that allocates tensor memory is added to the list above, or to the
    head-score kernels, which need no such order."""
    found = set()
    for f in os.listdir(CSRC):
        if f.endswith(".cu") and not f.startswith("head_scores"):
            src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for k in re.findall(r"__global__[^{;]*?\b(\w+)\(const", src):
                if "tmem_alloc" in _body(f, k):
                    found.add((f, k))
    assert found == set(KERNELS)
