"""Bounded device waits leave no thread behind, read off the CUDA source (a
wait that runs out is never provoked on a GPU).

A lane whose wait runs out must not part from its warp before a warp-collective
instruction, and a CTA must not start its barriers with some of its threads
gone.  So in every kernel that uses tensor memory:
  - a wait on a barrier is made by one thread, by the whole warp with one
    answer (mbar_wait_warp), or is followed by __syncthreads_and before
    anything collective;
  - the word that stops a launch is read once per CTA (tc::stopped).
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1701_08475_gb300", "csrc")
TENSOR_FILES = ("screen.cu", "leaf_tc.cu", "join_tc.cu")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _blocks(text):
    """(position, condition) of the braces open at every position of interest: the text between the previous
    statement and each '{'."""
    stack, at = [], {}
    last = 0
    for i, ch in enumerate(text):
        if ch == "{":
            stack.append(text[last:i])
            last = i + 1
        elif ch == "}":
            if stack:
                stack.pop()
            last = i + 1
        elif ch == ";":
            last = i + 1
        at[i] = tuple(stack)
    return at


@pytest.mark.parametrize("name", TENSOR_FILES)
def test_a_wait_is_one_thread_s_or_the_whole_warp_s(name):
    text = _source(name)
    at = _blocks(text)
    calls = [m.start() for m in re.finditer(r"tc::mbar_wait\(", text)]
    assert calls
    for c in calls:
        one_thread = any(re.search(r"\b(lane|tid) == 0\b", cond) for cond in at[c])
        one_thread |= re.search(r"\btid == 0 \?", text[text.rfind("\n", 0, c):c]) is not None
        # else the next collective of the CTA takes the answers together
        rest = re.search(r"__syncthreads_and|__syncthreads|__syncwarp|tmem_ld|epi_all|epi_sync|mbar_arrive|_sync\(", text[c:])
        together = rest is not None and rest.group(0) == "__syncthreads_and"
        assert one_thread or together, "%s: %s" % (name, text[c:text.find(";", c)])


@pytest.mark.parametrize("name", TENSOR_FILES)
def test_a_cta_with_tensor_memory_returns_whole(name):
    text = _source(name)
    kernels = re.split(r"(?=__global__)", text)
    users = [k for k in kernels if "tmem_alloc" in k]
    assert users
    for k in users:
        head = k[:k.index("tmem_alloc")]
        assert "tc::stopped(" in head
        assert not re.search(r"\*\s*(P\.)?status\s*&\s*kStatusStop", head)
