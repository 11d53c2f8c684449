"""Rules of the kernel sources that neither the compiler nor a run shows broken."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_28726_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", FILES)
def test_dynamic_shared_memory_declares_its_alignment(name):
    """Dynamic shared memory is read in 16-byte words: without a declared alignment
    it starts wherever the static part ends.  (head_attn aligns its base itself.)"""
    for decl in re.findall(r"extern\s+__shared__[^;]*;", code(name)):
        assert "__align__(16)" in decl or "ha_raw" in decl, decl


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_loads_of_the_callers_data(name):
    """Kernels are resident before the kernel ahead of them has ended, so what that
    one may write is not read through the path for read-only memory.  The scorer
    head's weights may be: its row kernels start once what precedes the call is
    complete."""
    found = re.findall(r"[^\n]*(?:__ldg\s*\(|ld\.global\.nc|__restrict__)[^\n]*", code(name))
    if name == "pr_head.cuh":
        found = [f for f in found
                 if not re.search(r"a\.lnext|\bL \+ H|__ldg\(wout|ht_copy_w", f)]
    assert not found, found
