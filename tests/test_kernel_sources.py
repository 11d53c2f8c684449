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
