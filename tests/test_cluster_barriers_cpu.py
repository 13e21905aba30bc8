"""Cluster barriers in the CUDA sources (read as text, CPU only): barrier.cluster's .aligned forms are defined
only when all threads of a warp execute them together, so every place that issues one reconverges
its warp first, instead of leaving that to the compiler after code whose lanes diverge."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_29029_gb300" / "csrc"
FILES = sorted(p for p in CSRC.iterdir() if "barrier.cluster" in p.read_text())


def _code(text):
    """The source's statements one per line, without comments and blank lines."""
    lines = (re.sub(r"//.*", "", line).strip() for line in text.splitlines())
    return [line for line in lines if line]


@pytest.mark.parametrize("path", FILES, ids=[p.name for p in FILES])
def test_aligned_cluster_barriers_follow_a_syncwarp(path):
    code = _code(path.read_text())
    at = [i for i, line in enumerate(code) if "barrier.cluster" in line]
    assert at
    for i in at:
        assert ".aligned" in code[i]
        k = i - 1
        while "barrier.cluster" in code[k]:  # an arrive and its wait, one after the other
            k -= 1
        assert code[k] == "__syncwarp();", (path.name, code[k:i + 1])
