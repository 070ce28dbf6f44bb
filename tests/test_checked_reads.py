"""CPU check that the plan and join kernels read their arrays through the helpers that the checked build
tests (csrc/checked.cuh), so that running the suites on that build covers every one of those reads."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1812_09141_gb300", "csrc")
BARE = re.compile(r"__ldg\(|\b(?:I\.(?:probe_ids|cand_offsets|cand_ids|r_desc|s_desc)|J\.(?:probes|size_end|toff|post)"
                  r"|P\.desc|R)\s*\[")


def _code(name, start=None, end=None):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    if start:
        s = s[s.index(start):s.index(end)]
    return [line for line in s.splitlines() if not line.lstrip().startswith("//")]


@pytest.mark.parametrize("name,start,end", [
    ("plan.cu", None, None),
    ("signature.cuh", None, None),
    ("candgen.cu", "join_kernel(const", "// GroupJoin expansion"),
    ("verify.cu", "uint32_t warp_lookup(", "// Warp-cooperative merge of one pair"),
])
def test_no_read_passes_the_helpers_by(name, start, end):
    bare = [line.strip() for line in _code(name, start, end) if BARE.search(line) and "in_bounds(" not in line]
    assert bare == []
