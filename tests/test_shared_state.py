"""CPU check that state which several threads' calls share is atomic or locked: a plain function-local
static that launches write would be a data race between serving threads."""
import glob
import os
import re

from conftest import ROOT

# a variable: no parenthesis (of a function or a static_assert) before its initialiser, extent or end
STATIC = re.compile(r"^\s+static\s+(?!const\b|constexpr\b|std::atomic)[^(]*[=;\[{]")


def test_function_local_statics_are_atomic_or_constant():
    bare = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_1812_09141_gb300", "csrc", "*"))):
        with open(path) as f:
            bare += [f"{os.path.basename(path)}: {line.strip()}" for line in f if STATIC.match(line)]
    assert bare == []
