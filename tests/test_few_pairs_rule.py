"""CPU check of the verify kernel's rule for few pairs (csrc/arith.h compiled for the host): a launch
with an instance that asks for one thread per pair never deals its pairs out one per warp."""
import os
import subprocess

from conftest import ROOT

HARNESS = r'''
#include <cstdint>
#include <cstdio>
#include <initializer_list>
#include "arith.h"
int main() {
    for (unsigned force = 0; force < 2; ++force)
        for (uint64_t n : {0ull, 1ull, 9727ull, 9728ull, 9729ull, 1ull << 40})
            for (uint64_t l : {0ull, 1ull, 5000ull, 9729ull})
                if (l <= n) printf("%u %llu %d\n", force, (unsigned long long)n, ssj::few_pairs(l, n - l, 4864, force) ? 1 : 0);
    return 0;
}
'''


def test_a_forced_thread_granularity_is_kept(tmp_path):
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1812_09141_gb300", "csrc"),
                           str(src), "-o", str(exe)])
    rows = [tuple(map(int, line.split())) for line in subprocess.check_output([str(exe)], text=True).splitlines()]
    assert len(rows) > 20
    for force, n, few in rows:
        assert few == (0 if force else int(n <= 2 * 4864)), (force, n, few)
