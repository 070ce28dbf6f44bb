"""CPU restatement of the set records at the sizes that the library uses (csrc/ssj_internal.h compiled for
the host) and of the saturated header: a set of 65,535 tokens or more has length 65,535 and loss 0 there,
and no pair with it is dropped."""
import os
import random
import shutil
import subprocess

import pytest

import oracle
from conftest import ROOT

BITS = [224, 480, 992, 2016]
SATURATED = 65_535

HARNESS = r'''
#include <cstdio>
#include "ssj_internal.h"
int main() {
    for (uint32_t c = 0; c < ssj::kRecClasses; ++c) printf("%u %u\n", ssj::rec_sectors(c), ssj::rec_bits(c));
    return 0;
}
'''


def test_bitmap_sizes_are_the_librarys(tmp_path):
    cuda = next((d for d in ("/usr/local/cuda", os.path.dirname(os.path.dirname(shutil.which("nvcc") or "")))
                 if os.path.exists(os.path.join(d, "include", "cuda_runtime.h"))), None)
    if cuda is None:
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1812_09141_gb300", "csrc"),
                           "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe)])
    rows = [tuple(map(int, r.split())) for r in subprocess.check_output([str(exe)], text=True).splitlines()]
    assert rows == [(1 << c, b) for c, b in enumerate(BITS)]


def _record(tokens, bits):
    m = 0
    for t in tokens:
        m |= 1 << (((t * 0x9E3779B1 & 0xFFFFFFFF) * bits) >> 32)
    n = len(tokens)
    return (SATURATED, 0, m) if n >= SATURATED else (n, n - m.bit_count(), m)


def _kept(r, s, p, q, sim):
    (nr, loss_r, mr), (ns, loss_s, ms) = r, s
    if SATURATED in (nr, ns):
        return True
    return oracle.sim_pass((mr & ms).bit_count() + min(loss_r, loss_s), nr, ns, p, q, sim)


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("sim", [0, 1, 2, 3])
def test_no_pair_that_passes_is_dropped(bits, sim):
    rng = random.Random(bits + sim)
    for _ in range(150):
        p, q = rng.choice([(3, 5), (4, 5), (19, 20), (1, 2), (999, 1000)]) if sim != 3 else (rng.randint(1, bits), 1)
        base = rng.sample(range(100_000), rng.choice([1, 20, bits // 2, bits, 3 * bits]))
        r = set(base)
        s = set(rng.sample(base, rng.randint(0, len(base)))) | set(rng.sample(range(100_000), rng.randint(0, 8)))
        if s and oracle.sim_pass(len(r & s), len(r), len(s), p, q, sim):
            assert _kept(_record(r, bits), _record(s, bits), p, q, sim)


@pytest.mark.parametrize("sizes", [(65_534, 65_534), (65_534, 65_535), (65_535, 65_535), (65_534, 70_000), (70_000, 70_000)])
def test_saturated_headers(sizes):
    """Headers fit their 16 bits up to 65,534 tokens; from 65,535 on the bound, too small there, is not used."""
    a, b = sizes
    r, s = _record(range(a), 224), _record(range(b), 224)
    for n, loss, m in (r, s):
        assert n <= SATURATED and loss < 1 << 16 and (n < SATURATED or loss == 0)
    assert _kept(r, s, 9, 10, 0)
    bound = (r[2] & s[2]).bit_count() + min(r[1], s[1])
    assert (bound < min(a, b)) == (max(a, b) >= SATURATED)
