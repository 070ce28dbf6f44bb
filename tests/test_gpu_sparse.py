"""Batches that list many probes without candidates: every candidate finds its probe across any
stretch of empty lists, and the plan kernel does not walk them one after the other."""
import numpy as np
import pytest

import oracle
import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    ctx = ssj.ssj_create(0, flags=ssj.SSJ_CTX_PROFILE)
    c = synth.collection(synth.tiny_self_join(n=600))
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    yield ctx, c, h
    ssj.ssj_destroy(ctx)


@pytest.mark.parametrize("gaps", [[31, 32, 33], [95, 96, 97, 127, 128, 129], [1, 160, 161, 1023, 1024, 1025],
                                  [0, 40, 5_000, 100_000]])
@pytest.mark.parametrize("each", [[1], [1, 2, 31], [31, 32, 33, 63, 64, 65, 200]])
@pytest.mark.parametrize("flags", [0, ssj.SSJ_EMIT_ALL])
def test_stretches_of_empty_lists(setup, gaps, each, flags):
    ctx, c, h = setup
    rng = np.random.default_rng(len(gaps) * 10 + len(each))
    counts = []
    for _ in range(300):
        counts += [0] * int(rng.choice(gaps)) + [int(rng.choice(each))]
    counts = np.array(counts + [0] * int(rng.choice(gaps)))
    co = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
    pr = rng.integers(0, c.n, len(counts)).astype(np.uint32)
    ci = rng.integers(0, c.n, int(co[-1])).astype(np.uint32)
    got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, h, h, 3, 5, pr, co, ci, flags=flags))
    if flags:  # every pair but a set with itself
        sets = [set(c.tokens[c.offsets[i]:c.offsets[i + 1]].tolist()) for i in range(c.n)]
        r = np.repeat(pr, counts)
        rows = [(min(x, y), max(x, y), len(sets[x] & sets[y])) for x, y in zip(r.tolist(), ci.tolist()) if x != y]
        want = oracle.sort_triples(np.array(rows, np.uint32).reshape(-1, 3))
    else:
        want = oracle.sort_triples(oracle.verify_batch(c.offsets, c.tokens, c.offsets, c.tokens, True, 3, 5, pr, co, ci))
    assert np.array_equal(got, want)


def test_empty_lists_are_not_walked(setup):
    """2,000,000 probes with 1,000 candidates: less than four times the plan kernel's time with one
    candidate each (over ten times when a warp walked all empty lists between two candidates)."""
    import torch
    ctx, c, h = setup
    n = 2_000_000
    pr = torch.arange(n, device="cuda", dtype=torch.int32) % c.n
    ms = []
    for cands in (1_000, n):
        co = torch.arange(n + 1, device="cuda", dtype=torch.int64) * cands // n
        ci = torch.arange(cands, device="cuda", dtype=torch.int32) % c.n
        t = []
        for _ in range(11):
            ssj.ssj_verify_batch(ctx, h, h, 3, 5, pr, co, ci, n_cands=cands,
                                 flags=ssj.SSJ_DEVICE_PTRS | ssj.SSJ_COUNT_ONLY)
            t.append(ssj.ssj_profile_read(ctx)[1])
        ms.append(np.median(t[2:]))
    assert ms[0] < 4 * ms[1], ms
