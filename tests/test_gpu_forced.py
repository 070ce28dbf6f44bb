"""Shapes that each path of the verify kernel has to get right, at counts of pairs where that path takes
them: tails of the last 16-byte block and extreme token values in more pairs than are dealt out one per
warp (one thread per pair, asked for or not), and a forced warp granularity's merge path around its
windows, with r whole in shared memory and without."""
import numpy as np
import pytest

import oracle
import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    h = ssj.ssj_create(0)
    yield h
    ssj.ssj_destroy(h)


def _all_ordered(n, times):
    """Every ordered pair of n sets, `times` times."""
    pr = np.tile(np.arange(n, dtype=np.uint32), times)
    return pr, np.arange(len(pr) + 1, dtype=np.uint64) * np.uint64(n), np.tile(np.arange(n, dtype=np.uint32), len(pr))


def _every(sets, b, p=0, q=1):
    """Triples of the batch (R x S), sorted, of the pairs with overlap / union at least p / q; empty
    sets only where every pair is asked for (p = 0)."""
    pr, co, ci = b
    rows = []
    py = [set(s) for s in sets]
    memo = {}
    for x, y in zip(np.repeat(pr, np.diff(co.astype(np.int64))).tolist(), ci.tolist()):
        if (x, y) not in memo:
            o = len(py[x] & py[y])
            keep = p == 0 or (py[x] and py[y] and o * (p + q) >= p * (len(py[x]) + len(py[y])))
            memo[x, y] = (x, y, o) if keep else None
        if memo[x, y]:
            rows.append(memo[x, y])
    return oracle.sort_triples(np.array(rows, np.uint32).reshape(-1, 3))


def _tails():
    top = 0xFFFFFFFF
    rng = np.random.default_rng(11)
    sets = [[], [0], [top], [0, top], [top - 1, top], [5, 6, 7, 8, 9], [4, 5, 6, 7], [4, 5, 6, 7, 8],
            [1, 2, 3, 4, 5, 6, 7, 8, 9], [3, 1 << 31, top], [1 << 31, top]]
    for n in range(1, 14):
        base = np.sort(rng.choice(40, size=n, replace=False)).tolist()
        sets += [base, sorted(set(base[:-1] + [top - n]))]
    return sets


@pytest.mark.parametrize("flags", [0, ssj.SSJ_FORCE_THREAD])
def test_tails_one_thread_per_pair(ctx, flags):
    sets = _tails()
    c = synth.from_lists(sets)
    h, g = (ssj.ssj_load_collection(ctx, c.offsets, c.tokens) for _ in range(2))
    try:
        few, many = _all_ordered(len(sets), 1), _all_ordered(len(sets), 12)
        assert len(many[2]) > 2 * 4864 + 5000 > 5000 > len(few[2])
        for b in (few, many):
            got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, h, g, 1, 2, *b, flags=flags | ssj.SSJ_EMIT_ALL))
            assert np.array_equal(got, _every(sets, b))
            for p, q in ((1, 1), (1, 2), (1, 100)):
                got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, h, g, p, q, *b, flags=flags))
                assert np.array_equal(got, _every(sets, b, p, q)), (p, q)
    finally:
        ssj.ssj_unload_collection(ctx, h)
        ssj.ssj_unload_collection(ctx, g)


@pytest.mark.parametrize("staging", [0, ssj.SSJ_BULK_STAGING])
@pytest.mark.parametrize("times", [1, 40])
def test_forced_warp_merges(ctx, times, staging):
    rng = np.random.default_rng(3)
    sets = [[], [7]]
    for n in (1, 4, 31, 128, 255, 256, 257, 511, 513, 1019, 1020, 1021, 1024, 1300):
        base = rng.choice(4_000, size=n, replace=False)
        sets += [sorted(base.tolist()), sorted(set(base[: n - n // 8].tolist()) | {4_001 + n})]
    c = synth.from_lists(sets)
    h, g = (ssj.ssj_load_collection(ctx, c.offsets, c.tokens) for _ in range(2))
    b = _all_ordered(len(sets), times)
    ssj.ssj_set_granularity(ctx, 0, 0, 0, 256 | staging)
    try:
        fl = ssj.SSJ_FORCE_WARP
        got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, h, g, 1, 2, *b, flags=fl | ssj.SSJ_EMIT_ALL))
        assert np.array_equal(got, _every(sets, b))
        for p, q in ((9, 10), (1, 2), (1, 100)):
            got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, h, g, p, q, *b, flags=fl))
            assert np.array_equal(got, _every(sets, b, p, q)), (p, q)
    finally:
        ssj.ssj_set_granularity(ctx, 0, 0, 0, 256)
        ssj.ssj_unload_collection(ctx, h)
        ssj.ssj_unload_collection(ctx, g)
