"""The plan kernel against the oracle where it can go wrong: every record class (and none), two
collections of different classes, probes without candidates, lists that end around the 32-candidate
rounds and the chunks, and probes whose near-duplicates all pass (early flushes, every kind of
work item).  Results are integers and must be equal."""
import numpy as np
import pytest

import oracle
import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu

SIMS = [(0, 3, 5), (0, 9, 10), (1, 4, 5), (2, 7, 10), (3, 9, 1)]


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    h = ssj.ssj_create(0)
    yield h
    ssj.ssj_destroy(h)


def _sets(rng, n, size, vocab, spread=0.5):
    """Random sets of about `size` tokens; every third is an edited copy of an earlier one."""
    out = []
    for i in range(n):
        if i % 3 == 2 and len(out[i // 2]):
            s = set(out[i // 2])
            for _ in range(rng.integers(0, 3 + size // 8)):
                s.discard(int(rng.choice(list(s)))) if s and rng.random() < 0.5 else s.add(int(rng.integers(vocab)))
        else:
            k = max(0, int(size * np.exp(spread * rng.standard_normal())))
            s = set(int(x) for x in rng.choice(vocab, min(k, vocab // 2), replace=False))
        out.append(sorted(s))
    return synth.from_lists(out)


def _check(ctx, cr, cs, hr, hs, b, sim, p, q):
    want = oracle.sort_triples(oracle.verify_batch(cr.offsets, cr.tokens, cs.offsets, cs.tokens, hr == hs, p, q,
                                                   b.probe_ids, b.cand_offsets, b.cand_ids, sim=sim))
    got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, hr, hs, p, q, b.probe_ids, b.cand_offsets, b.cand_ids,
                                                    flags=sim << 8))
    assert np.array_equal(got, want), (sim, p, q, len(got), len(want))
    return len(want)


@pytest.mark.parametrize("size", [1, 20, 100, 130, 250, 300, 600, 700, 1400, 4500])
def test_record_classes(ctx, size):
    rng = np.random.default_rng(size)
    c = _sets(rng, 160 if size < 1000 else 60, size, max(60, 8 * size), 0.1 if size > 1000 else 0.5)
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    try:
        found = [_check(ctx, c, c, h, h, synth.all_pairs_batch(c.n), *s) for s in SIMS]
        assert found[0] > 0
    finally:
        ssj.ssj_unload_collection(ctx, h)


@pytest.mark.parametrize("small,large", [(20, 200), (150, 400), (300, 5000)])
def test_two_collections_of_different_classes(ctx, small, large):
    rng = np.random.default_rng(small)
    big = _sets(rng, 80, large, 8 * large, 0.2)
    lists = [sorted(rng.choice(t, max(1, len(t) * 2 // 3), replace=False).tolist()) if i % 2 and len(t) else
             rng.choice(8 * large, small, replace=False).tolist() for i, t in
             enumerate(big.tokens[big.offsets[i]:big.offsets[i + 1]] for i in range(big.n))]
    lists = [sorted(int(x) for x in s) for s in lists] + [sorted(int(x) for x in rng.choice(8 * large, small, replace=False))
                                                          for _ in range(2000)]
    c = synth.from_lists(lists)
    hb, hc = ssj.ssj_load_collection(ctx, big.offsets, big.tokens), ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    try:
        for cr, cs, hr, hs in ((big, c, hb, hc), (c, big, hc, hb)):
            b = synth.random_batch(3, cr.n, cs.n, 120, 90)
            b = synth.Batch(np.concatenate([b.probe_ids, np.arange(80, dtype=np.uint32)]),
                            np.concatenate([b.cand_offsets, b.cand_offsets[-1] + np.arange(1, 81, dtype=np.uint64)]),
                            np.concatenate([b.cand_ids, np.arange(80, dtype=np.uint32)]))
            assert _check(ctx, cr, cs, hr, hs, b, 0, 3, 5) > 0
            _check(ctx, cr, cs, hr, hs, b, 2, 3, 5)
    finally:
        ssj.ssj_unload_collection(ctx, hb)
        ssj.ssj_unload_collection(ctx, hc)


@pytest.mark.parametrize("total", [1, 31, 32, 33, 64, 255, 256, 257, 1025, 80_000, 300_000])
@pytest.mark.parametrize("lists", ["one", "ones", "gaps"])
def test_list_ends_and_empty_probes(ctx, total, lists):
    """`total` candidates in one list, in lists of one, or in lists of 0 to 70 with runs of up to 200
    probes without candidates."""
    rng = np.random.default_rng(total)
    c = synth.collection(synth.tiny_self_join(n=600))
    if lists == "one":
        counts = np.array([total])
    elif lists == "ones":
        counts = np.ones(total, dtype=np.int64)
    else:
        counts, left = [], total
        while left:
            counts += [0] * int(rng.choice([0, 0, 1, 31, 32, 33, 200]))
            counts.append(min(int(rng.choice([1, 2, 31, 32, 33, 70])), left))
            left -= counts[-1]
        counts = np.array(counts + [0] * 40)
    offs = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
    b = synth.Batch(rng.integers(0, c.n, len(counts)).astype(np.uint32), offs,
                    rng.integers(0, c.n, total).astype(np.uint32))
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    try:
        _check(ctx, c, c, h, h, b, 0, 1, 10)
        _check(ctx, c, c, h, h, b, 3, 1, 1)
    finally:
        ssj.ssj_unload_collection(ctx, h)


@pytest.mark.parametrize("size", [12, 100, 300, 1100])
@pytest.mark.parametrize("raw", [False, True])
def test_probes_whose_candidates_all_pass(ctx, size, raw):
    """A cluster of near-duplicates: nothing is dropped, so chunks flush early and runs of every
    length become pairs, lane, block and index items (raw token values: no index items)."""
    rng = np.random.default_rng(size)
    base = rng.choice(4 * size, size, replace=False)
    n = 700
    lists = []
    for _ in range(n):
        s = set(int(x) for x in base)
        s.discard(int(base[rng.integers(size)]))
        s.add(int(rng.integers(4 * size)))
        lists.append(sorted((x * 2_654_435_761 + 7) & 0xFFFFFFFF if raw else x for x in s))
    c = synth.from_lists(lists)
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    counts = np.array([n, 1, 7, 15, 16, 17, n, 255, 256, 300, 0, n, 3] + [n] * 20)
    offs = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
    cands = np.concatenate([rng.permutation(n)[:k] for k in counts]).astype(np.uint32)
    b = synth.Batch(rng.integers(0, n, len(counts)).astype(np.uint32), offs, cands)
    try:
        assert _check(ctx, c, c, h, h, b, 0, 3, 5) > 0.9 * len(cands)
        _check(ctx, c, c, h, h, b, 2, 19, 20)
    finally:
        ssj.ssj_unload_collection(ctx, h)


@pytest.mark.parametrize("mean", [1, 12, 45, 700])
@pytest.mark.parametrize("size", [12, 300])
def test_offsets_that_fall_back_are_an_error(ctx, mean, size):
    """Offsets that are not nondecreasing, in batches whose chunks take several rounds: the call
    ends with SSJ_EINVAL (every round must still move on), and a valid batch works afterwards."""
    rng = np.random.default_rng(10 * mean + size)
    c = _sets(rng, 100, size, 20 * size)
    total = 1_000_000
    offs = np.sort(rng.integers(0, total + 1, total // mean + 1)).astype(np.uint64)
    offs[0], offs[-1] = 0, total
    good = synth.Batch(rng.integers(0, c.n, len(offs) - 1).astype(np.uint32), offs,
                       rng.integers(0, c.n, total).astype(np.uint32))
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    try:
        for back in (1, 5, 31, 200):
            bad = offs.copy()
            for at in rng.integers(len(offs) // 2, len(offs) - 1, 50):
                bad[at] = offs[int(at) - back] - 1 if back < 200 else offs[int(at)] // 2
            assert (np.diff(bad.astype(np.int64)) < 0).any()
            with pytest.raises(ssj.SsjError) as ei:
                ssj.ssj_verify_batch(ctx, h, h, 3, 5, good.probe_ids, bad, good.cand_ids)
            assert ei.value.status == ssj.SSJ_EINVAL
        _check(ctx, c, c, h, h, good, 0, 19, 20)
    finally:
        ssj.ssj_unload_collection(ctx, h)
