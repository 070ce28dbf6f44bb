"""Sets around the largest size that a record's header holds (65,534; 65,535 stands for that and more),
beside short sets that have the collection use records: near-duplicates of any such sizes are found, by
candidate batches and by the device's self-join, against the oracle."""
import numpy as np
import pytest

import oracle
import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu

VOCAB = 200_000


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    h = ssj.ssj_create(0)
    yield h
    ssj.ssj_destroy(h)


@pytest.fixture(scope="module")
def short():
    rng = np.random.default_rng(1)
    sets = [np.unique(rng.integers(0, VOCAB, 110)).tolist() for _ in range(26_000)]
    for i in range(0, 400, 2):
        sets[i] = sorted(set(sets[i + 1][3:]) | {int(rng.integers(VOCAB))})
    return sets


@pytest.mark.parametrize("a,b", [(65_534, 65_534), (65_534, 65_535), (65_535, 65_535), (65_535, 65_536), (65_534, 70_000)])
def test_near_duplicates_around_the_largest_header(ctx, short, a, b):
    rng = np.random.default_rng(a + b)
    order = rng.permutation(VOCAB)
    big = [sorted(order[:a].tolist()), sorted(order[500:b + 500].tolist())]
    sets = short + big
    sizes = np.array([len(s) for s in sets], dtype=np.float64)
    assert (sizes ** 2).sum() / sizes.sum() < 4_032  # the collection has records
    c = synth.from_lists(sets)
    n = c.n
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens, ssj.SSJ_RENUMBER_BY_FREQ)  # (the oracle's token order)
    try:
        # every set of a few hundred against the large ones and its neighbours
        pr = np.array([n - 1, n - 2] + list(range(400)), dtype=np.uint32)
        lists = [np.arange(n - 500, n), np.arange(n - 500, n)] + [np.array([i ^ 1, n - 1, n - 2, 7]) for i in range(400)]
        co = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.uint64)
        ci = np.concatenate(lists).astype(np.uint32)
        for sim, p, q in ((0, 9, 10), (0, 3, 5), (1, 9, 10), (2, 9, 10), (3, 60_000, 1)):
            want = oracle.sort_triples(oracle.verify_batch(c.offsets, c.tokens, c.offsets, c.tokens, True, p, q, pr, co, ci,
                                                           sim=sim))
            got = ssj.triples_to_array(ssj.ssj_verify_batch(ctx, h, h, p, q, pr, co, ci, flags=sim << 8))
            assert np.array_equal(got, want), (sim, p, q)
            assert (want[:, 0] == n - 2).any()
        want, cands = oracle.allpairs_self(c.offsets, c.tokens, 9, 10)[:2]
        got, found = ssj.ssj_self_join(ctx, h, 9, 10)
        assert np.array_equal(ssj.triples_to_array(got), oracle.sort_triples(want)) and found == cands
        assert (oracle.sort_triples(want)[:, 0] == n - 2).any()
    finally:
        ssj.ssj_unload_collection(ctx, h)
