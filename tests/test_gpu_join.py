"""ssj_self_join's probing kernel where it can go wrong, against the oracle's AllPairs join and its
candidate count: collections around a wave of warps and of every record class, windows of positions
beyond the bitmap (hash set and window by window), long index lists, clusters whose pairs all pass
(early flushes, a queue that has to grow), sizes beyond the shared-memory counting sort, forced
granularities (no signature test) and the positional filter."""
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


def _join(ctx, c, p, q, sim=0, flags=0, load=ssj.SSJ_RENUMBER_BY_FREQ, candidates=True):
    want, n_cands = oracle.allpairs_self(c.offsets, c.tokens, p, q, sim=sim)[:2]
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens, load)
    try:
        got, cands = ssj.ssj_self_join(ctx, h, p, q, (sim << 8) | flags)
        assert np.array_equal(ssj.triples_to_array(got), oracle.sort_triples(want)), (p, q, sim, flags)
        if candidates:
            assert cands == n_cands
        return len(want), cands
    finally:
        ssj.ssj_unload_collection(ctx, h)


@pytest.mark.parametrize("n", [0, 1, 2, 31, 33, 1000, 5000])
@pytest.mark.parametrize("sim,p,q", [(0, 3, 5), (1, 4, 5), (2, 7, 10), (3, 5, 1)])
def test_sizes_and_functions(ctx, n, sim, p, q):
    if n == 0:
        c = synth.from_lists([])
    else:
        spec = synth.short_sets(n=n)
        spec.plant_frac, spec.plant_edits = 0.3, 2
        c = synth.collection(spec)
    _join(ctx, c, p, q, sim)


@pytest.mark.parametrize("mean", [90, 200, 400, 800])
@pytest.mark.parametrize("flags", [0, ssj.SSJ_JOIN_POSITIONAL, ssj.SSJ_FORCE_WARP, ssj.SSJ_FORCE_LANE,
                                   ssj.SSJ_FORCE_BLOCK, ssj.SSJ_FORCE_INDEX])
def test_record_classes_and_granularities(ctx, mean, flags):
    spec = synth.long_sets(n=500)
    spec.a, spec.plant_frac, spec.plant_edits = float(mean), 0.3, 8
    assert _join(ctx, synth.collection(spec), 3, 5, flags=flags, candidates=flags != ssj.SSJ_JOIN_POSITIONAL)[0] > 0


@pytest.mark.parametrize("vocab", [80, 200_000])
def test_windows_beyond_the_bitmap(ctx, vocab):
    """70,000 sets of 3 to 6 tokens: up to 70,000 positions pass the length filter.  Few tokens: long
    lists, window by window; many: short lists, the hash set."""
    spec = synth.CollectionSpec(70_000, synth.SIZE_UNIFORM, 0, 0, 5, 6, 0.2, vocab, 77)
    c = synth.collection(spec)
    if vocab == 80:  # keep the oracle's work small: a high threshold has prefixes of one or two tokens
        _join(ctx, c, 9, 10)
    else:
        _join(ctx, c, 1, 2)


@pytest.mark.parametrize("size", [10, 120, 300])
def test_a_cluster_where_every_pair_passes(ctx, size):
    """2,500 near-duplicates: 3.1 million pairs pass, more than the queue's first size."""
    rng = np.random.default_rng(size)
    base = list(range(size))
    n = 2500 if size == 10 else 900
    c = synth.from_lists([sorted(base[:-1] + [size + int(rng.integers(3 * size))]) for _ in range(n)])
    found, cands = _join(ctx, c, 3, 5, load=0)
    assert found == cands == n * (n - 1) // 2


def test_sizes_beyond_the_shared_counters(ctx):
    rng = np.random.default_rng(5)
    lists = []
    for i, size in enumerate([4094, 4095, 4096, 4097, 5000, 9000, 3, 3, 2, 70, 4095, 4096]):
        s = set(int(x) for x in rng.choice(30_000, size, replace=False))
        lists += [sorted(s), sorted(set(list(s)[: size - size // 50]) | {30_001 + i})]
    _join(ctx, synth.from_lists(lists), 4, 5)
