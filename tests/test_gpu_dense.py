"""Batches whose candidates mostly pass, on the profiled kernels: work that the lists of such a batch
cause beside the merges (passing over the pairs of work items, queueing) stays small."""
import numpy as np
import pytest

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    h = ssj.ssj_create(0, flags=ssj.SSJ_CTX_PROFILE)
    yield h
    ssj.ssj_destroy(h)


def cluster(ctx, size, n, seed=1):
    """n near-duplicates of `size` tokens each: any two of them share at least size - 2."""
    rng = np.random.default_rng(seed)
    toks = np.tile(np.arange(size), (n, 1))
    toks[np.arange(n), rng.integers(0, size, n)] = size + rng.integers(0, 3 * size, n)
    toks.sort(axis=1)
    return ssj.ssj_load_collection(ctx, np.arange(n + 1, dtype=np.uint64) * np.uint64(size),
                                   toks.reshape(-1).astype(np.uint32))


def lists(n, probes, each, seed=2):
    """A device batch: `probes` lists of `each` random candidates."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.arange(probes, device="cuda", dtype=torch.int32) % n,
            torch.arange(probes + 1, device="cuda", dtype=torch.int64) * each,
            torch.randint(0, n, (probes * each,), generator=g, device="cuda", dtype=torch.int32))


def kernel_ms(ctx, h, b, flags, p=3, q=5, reps=9):
    """Medians (plan, verify) of the kernels' times, and the count."""
    times = []
    for _ in range(reps + 2):
        n = ssj.ssj_verify_batch(ctx, h, h, p, q, *b, n_cands=len(b[2]),
                                 flags=flags | ssj.SSJ_DEVICE_PTRS | ssj.SSJ_COUNT_ONLY)
        times.append(ssj.ssj_profile_read(ctx)[1:])
    return np.median(np.array(times[2:]), axis=0), int(n)


@pytest.mark.parametrize("size", [4, 20])
def test_pairs_of_work_items_are_passed_over_quickly(ctx, size):
    """5e6 pairs, all of them in index items: as many as one thread per pair would verify in about the
    same time, so the verify kernel takes less than twice that (three times when every pair of the
    list was read by a warp of its own)."""
    h = cluster(ctx, size, 20_000)
    try:
        b = lists(20_000, 500, 10_000)
        items, n = kernel_ms(ctx, h, b, ssj.SSJ_EMIT_ALL)
        threads, _ = kernel_ms(ctx, h, b, ssj.SSJ_FORCE_THREAD)
        assert n > 0.99 * len(b[2])
        assert items[1] < 1.9 * threads[1], (items, threads)
    finally:
        ssj.ssj_unload_collection(ctx, h)


@pytest.mark.parametrize("probes,each", [(500, 10_000), (160_000, 31)])
def test_queueing_pairs_costs_about_as_much_as_testing_them(ctx, probes, each):
    """5e6 pairs of 20 tokens that are all queued, against as many that the signature test (a 32-byte
    record per candidate) drops: a queued pair writes 8 bytes more, so the plan kernel takes less than
    2.5 times as long (over three times when each pair's run was searched for twice)."""
    h = cluster(ctx, 20, 20_000)
    try:
        b = lists(20_000, probes, each)
        queued, n = kernel_ms(ctx, h, b, ssj.SSJ_EMIT_ALL)
        dropped, left = kernel_ms(ctx, h, b, 0, 99, 100)
        assert n > 0.99 * len(b[2]) and left < 0.01 * len(b[2])
        assert queued[0] < 2.5 * dropped[0], (queued, dropped)
    finally:
        ssj.ssj_unload_collection(ctx, h)


def test_short_runs_of_cut_lists_of_long_sets(ctx):
    """Lists of 1,000 pairs of 1,500 tokens that all pass: most of the runs that chunks and buffers cut
    them into become index items as if they were asked for, so the verify kernel takes at most 1.4
    times as long (1.7 when runs below 256 pairs were verified by a block per pair)."""
    h = cluster(ctx, 1_500, 4_000)
    try:
        b = lists(4_000, 2_000, 1_000)
        default, n = kernel_ms(ctx, h, b, 0)
        items, m = kernel_ms(ctx, h, b, ssj.SSJ_FORCE_INDEX)
        assert n == m > 0.99 * len(b[2])
        assert default[1] < 1.4 * items[1], (default, items)
    finally:
        ssj.ssj_unload_collection(ctx, h)
