"""Prefix sums of the collection layout and of the group expansion at the edges of their tiles (4,096
values) and of the tiles whose totals each block sums itself (1,024): sets found where they were put,
and every pair of the groups expanded."""
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
    h = ssj.ssj_create(0)
    yield h
    ssj.ssj_destroy(h)


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 3 * 4096, 1024 * 4096, 1024 * 4096 + 1])
def test_layout(ctx, n):
    sizes = 1 + np.arange(n, dtype=np.uint64) * 7 % 9
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    r = ssj.ssj_load_collection(ctx, offs, np.arange(offs[-1], dtype=np.uint32))
    ids = np.unique(np.concatenate([np.arange(min(n, 2000)), n - 1 - np.arange(min(n, 2000)),
                                    np.random.default_rng(n).integers(0, n, 1000)]))
    sub = sizes[ids]
    s_offs = np.concatenate([[0], np.cumsum(sub)]).astype(np.uint64)
    s_toks = np.repeat(offs[ids] - s_offs[:-1], sub.astype(np.int64)) + np.arange(s_offs[-1], dtype=np.uint64)
    s = ssj.ssj_load_collection(ctx, s_offs, s_toks.astype(np.uint32))
    try:
        k = np.arange(len(ids), dtype=np.uint32)
        got = ssj.ssj_verify_batch(ctx, r, s, 1, 1, ids.astype(np.uint32), np.arange(len(ids) + 1, dtype=np.uint64), k,
                                   flags=ssj.SSJ_SORTED, cap=len(ids))
        assert np.array_equal(ssj.triples_to_array(got), np.stack([ids, k, sub], 1).astype(np.uint32))
    finally:
        ssj.ssj_unload_collection(ctx, r)
        ssj.ssj_unload_collection(ctx, s)


@pytest.mark.parametrize("n_groups,n_probe_groups", [(1, 0), (2730, 1364), (2730, 1365), (2731, 1365), (20000, 9999)])
def test_groups(ctx, n_groups, n_probe_groups):
    """Groups of two sets, groups 2 m and 2 m + 1 of four equal ones, some of them candidates of each other."""
    n = 2 * n_groups
    toks = (3 * (np.arange(n)[:, None] // 4) + np.arange(3)).astype(np.uint32)
    h = ssj.ssj_load_collection(ctx, 3 * np.arange(n + 1, dtype=np.uint64), toks.reshape(-1))
    m = np.arange(n_probe_groups)
    g = ssj.Groups(2 * np.arange(n_groups + 1, dtype=np.uint64), np.arange(n, dtype=np.uint32), 2 * m + 1,
                   np.arange(n_probe_groups + 1, dtype=np.uint64), 2 * m, n_groups + 4 * n_probe_groups)
    try:
        got, pairs = ssj.ssj_verify_groups(ctx, h, 1, 1, g, ssj.SSJ_SORTED)
    finally:
        ssj.ssj_unload_collection(ctx, h)
    inner = 2 * np.arange(n_groups)[:, None] + [0, 1]
    cross = (4 * m[:, None, None] + [[0, 2], [1, 2], [0, 3], [1, 3]]).reshape(-1, 2)  # (min id, max id)
    want = np.concatenate([inner, cross])
    want = want[np.lexsort((want[:, 1], want[:, 0]))]
    assert pairs == len(want)
    assert np.array_equal(ssj.triples_to_array(got), np.column_stack([want, np.full(len(want), 3)]).astype(np.uint32))
