"""SSJ_SORTED: results come back sorted by (r, s) at every size where the device sort changes its way
(one CTA's tile of 4,096, small tiles merged by sixteen, passes of two runs, odd runs) and where the
results stop coming along with their count (4,096; 16,384 for a group of ssj_verify_batches), through every
entry point.  A batch with
SSJ_EMIT_ALL lists as many results as it has pairs; repeated pairs are equal triples."""
import numpy as np
import pytest

import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu

SIZES = [0, 1, 2, 3, 64, 65, 4095, 4096, 4097, 5120, 5121, 8192, 8193, 12_289, 16_383, 16_384, 16_385,
         32_769, 70_000]


@pytest.fixture(scope="module")
def setup():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    ctx = ssj.ssj_create(0)
    c = synth.collection(synth.tiny_self_join(n=900))
    h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    g = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
    yield ctx, h, g, c
    ssj.ssj_destroy(ctx)


def _batch(n, seed):
    """n pairs of an R x S batch in lists of 0 to 60; some pairs repeat."""
    rng = np.random.default_rng(seed)
    counts = []
    while sum(counts) < n:
        counts.append(int(min(rng.integers(0, 61), n - sum(counts))))
    counts = np.array(counts + [0])
    pr = rng.integers(0, 900, len(counts)).astype(np.uint32)
    co = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
    ci = rng.integers(0, 900, n).astype(np.uint32)
    return pr, co, ci


def _want(c, b):
    pr, co, ci = b
    sets = [set(c.tokens[c.offsets[i]:c.offsets[i + 1]].tolist()) for i in range(c.n)]
    r = np.repeat(pr, np.diff(co.astype(np.int64)))
    t = np.array([(x, y, len(sets[x] & sets[y])) for x, y in zip(r.tolist(), ci.tolist())], np.uint32).reshape(-1, 3)
    return t[np.lexsort((t[:, 1], t[:, 0]))]


def _rows(t):
    return np.ascontiguousarray(t).view(np.uint32).reshape(-1, 3)


@pytest.mark.parametrize("n", SIZES)
def test_host_device_and_served_results_are_sorted(setup, n):
    import torch
    ctx, h, g, c = setup
    b = _batch(n, n)
    want = _want(c, b)
    fl = ssj.SSJ_EMIT_ALL | ssj.SSJ_SORTED
    assert np.array_equal(_rows(ssj.ssj_verify_batch(ctx, h, g, 1, 2, *b, flags=fl)), want)
    dev = [torch.from_numpy(x.astype(t)).cuda() for x, t in zip(b, (np.int32, np.int64, np.int32))]
    out = torch.full((n + 1, 3), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    got = ssj.ssj_verify_batch(ctx, h, g, 1, 2, *dev, n_cands=n, out=out, cap=n + 1, flags=fl | ssj.SSJ_DEVICE_PTRS)
    assert got == n and np.array_equal(out[:n].cpu().numpy().astype(np.uint32), want)
    assert int(out[n, 0]) == -1  # nothing past the results
    t = ssj.ssj_submit(ctx, h, g, 1, 2, *b, flags=fl)
    assert ssj.ssj_poll(ctx, t, -1)
    assert np.array_equal(_rows(ssj.ssj_results(ctx, t)), want)


@pytest.mark.parametrize("sizes", [[0, 3, 4096], [4097, 5, 0, 8193], [16_000, 384], [16_000, 385, 7], [9000, 9000, 9000]])
def test_several_batches_sorted_and_not(setup, sizes):
    ctx, h, g, c = setup
    bs = [_batch(n, 100 + i) for i, n in enumerate(sizes)]
    fl = [ssj.SSJ_EMIT_ALL | (ssj.SSJ_SORTED if i != 1 else 0) for i in range(len(sizes))]
    got = ssj.ssj_verify_batches(ctx, [(h, g, 1, 2, *b, f) for b, f in zip(bs, fl)])
    for i, (b, t) in enumerate(zip(bs, got)):
        rows = _rows(t)
        if i == 1:
            rows = rows[np.lexsort((rows[:, 1], rows[:, 0]))]
        assert np.array_equal(rows, _want(c, b))


def test_more_results_than_room_are_sorted_among_themselves(setup):
    import ctypes
    ctx, h, g, c = setup
    b = _batch(9000, 5)
    want = {tuple(x) for x in _want(c, b).tolist()}
    for cap in (1, 100, 4096, 5000):
        hb = ssj._make_batch(h, g, 1, 2, *b, ssj.SSJ_EMIT_ALL | ssj.SSJ_SORTED)
        out, n = np.zeros(cap + 1, dtype=ssj.TRIPLE_DTYPE), ctypes.c_uint64()
        assert ssj.lib().ssj_verify_batch(ctx, ctypes.byref(hb.batch), out.ctypes.data, cap, ctypes.byref(n)) == ssj.SSJ_ENOMEM
        rows = _rows(out[:cap])
        assert n.value == 9000 and {tuple(x) for x in rows.tolist()} <= want and out[cap]["r"] == 0
        assert np.array_equal(rows, rows[np.lexsort((rows[:, 1], rows[:, 0]))])
