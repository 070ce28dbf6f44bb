"""ssj_verify_batches with more batches than the CTAs that pack the results: every batch's own results,
and packing that grows with the number of batches, not with its square."""
import ctypes
import time

import numpy as np
import pytest

import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    import torch
    assert torch.cuda.is_available()
    _build.build()
    ctx = ssj.ssj_create(0)
    c = synth.collection(synth.tiny_self_join(n=200))
    h, g = (ssj.ssj_load_collection(ctx, c.offsets, c.tokens) for _ in range(2))
    yield ctx, h, g, c
    ssj.ssj_destroy(ctx)


class _Call:
    """A call of n batches of `each` candidates of one probe, as the C entry point takes it."""

    def __init__(self, setup, n, each, room, flags, seed=1):
        self.ctx, h, g, c = setup
        rng = np.random.default_rng(seed)
        self.probe = rng.integers(0, c.n, n).astype(np.uint32)
        self.cands = rng.integers(0, c.n, (n, each)).astype(np.uint32)
        self.offs = np.array([0, each], dtype=np.uint64)
        self.out = np.zeros((n, room + 1, 3), dtype=np.uint32)
        self.counts = (ctypes.c_uint64 * n)()
        self.batches = (ssj.ssj_batch * n)()
        for i in range(n):
            self.batches[i] = ssj.ssj_batch(h, g, 1, 2, 1, self.probe[i:].ctypes.data, self.offs.ctypes.data,
                                            self.cands[i].ctypes.data, each, flags)
        self.outs = (ctypes.c_void_p * n)(*[self.out[i].ctypes.data for i in range(n)])
        self.caps = (ctypes.c_uint64 * n)(*[room] * n)
        self.n = n

    def __call__(self):
        return ssj.lib().ssj_verify_batches(self.ctx, self.batches, self.n, self.outs, self.caps, self.counts)


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 2049, 5000])
@pytest.mark.parametrize("each", [3, 20])
def test_every_batch_gets_its_own_results(setup, n, each):
    c = setup[3]
    sets = [set(c.tokens[c.offsets[i]:c.offsets[i + 1]].tolist()) for i in range(c.n)]
    call = _Call(setup, n, each, each, ssj.SSJ_EMIT_ALL | ssj.SSJ_SORTED, seed=n)
    assert call() == ssj.SSJ_OK
    assert list(call.counts) == [each] * n
    for i in range(n):
        r, cands = int(call.probe[i]), sorted(call.cands[i].tolist())
        assert call.out[i, :each].tolist() == [[r, s, len(sets[r] & sets[s])] for s in cands]
        assert not call.out[i, each].any()


def test_packing_grows_with_the_batches(setup):
    """100,000 batches of one candidate: with room for results (packed on the device) against only
    counted, the call takes at most 15 ms longer (24 when each batch's CTA summed all counts
    before its own)."""
    best = {}
    for flags in (0, ssj.SSJ_COUNT_ONLY):
        call = _Call(setup, 100_000, 1, 1, flags)
        t = []
        for _ in range(7):
            a = time.perf_counter()
            assert call() == ssj.SSJ_OK
            t.append(time.perf_counter() - a)
        best[flags] = min(t[1:])
    assert best[0] - best[ssj.SSJ_COUNT_ONLY] < 0.015, best
