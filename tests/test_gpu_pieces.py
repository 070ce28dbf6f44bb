"""ssj_verify_batches calls whose candidates are planned in several pieces (more than a wave of plan chunks,
about five million candidates): read by the kernels over the host link, copied piece by piece, or some
batches one way and some the other, with batches that begin and end inside pieces."""
import numpy as np
import pytest

import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu


def test_pieces_of_direct_and_copied_batches():
    import torch
    _build.build()
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()
    spec = synth.tiny_self_join(seed=7, n=3_000)
    spec.plant_frac, spec.plant_edits = 0.3, 2
    c = synth.collection(spec)
    rng = np.random.default_rng(7)
    ctx = ssj.ssj_create(0)
    try:
        h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
        batches = []
        for n in (6_000_001, 1, 33, 4_000_000, 3_000_007, 700):
            counts = rng.integers(0, 2_001, max(2, n // 1_000))
            counts = counts * n // max(int(counts.sum()), 1)
            counts[-1] += n - int(counts.sum())
            co = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
            pr = rng.integers(0, c.n, len(counts)).astype(np.uint32)
            batches.append((h, h, 1, 2, pin(pr), pin(co), pin(rng.integers(0, c.n, n).astype(np.uint32))))
        want = [ssj.triples_to_array(ssj.ssj_verify_batch(ctx, *b)) for b in batches]
        assert len(want[0]) > 1_000
        for direct in ([0] * 6, [1] * 6, [0, 1, 0, 1, 0, 1], [1, 0, 1, 0, 1, 0]):
            got = ssj.ssj_verify_batches(ctx, [b + (ssj.SSJ_HOST_DIRECT * d,) for b, d in zip(batches, direct)],
                                         caps=[len(w) for w in want])
            for g, w in zip(got, want):
                assert np.array_equal(ssj.triples_to_array(g), w), direct
        assert ssj.ssj_device_error(ctx) == 0
    finally:
        ssj.ssj_destroy(ctx)
