"""Device memory after calls that take their own: what the library keeps mapped is bounded."""
import numpy as np
import pytest

import synth

import paper_1812_09141_gb300 as ssj
from paper_1812_09141_gb300 import _build

pytestmark = pytest.mark.gpu


def test_a_large_self_join_gives_its_memory_back():
    """Token values up to 2^27 make the prefix index take over 2 GB; afterwards the pool keeps at most
    256 MiB (and the workspace of a thousand sets, some 20 MB), and the next join finds the same pairs."""
    import torch
    _build.build()
    rng = np.random.default_rng(1)
    lists = [sorted(rng.choice(1 << 27, 20, replace=False).tolist()) for _ in range(1_000)]
    for i in range(0, 1_000, 2):
        lists[i] = sorted(set(lists[i + 1][:-1]) | {int(rng.integers(1 << 27))})
    c = synth.from_lists(lists)
    ctx = ssj.ssj_create(0)
    try:
        small = ssj.ssj_load_collection(ctx, c.offsets, c.tokens, ssj.SSJ_RENUMBER_BY_FREQ)
        want, _ = ssj.ssj_self_join(ctx, small, 4, 5, ssj.SSJ_SORTED)
        h = ssj.ssj_load_collection(ctx, c.offsets, c.tokens)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info(0)[0]
        for _ in range(2):
            got, _ = ssj.ssj_self_join(ctx, h, 4, 5, ssj.SSJ_SORTED)
            assert len(want) >= 400 and np.array_equal(got, want)
            assert free - torch.cuda.mem_get_info(0)[0] < (256 + 64) << 20
    finally:
        ssj.ssj_destroy(ctx)
