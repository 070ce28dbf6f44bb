"""CPU restatement of the signature test that the plan kernel applies to every candidate: a
record holds |x|, the loss |x| - popcount and a bitmap of the tokens' hash values; with a the
common bits of two bitmaps, a + min(loss_r, loss_s) is never below |r n s| and never above
min(|r|, |s|), so the exact similarity test of that bound drops no pair that passes."""
import random

import pytest

import oracle

BITS = [192, 448, 960, 1984]  # the record classes' bitmaps


def _record(tokens, bits):
    m = 0
    for t in tokens:
        m |= 1 << (((t * 0x9E3779B1 & 0xFFFFFFFF) * bits) >> 32)
    return len(tokens), len(tokens) - m.bit_count(), m


@pytest.mark.parametrize("bits", BITS)
def test_the_bound_holds_for_every_overlap(bits):
    rng = random.Random(bits)
    for trial in range(300):
        vocab = rng.choice([40, 500, 100_000, 1 << 32])
        n = rng.choice([0, 1, 2, 3, 31, 33, bits // 2, bits, 2 * bits])
        r = set(rng.randrange(vocab) for _ in range(n))
        keep = rng.random()
        s = {t for t in r if rng.random() < keep} | set(rng.randrange(vocab) for _ in range(rng.randrange(n + 2)))
        lr, loss_r, mr = _record(sorted(r), bits)
        ls, loss_s, ms = _record(sorted(s), bits)
        bound = (mr & ms).bit_count() + min(loss_r, loss_s)
        assert len(r & s) <= bound <= min(lr, ls)


@pytest.mark.parametrize("sim", [0, 1, 2, 3])
def test_no_pair_that_passes_is_dropped(sim):
    rng = random.Random(100 + sim)
    for trial in range(400):
        p, q = rng.choice([(3, 5), (4, 5), (19, 20), (1, 2), (999, 1000)]) if sim != 3 else (rng.randint(1, 30), 1)
        base = rng.sample(range(3000), rng.randint(1, 60))
        r = set(base)
        s = set(rng.sample(base, rng.randint(0, len(base)))) | set(rng.sample(range(3000), rng.randint(0, 8)))
        if not s:
            continue
        (nr, loss_r, mr), (ns, loss_s, ms) = _record(sorted(r), 192), _record(sorted(s), 192)
        bound = (mr & ms).bit_count() + min(loss_r, loss_s)
        if oracle.sim_pass(len(r & s), nr, ns, p, q, sim):
            assert oracle.sim_pass(bound, nr, ns, p, q, sim)
