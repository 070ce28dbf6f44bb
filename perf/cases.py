"""Timed cases: the verification work that a program has this library do.

Every case makes a seeded synthetic collection on the GPU (set sizes uniform or
lognormal, Zipf tokens, a share of near-duplicate sets), the prefix filter's
candidate pairs for it (the grouped batch that a filter hands to the library),
loads the collection once, and times one pass through a public entry point.
The shapes are those of the repository's benchmark and tests: all pairs of a
tiny collection, 200,000 short sets, 50,000 long sets, uneven independent
joins, a resident collection of 1,000,000 sets that serves batches.

Results come sorted where the entry point sorts (SSJ_SORTED); the order of
unsorted triples is unspecified, so the prepared launch's triples are put in
order on the device, as a consumer of several joins' results would.  Host
results are gathered into a buffer of the program's own.
"""
import math
import random

import numpy as np
import torch

import paper_1812_09141_gb300 as ssj

JACCARD, DICE, COSINE, OVERLAP = 0, 1, 2, 3
# the benchmark's thresholds
THRESHOLDS = [(3, 5), (13, 20), (7, 10), (3, 4), (4, 5), (17, 20), (9, 10), (19, 20)]
MAX_EXACT_LOOKUPS = 3_000_000_000  # token lookups of exact(): a few seconds


def _case(**kw):
    """A case with the defaults of the fields that it does not set."""
    c = {"call": "device",     # entry point, see run()
         "sets": 200_000,      # sets of the collection (of both collections of an R x S join)
         "r_sets": 0,          # R x S: the first r_sets sets are R, the others S; 0: self-join
         "law": "lognormal",   # set sizes: lognormal(mean, 0.6) or uniform in [lo, hi]
         "mean": 20.0, "lo": 2, "hi": 200,
         "zipf": 1.0, "vocab": 1_000_000,
         "dup": 0.01,          # share of sets that are edited copies of others
         "sim": JACCARD, "p": 3, "q": 5,
         "pairs": 0,           # most candidate pairs, cut as a run of probes (0: all of them)
         "all_pairs": False,   # every pair instead of the prefix filter's
         "raw": False,         # tokens are raw 32-bit values, renumbered by the library
         "room": 1 << 18,      # room for result triples (of one join of several)
         "instances": 1,       # independent joins (serving: batches) of one pass
         "shapes": 0}          # seed of the instances' shapes
    c.update(kw)
    return c


def listed():
    return [
        # a client checks a short candidate list from its own arrays: the smallest call, where latency counts
        _case(name="short_list_host", call="host", p=9, q=10, raw=True, pairs=10_000),
        # brute force over a tiny collection (no filter): every pair of 1,000 sets
        _case(name="tiny_all_pairs", sets=1_000, law="uniform", lo=5, hi=50, vocab=10_000, dup=0.05, p=4, q=5,
              all_pairs=True),
        # the ordinary join: the candidates of 200,000 short sets at a low threshold, on the device
        _case(name="short_sets"),
        # the same collection's size with Cosine, whose longer prefixes list many more candidates
        _case(name="short_sets_cosine", sets=100_003, sim=COSINE, p=7, q=10),
        # long documents: 50,000 sets of about 300 tokens, about 1e8 candidates; the largest pass
        _case(name="long_sets", sets=50_000, mean=300.0, lo=50, hi=2_000, zipf=0.8, vocab=100_000),
        # a join of two collections, only its size asked for (aggregation on top of the join), stream-ordered
        _case(name="rs_join_count", call="count", sets=250_000, r_sets=100_000, dup=0.1),
        # many independent joins of uneven shapes, prepared and tuned once, replayed as a graph
        _case(name="uneven_joins", call="multi", instances=48, shapes=1005, room=1 << 13),
        # the same kind of work in one call from pinned host arrays, results back on the host
        _case(name="uneven_joins_host", call="batches", instances=12, shapes=1006, room=1 << 14),
        # the whole join on the device, candidate generation included
        _case(name="self_join_short", call="self_join"),
        _case(name="self_join_long", call="self_join", sets=50_000, mean=300.0, lo=50, hi=2_000, zipf=0.8,
              vocab=100_000, p=4, q=5),
        # GroupJoin's candidates (groups of sets with equal prefixes) expanded and verified on the device
        _case(name="group_join", call="groups", sets=40_000, dup=0.2, p=4, q=5),
        # serving: batches of 1e3 to 1e6 pairs admitted one after another on a resident collection
        _case(name="serving", call="serve", sets=1_000_000, mean=12.0, vocab=2_000_000, p=7, q=10, instances=16,
              room=1 << 16),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng: random.Random):
    call = rng.choice(["device", "device", "device", "host", "count", "multi", "batches", "self_join", "groups",
                       "serve"])
    p, q = rng.choice(THRESHOLDS)
    mean = _log_uniform(rng, 8, 350)
    c = {"call": call, "p": p, "q": q, "mean": round(mean, 1), "lo": rng.choice([1, 2, 5]),
         "hi": int(min(2_000, rng.uniform(4, 9) * mean)) + 2, "zipf": round(rng.uniform(0.6, 1.1), 2),
         "vocab": int(_log_uniform(rng, 20_000, 2_000_000)), "dup": round(_log_uniform(rng, 0.02, 0.2), 3),
         "room": 1 << 21}
    most = 8_000_000 / mean  # sets: at most about 8e6 tokens
    if call in ("device", "host", "count"):
        c["sets"] = int(_log_uniform(rng, 15_000, min(250_000, most)))
        c["pairs"] = int(_log_uniform(rng, 300_000 if call == "count" else max(20_000, 1_500 * mean),
                                      2_000_000 if call == "host" else 30_000_000))
        c["sim"] = rng.choice([JACCARD, JACCARD, JACCARD, DICE, COSINE, OVERLAP])
        if c["sim"] == OVERLAP:
            c["p"], c["q"] = rng.randint(max(6, int(mean * 0.5)), max(8, int(mean * 0.9))), 1
            c["zipf"] = min(c["zipf"], 0.9)
        if rng.random() < 0.3:
            c["r_sets"] = int(c["sets"] * rng.uniform(0.2, 0.6))
        elif rng.random() < 0.3:
            c["raw"] = True
    elif call in ("multi", "batches"):
        c = {"call": call, "instances": rng.randint(4, 32), "shapes": rng.randrange(1 << 20), "dup": 0.03,
             "room": 1 << 18}
    elif call == "serve":
        c["sets"] = int(_log_uniform(rng, 50_000, max(60_000, min(500_000, most))))
        c["instances"] = rng.randint(4, 24)
        c["room"] = 1 << 18
    else:
        c["p"], c["q"] = rng.choice(THRESHOLDS[2:])
        c["mean"] = round(min(mean, 150.0), 1)
        c["hi"] = int(min(c["hi"], 900))
        c["zipf"] = round(rng.uniform(0.6, 1.0), 2)
        c["vocab"] = max(c["vocab"], 100_000)
        c["sets"] = int(_log_uniform(rng, 4_000, 60_000 if call == "self_join" else 25_000))
    return _case(**c)


# ----------------------------------------------------------------------------------------------
# inputs (torch only): collections and the prefix filter's candidates
# ----------------------------------------------------------------------------------------------

def _generator(*seeds):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.SeedSequence(seeds).generate_state(1, np.uint64)[0] >> np.uint64(1)))
    return g


def _zipf(g, cdf, n):
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, u).clamp_(max=len(cdf) - 1)


def _collection(g, n, law, mean, lo, hi, zipf, vocab, dup):
    """(offsets, tokens, raw tokens): token sets as ranks in ascending global frequency, each set ascending;
    raw: the same entries as scattered 32-bit values."""
    dev = "cuda"
    if law == "uniform":
        size = torch.randint(lo, hi + 1, (n,), generator=g, device=dev)
    else:
        z = torch.randn(n, generator=g, device=dev, dtype=torch.float64)
        size = torch.exp(math.log(mean) - 0.18 + 0.6 * z).round_().clamp_(lo, hi).long()
    size.clamp_(max=vocab // 2)
    cdf = torch.cumsum(torch.arange(1, vocab + 1, device=dev, dtype=torch.float64).pow_(-zipf), 0)
    ids = torch.arange(n, device=dev)
    keys = torch.empty(0, dtype=torch.int64, device=dev)
    for k in range(10):  # draws until the sets hold their sizes in distinct tokens
        have = torch.bincount(keys // vocab, minlength=n)
        short = (size - have).clamp_(min=0)
        if k and not bool((short > 0).any()):
            break
        rows = torch.repeat_interleave(ids, torch.where(short > 0, (short * 1.2 * 1.5 ** k).long() + 1, 0))
        keys = torch.unique(torch.cat([keys, rows * vocab + _zipf(g, cdf, len(rows))]))
    rows = keys // vocab  # drop what a set holds too much, at random
    mix = torch.randperm(len(keys), generator=g, device=dev)
    mix = mix[torch.argsort(rows[mix], stable=True)]
    start = torch.cumsum(torch.bincount(rows, minlength=n), 0) - torch.bincount(rows, minlength=n)
    keys = keys[mix][torch.arange(len(keys), device=dev) - start[rows[mix]] < size[rows[mix]]]
    copies = int(n * dup)
    if copies:  # the last sets of a random order become copies of others, about one token dropped and one added
        perm = torch.randperm(n, generator=g, device=dev)
        src = torch.full((n,), -1, dtype=torch.int64, device=dev)
        src[perm[n - copies:]] = perm[torch.randint(0, n - copies, (copies,), generator=g, device=dev)]
        keys = torch.sort(keys).values
        rows = keys // vocab
        cnt = torch.bincount(rows, minlength=n)
        start = torch.cumsum(cnt, 0) - cnt
        dst = (src >= 0).nonzero().squeeze(1)
        m = cnt[src[dst]]
        row = torch.repeat_interleave(dst, m)
        at = torch.arange(len(row), device=dev) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
        copied = row * vocab + keys[start[src[row]] + at] % vocab
        keep = torch.rand(len(row), generator=g, device=dev) * torch.repeat_interleave(m, m) >= 1
        keys = torch.unique(torch.cat([keys[src[rows] < 0], copied[keep], dst * vocab + _zipf(g, cdf, len(dst))]))
    rows, toks = keys // vocab, keys % vocab
    freq = torch.bincount(toks, minlength=vocab)
    order = torch.argsort(freq, stable=True)
    rank = torch.empty_like(order)
    rank[order] = torch.arange(vocab, device=dev) - int((freq == 0).sum())
    keys = torch.sort(rows * vocab + rank[toks]).values
    offs = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    offs[1:] = torch.cumsum(torch.bincount(keys // vocab, minlength=n), 0)
    toks = keys % vocab
    raw = torch.sort((keys // vocab << 32) + (order[toks + int((freq == 0).sum())] * 2654435761 + 97) % (1 << 32))
    return offs, toks, raw.values % (1 << 32)


def _least(sim, p, q, n):
    """Least overlap of a set of n tokens with any set that reaches the threshold."""
    if sim == DICE:
        return (n * p + 2 * q - p - 1) // (2 * q - p)
    if sim == COSINE:
        return (n * p * p + q * q - 1) // (q * q)
    if sim == OVERLAP:
        return torch.full_like(n, -(-p // q))
    return (n * p + q - 1) // q


def _candidates(g, offs, toks, r_sets, sim, p, q, pairs):
    """The prefix filter's grouped batch (probe ids, offsets, candidate ids); a run of probes of at most about
    `pairs` index matches if that is not 0.  R x S: R is the sets below r_sets, S the others (ids from 0)."""
    dev, n = offs.device, len(offs) - 1
    size = offs[1:] - offs[:-1]
    least = _least(sim, p, q, size)
    prefix = torch.where((least <= size) & (size > 0), size - least + 1, 0)
    prefix = torch.minimum(prefix, size)
    lo_id = r_sets
    order = torch.argsort(size[lo_id:], stable=True) + lo_id  # the indexed sets by size
    n_s = len(order)
    s_size = size[order]
    if r_sets:
        probes = torch.argsort(size[:r_sets], stable=True)
        hi = torch.searchsorted(least[order].contiguous(), size[probes].contiguous(), right=True)
    else:
        probes = order
        hi = torch.arange(n_s, device=dev)  # earlier sets only
    low = torch.searchsorted(s_size, least[probes].contiguous())

    def entries(of):  # (position in `of`, token) of the sets' prefixes
        m = prefix[of]
        row = torch.repeat_interleave(torch.arange(len(of), device=dev), m)
        at = torch.arange(len(row), device=dev) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
        return row, toks[offs[of[row]] + at]

    srow, stok = entries(order)
    index = torch.sort(stok * n_s + srow).values
    rrow, rtok = entries(probes)
    first = torch.searchsorted(index, rtok * n_s + low[rrow])
    count = (torch.searchsorted(index, rtok * n_s + hi[rrow]) - first).clamp_(min=0)
    if pairs:
        per = torch.zeros(len(probes), dtype=torch.int64, device=dev).scatter_add_(0, rrow, count)
        total = torch.cumsum(per, 0)
        whole = int(total[-1]) if len(total) else 0
        begin = int(torch.randint(0, max(whole - pairs, 0) + 1, (1,), generator=g, device=dev))
        a = int(torch.searchsorted(total, begin, right=True))
        b = max(int(torch.searchsorted(total, begin + pairs, right=True)), a + 1)
        pick = (rrow >= a) & (rrow < b)
        rrow, first, count = rrow[pick], first[pick], count[pick]
    which = torch.repeat_interleave(torch.arange(len(rrow), device=dev), count)
    at = torch.arange(len(which), device=dev) - (torch.cumsum(count, 0) - count)[which]
    found = index[first[which] + at] % n_s + rrow[which] * n_s
    del which, at
    found = torch.unique(found)
    k, per = torch.unique_consecutive(found // n_s, return_counts=True)
    out = torch.zeros(len(k) + 1, dtype=torch.int64, device=dev)
    out[1:] = torch.cumsum(per, 0)
    return probes[k].int(), out, (order[found % n_s] - lo_id).int()


def _all_pairs(n):
    i, j = torch.triu_indices(n, n, 1, device="cuda")
    offs = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    offs[1:] = torch.cumsum(torch.bincount(i, minlength=n), 0)
    return torch.arange(n, device="cuda", dtype=torch.int32), offs, j.int()


def _joins(case, seed):
    """The joins of a case: a list of dicts with the collection and the candidate batch (serving: several batches)."""
    if case["call"] in ("multi", "batches"):
        rng, specs = random.Random(case["shapes"]), []
        for _ in range(case["instances"]):
            mean = _log_uniform(rng, 8, 500)
            n = int(_log_uniform(rng, 500, min(50_000, 20_000_000 / mean)))
            p, q = rng.choice(THRESHOLDS)
            specs.append(dict(case, sets=n, law="lognormal", mean=mean, lo=2, hi=max(2, int(min(4 * mean, 2_000))),
                              zipf=rng.uniform(0.6, 1.1), vocab=100_000, p=p, q=q))
    else:
        specs = [case]
    joins = []
    for i, c in enumerate(specs):
        g = _generator(seed, i)
        offs, toks, raw = _collection(g, c["sets"], c["law"], c["mean"], c["lo"], c["hi"], c["zipf"], c["vocab"],
                                      c["dup"])
        j = {"offs": offs, "toks": toks, "raw": raw, "p": c["p"], "q": c["q"]}
        if c["all_pairs"]:
            j["batch"] = _all_pairs(c["sets"])
        elif c["call"] == "serve":
            rng = random.Random(c["sets"] + c["instances"])
            j["batches"] = [_candidates(g, offs, toks, 0, c["sim"], c["p"], c["q"], int(_log_uniform(rng, 1e3, 1e6)))
                            for _ in range(c["instances"])]
        elif c["call"] != "self_join" and c["call"] != "groups":
            j["batch"] = _candidates(g, offs, toks, c["r_sets"], c["sim"], c["p"], c["q"], c["pairs"])
        joins.append(j)
    return joins


# ----------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ----------------------------------------------------------------------------------------------

_shared = {}


def _context():
    """The program's context, on a stream of its own, for as long as the program runs."""
    if not _shared:
        _shared["stream"] = torch.cuda.Stream()
        _shared["ctx"] = ssj.ssj_create(0, max_inflight=8, stream=_shared["stream"].cuda_stream)
    return _shared["ctx"]


def _u32(t):
    return t.to(torch.int64).cpu().numpy().astype(np.uint32)


class _State:
    """Collections and launches of one state, given back with it."""

    def __init__(self):
        self.colls, self.multi = [], None

    def load(self, offs, toks, flags=0):
        h = ssj.ssj_load_collection(_context(), offs.cpu().numpy().astype(np.uint64), _u32(toks), flags)
        self.colls.append(h)
        return h

    def __del__(self):
        try:
            if self.multi is not None:
                ssj.ssj_multi_destroy(_context(), self.multi)
            for h in self.colls:
                ssj.ssj_unload_collection(_context(), h)
        except Exception:  # the interpreter is going down
            pass


def _pinned(batch):
    """A batch as page-locked host arrays."""
    pr, co, ci = (t.cpu().pin_memory().numpy() for t in batch)
    return pr.view(np.uint32), co.view(np.uint64), ci.view(np.uint32)


def prepare(case, seed):
    s = _State()
    s.case, call, ctx = case, case["call"], _context()
    s.flags = case["sim"] << 8
    joins = _joins(case, seed)
    for j in joins:
        if case["r_sets"]:  # R x S: tokens in their joint order
            cut = case["r_sets"]
            at = int(j["offs"][cut])
            j["R"] = s.load(j["offs"][:cut + 1], j["toks"][:at])
            j["S"] = s.load(j["offs"][cut:] - at, j["toks"][at:])
        elif case["raw"]:
            j["R"] = j["S"] = s.load(j["offs"], j["raw"], ssj.SSJ_RENUMBER_BY_FREQ)
        else:
            j["R"] = j["S"] = s.load(j["offs"], j["toks"])
    j = joins[0]
    s.ids = (j["R"], j["S"], case["p"], case["q"])
    if call == "host":
        s.batch = tuple(t.cpu().numpy() for t in j["batch"])
    elif call in ("device", "count"):
        s.batch = j["batch"]
        s.n_cands = len(s.batch[2])
        s.out = torch.zeros((case["room"], 3), dtype=torch.int32, device="cuda")
        s.count = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        ssj.ssj_reserve(ctx, len(s.batch[0]), s.n_cands)
    elif call == "batches":
        s.batches = [(j["R"], j["S"], j["p"], j["q"], *_pinned(j["batch"]), s.flags | ssj.SSJ_SORTED) for j in joins]
        s.caps = [case["room"]] * len(joins)
    elif call == "multi":
        keep = [(j["R"], j["S"], j["p"], j["q"], *j["batch"], len(j["batch"][2])) for j in joins]
        torch.cuda.synchronize()
        s.keep = keep
        s.out = torch.zeros((len(keep), case["room"], 3), dtype=torch.int32, device="cuda")
        s.owner = torch.arange(len(keep), device="cuda")[:, None] << 40
        s.count = torch.zeros(len(keep), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        s.multi = ssj.ssj_multi_create(ctx, [ssj.DeviceBatch(*b[:7], b[7], flags=s.flags) for b in keep], list(s.out),
                                       [case["room"]] * len(keep), s.count)
        ssj.ssj_multi_autotune(ctx, s.multi, reps=3)
    elif call == "groups":
        s.groups = ssj.group_candidates(j["offs"].cpu().numpy(), _u32(j["toks"]), case["p"], case["q"], case["sim"])
    elif call == "serve":
        s.batches = [_pinned(b) for b in j["batches"]]
    if call not in ("device", "count", "multi"):
        s.host = np.zeros((case["instances"], case["room"], 3), dtype=np.int32)
        s.counts = np.zeros(case["instances"], dtype=np.int64)
    torch.cuda.synchronize()
    return s


def _gather(s, i, triples):
    s.counts[i] = len(triples)
    s.host[i, :len(triples)] = triples.view(np.int32).reshape(-1, 3)


def run(s):
    ctx, call, room = _context(), s.case["call"], s.case["room"]
    if call == "device":
        n = ssj.ssj_verify_batch(ctx, *s.ids, *s.batch, n_cands=s.n_cands, out=s.out, cap=room,
                                 flags=s.flags | ssj.SSJ_SORTED | ssj.SSJ_DEVICE_PTRS)
        return {"counts": n, "triples": s.out}
    if call == "count":
        ssj.ssj_verify_batch_async(ctx, *s.ids, *s.batch, s.n_cands, None, 0, s.count,
                                   flags=s.flags | ssj.SSJ_COUNT_ONLY)
        return {"counts": s.count}
    if call == "multi":
        ssj.ssj_multi_graph_launch(ctx, s.multi)
        with torch.cuda.stream(_shared["stream"]):  # every join's triples in order: (join, r, s) and the overlap
            key = s.owner + (s.out[:, :, 0].long() << 20) + s.out[:, :, 1]
            key, at = torch.sort(key.view(-1))
            return {"counts": s.count, "pairs": key, "overlaps": s.out.view(-1, 3)[at, 2]}
    out = {"counts": s.counts, "triples": s.host}
    if call == "host":
        _gather(s, 0, ssj.ssj_verify_batch(ctx, *s.ids, *s.batch, flags=s.flags | ssj.SSJ_SORTED, cap=room))
    elif call == "batches":
        for i, t in enumerate(ssj.ssj_verify_batches(ctx, s.batches, s.caps)):
            _gather(s, i, t)
    elif call == "groups":
        t, out["pairs"] = ssj.ssj_verify_groups(ctx, s.ids[0], s.ids[2], s.ids[3], s.groups, s.flags | ssj.SSJ_SORTED,
                                                room)
        _gather(s, 0, t)
    elif call == "self_join":
        t, out["pairs"] = ssj.ssj_self_join(ctx, s.ids[0], s.ids[2], s.ids[3], s.flags | ssj.SSJ_SORTED, room)
        _gather(s, 0, t)
    else:  # serving: admit while there is room, collect in order
        flying = []
        for i, b in enumerate(s.batches):
            while (t := ssj.ssj_submit(ctx, *s.ids, *b, flags=s.flags | ssj.SSJ_SORTED)) is None:
                _collect(s, *flying.pop(0))
            flying.append((i, t))
        for i, t in flying:
            _collect(s, i, t)
    return out


def _collect(s, i, ticket):
    ssj.ssj_poll(_context(), ticket, -1)
    _gather(s, i, ssj.ssj_results(_context(), ticket))


def work(case):
    """Batch arrays and the tokens (with a descriptor each) of the sets that the batch names, read once; the triples,
    few beside them, are left out.  Integer compares: no floating-point operations."""
    total = 0
    for j in _joins(case, 0):
        size = j["offs"][1:] - j["offs"][:-1]
        batches = j.get("batches") or ([j["batch"]] if "batch" in j else [])
        named = torch.zeros(len(size), dtype=torch.bool, device=size.device)
        for pr, co, ci in batches:
            named[pr.long()] = True
            named[ci.long() + case["r_sets"]] = True
            total += 4 * len(pr) + 8 * len(co) + 4 * len(ci)
        if not batches:
            named[:] = True
        total += 4 * int(size[named].sum()) + 8 * int(named.sum())
    return {"bytes": total, "flops": 0}


# ----------------------------------------------------------------------------------------------
# the same results in plain torch
# ----------------------------------------------------------------------------------------------

def _verified(j, batch, case):
    """Triples of one batch, sorted by (r, s), from a lookup of every candidate's tokens in its probe's set."""
    pr, co, ci = batch
    offs, toks = j["offs"], j["toks"]
    size, width = offs[1:] - offs[:-1], int(toks.max()) + 1 if len(toks) else 1
    keys = torch.repeat_interleave(torch.arange(len(size), device=offs.device), size) * width + toks
    r = torch.repeat_interleave(pr.long(), co[1:] - co[:-1])
    s = ci.long() + case["r_sets"]
    o = torch.zeros(len(s), dtype=torch.int64, device=offs.device)
    ends = torch.cumsum(size[s], 0)
    a = 0
    while a < len(s):
        b = max(int(torch.searchsorted(ends, (int(ends[a - 1]) if a else 0) + 200_000_000, right=True)), a + 1)
        m = size[s[a:b]]
        row = torch.repeat_interleave(torch.arange(b - a, device=offs.device), m)
        at = torch.arange(len(row), device=offs.device) - (torch.cumsum(m, 0) - m)[row]
        key = r[a:b][row] * width + toks[offs[s[a:b][row]] + at]
        hit = keys[torch.searchsorted(keys, key).clamp_(max=len(keys) - 1)] == key
        o[a:b].scatter_add_(0, row, hit.long())
        a = b
    x, y, p, q = size[r], size[s], j["p"], j["q"]
    if case["sim"] == DICE:
        ok = 2 * q * o >= p * (x + y)
    elif case["sim"] == COSINE:
        ok = (q * o) * (q * o) >= p * p * x * y
    elif case["sim"] == OVERLAP:
        ok = q * o >= p
    else:
        ok = o * (p + q) >= p * (x + y)
    ok &= (x > 0) & (y > 0)
    s = s - case["r_sets"]
    if not case["r_sets"]:
        r, s = torch.minimum(r, s), torch.maximum(r, s)
    t = torch.stack([r[ok], s[ok], o[ok]], 1)
    return t[torch.argsort((t[:, 0] << 32) + t[:, 1])]


def exact(case, seed):
    joins, call = _joins(case, seed), case["call"]
    lookups = 0
    for j in joins:
        if call in ("self_join", "groups"):
            j["batch"] = _candidates(None, j["offs"], j["toks"], 0, case["sim"], case["p"], case["q"], 0)
        size = j["offs"][1:] - j["offs"][:-1]
        for b in j.get("batches") or [j["batch"]]:
            lookups += int(size[b[2].long() + case["r_sets"]].sum())
    if lookups > MAX_EXACT_LOOKUPS:
        return None
    found = [_verified(j, b, case) for j in joins for b in j.get("batches") or [j["batch"]]]
    counts = torch.tensor([len(t) for t in found])
    if call == "count":
        return {"counts": counts}
    room = torch.zeros((len(found), case["room"], 3), dtype=torch.int64)
    for i, t in enumerate(found):
        room[i, :len(t)] = t.cpu()
    if call == "device":
        return {"counts": int(counts[0]), "triples": room[0].int()}
    if call == "multi":
        key, at = torch.sort(((torch.arange(len(found))[:, None] << 40) + (room[:, :, 0] << 20) + room[:, :, 1]).view(-1),
                             stable=True)
        return {"counts": counts, "pairs": key, "overlaps": room.view(-1, 3)[at, 2].int()}
    out = {"counts": counts.numpy(), "triples": room.numpy().astype(np.int32)}
    if call in ("self_join", "groups"):
        out["pairs"] = len(joins[0]["batch"][2])
    return out
