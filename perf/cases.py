"""The work a user of the library has it do, as cases that can be timed.

Every case is one recording session's work through the public entry points: mining a
recording level by level, counting a candidate set (relaxed, exact or two-pass), many
recordings in one batch, window frequencies, a live recording that grows in chunks, and
requests to the server.  The sizes come from the repository's named workloads
(``synth``), its tests and its benchmark; ``draw`` spreads over the ranges between them.

The recordings are Poisson spike trains with embedded chains (and, for a bursting
culture, network bursts) like those of ``synth``, drawn here from the seed alone and
sorted on the GPU, so that an hour of spikes is ready in a moment.
"""
import math

import numpy as np
import torch

from paper_0905_2200_gb300 import fem

# Interval sets in microseconds: of the recordings, of a bursting culture (its last one
# has hi < 2 lo) and of the 5 ms cascade.
INTERVALS = {
    "ms4": [[0, 2000], [2000, 5000], [5000, 10000], [10000, 20000]],
    "burst": [[0, 2000], [2000, 5000], [5000, 10000], [15000, 20000]],
    "cascade": [[4000, 6000]],
}


# ----------------------------------------------------------------------------- cases
def listed():
    return [
        # A first look at a small culture: one 10 s recording, loaded and mined.  All latency.
        dict(name="mine_10s", kind="mine", types=16, seconds=10.0, rate=20.0, bursts=False,
             intervals="cascade", theta=15, max_len=4),
        # The benchmark's recording: five minutes of 64 neurons at five times chance.
        dict(name="mine_300s", kind="mine", types=64, seconds=300.0, rate=20.0, bursts=False,
             intervals="ms4", theta=1177, max_len=6),
        # The same recording searched down to a low support: millions of level-3 candidates.
        dict(name="mine_300s_deep", kind="mine", types=64, seconds=300.0, rate=20.0, bursts=False,
             intervals="ms4", theta=300, max_len=6),
        # A short list of hypotheses checked on a short recording: the smallest two-pass call.
        dict(name="two_pass_100", kind="two_pass", types=16, seconds=10.0, rate=20.0, bursts=False,
             intervals="ms4", theta=15, m=100, min_len=2, max_len=4),
        # A network-bursting culture, whose bursts overfill the counters' lists.
        dict(name="two_pass_bursts", kind="two_pass", types=64, seconds=300.0, rate=5.0, bursts=True,
             intervals="burst", theta=903, m=36000, min_len=2, max_len=4),
        # An hour-long recording against 100,000 candidates: the largest single call.
        dict(name="two_pass_hour", kind="two_pass", types=64, seconds=3600.0, rate=50.0,
             bursts=False, intervals="ms4", theta=8151, m=100000, min_len=3, max_len=5),
        # Exact counts of every ordered pair with every interval (a connectivity map).
        dict(name="exact_pairs", kind="count", exact=True, types=64, seconds=300.0, rate=20.0,
             bursts=False, intervals="ms4", m=0, min_len=2, max_len=2),
        # Upper bounds of a mixed candidate list, every length, on a ragged recording.
        dict(name="relaxed_mixed", kind="count", exact=False, types=37, seconds=171.3, rate=31.0,
             bursts=False, intervals="ms4", m=20011, min_len=2, max_len=8),
        # The alternative measure: window frequencies of every pair, 40 ms windows.
        dict(name="windows_pairs", kind="windows", types=64, seconds=300.0, rate=20.0, bursts=False,
             intervals="ms4", m=0, min_len=2, max_len=2, window_us=40000),
        # An archive of recordings of uneven length, counted in one batch.
        dict(name="batch_48", kind="batch", recordings=48, max_seconds=600.0, max_m=20000,
             min_len=2, max_len=8),
        # A live recording: a minute of history, then chunks of 100 ms, each followed by the
        # exact counts of a watched set.
        dict(name="live", kind="live", types=60, seconds=60.0, rate=20.0, intervals="ms4",
             chunks=8, m=1000, min_len=2, max_len=4),
        # The server with a burst of one-shot requests over its streams' last minute.
        dict(name="serve_16", kind="serve", streams=8, seconds=70.0, requests=16, max_m=50000,
             min_len=2, max_len=6),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _chance(rate, seconds, window_s, power=1):
    return rate * seconds * (1 - math.exp(-rate * window_s)) ** power


def draw(rng):
    kind = rng.choice(["mine", "mine", "two_pass", "two_pass", "count", "count", "windows",
                       "batch", "live", "serve"])
    types, rate = rng.randint(16, 64), rng.uniform(5.0, 50.0)
    if kind == "mine":
        seconds = min(round(_log(rng, 10.0, 300.0), 2), 6000.0 / rate)
        # at least 1.5 times the chance count of three nodes, as the deep search has
        theta = max(15, math.ceil(_log(rng, 1.27, 5.0) * _chance(rate, seconds, 0.002)),
                    math.ceil(1.52 * _chance(rate, seconds, 0.010, 2)))
        return dict(kind=kind, types=types, seconds=seconds, rate=rate, bursts=False,
                    intervals=rng.choice(["ms4", "ms4", "cascade"]), theta=theta,
                    max_len=rng.randint(4, 6))
    if kind in ("two_pass", "count"):
        bursts = kind == "two_pass" and rng.random() < 0.25
        seconds = round(_log(rng, 10.0, 300.0 if bursts or kind == "count" else 3600.0), 2)
        rate = 5.0 if bursts else rate
        lo = rng.randint(2, 6)
        hi = rng.randint(lo, 4 if bursts and lo <= 4 else 8)
        lo, hi = (2, 4) if bursts else (lo, hi)
        m = int(_log(rng, 100, 36000 if bursts else 100000))
        # no more (candidate, event) work than the hour's, 100,000 x 4 x 180,000
        m = max(100, min(m, int(7.2e10 / ((lo + hi) / 2 * rate * seconds))))
        case = dict(kind=kind, types=types, seconds=seconds, rate=rate, bursts=bursts,
                    intervals="burst" if bursts else "ms4", m=m, min_len=lo, max_len=hi)
        if kind == "count":
            return dict(case, exact=rng.random() < 0.5)
        mean = rate + (12.5 if bursts else 0.0)
        return dict(case, theta=max(2, math.ceil(5 * _chance(mean, seconds, 0.002, lo - 1))))
    if kind == "windows":
        # (an edge holds at most 32 pending entries: no types that fire far less than others)
        lo = rng.randint(2, 4)
        return dict(kind=kind, types=rng.randint(32, 64), seconds=round(_log(rng, 10.0, 300.0), 2),
                    rate=rng.uniform(20.0, 50.0), bursts=False, intervals="ms4",
                    m=int(_log(rng, 100, 8000)), min_len=lo,
                    max_len=rng.randint(lo, 4), window_us=rng.randint(20000, 100000))
    if kind == "batch":
        lo = rng.randint(2, 6)
        return dict(kind=kind, recordings=rng.randint(5, 48), max_seconds=round(_log(rng, 30.0, 600.0), 2),
                    max_m=int(_log(rng, 1000, 20000)), min_len=lo, max_len=rng.randint(lo, 8))
    if kind == "live":
        lo = rng.randint(2, 4)
        return dict(kind=kind, types=rng.randint(16, 128), seconds=round(_log(rng, 6.0, 60.0), 2),
                    rate=rng.uniform(10.0, 100.0), intervals="ms4", chunks=rng.randint(2, 12),
                    m=int(_log(rng, 100, 4000)), min_len=lo, max_len=rng.randint(lo, 5))
    lo = rng.randint(2, 4)
    return dict(kind=kind, streams=rng.randint(1, 8), seconds=round(rng.uniform(20.0, 70.0), 2),
                requests=rng.randint(1, 16), max_m=int(_log(rng, 1000, 50000)), min_len=lo,
                max_len=rng.randint(lo, 6))


# ---------------------------------------------------------------------------- inputs
def _recording(rng, types, seconds, rate, intervals, bursts=False, chains=8):
    """(types uint8[n], times uint32[n]) on the GPU, sorted by time (ties by type):
    Poisson firing at `rate` (one number, or one per type), embedded chains of 4 to 6
    nodes at 1 to 3 Hz and, if asked, network bursts (0.5 Hz, 50 to 200 ms, every type
    at 200 Hz)."""
    span = int(round(seconds * 1e6))
    k = rng.poisson(np.broadcast_to(rate, types) * seconds)
    t = [rng.integers(0, span, int(k.sum()))]
    ty = [np.repeat(np.arange(types), k)]
    for _ in range(chains):
        nodes = rng.choice(types, size=int(rng.integers(4, 7)), replace=False)
        at = rng.integers(0, span, int(rng.poisson(rng.uniform(1.0, 3.0) * seconds)))
        for j, a in enumerate(nodes):
            if j:
                lo, hi = intervals[int(rng.integers(0, len(intervals)))]
                at = at + np.clip((lo + hi) // 2 + rng.integers(-500, 501, at.size), lo + 1, hi)
            t.append(at)
            ty.append(np.full(at.size, a))
    if bursts:
        for _ in range(int(rng.poisson(0.5 * seconds))):
            start, length = int(rng.integers(0, span)), int(rng.uniform(50e3, 200e3))
            k = rng.poisson(200.0 * length * 1e-6, types)
            t.append(start + rng.integers(0, length, int(k.sum())))
            ty.append(np.repeat(np.arange(types), k))
    key = torch.from_numpy(np.concatenate(t).astype(np.int64) * 256 + np.concatenate(ty)).cuda()
    key = key[key < span * 256].sort().values
    out = (key & 255).to(torch.uint8), (key >> 8).to(torch.int32)
    torch.cuda.synchronize()  # the library reads them on its context's own stream
    return out


def _candidates(rng, m, types, lo, hi, n_intervals):
    """uint8[m, 16] episode records on the GPU: lengths lo..hi in equal shares and random
    order, distinct types, random intervals; m = 0: every ordered pair with every
    interval, in order."""
    if m == 0:
        a, v, b = (x.reshape(-1) for x in np.meshgrid(np.arange(types), np.arange(n_intervals),
                                                      np.arange(types), indexing="ij"))
        keep = a != b
        rec = np.zeros((int(keep.sum()), 16), np.uint8)
        rec[:, 0], rec[:, 1], rec[:, 8], rec[:, 15] = a[keep], b[keep], v[keep], 2
        return torch.from_numpy(rec).cuda()
    length = rng.permutation(lo + np.arange(m) % (hi - lo + 1))
    order = torch.from_numpy(rng.random((m, types), dtype=np.float32)).cuda().argsort(dim=1)
    rec = np.zeros((m, 16), np.uint8)
    rec[:, :8] = order[:, :8].cpu().numpy()
    rec[:, 8:15] = rng.integers(0, n_intervals, (m, 7))
    at = np.arange(8)
    rec[:, :8][at >= length[:, None]] = 0
    rec[:, 8:15][at[:7] >= length[:, None] - 1] = 0
    rec[:, 15] = length
    return torch.from_numpy(rec).cuda()


def _sizes(case):
    """The sizes within a case that its numbers alone fix: each recording's or request's."""
    return np.random.default_rng([int(1000 * v) for _, v in sorted(case.items())
                                  if isinstance(v, (int, float))])


def _host(types, t):
    return types.cpu().numpy(), t.cpu().numpy().view(np.uint32)


ROWS = 1 << 16  # the table that a mining program keeps its episodes and their counts in


class _State:
    """What a program holds between calls; the handles are given back with it."""

    def __init__(self, case):
        self.case = case
        self.intervals = np.array(INTERVALS[case.get("intervals", "ms4")], np.uint32)
        self.batch = self.server = None
        self.found = np.zeros((ROWS, 20), np.uint8) if case["kind"] == "mine" else None
        self.ctx = fem.Context(torch.cuda.current_device())

    def __del__(self):
        if self.server:
            fem.fem_server_destroy(self.server)
        if self.batch:
            fem.fem_batch_destroy(self.batch)
        self.ctx.close()


def prepare(case, seed):
    s = _State(case)
    rng = np.random.default_rng(int(seed))
    kind, iv = case["kind"], s.intervals.astype(np.int64)
    if kind == "batch":
        jobs, sizes = [], _sizes(case)
        for _ in range(case["recordings"]):
            seconds = math.exp(sizes.uniform(math.log(10.0), math.log(case["max_seconds"])))
            types = int(sizes.integers(16, 65))
            rates = rng.uniform(5.0, 50.0, types)
            ty, t = _recording(rng, types, seconds, rates, iv, chains=4)
            m = int(math.exp(sizes.uniform(math.log(100), math.log(case["max_m"]))))
            rec = _candidates(rng, m, types, case["min_len"], case["max_len"], len(iv))
            sid = fem.fem_load_stream(s.ctx.h, ty, t, types)
            for n in range(case["min_len"], case["max_len"] + 1):
                own = rec[rec[:, 15] == n].contiguous()
                theta = max(2, math.ceil(5 * _chance(float(rates.mean()), seconds, 0.002, n - 1)))
                if len(own):
                    jobs.append(dict(stream_id=sid, len=n, theta=theta, cands=own))
        total = sum(len(j["cands"]) for j in jobs)
        s.counts = torch.zeros(total, dtype=torch.int32, device="cuda")
        s.survived = torch.zeros(total, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        at = 0
        for j in jobs:
            j["exact_out"] = s.counts[at:at + len(j["cands"])]
            j["survived_out"] = s.survived[at:at + len(j["cands"])]
            at += len(j["cands"])
        s.jobs = jobs
        s.batch = fem.fem_batch_create(s.ctx.h, jobs, s.intervals)
        return s
    if kind == "serve":
        s.server = fem.fem_server_create(s.ctx.h, mem_budget_bytes=8 << 30)
        streams, sizes = [], _sizes(case)
        for _ in range(case["streams"]):
            types, rate = int(sizes.integers(16, 129)), float(sizes.uniform(10.0, 100.0))
            ty, t = _host(*_recording(rng, types, case["seconds"], rate, iv, chains=4))
            sid = fem.fem_server_open_stream(s.server, types, len(t) + 16)
            fem.fem_server_append(s.server, sid, ty, t)
            streams.append((sid, types, rate))
        s.requests = []
        for _ in range(case["requests"]):
            sid, types, rate = streams[int(sizes.integers(0, len(streams)))]
            m = int(math.exp(sizes.uniform(math.log(1000), math.log(case["max_m"]))))
            rec = _candidates(rng, m, types, case["min_len"], case["max_len"], len(iv)).cpu().numpy()
            s.requests.append((sid, rec, math.ceil(5 * _chance(rate, min(60.0, case["seconds"]), 0.002,
                                                               case["min_len"] - 1))))
        fem.fem_server_drain(s.server)
        return s
    if kind == "live":
        tail = case["chunks"] * 0.1
        ty, t = _host(*_recording(rng, case["types"], case["seconds"] + tail, case["rate"], iv))
        cut = np.searchsorted(t, (case["seconds"] + np.arange(case["chunks"] + 1) * 0.1) * 1e6)
        s.chunks = [(ty[a:b], t[a:b]) for a, b in zip([0] + list(cut[:-1]), cut)]
        s.cands = _candidates(rng, case["m"], case["types"], case["min_len"], case["max_len"], len(iv))
        return s
    s.types, s.t = _recording(rng, case["types"], case["seconds"], case["rate"], iv, case["bursts"])
    if kind != "mine":
        s.sid = fem.fem_load_stream(s.ctx.h, s.types, s.t, case["types"])
        s.cands = _candidates(rng, case["m"], case["types"], case["min_len"], case["max_len"], len(iv))
        m = len(s.cands)
        s.counts = torch.zeros(m, dtype=torch.int64 if kind == "windows" else torch.int32, device="cuda")
        s.survived = torch.zeros(m, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------- one pass
def run(s):
    case, ctx, iv = s.case, s.ctx.h, s.intervals
    kind = case["kind"]
    if kind == "mine":
        sid = fem.fem_load_stream(ctx, s.types, s.t, case["types"])
        found = fem.fem_mine_levelwise(ctx, sid, iv, case["theta"], case["max_len"], raw=True)
        fem.fem_free_stream(ctx, sid)
        per_level, at = np.zeros(fem.MAX_LEN + 1, np.int64), 0
        for level, (records, counts) in found.items():
            end = at + len(counts)
            s.found[at:end, :16] = records
            s.found[at:end, 16:] = counts.view(np.uint8).reshape(-1, 4)
            per_level[level], at = len(counts), end
        return s.found, per_level
    if kind == "two_pass":
        return fem.fem_count_two_pass(ctx, s.sid, s.cands, iv, case["theta"],
                                      exact_out=s.counts, survived_out=s.survived)
    if kind == "count":
        return fem.fem_count_candidates(ctx, s.sid, s.cands, iv,
                                        fem.PASS_EXACT if case["exact"] else fem.PASS_RELAXED,
                                        out=s.counts)
    if kind == "windows":
        return fem.fem_count_windows(ctx, s.sid, s.cands, iv, case["window_us"], out=s.counts)
    if kind == "batch":
        fem.fem_batch_run(s.batch)
        return s.counts, s.survived
    if kind == "live":
        out = []
        sid = fem.fem_load_stream(ctx, *s.chunks[0], case["types"])
        for ty, t in s.chunks[1:]:
            fem.fem_append_stream(ctx, sid, ty, t)
            out.append(fem.fem_count_candidates(ctx, sid, s.cands, iv, fem.PASS_EXACT))
        fem.fem_free_stream(ctx, sid)
        return out
    ids = [fem.fem_server_submit(s.server, sid, rec, iv, theta, fem.REQ_ONESHOT, 60_000_000)
           for sid, rec, theta in s.requests]
    fem.fem_server_drain(s.server)
    out = []
    for rid, (_, rec, _) in zip(ids, s.requests):
        counts, flags, events, status = fem.fem_server_result(s.server, rid, len(rec))
        if status:
            raise fem.FemError(status, "fem_server_result")
        out.append((counts, flags))
        fem.fem_server_release(s.server, rid)
    return out


# ----------------------------------------------------------------------------- work
def work(case):
    """Bytes: the events (5 each), the candidate records (16) and the outputs, once.
    Operations: one integer update per (candidate, event of one of its types), the
    machines' steps; for mining, those of level 2's candidates (deeper levels depend on
    what is found)."""
    kind = case["kind"]
    mean_len = (case.get("min_len", 2) + case.get("max_len", 2)) / 2
    if kind == "batch":  # log-uniform lengths and set sizes, 16 to 64 types at 5 to 50 Hz
        seconds = (case["max_seconds"] - 10) / math.log(case["max_seconds"] / 10)
        m = (case["max_m"] - 100) / math.log(case["max_m"] / 100)
        r = case["recordings"]
        return dict(bytes=r * (5 * 40 * 27.5 * seconds + 21 * m), flops=r * m * mean_len * 27.5 * seconds)
    if kind == "serve":
        m = (case["max_m"] - 1000) / math.log(max(1.001, case["max_m"] / 1000))
        events = 72 * 55 * min(60.0, case["seconds"])
        return dict(bytes=case["streams"] * 5 * events + case["requests"] * 21 * m,
                    flops=case["requests"] * m * mean_len * events / 72)
    rate = case["rate"] + (12.5 if case.get("bursts") else 0.0)
    events = case["types"] * rate * case["seconds"]
    m = case.get("m", 0)
    if m == 0:
        m, mean_len = case["types"] * (case["types"] - 1) * len(INTERVALS[case["intervals"]]), 2
    times = case["chunks"] if kind == "live" else 1  # a watched set is counted at each chunk
    return dict(bytes=5 * events + times * 21 * m,
                flops=times * m * mean_len * rate * case["seconds"])


# ---------------------------------------------------------------------------- exact
def _count_one(where, t, rec, iv, exact):
    """Non-overlapped occurrences of one episode: the exact machine, whose node k keeps
    the times that may still be followed, or the relaxed one, which keeps the newest and
    asks no lower bound."""
    n = int(rec[15])
    nodes = [int(x) for x in rec[:n]]
    edges = [(int(iv[int(v)][0]), int(iv[int(v)][1])) for v in rec[8:7 + n]]
    at = np.concatenate([where[a] for a in nodes])
    node = np.repeat(np.arange(n), [len(where[a]) for a in nodes])
    order = np.argsort(at, kind="stable")
    lists, count = [[] for _ in range(n)], 0
    for k, now in zip(node[order].tolist(), t[at[order]].tolist()):
        if k:
            lo, hi = edges[k - 1] if exact else (-1, edges[k - 1][1])
            before = lists[k - 1] if exact else lists[k - 1][-1:]
            if not any(lo < now - x <= hi for x in before):
                continue
            if k == n - 1:
                count += 1
                lists = [[] for _ in range(n)]
                continue
        hi = edges[k][1]
        lists[k] = [x for x in lists[k] if now - x <= hi] + [now]
    return count


def exact(case, seed):
    """The counts from plain loops over the events, for cases small enough."""
    kind = case["kind"]
    if kind not in ("two_pass", "count") or work(case)["flops"] > 1.5e6:
        return None
    s = prepare(case, seed)
    ty, t = s.types.cpu().numpy(), s.t.cpu().numpy().view(np.uint32).astype(np.int64)
    where = [np.nonzero(ty == a)[0] for a in range(case["types"])]
    recs, iv = s.cands.cpu().numpy(), INTERVALS[case["intervals"]]
    if kind == "count":
        return np.array([_count_one(where, t, r, iv, case["exact"]) for r in recs], np.int64)
    kept = np.array([_count_one(where, t, r, iv, False) >= case["theta"] for r in recs])
    counts = [_count_one(where, t, r, iv, True) if k else 0 for r, k in zip(recs, kept)]
    return np.array(counts, np.int64), kept.astype(np.int64)
