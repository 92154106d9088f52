"""Streams that are sparse on average and, in a burst, denser than the hit tables' words: the
tables are built and read before their build is found out, and the other kernels then count.
"""
import numpy as np
import pytest

import oracle
from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu
PASSES = (fem.PASS_RELAXED, fem.PASS_EXACT)
K = 16
I = np.array([[0, 5000], [0, 10000], [100, 12000], [15000, 40000]], np.uint32)


def burst_stream(seed, n=3000, seconds=10.0, bursts=2, first_us=0):
    """n events of K types over `seconds`; in each burst 100 of type 0, 400 us apart, one of type
    1 every 2 ms among them, and 20 of type 1 after them: 30 of type 0 in 12 ms, 100 in 40 ms,
    and the last 32 of them all less than 15 ms before the first type 1 that follows."""
    rng = np.random.default_rng(seed)
    ty, t = [rng.integers(0, K, n)], [rng.integers(0, int(seconds * 1e6), n)]
    for k in range(bursts):
        at = int(seconds * 1e6 * (k + 0.5) / bursts)
        ty += [np.zeros(100, int), np.ones(20, int), np.ones(20, int)]
        t += [at + 400 * np.arange(100), at + 1001 + 2000 * np.arange(20),
              at + 400 * 99 + 50 + 100 * np.arange(20)]
    ty, t = np.concatenate(ty), np.concatenate(t)
    order = np.argsort(t, kind="stable")
    return ty[order].astype(np.uint8), (t[order] + first_us).astype(np.uint32)


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    fem.fem_destroy(c)


def with_edge(cands, ivl):
    """The set with the candidates (0, I[0], 1) to (0, I[ivl], 1) first: with all four a type 1
    after a burst has more hits than the events of its slab."""
    L, E, iv = (a.copy() for a in cands)
    k = ivl + 1
    L[:k], E[:k], E[:k, 1], iv[:k, 0] = 2, 0, 1, np.arange(k)
    return L, E, iv


@pytest.mark.parametrize("first_us", [0, 70000])
def test_windows(ctx, first_us):
    """With the edges of the shorter intervals the other kernel counts; with the longest one its
    lists run over, which is an error as it is without tables."""
    ty, t = burst_stream(1, first_us=first_us)
    sid = fem.fem_load_stream(ctx, ty, t, K)
    L, E, iv = synth.random_candidates(1, 300, K - 2, [2, 3], 3)
    E = np.where(np.arange(E.shape[1]) < L[:, None], E + 2, 0)
    for ivl in (2, 3):
        cands = with_edge((L, E, iv), ivl)
        rec = fem.pack_episodes(*cands)
        if ivl == 3:
            with pytest.raises(fem.FemError) as e:
                fem.fem_count_windows(ctx, sid, rec, I, 30000)
            assert e.value.status == -9
        else:
            assert_counts_equal(fem.fem_count_windows(ctx, sid, rec, I, 30000),
                                oracle.count_windows_batch(ty, t, *cands, I, 30000), "windows")
    fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("m", [200, 700])
def test_counts(ctx, m):
    ty, t = burst_stream(2)
    sid = fem.fem_load_stream(ctx, ty, t, K)
    cands = with_edge(synth.random_candidates(2, m, K, [2, 3, 4], 4), 3)
    rec = fem.pack_episodes(*cands)
    for p in PASSES:
        want = oracle_counts(ty, t, *cands, I, p)
        for call in range(3):
            assert_counts_equal(fem.fem_count_candidates(ctx, sid, rec, I, p), want, f"pass {p} call {call}")
    fem.fem_free_stream(ctx, sid)


@pytest.fixture()
def told(monkeypatch, capfd):
    """What became of the hit tables since the last look, one word each."""
    monkeypatch.setenv("FEM_DEBUG", "1")

    def look():
        return [x.split(": ")[-1] for x in capfd.readouterr().err.splitlines() if "hit tables of" in x]

    return look


@pytest.mark.parametrize("m", [100, 700])
def test_a_dense_type_is_remembered(ctx, told, m):
    """Tables that turned out too dense are not built again for sets with an edge from that type
    and an interval as long, also after events were appended; other sets still go over them."""
    ty, t = burst_stream(3)
    sid = fem.fem_load_stream(ctx, ty, t, K)
    L, E, iv = synth.random_candidates(3, m, K - 2, [2, 3], 4)
    quiet = L, np.where(np.arange(E.shape[1]) < L[:, None], E + 2, 0).astype(np.uint8), iv
    dense = with_edge(quiet, 3)

    def counts(cands, intervals=I):
        told()
        for p in PASSES:
            assert_counts_equal(fem.fem_count_candidates(ctx, sid, fem.pack_episodes(*cands), intervals, p),
                                oracle_counts(ty, t, *cands, intervals, p), f"pass {p}")
        return told()

    assert counts(dense) == ["too dense"]
    assert counts(dense) == []
    assert counts(quiet) == ["counted"] * 2
    assert counts(dense, I // 4) == ["counted"] * 2  # up to 25 of type 0 in the longest
    more = np.arange(200, dtype=np.uint32) * 30000 + t[-1] + 1
    for k in range(3):  # (the stream's buffers grow)
        fem.fem_append_stream(ctx, sid, np.full(200, 2 + k, np.uint8), more)
        ty, t = np.append(ty, np.full(200, 2 + k, np.uint8)), np.append(t, more)
        more = more + np.uint32(7_000_000)
        assert counts(dense) == [] and counts(quiet) == ["counted"] * 2
    assert fem.fem_count_windows(ctx, sid, fem.pack_episodes(*quiet), I, 9000).sum() > 0
    assert told() == ["counted"]
    with pytest.raises(fem.FemError):
        fem.fem_count_windows(ctx, sid, fem.pack_episodes(*dense), I, 9000)
    assert told() == []
    fem.fem_free_stream(ctx, sid)


def test_mining_a_dense_stream(ctx, told):
    ty, t = burst_stream(4)
    sid = fem.fem_load_stream(ctx, ty, t, K)
    want = oracle.mine(ty, t, K, I[:2], 20, 4)
    long = np.array([[0, 5000], [0, 40000]], np.uint32)
    for intervals, first, second in ((I[:2], None, None), (long, 1, 0)):
        for expected in (first, second):
            got = fem.fem_mine_levelwise(ctx, sid, intervals, 20, 4)
            assert got == (want if expected is None else oracle.mine(ty, t, K, intervals, 20, 4))
            words = told()
            if expected is None:
                assert set(words) == {"counted"}
            else:
                assert words == ["too dense"] * expected
    fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("appended", [False, True])
def test_streams_that_start_late(ctx, told, appended):
    """How dense a stream is, is told by the time from its first to its last event: an hour after
    time 0 as at time 0, also where it was empty when it was loaded."""
    rng = np.random.default_rng(8)
    dense = rng.integers(0, 3, 6000).astype(np.uint8), np.cumsum(rng.integers(1, 60, 6000)).astype(np.uint32)
    even = rng.integers(0, K, 60000).astype(np.uint8), np.cumsum(rng.integers(1, 700, 60000)).astype(np.uint32)
    for (ty, t), types, ivls, words in ((dense, 3, np.array([[500, 9000]], np.uint32), []),
                                        (even, K, I[2:3], ["counted"])):
        cands = synth.random_candidates(8, 200, types, [2, 3], 1)
        for first_us in (0, 3_600_000_000):
            t1 = (t + np.uint32(first_us)).astype(np.uint32)
            n0 = 0 if appended else len(t)
            sid = fem.fem_load_stream(ctx, ty[:n0], t1[:n0], types)
            if appended:
                fem.fem_append_stream(ctx, sid, ty, t1)
            told()
            got = fem.fem_count_candidates(ctx, sid, fem.pack_episodes(*cands), ivls, 0)
            assert told() == words
            assert_counts_equal(got, oracle_counts(ty, t1, *cands, ivls, 0), f"from {first_us}")
            fem.fem_free_stream(ctx, sid)
