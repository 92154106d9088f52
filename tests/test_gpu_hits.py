"""The hit-table counting kernels (fem_hits.cu) against the oracle, element by element, at the
places where they can go wrong: types with more events in a slab than a word holds (the
slabs shrink to 32 events), equal times across slab and chunk ends, every length 1-8 with one
segment up to more segments than chunks, overlapping intervals and more than four of them,
256 types, windows denser than the tables' words (counted by the other kernels), more hits
than the table was sized for, and a memory budget without room for the tables."""
import numpy as np
import pytest

import oracle
from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu
PASSES = (fem.PASS_RELAXED, fem.PASS_EXACT)


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    fem.fem_destroy(c)


@pytest.fixture(autouse=True)
def _reset_config(ctx):
    yield
    fem.fem_set_config(ctx, reset=True)


def stream(seed, n, K, skew=0.0, tie=0.3, gap=400):
    """n events of K types, gaps up to `gap` us, a share `tie` of equal times; type 0 takes
    `skew` of the events."""
    rng = np.random.default_rng(seed)
    g = rng.integers(1, gap + 1, n)
    g[rng.random(n) < tie] = 0
    ty = rng.integers(0, K, n)
    ty[rng.random(n) < skew] = 0
    return ty.astype(np.uint8), np.cumsum(g).astype(np.uint32)


def check(ctx, ty, t, K, cands, I, segments=(0,), what=""):
    sid = fem.fem_load_stream(ctx, ty, t, K)
    L, E, iv = cands
    rec = fem.pack_episodes(L, E, iv)
    for p in PASSES:
        want = oracle_counts(ty, t, L, E, iv, I, p)
        for seg in segments:
            fem.fem_set_config(ctx, segments=seg)
            assert_counts_equal(fem.fem_count_candidates(ctx, sid, rec, I, p), want,
                                f"{what} pass {p} segments {seg}")
    fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("n", [1, 31, 33, 2047, 2048, 2049, 4096, 9000])
def test_sizes_and_segments(ctx, n):
    ty, t = stream(n, n, 12)
    cands = synth.random_candidates(n, 240, 12, [1, 2, 3, 4, 5, 6, 7, 8], 4)
    check(ctx, ty, t, 12, cands, I_MS4, (0, 1, 2, 7, 50), f"n {n}")


@pytest.mark.parametrize("K,skew", [(2, 0.0), (5, 0.95), (40, 0.6)])
def test_skewed_types(ctx, K, skew):
    """A type with most of the events: up to 64 slabs per chunk."""
    ty, t = stream(K, 7000, K, skew, gap=3000)
    I = np.array([[0, 3000], [1000, 9000]], np.uint32)
    check(ctx, ty, t, K, synth.random_candidates(K, 150, K, [2, min(3, K)], 2), I, (0, 3), "skewed")


@pytest.mark.parametrize("K", [64, 256])
def test_overlapping_intervals(ctx, K):
    I = np.array([[0, 30000], [10000, 12000], [5000, 60000]] + ([[0, 1], [59999, 60000], [7, 9000]]
                                                               if K == 64 else []), np.uint32)
    ty, t = stream(K, 12000, K, gap=900)
    check(ctx, ty, t, K, synth.random_candidates(K, 500, K, [2, 3, 5], len(I)), I, (0, 4), f"K {K}")


def test_windows_denser_than_a_word(ctx):
    ty, t = stream(1, 6000, 3, gap=60)
    I = np.array([[0, 2000], [500, 9000]], np.uint32)  # up to 100 events of a type
    check(ctx, ty, t, 3, synth.random_candidates(1, 60, 3, [2, 3], 2), I, (0, 2), "dense")


def test_more_hits_than_estimated(ctx):
    """Bursts in a quiet stream: far more hits than its mean rate gives, and entry classes
    past eight."""
    ty, t = synth.sparse_bursts(seed=5, n_types=16, base_hz=0.5, duration_s=200.0, n_bursts=40)
    I = np.array([[0, 2000], [2000, 20000]], np.uint32)
    check(ctx, ty, t, 16, synth.random_candidates(2, 700, 16, [2, 3, 4, 5], 2), I, (0, 1, 5), "bursts")


def test_no_room_for_the_tables():
    ty, t = stream(9, 20000, 32, gap=1500)
    L, E, iv = synth.random_candidates(9, 300, 32, [2, 3, 4], 4)
    rec = fem.pack_episodes(L, E, iv)
    for budget in (600 << 10, 4 << 20):
        c = fem.fem_create(0, mem_budget_bytes=budget)
        try:
            sid = fem.fem_load_stream(c, ty, t, 32)
            for p in PASSES:
                assert_counts_equal(fem.fem_count_candidates(c, sid, rec, I_MS4, p),
                                    oracle_counts(ty, t, L, E, iv, I_MS4, p), f"budget {budget}")
            assert fem.fem_mem_usage(c)[0] <= budget
            # the tables make room for a stream
            other = fem.fem_load_stream(c, ty[:5000], t[:5000], 32)
            fem.fem_free_stream(c, other)
        finally:
            fem.fem_destroy(c)


@pytest.mark.parametrize("n,w_us", [(1, 5), (33, 900), (2049, 1), (7000, 2500), (9000, 400000)])
@pytest.mark.parametrize("segments", [0, 1, 5, 60])
def test_window_frequency(ctx, n, w_us, segments):
    """Window frequencies over segments: windows shorter and longer than a segment, one event,
    equal times at the cuts."""
    ty, t = stream(n + 1, n, 9)
    cands = synth.random_candidates(n, 150, 9, [1, 2, 3, 4, 6, 8], 4)
    sid = fem.fem_load_stream(ctx, ty, t, 9)
    fem.fem_set_config(ctx, segments=segments)
    got = fem.fem_count_windows(ctx, sid, fem.pack_episodes(*cands), I_MS4, w_us)
    assert_counts_equal(got, oracle.count_windows_batch(ty, t, *cands, I_MS4, w_us), "windows")
    fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("dense", [False, True])
def test_batch(ctx, dense):
    """A batch over streams of 1 to several chunks: a bursting one (more hits than estimated),
    interleaved jobs, lengths 1-8, and with `dense` a stream the tables do not fit, for which
    the whole batch takes the other kernels."""
    torch = pytest.importorskip("torch")
    I = np.array([[0, 2000], [2000, 20000]], np.uint32)
    streams = [synth.sparse_bursts(seed=5, n_types=16, base_hz=0.5, duration_s=200.0, n_bursts=20),
               stream(3, 1, 16), stream(4, 6000, 16)]
    if dense:
        streams.append(stream(6, 6000, 16, gap=5))
    sids = [fem.fem_load_stream(ctx, ty, t, 16) for ty, t in streams]
    jobs, want = [], []
    for n in (2, 5, 1, 8, 3):
        for k, (ty, t) in enumerate(streams):
            cands = synth.random_candidates(10 * n + k, 90 + 37 * k, 16, [n], 2)
            theta = 2 + 5 * k
            jobs.append(dict(stream_id=sids[k], len=n, theta=theta,
                             cands=torch.from_numpy(fem.pack_episodes(*cands)).cuda(),
                             exact_out=torch.zeros(len(cands[0]), dtype=torch.int32, device="cuda"),
                             survived_out=torch.zeros(len(cands[0]), dtype=torch.uint8, device="cuda")))
            keep = oracle_counts(ty, t, *cands, I, fem.PASS_RELAXED) >= theta
            want.append((np.where(keep, oracle_counts(ty, t, *cands, I, fem.PASS_EXACT), 0), keep))
    torch.cuda.synchronize()
    b = fem.fem_batch_create(ctx, jobs, I)
    for _ in range(2):
        for j in jobs:
            j["exact_out"].fill_(-1)
        torch.cuda.synchronize()
        fem.fem_batch_run(b)
        for i, (j, (ex, keep)) in enumerate(zip(jobs, want)):
            assert_counts_equal(j["exact_out"].cpu().numpy(), ex, f"job {i}")
            assert_counts_equal(j["survived_out"].cpu().numpy(), keep.astype(np.uint8), f"job {i}")
    fem.fem_batch_destroy(b)
    jobs[0]["len"] = 3  # candidates of another length than the job's
    with pytest.raises(fem.FemError) as e:
        fem.fem_batch_create(ctx, jobs, I)
    assert e.value.status == -1
    for sid in sids:
        fem.fem_free_stream(ctx, sid)


I_LONG = np.array([[0, 9000], [9000, 18000]], np.uint32)
MINES = {  # events, types, theta, gap, share of type 0, intervals
    "long lists, several chunks": (5000, 24, 3, 400, 0.0, I_LONG),
    "one more than a chunk": (2049, 24, 3, 300, 0.0, I_LONG),
    "one interval": (2500, 36, 2, 300, 0.0, np.array([[0, 9000]], np.uint32)),
    "too dense for the tables": (3000, 24, 3, 400, 0.5, I_LONG),
}


@pytest.mark.parametrize("name", list(MINES))
def test_mine_joined(ctx, name):
    """Level 3 of mining over 40,000 or more candidates joins the lists of pairs: lists shorter
    and longer than a warp's 64 entries, more hits in a slab than the queue holds, and a
    stream that is too dense, for which the other kernels count."""
    n, K, theta, gap, skew, I = MINES[name]
    ty, t = stream(n + K, n, K, skew=skew, gap=gap)
    sid = fem.fem_load_stream(ctx, ty, t, K)
    got = fem.fem_mine_levelwise(ctx, sid, I, theta, 3)
    stats = fem.fem_last_mine_stats(ctx)
    fem.fem_free_stream(ctx, sid)
    assert stats[1]["level"] == 3 and stats[1]["candidates"] >= 40000
    assert (stats[1]["kernel_relaxed"] == fem.KERNEL_HITS) == ("dense" not in name)
    assert got == oracle.mine(ty, t, K, I, theta, 3)


def test_mine_levels_and_budgets(ctx):
    """Levels 2-6 over hit tables equal the oracle's; under a memory budget whatever the
    latest-chain kernels can mine is mined too, with or without room for the tables."""
    ty, t = stream(77, 4000, 24, tie=0.0, gap=2000)
    ty[:2400] = np.tile(np.arange(24, dtype=np.uint8), 100)  # long chains
    sid = fem.fem_load_stream(ctx, ty, t, 24)
    want = fem.fem_mine_levelwise(ctx, sid, I_MS4[:2], 40, 6)
    assert want == oracle.mine(ty, t, 24, I_MS4[:2], 40, 6)
    kinds = [s["kernel_exact"] for s in fem.fem_last_mine_stats(ctx)]
    assert len(kinds) >= 3 and kinds.count(fem.KERNEL_HITS) >= 2
    fem.fem_free_stream(ctx, sid)
    mined = 0
    for mb in (1, 2, 3, 4, 6, 9, 13, 20, 30, 45, 70):
        c = fem.fem_create(0, mem_budget_bytes=mb << 20)
        try:
            try:
                sid = fem.fem_load_stream(c, ty, t, 24)
                fem.fem_set_config(c, kernel=fem.KERNEL_CHAIN)
                fem.fem_mine_levelwise(c, sid, I_MS4[:2], 40, 6)
            except fem.FemError as e:
                assert e.status == -5
                continue
        finally:
            fem.fem_destroy(c)
        c = fem.fem_create(0, mem_budget_bytes=mb << 20)
        try:
            sid = fem.fem_load_stream(c, ty, t, 24)
            assert fem.fem_mine_levelwise(c, sid, I_MS4[:2], 40, 6) == want
            mined += 1
        finally:
            fem.fem_destroy(c)
    assert mined >= 3


@pytest.mark.parametrize("n5", range(60, 72))
def test_many_calls(ctx, n5):
    """Call after call in a new context: a set's count of one length passes the sequence number
    of the words the host waits for, which must not be taken for it."""
    torch = pytest.importorskip("torch")
    ty, t = stream(5, 3000, 12)
    parts = [synth.random_candidates(m, m, 12, [n], 4) for m, n in ((n5, 5), (127, 4), (120, 3))]
    cands = tuple(np.concatenate(p) for p in zip(*parts))
    keep = oracle_counts(ty, t, *cands, I_MS4, fem.PASS_RELAXED) >= 0
    want = np.where(keep, oracle_counts(ty, t, *cands, I_MS4, fem.PASS_EXACT), 0)
    rec = torch.from_numpy(fem.pack_episodes(*cands)).cuda()
    ex = torch.zeros(len(keep), dtype=torch.int32, device="cuda")
    kept = torch.zeros(len(keep), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    c = fem.fem_create(0)
    try:
        sid = fem.fem_load_stream(c, ty, t, 12)
        for k in range(60):
            fem.fem_count_two_pass(c, sid, rec, I_MS4, 0, ex, kept)
            assert_counts_equal(ex.cpu().numpy(), want, f"call {k}")
            assert_counts_equal(kept.cpu().numpy(), keep.astype(np.uint8), f"call {k}")
    finally:
        fem.fem_destroy(c)
