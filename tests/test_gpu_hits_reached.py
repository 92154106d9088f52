"""The hit-table kernels against the oracle at the edges of slabs, chunks and segments, on
streams sparse enough for them; every test looks at what the library says of its tables (the
FEM_DEBUG lines), so that it cannot pass on the other kernels' counts."""
import numpy as np
import pytest

import oracle
from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts
from tests.test_gpu_hits import stream

pytestmark = pytest.mark.gpu
PASSES = (fem.PASS_RELAXED, fem.PASS_EXACT)
GAP = 1500  # microseconds at most between events: on average 4 of a type in 20 ms, of 9 to 12 types
SHORT = np.array([[0, 2], [2, 5], [5, 10], [10, 20]], np.uint32)  # for a stream of one event


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    fem.fem_destroy(c)


@pytest.fixture(autouse=True)
def _reset_config(ctx):
    yield
    fem.fem_set_config(ctx, reset=True)


@pytest.fixture()
def told(monkeypatch, capfd):
    """What became of the hit tables since the last look, one word each."""
    monkeypatch.setenv("FEM_DEBUG", "1")

    def look():
        return [x.split(": ")[-1] for x in capfd.readouterr().err.splitlines() if "hit tables of" in x]

    return look


@pytest.mark.parametrize("n", [1, 31, 33, 2047, 2048, 2049, 4096, 9000])
@pytest.mark.parametrize("m", [240, 600])
def test_sizes_and_segments(ctx, told, n, m):
    """Every length 1-8, equal times across slab and chunk ends, one segment up to more segments
    than chunks; sets that are validated first and sets that are not."""
    ty, t = stream(n, n, 12, gap=GAP)
    I = SHORT if n == 1 else I_MS4
    L, E, iv = synth.random_candidates(n, m, 12, [1, 2, 3, 4, 5, 6, 7, 8], 4)
    rec = fem.pack_episodes(L, E, iv)
    sid = fem.fem_load_stream(ctx, ty, t, 12)
    for p in PASSES:
        want = oracle_counts(ty, t, L, E, iv, I, p)
        for seg in (0, 1, 2, 7, 50):
            fem.fem_set_config(ctx, segments=seg)
            told()
            got = fem.fem_count_candidates(ctx, sid, rec, I, p)
            words = told()
            assert words[-1] == "counted" and set(words[:-1]) <= {"too small"}
            assert_counts_equal(got, want, f"n {n} pass {p} segments {seg}")
    fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("n,w_us", [(1, 5), (33, 900), (2049, 1), (7000, 2500), (9000, 400000), (2048, 70000)])
@pytest.mark.parametrize("segments", [0, 1, 5, 60])
def test_window_frequency(ctx, told, n, w_us, segments):
    """Windows shorter and longer than a segment, one-node episodes, one event, equal times at
    the cuts."""
    ty, t = stream(n + 1, n, 9, gap=GAP)
    I = SHORT if n == 1 else I_MS4
    cands = synth.random_candidates(n, 150, 9, [1, 2, 3, 4, 6, 8], 4)
    sid = fem.fem_load_stream(ctx, ty, t, 9)
    fem.fem_set_config(ctx, segments=segments)
    told()
    got = fem.fem_count_windows(ctx, sid, fem.pack_episodes(*cands), I, w_us)
    words = told()
    assert words[-1] == "counted" and set(words[:-1]) <= {"too small"}
    assert_counts_equal(got, oracle.count_windows_batch(ty, t, *cands, I, w_us), "windows")
    fem.fem_free_stream(ctx, sid)


def test_batch(ctx, monkeypatch, capfd):
    """A batch over a stream of bursts (more hits than estimated), one of one slab and one of
    several chunks; interleaved jobs, lengths 1-8."""
    torch = pytest.importorskip("torch")
    monkeypatch.setenv("FEM_DEBUG", "1")
    I = np.array([[0, 2000], [2000, 20000]], np.uint32)
    streams = [synth.sparse_bursts(seed=5, n_types=16, base_hz=0.5, duration_s=200.0, n_bursts=20),
               stream(3, 40, 16, gap=GAP), stream(4, 6000, 16, gap=GAP)]
    sids = [fem.fem_load_stream(ctx, ty, t, 16) for ty, t in streams]
    jobs, want = [], []
    for n in (2, 5, 1, 8, 3):
        for k, (ty, t) in enumerate(streams):
            cands = synth.random_candidates(10 * n + k, 90 + 37 * k, 16, [n], 2)
            theta = 1 + k
            jobs.append(dict(stream_id=sids[k], len=n, theta=theta,
                             cands=torch.from_numpy(fem.pack_episodes(*cands)).cuda(),
                             exact_out=torch.zeros(len(cands[0]), dtype=torch.int32, device="cuda"),
                             survived_out=torch.zeros(len(cands[0]), dtype=torch.uint8, device="cuda")))
            keep = oracle_counts(ty, t, *cands, I, fem.PASS_RELAXED) >= theta
            want.append((np.where(keep, oracle_counts(ty, t, *cands, I, fem.PASS_EXACT), 0), keep))
    torch.cuda.synchronize()
    b = fem.fem_batch_create(ctx, jobs, I)
    assert "over hit tables" in capfd.readouterr().err
    for _ in range(2):
        for j in jobs:
            j["exact_out"].fill_(-1)
        torch.cuda.synchronize()
        fem.fem_batch_run(b)
        for i, (j, (ex, keep)) in enumerate(zip(jobs, want)):
            assert_counts_equal(j["exact_out"].cpu().numpy(), ex, f"job {i}")
            assert_counts_equal(j["survived_out"].cpu().numpy(), keep.astype(np.uint8), f"job {i}")
    fem.fem_batch_destroy(b)
    for sid in sids:
        fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("m", [100, 700])
def test_too_dense_across_a_chunk_end(ctx, monkeypatch, capfd, m):
    """35 events of a type in an interval, 15 of them before a chunk's end: the plan, which looks
    within chunks, does not see it, the build does, and the other kernels count."""
    monkeypatch.setenv("FEM_DEBUG", "1")
    ty, t = stream(12, 6000, 12, gap=GAP)
    burst = 4096 - 15 + np.arange(35)
    ty = np.where(ty == 0, 1, ty)
    ty[burst] = 0
    t[burst] = t[burst[0]] + 100 * np.arange(35)
    t = np.maximum.accumulate(t).astype(np.uint32)
    ty[burst[-1] + 1:burst[-1] + 40:2] = 1  # soon after the burst
    t[burst[-1] + 1:] -= t[burst[-1] + 1] - t[burst[-1]] - np.uint32(50)
    sid = fem.fem_load_stream(ctx, ty, t, 12)
    L, E, iv = synth.random_candidates(7, m, 12, [2, 3, 4], 4)
    L[:4], E[:4], E[:4, 1], iv[:4, 0] = 2, 0, 1, np.arange(4)
    for p in PASSES:
        capfd.readouterr()
        got = fem.fem_count_candidates(ctx, sid, fem.pack_episodes(L, E, iv), I_MS4, p)
        err = capfd.readouterr().err
        assert ("edges in" in err and "too dense" in err) == (p == PASSES[0])
        assert_counts_equal(got, oracle_counts(ty, t, L, E, iv, I_MS4, p), f"pass {p}")
    fem.fem_free_stream(ctx, sid)


@pytest.mark.parametrize("n5", range(60, 72))
def test_many_calls(told, n5):
    """Call after call in a new context: the number of a set's candidates of five nodes, a word
    of its plan, passes the sequence numbers that the host waits for."""
    torch = pytest.importorskip("torch")
    ty, t = stream(5, 3000, 12, gap=GAP)
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
        assert told().count("counted") == 120
    finally:
        fem.fem_destroy(c)
