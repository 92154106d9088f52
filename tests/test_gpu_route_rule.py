"""Which way a candidate set is counted: over hit tables where they pay, by the other kernels
where the edges that a plan numbers, the types and the events cost more than the episodes, and
the counts by either way."""
import numpy as np
import pytest

from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu

CASES = {  # types, events, Hz a type, candidates, lengths, whether (relaxed, exact) go over tables
    "many types, short stream": (128, 5000, 20, 2000, [2], (False, False)),
    "more types than fit a build's block twice": (200, 20000, 10, 700, [3, 4], (False, False)),
    "pairs on a long stream": (64, 400000, 20, 5000, [2], (False, True)),
    "long episodes on a long stream": (64, 400000, 20, 5000, [7], (True, True)),
    "exact but not relaxed": (48, 300000, 20, 3000, [4], (False, True)),
    "several lengths": (64, 20000, 20, 2000, [2, 3, 4, 5], (True, True)),
    "few types": (12, 30000, 20, 300, [3], (True, True)),
    "a small set of one length": (64, 60000, 20, 100, [2], (False, False)),
    "a small set of several": (24, 6000, 20, 100, [2, 3, 4], (True, True)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_route(monkeypatch, capfd, name):
    K, n, hz, m, lens, expected = CASES[name]
    monkeypatch.setenv("FEM_DEBUG", "1")
    rng = np.random.default_rng(n + K)
    ty = rng.integers(0, K, n).astype(np.uint8)
    t = np.cumsum(rng.integers(1, int(2e6 / (K * hz)), n)).astype(np.uint32)
    cands = synth.random_candidates(3, m, K, lens, 4)
    ctx = ctx_fixture()
    try:
        sid = fem.fem_load_stream(ctx, ty, t, K)
        for p in (fem.PASS_RELAXED, fem.PASS_EXACT):
            capfd.readouterr()
            got = fem.fem_count_candidates(ctx, sid, fem.pack_episodes(*cands), I_MS4, p)
            assert ("hit tables of" in capfd.readouterr().err) == expected[p]
            some = rng.choice(m, min(m, 300), replace=False)
            assert_counts_equal(got[some], oracle_counts(ty, t, *(a[some] for a in cands), I_MS4, p), f"pass {p}")
    finally:
        fem.fem_destroy(ctx)
