"""Window frequencies: over hit tables or by the kernel that walks the stream, whichever is
estimated to be faster, with the same results; and over the tables where that kernel's lists
would run over."""
import numpy as np
import pytest

import oracle
from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture

pytestmark = pytest.mark.gpu

CASES = {  # types, events, candidates, lengths, over tables
    "short stream": (16, 100, 100, [2], False),
    "many types": (128, 1000, 2000, [2], False),
    "many types, longer": (128, 20000, 2000, [2], True),
    "longer episodes": (64, 1000, 2000, [4], True),
    "several lengths": (64, 1000, 500, [2, 3, 4], True),
    "few types": (16, 1000, 100, [2], True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_route(monkeypatch, capfd, name):
    K, n, m, lens, tables = CASES[name]
    monkeypatch.setenv("FEM_DEBUG", "1")
    rng = np.random.default_rng(n + K)
    ty = rng.integers(0, K, n).astype(np.uint8)
    t = np.cumsum(rng.integers(1, int(1e5 / K), n)).astype(np.uint32)
    cands = synth.random_candidates(3, m, K, lens, 4)
    ctx = ctx_fixture()
    try:
        sid = fem.fem_load_stream(ctx, ty, t, K)
        got = fem.fem_count_windows(ctx, sid, fem.pack_episodes(*cands), I_MS4, 40000)
        assert ("hit tables of" in capfd.readouterr().err) == tables
        assert_counts_equal(got, oracle.count_windows_batch(ty, t, *cands, I_MS4, 40000), name)
    finally:
        fem.fem_destroy(ctx)


def test_lists_that_run_over(monkeypatch, capfd):
    """40 events of one type and then, much later, one of the next: more than the walking kernel's
    lists hold, far fewer than 32 in an interval."""
    monkeypatch.setenv("FEM_DEBUG", "1")
    ty = np.array([0] * 40 + [1, 2, 3, 1], np.uint8)
    t = (5000 * np.arange(44)).astype(np.uint32)
    K, I = 24, np.array([[0, 20000]], np.uint32)
    L, E, iv = np.array([2, 2]), np.zeros((2, 8), int), np.zeros((2, 7), int)
    E[:, 1] = 1, 2
    ctx = ctx_fixture()
    try:
        sid = fem.fem_load_stream(ctx, ty, t, K)
        got = fem.fem_count_windows(ctx, sid, fem.pack_episodes(L, E, iv), I, 30000)
        assert "counted" in capfd.readouterr().err
        assert_counts_equal(got, oracle.count_windows_batch(ty, t, L, E, iv, I, 30000), "run over")
    finally:
        fem.fem_destroy(ctx)
