"""Which way a batch runs: over hit tables where that is estimated to be faster, with the same
results by either way."""
import numpy as np
import pytest

from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu

CASES = {  # types, events a stream, streams, candidates a job, lengths, over tables
    "many types": (128, 30000, 4, 300, [5], False),
    "one length, few candidates": (100, 100000, 4, 70, [2], False),
    "several lengths": (16, 12000, 6, 300, [2, 3, 4, 5], True),
    "one long stream": (8, 40000, 1, 120, [5], True),
    "short streams": (64, 3000, 8, 100, [3], False),
}


@pytest.mark.parametrize("name", list(CASES))
def test_route(monkeypatch, capfd, name):
    torch = pytest.importorskip("torch")
    K, n, S, m, lens, tables = CASES[name]
    monkeypatch.setenv("FEM_DEBUG", "1")
    ctx = ctx_fixture()
    try:
        jobs, want = [], []
        for k in range(S):
            rng = np.random.default_rng(n + K + k)
            ty = rng.integers(0, K, n).astype(np.uint8)
            t = np.cumsum(rng.integers(1, int(1e5 / K), n)).astype(np.uint32)
            sid = fem.fem_load_stream(ctx, ty, t, K)
            cands = synth.random_candidates(k, m, K, [lens[k % len(lens)]], 4)
            theta = max(1, n // K // 40)
            jobs.append(dict(stream_id=sid, len=lens[k % len(lens)], theta=theta,
                             cands=torch.from_numpy(fem.pack_episodes(*cands)).cuda(),
                             exact_out=torch.zeros(m, dtype=torch.int32, device="cuda"),
                             survived_out=torch.zeros(m, dtype=torch.uint8, device="cuda")))
            keep = oracle_counts(ty, t, *cands, I_MS4, fem.PASS_RELAXED) >= theta
            want.append((np.where(keep, oracle_counts(ty, t, *cands, I_MS4, fem.PASS_EXACT), 0), keep))
        torch.cuda.synchronize()
        capfd.readouterr()
        b = fem.fem_batch_create(ctx, jobs, I_MS4)
        assert ("over hit tables" in capfd.readouterr().err) == tables
        fem.fem_batch_run(b)
        for j, (ex, keep) in zip(jobs, want):
            assert_counts_equal(j["exact_out"].cpu().numpy(), ex, "exact")
            assert_counts_equal(j["survived_out"].cpu().numpy(), keep.astype(np.uint8), "survived")
        fem.fem_batch_destroy(b)
    finally:
        fem.fem_destroy(ctx)
