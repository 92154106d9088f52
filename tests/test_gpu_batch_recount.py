"""A batch over hit tables with a job whose candidates need more entry classes than a table has
slots: in a second of eight types that each fire every millisecond, the exact chains of eight
nodes start 140 ms and more before they end, and completions out of phase stay apart."""
import numpy as np
import pytest

from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu
K, I = 64, np.array([[0, 2000], [20000, 30000]], np.uint32)


def recording():
    rng = np.random.default_rng(11)
    ty = np.concatenate([np.tile(np.arange(8), 1000), rng.integers(8, K, 20000)])
    t = np.concatenate([9_000_000 + 125 * np.arange(8000), rng.integers(0, 20_000_000, 20000)])
    order = np.argsort(t, kind="stable")
    return ty[order].astype(np.uint8), t[order].astype(np.uint32)


def job(torch, sid, cands, theta):
    m = len(cands[0])
    return dict(stream_id=sid, len=int(cands[0][0]), theta=theta, cands=torch.from_numpy(fem.pack_episodes(*cands)).cuda(),
                exact_out=torch.zeros(m, dtype=torch.int32, device="cuda"),
                survived_out=torch.zeros(m, dtype=torch.uint8, device="cuda"))


def test_only_the_flagged_jobs_are_counted_again(monkeypatch, capfd):
    torch = pytest.importorskip("torch")
    monkeypatch.setenv("FEM_DEBUG", "1")
    ctx = ctx_fixture()
    try:
        ty, t = recording()
        sid = fem.fem_load_stream(ctx, ty, t, K)
        rng = np.random.default_rng(3)
        m = 20
        flagged = (np.full(m, 8), np.stack([rng.permutation(8) for _ in range(m)]),
                   np.ones((m, 7), int))
        # (lengths 6 and 7, counted by the same launch)
        quiet = [(np.full(50 + k, 6 + k % 2),
                  np.stack([8 + rng.permutation(K - 8)[:8] for _ in range(50 + k)]) * (np.arange(8) < 6 + k % 2),
                  rng.integers(0, 2, (50 + k, 7)) * (np.arange(7) < 5 + k % 2)) for k in range(24)]
        launches = []
        for sets in (quiet, [flagged] + quiet[:1], quiet[:-1] + [flagged] + quiet[-1:]):
            jobs = [job(torch, sid, c, 1) for c in sets]
            torch.cuda.synchronize()
            b = fem.fem_batch_create(ctx, jobs, I)
            before = fem.fem_kernel_launches()
            fem.fem_batch_run(b)
            launches.append(fem.fem_kernel_launches() - before)
            for c, j in zip(sets, jobs):
                keep = oracle_counts(ty, t, *c, I, fem.PASS_RELAXED) >= 1
                want = np.where(keep, oracle_counts(ty, t, *c, I, fem.PASS_EXACT), 0)
                assert_counts_equal(j["exact_out"].cpu().numpy(), want, "exact")
                assert_counts_equal(j["survived_out"].cpu().numpy(), keep.astype(np.uint8), "survived")
            fem.fem_batch_destroy(b)
        assert capfd.readouterr().err.count("over hit tables") == 3
        assert launches[0] < launches[1] == launches[2]
    finally:
        fem.fem_destroy(ctx)
