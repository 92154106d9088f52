"""One-shot requests whose first count runs out of entry classes or list room: the flagged
candidates (or, where they are most, all) are counted again on the request's lane while
other requests run.  Every result equals the oracle's two passes on the request's range,
with few candidates flagged, many, none, and with events appended meanwhile."""
import numpy as np
import pytest

import oracle
from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu
I = synth.I_BURST


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    fem.fem_destroy(c)


def two_passes(ty, t, cands, theta):
    keep = oracle_counts(ty, t, *cands, I, oracle.RELAXED) >= theta
    return np.where(keep, oracle_counts(ty, t, *cands, I, oracle.EXACT), 0), keep


@pytest.mark.parametrize("bursts,burst_ms", [(1, 100.0), (4, 300.0), (40, 1000.0), (0, 0.0)])
@pytest.mark.parametrize("append", [False, True])
def test_recounts_equal_oracle(ctx, bursts, burst_ms, append):
    ty, t = synth.sparse_bursts(seed=bursts + 7, n_types=16, base_hz=8.0, duration_s=60.0, n_bursts=bursts,
                                burst_ms=burst_ms, burst_rate_hz=120.0)
    n = len(t) - (len(t) // 10 if append else 0)
    srv = fem.fem_server_create(ctx, mem_budget_bytes=512 << 20, max_active=16, n_lanes=4)
    try:
        sid = fem.fem_server_open_stream(srv, 16, len(t) + 4096)
        fem.fem_server_append(srv, sid, ty[:n], t[:n])
        reqs = []
        for k, (m, lens, theta) in enumerate([(3, [2], 1), (700, [2, 3, 4, 5], 2), (2000, [2, 6], 30),
                                              (501, [3, 8], 1)]):
            cands = synth.random_candidates(90 + k, m, 16, lens, 4)
            rid = fem.fem_server_submit(srv, sid, fem.pack_episodes(*cands), I, theta, fem.REQ_ONESHOT, 0)
            reqs.append((rid, cands, theta, m))
        if append:
            fem.fem_server_append(srv, sid, ty[n:], t[n:])
        fem.fem_server_drain(srv)
        for rid, cands, theta, m in reqs:
            counts, flags, events, status = fem.fem_server_result(srv, rid, m)
            assert status == 0 and events == n
            ex, keep = two_passes(ty[:n], t[:n], cands, theta)
            assert_counts_equal(counts, ex, f"{m} candidates")
            assert_counts_equal(flags, keep.astype(np.uint8), f"{m} candidates' flags")
            fem.fem_server_release(srv, rid)
    finally:
        fem.fem_server_destroy(srv)
