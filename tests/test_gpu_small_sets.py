"""Small sets to which the hit tables do not apply: repeated types, few episodes of many types
on a long stream, chunks shorter than an interval.  They are counted by the other kernels, and
are looked at once on the way there."""
import numpy as np
import pytest

from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts
from tests.test_gpu_hits import stream

pytestmark = pytest.mark.gpu


def lumps(n, K):
    """4,000 events in 10 ms every 100 s: sparse on average, the first chunk of each lump 5 ms."""
    rng = np.random.default_rng(1)
    t = np.arange(n) // 4000 * 100_000_000 + np.sort(rng.integers(0, 10000, (n // 4000 + 1, 4000)), axis=1).ravel()[:n]
    return rng.integers(0, K, n).astype(np.uint8), t.astype(np.uint32)


def repeated(cands):
    L, E, iv = (a.copy() for a in cands)
    E[:, 1] = E[:, 0]
    return L, E, iv


CASES = {  # stream, types, candidates, launches more than with the per-thread kernels configured
    # (a plan's four in place of a validation's two)
    "repeated types": (lambda: stream(5, 6000, 16, gap=1500), 16,
                       lambda: repeated(synth.random_candidates(1, 100, 16, [2, 3], 4)), 2),
    "few on a long stream": (lambda: stream(6, 160000, 64, gap=1000), 64,
                             lambda: synth.random_candidates(1, 200, 64, [3], 4), 2),
    "short chunks": (lambda: lumps(40000, 250), 250, lambda: synth.random_candidates(1, 200, 250, [3], 4), 0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_small_sets(name):
    make, K, candidates, more = CASES[name]
    ty, t = make()
    cands = candidates()
    rec = fem.pack_episodes(*cands)
    ctx = ctx_fixture()
    try:
        sid = fem.fem_load_stream(ctx, ty, t, K)
        for p in (fem.PASS_RELAXED, fem.PASS_EXACT):
            want = oracle_counts(ty, t, *cands, I_MS4, p)
            launches = []
            for kernel in (0, 0, fem.KERNEL_MACHINE):
                fem.fem_set_config(ctx, kernel=kernel)
                before = fem.fem_kernel_launches()
                assert_counts_equal(fem.fem_count_candidates(ctx, sid, rec, I_MS4, p), want, f"pass {p}")
                launches.append(fem.fem_kernel_launches() - before)
            assert launches[1] == launches[2] + more, launches
    finally:
        fem.fem_destroy(ctx)
