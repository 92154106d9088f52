"""Level-wise mining of a short, dense recording without structure: the relaxed pass of level 4
over more than a million candidates, whose prefixes the latest-chain kernel shares, is that
kernel's; level 3 is joined.  The results equal those of the latest-chain kernels alone."""
import numpy as np
import pytest

from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import ctx_fixture

pytestmark = pytest.mark.gpu


def test_large_relaxed_level():
    rng = np.random.default_rng(4)
    K, n, hz, theta = 32, 10000, 40, 18
    I = synth.I_MS4
    ty = rng.integers(0, K, n).astype(np.uint8)
    t = np.cumsum(rng.integers(1, int(2e6 / (K * hz)), n)).astype(np.uint32)
    ctx = ctx_fixture()
    try:
        sid = fem.fem_load_stream(ctx, ty, t, K)
        got = fem.fem_mine_levelwise(ctx, sid, I, theta, 4, raw=True)
        stats = {s["level"]: s for s in fem.fem_last_mine_stats(ctx)}
        assert stats[3]["kernel_relaxed"] == fem.KERNEL_HITS and stats[3]["candidates"] >= 40000
        assert stats[4]["candidates"] * 4 * n / K >= 1e9
        assert stats[4]["kernel_relaxed"] == fem.KERNEL_CHAIN
        fem.fem_set_config(ctx, kernel=fem.KERNEL_CHAIN)
        want = fem.fem_mine_levelwise(ctx, sid, I, theta, 4, raw=True)
        assert list(got) == list(want)
        for level in want:
            assert all(np.array_equal(a, b) for a, b in zip(got[level], want[level]))
    finally:
        fem.fem_destroy(ctx)
