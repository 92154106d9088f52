"""A hit-table count whose transfer tables would pass a 64th of the device's memory runs over
a part of the candidates after the other, with the same counts."""
import numpy as np
import pytest

from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts

pytestmark = pytest.mark.gpu


def test_counts_in_parts_of_the_set():
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(2)
    chunks, K, m = 420, 32, 130001
    n = chunks * 2048
    ty = rng.integers(0, K, n).astype(np.uint8)
    t = np.cumsum(rng.integers(1, 1000, n)).astype(np.uint32)
    L, E, iv = synth.random_candidates(5, m, K, [3], 4)
    rec = torch.from_numpy(fem.pack_episodes(L, E, iv)).cuda()
    ctx = ctx_fixture()
    try:
        sid = fem.fem_load_stream(ctx, ty, t, K)
        some = rng.choice(m, 200, replace=False)
        some[:3] = 0, m - 1, m - 2
        for p in (fem.PASS_RELAXED, fem.PASS_EXACT):
            got, launches = [], []
            for segments in (0, chunks):  # (tables of 5.7 GB where a 64th is 4.4)
                fem.fem_set_config(ctx, segments=segments)
                out = torch.full((m,), -1, dtype=torch.int32, device="cuda")
                before = fem.fem_kernel_launches()
                fem.fem_count_candidates(ctx, sid, rec, I_MS4, p, out=out)
                launches.append(fem.fem_kernel_launches() - before)
                got.append(out.cpu().numpy())
                assert fem.fem_mem_usage(ctx)[0] < torch.cuda.mem_get_info()[1] // 64 + (700 << 20)
            assert launches[1] >= launches[0] + 2  # a count and a stitch more, and recounts
            assert_counts_equal(got[1], got[0], f"pass {p}")
            assert_counts_equal(got[0][some], oracle_counts(ty, t, L[some], E[some], iv[some], I_MS4, p), "some")
    finally:
        fem.fem_destroy(ctx)
