"""Tuning and the hit tables: where the rule takes the tables the choice is measured, kept,
saved and loaded; a shape cached for mining's sets in runs does not decide for others."""
import json
import math

import numpy as np
import pytest

import oracle
from paper_0905_2200_gb300 import fem, synth
from tests.gpu_common import I_MS4, assert_counts_equal, ctx_fixture, oracle_counts
from tests.test_gpu_hits import stream

pytestmark = pytest.mark.gpu
K = 16


@pytest.fixture()
def ctx():
    c = ctx_fixture()
    yield c
    fem.fem_destroy(c)


@pytest.fixture()
def told(monkeypatch, capfd):
    """What became of the hit tables since the last look, one word each."""
    monkeypatch.setenv("FEM_DEBUG", "1")

    def look():
        return [x.split(": ")[-1] for x in capfd.readouterr().err.splitlines() if "hit tables of" in x]

    return look


def key(N, pass_, kind, m, n):
    return f"{N}/{pass_}/{kind}/{math.ceil(math.log2(m))}/{math.ceil(math.log2((n + 2047) // 2048))}/{K}"


def load(ctx, tmp_path, *lines):
    path = tmp_path / "in.jsonl"
    path.write_text("".join(json.dumps(dict(key=k, segments=s, threads=t, ms=0.5, kernel=kernel)) + "\n"
                            for k, s, t, kernel in lines))
    fem.fem_tune_load(ctx, path)


@pytest.mark.parametrize("m", [100, 600])
@pytest.mark.parametrize("lens", [[3], [2, 3, 5]])
def test_a_sets_choice(ctx, told, tmp_path, m, lens):
    ty, t = stream(31, 9000, K, gap=1500)
    cands = synth.random_candidates(31, m, K, lens, 4)
    rec = fem.pack_episodes(*cands)
    N = lens[0] if len(lens) == 1 else 0
    keys = [key(N, p, 2, m, len(t)) for p in (0, 1)]
    want = [oracle_counts(ty, t, *cands, I_MS4, p) for p in (0, 1)]

    def counts(c, sid):
        told()
        for p in (0, 1):
            assert_counts_equal(fem.fem_count_candidates(c, sid, rec, I_MS4, p), want[p], f"pass {p}")
        return told().count("counted")

    # tuning on: measured once, kept, saved
    sid = fem.fem_load_stream(ctx, ty, t, K)
    fem.fem_tune_enable(ctx, True)
    assert counts(ctx, sid) >= 4
    path = tmp_path / "out.jsonl"
    fem.fem_tune_save(ctx, path)
    saved = {x["key"]: x["kernel"] for x in map(json.loads, path.read_text().splitlines())}
    assert all(saved[k] in (fem.KERNEL_HITS, fem.KERNEL_MACHINE) for k in keys)
    over = sum(saved[k] == fem.KERNEL_HITS for k in keys)
    assert counts(ctx, sid) == over
    # loaded: the choice holds without tuning; another one is taken as it stands
    for choice, expected in ((None, over), ((fem.KERNEL_HITS,) * 2, 2), ((fem.KERNEL_MACHINE,) * 2, 0)):
        c = ctx_fixture()
        try:
            if choice is None:
                fem.fem_tune_load(c, path)
            else:
                load(c, tmp_path, *[(k, 1, 32, ch) for k, ch in zip(keys, choice)])
            assert counts(c, fem.fem_load_stream(c, ty, t, K)) == expected
        finally:
            fem.fem_destroy(c)
    # a shape of the other kernels for the same length and size does not decide
    c = ctx_fixture()
    try:
        load(c, tmp_path, *[(key(n, p, 1, m, len(t)), 2, 64, 1) for p in (0, 1) for n in lens])
        assert counts(c, fem.fem_load_stream(c, ty, t, K)) == 2
    finally:
        fem.fem_destroy(c)


def test_mining_levels(ctx, told, tmp_path):
    """Mining with tuning on measures what the rule sends over the tables, once; a level's shape
    from an earlier file is kept, without a plan made for nothing."""
    I = I_MS4[:2]
    ty, t = stream(77, 4000, K, tie=0.0, gap=2000)
    ty[:2400] = np.tile(np.arange(K, dtype=np.uint8), 150)  # long chains
    want = oracle.mine(ty, t, K, I, 40, 5)
    sid = fem.fem_load_stream(ctx, ty, t, K)
    assert fem.fem_mine_levelwise(ctx, sid, I, 40, 5) == want
    stats = fem.fem_last_mine_stats(ctx)
    plain = told()
    assert plain.count("counted") >= 3
    fem.fem_tune_enable(ctx, True)
    assert fem.fem_mine_levelwise(ctx, sid, I, 40, 5) == want
    first = told()
    assert first.count("counted") >= 2 * plain.count("counted")
    path = tmp_path / "out.jsonl"
    fem.fem_tune_save(ctx, path)
    kinds = [x["key"].split("/")[2] for x in map(json.loads, path.read_text().splitlines())]
    assert kinds.count("3") >= 3
    assert fem.fem_mine_levelwise(ctx, sid, I, 40, 5) == want
    assert len(told()) <= len(plain)
    c = ctx_fixture()
    try:
        lines = []
        for s in stats:
            for p, m, kernel in ((0, s["candidates"], s["kernel_relaxed"]), (1, s["survivors"], s["kernel_exact"])):
                if m:
                    lines.append((key(s["level"], p, 1, m, len(t)), 1, 64, 1))
        load(c, tmp_path, *lines)
        sid = fem.fem_load_stream(c, ty, t, K)
        assert fem.fem_mine_levelwise(c, sid, I, 40, 5) == want
        assert told() == []
        assert all(x["kernel_relaxed"] != fem.KERNEL_HITS for x in fem.fem_last_mine_stats(c))
    finally:
        fem.fem_destroy(c)


def test_joined_level_with_tuning(ctx, told):
    ty, t = stream(2500 + 36, 2500, 36, gap=300)
    I = np.array([[0, 9000]], np.uint32)
    sid = fem.fem_load_stream(ctx, ty, t, 36)
    want = oracle.mine(ty, t, 36, I, 2, 3)
    fem.fem_tune_enable(ctx, True)
    for _ in range(2):
        assert fem.fem_mine_levelwise(ctx, sid, I, 2, 3) == want
        assert fem.fem_last_mine_stats(ctx)[1]["candidates"] >= 40000


def test_tables_are_no_shape(ctx, tmp_path):
    path = tmp_path / "bad.jsonl"
    path.write_text('{"key": "2/0/1/14/8/64", "segments": 1, "threads": 64, "ms": 0, "kernel": 4}\n')
    with pytest.raises(fem.FemError) as e:
        fem.fem_tune_load(ctx, path)
    assert e.value.status == -1
