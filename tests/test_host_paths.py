"""Host code of the library where calls of the runtime fail: every fault is the fake
runtime's (host_cuda.c), no GPU is needed."""
import ctypes

import numpy as np
import pytest

from paper_0905_2200_gb300 import fem
from tests.host_cuda import PLAN_EDGES, PLAN_PARTS_MIN, PLAN_SLABS, Host

vp = ctypes.c_void_p


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return Host(str(tmp_path_factory.mktemp("host_cuda")))


@pytest.fixture()
def ctx(host):
    host.plan = {2: 40, PLAN_EDGES: 50, PLAN_SLABS: 1, PLAN_PARTS_MIN: 1}  # 40 of three nodes
    host.error = 0
    c = vp()
    assert host.lib.fem_create(ctypes.byref(c), 0, ctypes.c_size_t(0)) == 0
    yield c
    assert host.lib.fem_destroy(c) == 0


def load(host, ctx, n, K):
    """A stream of n events a millisecond apart; its id."""
    ty = (np.arange(n) % K).astype(np.uint8)
    t = (1000 * np.arange(n)).astype(np.uint32)
    sid = ctypes.c_int32()
    assert host.lib.fem_load_stream(ctx, ty.ctypes.data_as(vp), t.ctypes.data_as(vp), ctypes.c_uint64(n), K, 0,
                                    None, ctypes.byref(sid)) == 0
    return sid


def count(host, ctx, sid, m=40, pass_=1, K=8):
    """A count of m candidates of three nodes; the kernels that it launched."""
    rec = fem.pack_episodes(np.full(m, 3), np.tile([0, 1, 2] + [0] * 5, (m, 1)), np.zeros((m, 7), int))
    I = np.array([[0, 4000]], np.uint32)
    out = np.zeros(m, np.uint32)
    at = len(host.launches)
    rc = host.lib.fem_count_candidates(ctx, sid, rec.ctypes.data_as(vp), m, 0, I.ctypes.data_as(vp), 1, pass_,
                                       out.ctypes.data_as(vp), 0, None)
    assert rc == 0
    return host.launches[at:]


@pytest.mark.parametrize("failing", [1, 2, 6])
def test_stream_loaded_after_the_tables_made_room(host, ctx, failing):
    """The device is full when a stream is loaded, and the hit tables of an earlier count are
    given up for it: the stream is then the one that was asked for."""
    sid = load(host, ctx, 4000, 8)
    assert any("k_hit_count" in k for k in count(host, ctx, sid))
    at = len(host.launches)
    host.number("host_fail_malloc").value = failing  # of the stream's six allocations
    other = load(host, ctx, 50000, 8)
    assert host.number("host_fail_malloc").value == 0
    assert any("k_bucket" in k for k in host.launches[at:])
    counts = np.full(8, 7, np.uint32)
    assert host.lib.fem_type_counts(ctx, other, counts.ctypes.data_as(vp)) == 0
    assert (counts == 0).all()  # (of all eight types; the fake runtime counts none)
    assert any("k_hit_count" in k for k in count(host, ctx, other))


class Job(ctypes.Structure):
    _fields_ = fem.fem_job._fields_


def batch_jobs(sids, m=40):
    """One job of m candidates of three nodes per stream; the array and what it points to."""
    rec = fem.pack_episodes(np.full(m, 3), np.tile([0, 1, 2] + [0] * 5, (m, 1)), np.zeros((m, 7), int))
    out, kept = np.zeros((len(sids), m), np.uint32), np.zeros((len(sids), m), np.uint8)
    jobs = (Job * len(sids))()
    for k, sid in enumerate(sids):
        jobs[k] = Job(sid.value, 3, m, rec.ctypes.data, 1, out[k].ctypes.data, kept[k].ctypes.data)
    return jobs, (rec, out, kept)


def create_batch(host, ctx, jobs):
    I = np.array([[0, 4000]], np.uint32)
    b = vp()
    assert host.lib.fem_batch_create(ctx, jobs, len(jobs), I.ctypes.data_as(vp), 1, None, ctypes.byref(b)) == 0
    return b


def test_batch_uploads_in_its_streams_order(host, ctx):
    """What the kernels of a batch read is uploaded on their stream: a plain copy from pageable
    memory goes over the default stream, which a stream of the context's kind does not wait for."""
    jobs, kept = batch_jobs([load(host, ctx, 4000, 8), load(host, ctx, 5000, 8)])
    plain = host.number("host_plain_uploads", ctypes.c_uint64)
    at, before = len(host.launches), plain.value
    b = create_batch(host, ctx, jobs)
    assert any("k_hit_count_batch" in k for k in host.launches[at:])
    assert plain.value == before
    assert host.lib.fem_batch_destroy(b) == 0


def join(host):
    """The launches of a level-3 join over one slab of 4 types; the status."""
    fn = getattr(host.lib, "_ZN3fem11launch_joinERKNS_9HitTablesERKNS_10JoinTablesEPKjjjjPjS8_S8_P11CUstream_st")
    h, g = (ctypes.c_uint32 * 64)(), (ctypes.c_uint32 * 64)()
    ctypes.c_uint32.from_buffer(h, 64).value = 1  # n_slabs
    words = (ctypes.c_uint32 * 4096)()
    for k in range(0, 64, 2):
        ctypes.c_uint64.from_buffer(g, 4 * k).value = ctypes.addressof(words)
    return fn(h, g, words, 100, 4, 1, words, words, words, None)


@pytest.mark.parametrize("failing", [1, 2, 3, 4, 5])
def test_a_failed_join_is_not_remembered(host, failing):
    """One of a join's launches (the third is its lists' scan) fails once: that call says so,
    the next one runs."""
    assert join(host) == 0
    host.number("host_fail_launch").value = failing
    assert join(host) == 719
    assert host.number("host_fail_launch").value == 0
    assert join(host) == 0


def test_shared_memory_limits_on_each_device(host):
    """A kernel's limit holds on the device that it was set on: the first launch on another
    device sets it there too, the second does not."""
    attributes = host.number("host_attributes", ctypes.c_uint64)
    host.number("host_devices").value = 2

    def work(device):
        before, c = attributes.value, vp()
        assert host.lib.fem_create(ctypes.byref(c), device, ctypes.c_size_t(0)) == 0
        jobs, kept = batch_jobs([load(host, c, 4000, 8)])
        assert host.lib.fem_batch_destroy(create_batch(host, c, jobs)) == 0
        assert join(host) == 0
        assert host.lib.fem_destroy(c) == 0
        return attributes.value - before

    try:
        work(0)
        assert work(0) == 0
        assert work(1) >= 4  # two builds, a batch's count, the join
        assert work(1) == 0
    finally:
        host.number("host_devices").value = 1
        host.rt.cudaSetDevice(0)


@pytest.mark.parametrize("m", [300000, 65536, 65537])
def test_batch_of_many_candidates_on_the_host(host, ctx, m):
    """Creating a batch takes little host memory whatever the number of its candidates (none of
    it can be refused across the C boundary), and every candidate's length is looked at."""
    host.plan[2] = m
    sid = load(host, ctx, 4000, 8)
    jobs, kept = batch_jobs([sid, sid], m)
    taken = host.number("host_new_max", ctypes.c_size_t)
    taken.value = 0
    b = create_batch(host, ctx, jobs)
    assert 0 < taken.value <= 2 << 20
    assert host.lib.fem_batch_destroy(b) == 0
    for at in (0, 65535, m - 1):
        kept[0][at, 15] = 2
        I = np.array([[0, 4000]], np.uint32)
        assert host.lib.fem_batch_create(ctx, jobs, 2, I.ctypes.data_as(vp), 1, None, ctypes.byref(vp())) == -1
        kept[0][at, 15] = 3


def used(host, ctx):
    n = ctypes.c_size_t()
    assert host.lib.fem_mem_usage(ctx, ctypes.byref(n), None) == 0
    return n.value


def many(m, edges, slabs):
    """The words of a plan, and of a validation, of m candidates of three nodes not in runs."""
    return {2: m, PLAN_EDGES: edges, PLAN_SLABS: slabs, PLAN_PARTS_MIN: 1, ("info", 0): 8, ("info", 2): m}


def context(host, budget=0):
    c = vp()
    assert host.lib.fem_create(ctypes.byref(c), 0, ctypes.c_size_t(budget)) == 0
    return c


def test_transfer_tables_are_bounded_in_bytes(host):
    """Many candidates on a long stream: the tables between its segments take at most a 64th of
    the device's memory, and no more than a 16th is kept in all."""
    total, largest = host.number("host_total", ctypes.c_size_t), host.number("host_malloc_max", ctypes.c_size_t)
    was, total.value = total.value, 16 << 30
    host.error = 0
    try:
        c = context(host)
        for slabs, edges in ((2000, 30000), (4000, 60000)):  # 0.5 and 1.9 GB of edges
            host.plan = many(100000, edges, slabs)
            sid = load(host, c, 4000, 8)
            largest.value = 0
            assert any("k_hit_count" in k for k in count(host, c, sid, 100000))
            assert largest.value <= max(slabs * edges * 8, total.value // 64) + 4096
            assert used(host, c) <= total.value // 16 + (16 << 20)
        assert host.lib.fem_destroy(c) == 0
    finally:
        total.value = was


def test_transfer_tables_make_room_for_a_stream(host):
    """Under a budget a stream that fits beside the other one is loaded, whatever was counted
    before."""
    host.error = 0
    host.plan = many(100000, 6000, 400)
    c = context(host, 110 << 20)
    sid = load(host, c, 4000, 8)
    assert any("k_hit_count" in k for k in count(host, c, sid, 100000))
    assert used(host, c) > 70 << 20
    load(host, c, 4_000_000, 8)  # 55 MB
    assert host.lib.fem_destroy(c) == 0


def test_tables_make_room_for_a_server(host, ctx):
    sid = load(host, ctx, 4000, 8)
    assert any("k_hit_count" in k for k in count(host, ctx, sid))
    v, before = vp(), used(host, ctx)
    host.number("host_fail_malloc").value = 1
    assert host.lib.fem_server_create(ctx, None, ctypes.byref(v)) == 0
    assert used(host, ctx) < before
    assert host.lib.fem_server_destroy(v) == 0


def test_tables_of_a_count_make_room_for_a_batch(host):
    """A batch goes over hit tables of its own under a budget that the tables of an earlier count
    would leave no room in."""
    host.error = 0
    host.plan = many(100000, 6000, 400)
    c = context(host, 110 << 20)
    sid = load(host, c, 4000, 8)
    assert any("k_hit_count" in k for k in count(host, c, sid, 100000))
    assert used(host, c) > 70 << 20
    host.plan = many(40, 6000, 400)
    jobs, kept = batch_jobs([sid, sid, sid])
    at = len(host.launches)
    b = create_batch(host, c, jobs)
    assert any("k_hit_count_batch" in k for k in host.launches[at:])
    assert host.lib.fem_batch_destroy(b) == 0
    assert host.lib.fem_destroy(c) == 0


def test_only_the_sequence_word_ends_a_wait(host, ctx):
    """Whatever the published words are, also the sequence number that is waited for, the host
    takes them when the word behind them says so and not before (here it never does)."""
    sid = load(host, ctx, 4000, 8)
    assert any("k_hit_count" in k for k in count(host, ctx, sid))
    publish = host.publish_seq

    def count_rc(m):
        rec = fem.pack_episodes(np.full(m, 3), np.tile([0, 1, 2] + [0] * 5, (m, 1)), np.zeros((m, 7), int))
        I, out = np.array([[0, 4000]], np.uint32), np.zeros(m, np.uint32)
        return host.lib.fem_count_candidates(ctx, sid, rec.ctypes.data_as(vp), m, 0, I.ctypes.data_as(vp), 1, 0,
                                             out.ctypes.data_as(vp), 0, None)

    try:
        host.publish_seq = False
        assert count_rc(40) == -8   # the plan's words
        assert count_rc(300) == -8  # a validation's
    finally:
        host.publish_seq = publish
    assert count_rc(40) == 0
