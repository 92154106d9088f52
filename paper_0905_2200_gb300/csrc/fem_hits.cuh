// fem_hits.cuh -- the counting passes over hit tables, for candidate sets whose episodes
// share edges rather than prefixes (any set a user brings); lengths 1..8.
//
// The rule is the latest-chain one (fem_chain.cuh): a last-node event i completes an
// occurrence iff a chain reaches it whose first event is at or after st (one past the
// last completion), the chain taking at every edge the latest admitted event before i
// (relaxed pass; within hi) or the latest one older than lo (exact pass; within hi).
// Which events of type b lie in the interval before an event of type c depends on the
// edge (b, interval, c) alone, and a set has far fewer edges than (episode, node) pairs:
// 100,000 random episodes of 64 types and four intervals have 375,000 edges, 16,128 of
// them different.  So the passes run in two steps:
//
//   * The stream is cut into slabs in which no type has more than 32 events, so that a
//     set of a type's events in a slab is a word.  k_hit_build, one block per slab (several
//     where there are few), gives a warp to a next type and a lane to each earlier type; the
//     lane goes through the next type's events and from each a few steps back down its own
//     type's, and writes every edge's hits: a mask of the next type's events that have one of
//     the earlier type in the interval, and per such event the range of those (as bits of a
//     64-bit word: the 32 events before the slab, then the slab's own) and the latest of them.
//   * k_hit_count, one thread per (episode, segment), goes through the slabs with the
//     admitted events of every node as a 64-bit word.  A node's admitted events are those
//     of its edge's hits whose range meets the node before's word; the highest bit of the
//     meet is the latest admitted event, whose chain's start the event takes over.
//
// A thread therefore does work only for hits (a tenth to a third of the events), where the
// per-thread machine spends 60 to 150 issue slots on every event of every node, and the cost
// of an episode hardly grows with its length: a node after one without admitted events is
// passed over.  Measured (two-pass and single-pass counts, without tables -> over them): an
// hour of 64 types at 50 Hz, 100,000 episodes of 3-5 nodes, 332 -> 147 ms; 20,011 episodes
// of 2-8 nodes on 196,000 events, 6.02 -> 1.54 ms; a bursting recording 31.4 -> 6.8 ms (no
// rings, and twice the entry classes in the first try); 100 episodes on 3,400 events, 0.95 ->
// 0.27 ms (all lengths planned in one host wait).  What bounds it: in the count, the latency
// of the tables' L2 reads and warp issue slots (35-45% used at 15 to 22 warps per SM, about
// half of the lanes active: lanes wait for the one with the most hits, so the candidates are
// ordered by their last three intervals); in the build, issue slots (62% used).
//
// MapConcatenate (template flag MC): the entry classes and transfer tables are those of
// the other counting kernels, so the same stitch composes them; segments are runs of
// slabs.  An episode that needs more classes than its table has slots is marked for the
// host's recount.  A window that may hold more than 32 events of a type sets ERR_DENSE
// (the whole count is then done by the other kernels).
#pragma once

#include <string.h>

#include "fem_internal.cuh"

namespace fem {

constexpr uint32_t HIT_CLASSES = 32;   // most entry classes per table
constexpr uint32_t HIT_PARTS = 64;     // most slabs per chunk (32 events each)
constexpr uint32_t HIT_ROW = 65;       // words per type of a slab's rank tables (64 and a pad)
constexpr uint32_t HIT_BUILD_T = 256;  // threads of a build block

// inner nodes of an episode of up to nmax nodes, and those whose chains' starts are in
// shared memory
__host__ __device__ constexpr int hit_inner(int nmax) { return nmax > 2 ? nmax - 2 : 0; }
__host__ __device__ constexpr int hit_shared(int nmax) { return nmax <= 5 ? hit_inner(nmax) : 2; }

// The stored form of a hit: bits 0-5 the first event of the range, 6-11 their number (1 to
// 32; start + number at most 64), from bit 16 on the low half of the latest one's index in
// the stream.  That holds for every stored hit, also on streams too dense for the tables:
// the host learns of those only after the kernels that read them have run.
__device__ __forceinline__ uint32_t hit_pack(uint32_t start, uint32_t len, uint32_t latest) {
    return latest << 16 | len << 6 | start;
}

extern __shared__ __align__(128) uint8_t fem_hit_smem[];

// One thread's episode going through the slabs.  NMAX: most nodes of an episode.  Shared
// memory: the chains' starts (low half) of the inner nodes' last 64 events,
// [node][event & 63][thread]; of long episodes the later nodes', which few chains reach,
// are in local memory (all of eight nodes' in shared memory left an SM two blocks).
template <int NMAX>
struct HitEpisode {
    uint32_t N, last;                 // nodes, last type
    uint64_t W;                       // sum of hi
    uint32_t edge[NMAX], type[NMAX];  // edge d joins node d - 1 to node d

    // The candidate of the thread's slot; false if there is none or it is malformed.
    __device__ __forceinline__ bool load(const CountParams &p, uint32_t ci) {
        N = 0, last = 0, W = 0;
#pragma unroll
        for (int d = 0; d < NMAX; ++d) edge[d] = 0, type[d] = 0;
        if (ci >= p.m) return false;
        const uint4 v = reinterpret_cast<const uint4 *>(p.cands)[p.gather ? p.gather[ci] : ci];
        fem_episode rec;
        memcpy(&rec, &v, sizeof(rec));
        bool ok = rec.len >= 1 && rec.len <= NMAX;
#pragma unroll
        for (int d = 0; d < NMAX; ++d) {
            if (ok && d < (int)rec.len) {
                type[d] = rec.types[d];
                ok = type[d] < p.K;
                last = type[d];
                if (ok && d > 0) {
                    const uint32_t iv = rec.ivl[d > 0 ? d - 1 : 0];
                    ok = iv < p.n_ivl;
                    if (ok) {
                        W += p.ivl[iv].y;
                        edge[d] = p.hits.edge_id[(type[d] * p.K + type[d > 0 ? d - 1 : 0]) * p.n_ivl + iv];
                    }
                }
            }
        }
        if (ok) N = rec.len;
        else atomicOr(p.err, ERR_BADEP);
        return ok;
    }

    // Slabs [s_w, s1) (the same in every lane of the warp): slab(s) before each, then
    // leaf(s, r, S) for every last-node event (the slab's r-th of its type) that a chain
    // reaches, in order; S is the index of the latest chain's first event.
    template <typename SLAB, typename LEAF>
    __device__ __forceinline__ void walk(const HitTables &h, uint32_t s_w, uint32_t s1, SLAB &&slab,
                                         LEAF &&leaf) const {
        constexpr int SHARED = hit_shared(NMAX);
        const uint32_t T = blockDim.x;
        uint16_t *starts = reinterpret_cast<uint16_t *>(fem_hit_smem) + threadIdx.x;
        uint16_t deep[hit_inner(NMAX) > SHARED ? (hit_inner(NMAX) - SHARED) * 64 : 1];
        auto start_of = [&](int d, uint32_t at) -> uint16_t & {
            if (hit_inner(NMAX) <= SHARED || d <= SHARED)
                return starts[((uint32_t)(d - 1) * 64u + (at & 63u)) * T];
            return deep[(uint32_t)(d - 1 - SHARED) * 64u + (at & 63u)];
        };
        // Per inner node: its admitted events among the 32 before the slab, and where the
        // event 32 before the slab's first sits in `starts`.
        uint32_t hist[NMAX], at[NMAX];
#pragma unroll
        for (int d = 0; d < NMAX; ++d) hist[d] = 0, at[d] = 0;
        // An edge's mask is asked for a slab ahead, its first ranges before any edge's are
        // used; in episodes of six or more nodes only the first edges', the others' when the
        // node before has any admitted event, which is seldom so.
        constexpr int MASKS = NMAX <= 5 ? NMAX : 4, HEADS = NMAX <= 5 ? NMAX : 3, G = 4;
        uint2 nxt[MASKS];
#pragma unroll
        for (int d = 1; d < MASKS; ++d)
            nxt[d] = d < (int)N ? h.edge[(uint64_t)s_w * h.n_edges + edge[d]] : make_uint2(0u, 0u);
        for (uint32_t s = s_w; s < s1; ++s) {
            uint2 now[MASKS];
            uint32_t cn[NMAX];
            const uint8_t *crow = h.count + (uint64_t)s * h.types;
            const uint2 *erow = h.edge + (uint64_t)s * h.n_edges;
#pragma unroll
            for (int d = 1; d < NMAX; ++d) {
                cn[d] = d + 1 < NMAX && d + 1 < (int)N ? crow[type[d]] : 0u;
                if (d >= MASKS) continue;
                now[d] = nxt[d];
                if (s + 1 < s1 && d < (int)N) nxt[d] = erow[h.n_edges + edge[d]];
            }
            slab(s);
            const uint32_t end = h.begin[s + 1];  // a low half names one of the 65,536 before it
            uint32_t head[HEADS][G];
#pragma unroll
            for (int d = 1; d < HEADS; ++d) {
                const uint32_t k = d < (int)N ? __popc(now[d].x) : 0u;
#pragma unroll
                for (int g = 0; g < G; ++g) head[d][g] = (uint32_t)g < k ? __ldg(h.range + now[d].y + g) : 0u;
            }
            uint64_t before = 0;  // admitted events of the node before
#pragma unroll
            for (int d = 1; d < NMAX; ++d) {
                if (d >= (int)N) continue;
                const bool is_leaf = d + 1 == (int)N;
                uint32_t bits = 0, rg = 0, cur = 0, e4[G];
                if (d == 1 || before) {
                    const uint2 e = d < MASKS ? now[d < MASKS ? d : 0] : erow[edge[d]];
                    bits = e.x, rg = e.y;
                    const uint32_t k = __popc(bits);
#pragma unroll
                    for (int g = 0; g < G; ++g)
                        e4[g] = d < HEADS ? head[d < HEADS ? d : 0][g]
                                          : (uint32_t)g < k ? __ldg(h.range + rg + g) : 0u;
                }
                while (bits) {
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        if (!bits) break;
                        const uint32_t r = __ffs(bits) - 1;
                        bits &= bits - 1u;
                        const uint32_t e = e4[g];
                        uint32_t S = e >> 16;
                        if (d > 1) {
                            const uint32_t start = e & 63u, len = (e >> 6) & 63u;
                            const uint32_t w = (uint32_t)(before >> start) & (0xFFFFFFFFu >> (32u - len));
                            if (!w) continue;
                            S = start_of(d - 1, at[d - 1] + start + 31u - (uint32_t)__clz(w));
                        }
                        if (!is_leaf) {
                            cur |= 1u << r;
                            if (d + 1 < NMAX) start_of(d, at[d] + 32u + r) = (uint16_t)S;
                        } else {
                            leaf(s, r, end - ((end - S) & 0xFFFFu));
                        }
                    }
                    if (!bits) break;
                    rg += G;
                    const uint32_t k = __popc(bits);
#pragma unroll
                    for (int g = 0; g < G; ++g) e4[g] = (uint32_t)g < k ? __ldg(h.range + rg + g) : 0u;
                }
                if (!is_leaf) {
                    before = (uint64_t)cur << 32 | hist[d];
                    hist[d] = (uint32_t)(before >> cn[d]);
                }
            }
#pragma unroll
            for (int d = 1; d < NMAX; ++d) at[d] += cn[d];
        }
    }

    // The index of the slab's r-th event of the last type.
    __device__ __forceinline__ uint32_t index(const HitTables &h, uint32_t s, uint32_t r) const {
        const uint32_t end = h.begin[s + 1];
        const uint32_t i = h.index[h.begin[s] + h.place[(uint64_t)s * h.types + last] + r];
        return end - ((end - i) & 0xFFFFu);
    }
};

// Count one tile of candidates over segment `seg`.
template <int NMAX, bool MC>
__device__ __forceinline__ void hit_count_tile(const CountParams &p, uint32_t tile, uint32_t seg) {
    const uint32_t ci = tile * blockDim.x + threadIdx.x;
    const HitTables &h = p.hits;
    // tables that are too dense (the build before said so) are not worth a count
    const uint32_t e0 = *reinterpret_cast<const volatile uint32_t *>(p.err);
    HitEpisode<NMAX> ep;
    const bool ok = ep.load(p, ci);
    if (e0 & ERR_DENSE) return;
    const uint64_t W = ep.W;

    // ------------------------------------------------------------ segment and window
    const uint32_t s0 = seg * p.cps, s1 = min(s0 + p.cps, h.n_slabs);
    const bool last_seg = s1 >= h.n_slabs;
    const uint32_t L = h.begin[s0];
    uint32_t X = 0, Xn = 0, s_w = s0;
    uint32_t st = 0;  // class "none" (or the only class): one past its last completion
    if (MC) {
        if (ok && seg > 0) {
            // class "none" is a machine started at the window start X = t[L] - W; chains
            // of the window's events start no earlier than X - W
            const uint32_t tL = p.t[L];
            X = (uint64_t)tL >= W ? (uint32_t)(tL - W) : 0u;
            const uint32_t X2 = (uint64_t)tL >= 2 * W ? (uint32_t)(tL - 2 * W) : 0u;
            while (s_w > 0 && h.t0[s_w] >= X2) --s_w;
            uint32_t a = h.begin[s_w], b = L;  // the first event at or after X
            while (a < b) {
                const uint32_t mid = a + (b - a) / 2;
                if (p.t[mid] >= X) b = mid;
                else a = mid + 1;
            }
            st = a;
        }
        if (!last_seg) {
            const uint32_t tR = h.t0[s1];
            Xn = (uint64_t)tR >= W ? (uint32_t)(tR - W) : 0u;
        }
        s_w = __reduce_min_sync(0xffffffffu, ok ? s_w : s0);
    }
    const uint32_t first = st;  // nothing before it is looked at in the window

    // ------------------------------------------------------------ counting state
    uint32_t cnt = 0;
    // entry classes 1 .. classes - 1 (local memory: they are touched near the segment's
    // start and in its result only); class j restarts after the last-node event c_key[j]
    // of the window, and a class that has merged into class "none" keeps its count
    // relative to it
    constexpr uint32_t SC = MC ? HIT_CLASSES : 1;
    const uint32_t classes = p.hit_classes;
    uint32_t c_st[SC], c_cnt[SC], c_key[SC], c_t[SC];
    uint32_t used = 0, umask = 0, t_none = X;  // t_none: no chain from before it reaches class "none"
    bool c0_done = false, class_overflow = false;
    // Every chain that ends at time t or later starts at t - W or later: two classes whose
    // last completions are both older see the same chains.  Their exits agree too while
    // neither completion reaches into the next segment's window.
    auto merge_before = [&](uint32_t t, bool window) {
        const uint32_t tw = (uint64_t)t > W ? (uint32_t)(t - W) : 0u;
        for (uint32_t u = umask; u; u &= u - 1u) {
            const uint32_t j = __ffs(u) - 1;
            const uint32_t tm = max(t_none, c_t[j]);
            if (tm < tw && (last_seg || tm < Xn)) {
                c_cnt[j] -= cnt;
                umask &= ~(1u << j);
                if (window) used &= ~(1u << j);
            }
        }
    };
    // a last-node event with a chain from S on, while classes are apart
    auto slow_event = [&](uint32_t gidx, uint32_t S) {
        const uint32_t t = p.t[gidx];
        const uint32_t inc = gidx >= L ? 1u : 0u;
        if (!inc && gidx < first) return;
        merge_before(t, !inc);
        if (S >= st) st = gidx + 1, cnt += inc, c0_done = true, t_none = t;
        for (uint32_t u = umask; u; u &= u - 1u) {
            const uint32_t j = __ffs(u) - 1;
            if (S >= c_st[j]) {
                if (!inc) {  // refuted: the serial machine completes again before L
                    used &= ~(1u << j), umask &= ~(1u << j);
                    continue;
                }
                c_st[j] = gidx + 1, c_t[j] = t, ++c_cnt[j];
            }
            if (c_st[j] == st) {
                c_cnt[j] -= cnt;
                umask &= ~(1u << j);
                if (!inc) used &= ~(1u << j);
            }
        }
        if (!inc && st != gidx + 1) {  // entry class r = gidx: the chains after it
            const uint32_t free_slots = ~used & (classes >= 32 ? ~1u : ((1u << classes) - 2u));
            if (free_slots) {
                const uint32_t j = __ffs(free_slots) - 1;
                c_key[j] = gidx, c_st[j] = gidx + 1, c_cnt[j] = 0, c_t[j] = t;
                used |= 1u << j;
                umask |= 1u << j;
            } else {
                class_overflow = true;
            }
        }
    };

    // ------------------------------------------------------------ slabs
    if (ep.N == 1) {
        for (uint32_t s = s0; s < s1; ++s) cnt += h.count[(uint64_t)s * h.types + ep.last];
        ep.N = 0;
    }
    ep.walk(
        h, s_w, s1,
        [&](uint32_t s) {
            if (MC && umask) merge_before(h.t0[s], s < s0);
        },
        [&](uint32_t s, uint32_t r, uint32_t S) {
            const bool slow = MC && (s < s0 || umask);
            if (!slow && S < st) return;
            const uint32_t gidx = ep.index(h, s, r);
            if (slow) {
                slow_event(gidx, S);
            } else {
                st = gidx + 1u;
                ++cnt;
                if (MC) c0_done = true;
            }
        });

    // ------------------------------------------------------------ results
    if (ci >= p.m) return;
    if (class_overflow) {
        atomicOr(p.err, ERR_CLASS);
        p.redo[ci] = 1;
    }
    if constexpr (!MC) {
        p.out[ci] = cnt;
    } else {
        uint4 *tab = p.tables + ((uint64_t)seg * p.m + ci) * classes;
        const uint32_t n_slots = used ? 32u - __clz(used) : 1u;
        for (uint32_t j = 0; j < n_slots; ++j) {
            uint4 e = make_uint4(CLS_EMPTY, 0, CLS_NONE, j == 0 ? n_slots : 0u);
            if (j == 0 || ((used >> j) & 1u)) {
                const bool own = j > 0 && ((umask >> j) & 1u);  // not merged into class "none"
                const uint32_t cj = j == 0 ? cnt : own ? c_cnt[j] : cnt + c_cnt[j];
                uint32_t ex = own ? c_st[j] - 1u : c0_done ? st - 1u : CLS_NONE;
                if (ex != CLS_NONE && !last_seg && p.t[ex] < Xn) ex = CLS_NONE;
                e = make_uint4(j == 0 ? CLS_NONE : c_key[j], cj, ex, j == 0 ? n_slots : 0u);
            }
            tab[j] = e;
        }
    }
}

template <int NMAX, bool MC>
__global__ void __launch_bounds__(128) k_hit_count(const CountParams p) {
    hit_count_tile<NMAX, MC>(p, blockIdx.x, blockIdx.y);
}

// The same for a batch: list[i] names a part (z) whose items are the blocks from list[i].x on,
// the list[i].y tiles of a segment one after the other.  A part's candidate count may be
// the device's (survivors); its items are for the most there can be.
template <int NMAX>
__global__ void __launch_bounds__(128) k_hit_count_batch(const CountParams *__restrict__ parts,
                                                         const uint4 *__restrict__ list, uint32_t n_list) {
    __shared__ CountParams p;
    uint32_t lo = 0, hi = n_list;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (list[mid].x <= blockIdx.x) lo = mid;
        else hi = mid;
    }
    const uint4 e = list[lo];
    const uint32_t r = blockIdx.x - e.x, tile = r % e.y;
    if (tile * blockDim.x >= parts[e.z].m) return;  // uniform
    if (threadIdx.x == 0) p = parts[e.z];
    __syncthreads();
    hit_count_tile<NMAX, true>(p, tile, r / e.y);
}

// Window-based frequency (fem_windows.cu) of one tile of candidates over segment `seg`: the
// starts whose window holds a chain ending at last-node event j are (t[j] - w, t[S]], S the
// latest chain's first event (the exact pass's chains).  The ranges' left ends increase, so
// what is at or below the greatest right end so far is covered, and event j adds what lies
// above it.  A segment finds that end from the last-node events of the w before it (an
// earlier one's range ends before its own ranges begin), and the segments' sums add up: no
// stitch.  One thread per episode walked the whole stream before (fem_windows.cu), few warps
// and long chains of loads: 16,128 pairs on 406,000 events 15.5 ms, now 0.10 ms and 0.26
// for the tables.
template <int NMAX>
__global__ void __launch_bounds__(128) k_hit_windows(const CountParams p, const uint32_t *order,
                                                     uint32_t w, unsigned long long *out) {
    const uint32_t ci = blockIdx.x * blockDim.x + threadIdx.x, seg = blockIdx.y;
    const HitTables &h = p.hits;
    HitEpisode<NMAX> ep;
    const bool ok = ep.load(p, ci);
    const uint32_t s0 = seg * p.cps, s1 = min(s0 + p.cps, h.n_slabs);
    uint32_t s_w = s0;
    if (ok) {
        // chains of the events of the w before the segment: none starts before back
        const uint64_t t = h.t0[s0], reach = (uint64_t)w + ep.W;
        const uint32_t back = t >= reach ? (uint32_t)(t - reach) : 0u;
        while (s_w > 0 && h.t0[s_w] >= back) --s_w;
    }
    s_w = __reduce_min_sync(0xffffffffu, s_w);
    int64_t covered = -0x7FFFFFFFFFFFFFFFll;
    uint64_t sum = 0;
    auto add = [&](uint32_t s, int64_t t, int64_t right) {
        const int64_t left = t - (int64_t)w;  // starts left + 1 .. right
        if (left >= right) return;            // the chain is longer than the window
        if (s >= s0) sum += (uint64_t)max((int64_t)0, right - max(left, covered));
        covered = max(covered, right);
    };
    if (ep.N == 1) {
        for (uint32_t s = s_w; s < s1; ++s) {
            const uint32_t n = h.count[(uint64_t)s * h.types + ep.last];
            for (uint32_t r = 0; r < n; ++r) {
                const int64_t t = p.t[ep.index(h, s, r)];
                add(s, t, t);
            }
        }
        ep.N = 0;
    }
    ep.walk(
        h, s_w, s1, [](uint32_t) {},
        [&](uint32_t s, uint32_t r, uint32_t S) { add(s, p.t[ep.index(h, s, r)], p.t[S]); });
    if (ok && sum) atomicAdd(&out[order[ci]], (unsigned long long)sum);
}

// Level-3 counts of level-wise mining, all at once: every frequent pair (a, v, b) joined with
// every frequent pair (b, u, c), edges numbered by the tables.  Each b event gets the list
// of the pairs (a, v, b) that admit it, with the low half of the index of its latest a
// event; the lists stand by type and then time, so that a range of b events is one run of
// entries.  A warp takes a pair (b, u, c) and goes through its hits, c events with the range
// of b events before them, 32 list entries at a time: an entry names a candidate, whose
// threshold and count are the warp's own in shared memory.  A candidate that comes twice in
// a run (two b events admitted) needs no order: the later b event's chain starts no earlier,
// so some entry passes the threshold exactly if the latest one does, and after it none does.
//
// What bounds it: issue slots, about 12 for 32 entries, and the lists' latency.  Measured on
// the deep search of 64 types, 300 s (2.4 million candidates from 12,400 frequent pairs):
// 2.4 ms relaxed and 1.2 ms exact, after 0.4 ms for the tables and lists.  A thread for each
// (a, v, b) that looked at every hit of (b, u, c) took 7.3 ms: one in five admits it.  The
// latest-chain kernel, which looks up every last-node event of every candidate: 31.2 ms
// relaxed and 15.1 ms exact.
constexpr uint32_t JOIN_QUEUE = 64;  // hits a warp takes at a time, at least a slab's 32

__global__ void __launch_bounds__(256) k_join(const HitTables h, const JoinTables g, uint32_t n_events,
                                              uint32_t K, uint32_t n_ivl, uint32_t *__restrict__ out) {
    if (*g.err & ERR_DENSE) return;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x / 32;
    const uint32_t slots = K * n_ivl, b = blockIdx.x, second = blockIdx.y * NW + warp;
    if (second >= g.n_begins[b]) return;  // (warps are on their own)
    const uint2 pair = g.begins[b * slots + second];
    const uint32_t n_first = g.n_ends[b], c = pair.y / n_ivl, e2 = pair.x;
    if (n_first == 0) return;
    uint4 *queue = reinterpret_cast<uint4 *>(fem_hit_smem) + warp * JOIN_QUEUE;
    uint2 *state = reinterpret_cast<uint2 *>(reinterpret_cast<uint4 *>(fem_hit_smem) + NW * JOIN_QUEUE) +
                   (size_t)warp * slots;  // threshold, count
    for (uint32_t i = lane; i < n_first; i += 32) state[i] = make_uint2(0u, 0u);
    const uint32_t *rank = g.rank + (uint64_t)b * h.n_slabs;
    // 32 list entries: the c event i completes the candidates whose chain starts late enough
    auto meet = [&](bool in, uint32_t v, uint32_t i) {
        uint2 z = make_uint2(~0u, 0u);
        if (in) z = state[v >> 16];
        __syncwarp();
        if (i - ((i - v) & 0xFFFFu) >= z.x) state[v >> 16] = make_uint2(i + 1u, z.y + 1u);
        __syncwarp();
    };
    uint2 e = lane < h.n_slabs ? h.edge[(uint64_t)lane * h.n_edges + e2] : make_uint2(0u, 0u);
    for (uint32_t s = 0; s < h.n_slabs;) {
        // lane k: slab s + k; as many slabs as the queue has room for
        uint32_t at = __popc(e.x);
#pragma unroll
        for (int d = 1; d < 32; d *= 2) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, at, d);
            if (lane >= (uint32_t)d) at += o;
        }
        const uint32_t take = __popc(__ballot_sync(0xffffffffu, at <= JOIN_QUEUE));
        const uint32_t n = __shfl_sync(0xffffffffu, at, take - 1);
        const uint32_t sl = s + lane;
        if (lane < take && e.x) {
            const uint32_t r0 = rank[sl];
            const uint32_t end = h.begin[sl + 1], place = h.begin[sl] + h.place[(uint64_t)sl * h.types + c];
            uint32_t q = at - __popc(e.x), rg = e.y;
            for (uint32_t bits = e.x; bits; bits &= bits - 1u)
                queue[q++] = make_uint4(rg++, place + __ffs(bits) - 1u, r0, end);
        }
        s += take;
        e = s + lane < h.n_slabs ? h.edge[(uint64_t)(s + lane) * h.n_edges + e2] : make_uint2(0u, 0u);
        __syncwarp();
#pragma unroll
        for (uint32_t q = lane; q < JOIN_QUEUE; q += 32) {
            if (q < n) {
                const uint4 z = queue[q];
                const uint32_t r = h.range[z.x], i = h.index[z.y];
                const uint32_t p0 = min(z.z + (r & 63u) - 32u, n_events), p1 = min(p0 + ((r >> 6) & 63u), n_events);
                const uint32_t from = g.off[p0];
                queue[q] = make_uint4(from, g.off[p1] - from, z.w - ((z.w - i) & 0xFFFFu), 0u);
            }
        }
        __syncwarp();
        constexpr int G = 4;
        for (uint32_t q0 = 0; q0 < n; q0 += G) {
            uint4 z[G];
            uint32_t v[G], w[G];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                z[k] = q0 + k < n ? queue[q0 + k] : make_uint4(0u, 0u, 0u, 0u);
                v[k] = lane < z[k].y ? g.list[z[k].x + lane] : 0u;
                w[k] = lane + 32u < z[k].y ? g.list[z[k].x + lane + 32u] : 0u;
            }
#pragma unroll
            for (int k = 0; k < G; ++k) {
                meet(lane < z[k].y, v[k], z[k].z);
                if (z[k].y > 32) meet(lane + 32u < z[k].y, w[k], z[k].z);
                for (uint32_t l = lane + 64; l - lane < z[k].y; l += 32)
                    meet(l < z[k].y, l < z[k].y ? g.list[z[k].x + l] : 0u, z[k].z);
            }
        }
        __syncwarp();
    }
    for (uint32_t i = lane; i < n_first; i += 32)
        out[((uint64_t)b * slots + pair.y) * slots + g.ends[b * slots + i].y] = state[i].y;
}

}  // namespace fem
