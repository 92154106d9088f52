// fem_hits.cu -- the hit tables of a stream and an edge set, the launches of the counting
// kernels that read them, and the plan both need: the candidates checked and ordered, the
// edges they use numbered, the stream cut into slabs.
#include <algorithm>

#include "fem_hits.cuh"

namespace fem {

namespace {

// Exclusive sum of one value per thread over a block of 1024; *total = the sum.
__device__ __forceinline__ uint32_t block_scan_1024(uint32_t v, uint32_t *total) {
    __shared__ uint32_t wsum[33];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= (uint32_t)d) inc += y;
    }
    __syncthreads();
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint32_t x = wsum[lane];
        uint32_t s = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= (uint32_t)d) s += y;
        }
        wsum[lane] = s - x;
        if (lane == 31) wsum[32] = s;
    }
    __syncthreads();
    *total = wsum[32];
    return wsum[w] + inc - v;
}

// Exclusive sums of f(w[i]) over i < n by one block of 1024: g(i, w[i], sum before i) for
// every i, *total = the whole sum.  A warp takes a run of words and goes through it 32 at
// a time, twice.
template <typename F, typename G>
__device__ __forceinline__ void scan_words(const uint32_t *w, uint32_t n, uint32_t *total, F &&f, G &&g) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t per = ((n + 31) / 32 + 31) & ~31u, lo = min(warp * per, n), hi = min(lo + per, n);
    uint32_t sum = 0;
#pragma unroll 4
    for (uint32_t i = lo + lane; i < hi; i += 32) sum += f(w[i]);
    sum = __reduce_add_sync(0xffffffffu, sum);
    uint32_t at = block_scan_1024(lane == 0 ? sum : 0u, total);
    at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll 4
    for (uint32_t i0 = lo; i0 < hi; i0 += 32) {
        const uint32_t i = i0 + lane, v = i < hi ? w[i] : 0u, x = i < hi ? f(v) : 0u;
        uint32_t inc = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (uint32_t)d) inc += y;
        }
        if (i < hi) g(i, v, at + inc - x);
        at += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncthreads();
}

// Bin of a valid candidate: the launch that counts it (plan_group), the places of its last
// three intervals in the set (in `parts` parts each, the last first: the longest work
// first), its last type.
__device__ __forceinline__ uint32_t plan_bin(const fem_episode &e, const PlanArgs &a) {
    const uint32_t N = e.len;
    uint32_t bin = plan_group(N, a.fine);
    for (uint32_t k = 1; k <= 3; ++k)
        bin = bin * a.parts + (N > k ? a.parts - 1u - e.ivl[N - 1 - k] * a.parts / a.n_ivl : 0u);
    return bin * a.K + e.types[N - 1];
}

// Each candidate's bin and its place in the bin (the order within a bin is arbitrary: a
// candidate's count does not depend on it), the bins' sizes, the edges in use, and the
// plan words: per length 1..8 the candidates, [PLAN_REP] those with a repeated type,
// [PLAN_SPAN] 2^32 - 1 less the least time that a chunk spans (and of k_plan_scan [PLAN_DENSE]:
// an edge in use leads from a type too dense for the tables), [PLAN_RUNS] where asked for.
__global__ void __launch_bounds__(256) k_plan_bins(const PlanArgs a) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t rep = 0, bad = 0, len = 0, brk = 0;
    if (i < a.m) {
        const fem_episode e = a.cands[a.gather ? a.gather[i] : i];
        const uint32_t N = e.len;
        if (a.runs && i > 0) {  // a run of candidates sharing the prefix of a last node ends here
            const fem_episode q = a.cands[a.gather ? a.gather[i - 1] : i - 1];
            brk = q.len != N;
            for (uint32_t k = 0; k + 1 < N && k < FEM_MAX_LEN; ++k) brk |= q.types[k] != e.types[k];
            for (uint32_t k = 0; k + 2 < N && k < FEM_MAX_LEN - 1; ++k) brk |= q.ivl[k] != e.ivl[k];
        }
        if (N < 1 || N > FEM_MAX_LEN) {
            bad = ERR_BADEP;
        } else {
            for (uint32_t k = 0; k < N; ++k)
                if (e.types[k] >= a.K) bad = ERR_BADEP;
            for (uint32_t k = 0; k + 1 < N; ++k)
                if (e.ivl[k] >= a.n_ivl) bad = ERR_BADEP;
            for (uint32_t x = 0; x < N; ++x)
                for (uint32_t y = x + 1; y < N; ++y)
                    if (e.types[x] == e.types[y]) rep = 1;
        }
        if (!bad) {
            len = N;
            const uint32_t bin = plan_bin(e, a);
            a.bin[i] = bin;
            a.rank[i] = atomicAdd(&a.hist[bin], 1u);
            if (!rep)
                for (uint32_t k = 0; k + 1 < N; ++k)
                    a.edge_id[(e.types[k + 1] * a.K + e.types[k]) * a.n_ivl + e.ivl[k]] = 1u;
        }
    }
    for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N) {
        const uint32_t k = __popc(__ballot_sync(0xffffffffu, len == N));
        if (k && (threadIdx.x & 31) == 0) atomicAdd(&a.words[N - 1], k);
    }
    rep = __reduce_add_sync(0xffffffffu, rep);
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (a.runs) brk = __reduce_add_sync(0xffffffffu, brk);
    if ((threadIdx.x & 31) == 0) {
        if (rep) atomicAdd(&a.words[PLAN_REP], rep);
        if (brk) atomicAdd(&a.words[PLAN_RUNS], brk);
        if (bad) atomicOr(a.err, bad);
    }
    // the least span, over the whole grid
    uint32_t span = 0;
    for (uint32_t c = i + 1; c < a.n_chunks; c += gridDim.x * blockDim.x)
        span = max(span, ~(a.cfirst[c] - a.cfirst[c - 1]));
    span = __reduce_max_sync(0xffffffffu, span);
    if (span && (threadIdx.x & 31) == 0) atomicMax(&a.words[PLAN_SPAN], span);
}

// Slabs per chunk: the fewest equal parts (a power of two) in none of which a type has
// more than 32 events.  One block per chunk, a warp per type.  Types with more than 32 events
// of the chunk in the longest interval are told too: their tables would be too dense (all
// but certainly: it takes an event of the edge's next type at the right time), and the set
// need not wait for the build to find out.
__global__ void __launch_bounds__(256) k_hit_cuts(const uint2 *bev, const uint16_t *boff, uint32_t offs,
                                                  uint32_t K, uint32_t *parts_of, uint32_t max_hi,
                                                  uint32_t *dense) {
    __shared__ uint32_t need;
    const uint32_t c = blockIdx.x, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) need = 1;
    __syncthreads();
    const uint16_t *off = boff + (uint64_t)c * offs;
    const uint2 *ev = bev + (uint64_t)c * CHUNK;
    for (uint32_t b = threadIdx.x >> 5; b < K; b += blockDim.x >> 5) {
        const uint32_t g0 = off[b], g1 = off[b + 1];
        // a part holds more than 32 of the type iff two of its events 32 apart lie in it: the
        // parts must be finer than the highest bit in which their places differ
        uint32_t q = 1, span = ~0u;
        for (uint32_t j = g0 + lane; j + 32 < g1; j += 32) {
            const uint2 e = ev[j], f = ev[j + 32];
            const uint32_t x = e.y ^ f.y;          // not zero
            q = max(q, CHUNK >> (31 - __clz(x)));  // parts of half the size of that bit's
            span = min(span, f.x - e.x);
        }
        q = __reduce_max_sync(0xffffffffu, q);
        span = __reduce_min_sync(0xffffffffu, span);
        if (lane == 0 && q > 1) atomicMax(&need, q);
        if (lane == 0 && span <= max_hi) atomicMin(&dense[b], max_hi);
    }
    __syncthreads();
    if (threadIdx.x == 0) parts_of[c] = need;
}

// One block of 1024: the bins' and the edges' numbers scanned in place (an edge in use
// gets its number, the others none), the slabs' first events and times, and everything
// the host plans with published.
__global__ void __launch_bounds__(1024) k_plan_scan(const PlanArgs a, uint32_t bins, uint32_t edges,
                                                    Publish pub) {
    const uint32_t tid = threadIdx.x;
    const bool too_dense = tid < a.K && a.dense[tid] <= a.max_hi;
    uint32_t total, n_edges, n_slabs, per;
    scan_words(a.hist, bins, &total, [](uint32_t v) { return v; },
               [&](uint32_t i, uint32_t, uint32_t at) { a.hist[i] = at; });
    scan_words(a.edge_id, edges, &n_edges, [](uint32_t v) { return v; },
               [&](uint32_t i, uint32_t v, uint32_t at) { a.edge_id[i] = v ? at : ~0u; });
    {
        per = (a.n_chunks + 1023) / 1024;
        const uint32_t lo = min(tid * per, a.n_chunks), hi = min(lo + per, a.n_chunks);
        auto slabs = [&](uint32_t c) {  // (the last chunk's parts end with the stream)
            const uint32_t q = a.parts_of[c], size = CHUNK / q;
            const uint64_t left = a.n - (uint64_t)c * CHUNK;
            return left >= CHUNK ? q : (uint32_t)((left + size - 1) / size);
        };
        uint32_t v = 0;
        for (uint32_t c = lo; c < hi; ++c) v += slabs(c);
        uint32_t at = block_scan_1024(v, &n_slabs);
        for (uint32_t c = lo; c < hi; ++c) {
            const uint32_t q = slabs(c), size = CHUNK / a.parts_of[c];
            for (uint32_t k = 0; k < q; ++k, ++at) {
                a.begin[at] = c * CHUNK + k * size;
                a.t0[at] = a.t[c * CHUNK + k * size];
            }
        }
        if (tid == 0) a.begin[n_slabs] = (uint32_t)a.n, a.t0[n_slabs] = 0xFFFFFFFFu;
    }
    // the largest slab (the fewest parts of a chunk)
    uint32_t fewest = HIT_PARTS;
    for (uint32_t c = tid; c < a.n_chunks; c += 1024) fewest = min(fewest, a.parts_of[c]);
    fewest = __reduce_min_sync(0xffffffffu, fewest);
    __shared__ uint32_t least, dense;
    if (tid == 0) least = HIT_PARTS, dense = 0;
    __syncthreads();
    if ((tid & 31) == 0) atomicMin(&least, fewest);
    // whether an edge in use leads from a type that is too dense (else none is told)
    if (__syncthreads_or(too_dense)) {
        for (uint32_t i = tid; i < edges; i += 1024)
            if (a.edge_id[i] != ~0u && a.dense[i / a.n_ivl % a.K] <= a.max_hi) dense = 1;
        __syncthreads();
        if (!dense && tid < a.K) a.dense[tid] = ~0u;
    }
    if (tid == 0) {
        volatile uint32_t *h = pub.host;
        for (uint32_t k = 0; k < PLAN_EDGES; ++k) h[k] = a.words[k];
        h[PLAN_PARTS_MIN] = least;
        h[PLAN_DENSE] = dense;
        h[PLAN_RUNS] = a.words[PLAN_RUNS];
        h[PLAN_EDGES] = n_edges;
        h[PLAN_SLABS] = n_slabs;
        h[PLAN_WORDS] = *reinterpret_cast<const volatile uint32_t *>(pub.err);
        __threadfence_system();
        h[PLAN_WORDS + 1] = pub.seq;
    }
}

// order[slot] = i and gather[slot] = candidate record of i, by the scanned bins
__global__ void __launch_bounds__(256) k_plan_place(const PlanArgs a, uint32_t *order,
                                                    uint32_t *gather) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.m || (*a.err & ERR_BADEP)) return;
    const uint32_t s = a.hist[a.bin[i]] + a.rank[i];
    order[s] = i;
    gather[s] = a.gather ? a.gather[i] : i;
}

// The words of k_validate_cands and the error word, published; the error word and the
// sequence number where a plan's are, so that no other word is ever taken for the number.
__global__ void k_publish_info(const uint32_t *info, uint32_t n, Publish pub) {
    volatile uint32_t *h = pub.host;
    for (uint32_t k = 0; k < n; ++k) h[k] = info[k];
    h[PLAN_WORDS] = *reinterpret_cast<const volatile uint32_t *>(pub.err);
    __threadfence_system();
    h[PLAN_WORDS + 1] = pub.seq;
}

// (a count above 32 bits as 2^32 - 1)
__global__ void k_publish_count(const unsigned long long *src, Publish pub) {
    volatile uint32_t *h = pub.host;
    const unsigned long long v = *reinterpret_cast<const volatile unsigned long long *>(src);
    h[0] = v > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)v;
    h[1] = *reinterpret_cast<const volatile uint32_t *>(pub.err);
    __threadfence_system();
    h[2] = pub.seq;
}

// The hit tables of one slab (a block; of a few slabs several, which share the types).
// Every type's events in the slab and the 32 before it go into shared memory as rank rows
// (rank 32 is the slab's first; the types' own order in the chunk gives the ranks), with a
// bit per position of the slab and, per 32 positions, the events before them, so that the
// number of a type's events before any event of the slab is two reads and a popc.  Then a
// warp takes a type y, a lane a type x: for each of y's events, the x events before it as far
// back as the longest interval reaches, a few steps down the row, give the masks of four
// edges.  The warp reserves room for its hits in the table, and the ranges are found again:
// by each lane for its own hits where these are few, else event by event for all four
// intervals.  What bounds it: issue slots, 62% of them used, half the lanes in the
// walks.  Measured on the 406,000 events of 64 types at 20 Hz, all 16,128 edges, exact pass:
// 258 us (48 recordings, 16 to 64 types: 3.1 ms exact, 3.3 relaxed; bursts of 64 types,
// 635 us).  Lanes on the events of a few y, all x one after the other, with ballots for the
// masks: 467 us (3.6 and 3.5 ms; 671 us).  Masks first, then one reservation a block and the
// ranges: 272 us (3.3 and 3.8 ms; 950 us).  Without the walk event by event, bursts take
// 837 us.  A thread per edge, merging its two rows: 983 us.
constexpr int U = 4;                   // intervals taken at once

template <int PASS>
__device__ __forceinline__ void hit_build_slab(const HitBuild &b, uint32_t s, uint32_t part, uint32_t parts) {
    const uint32_t T = HIT_BUILD_T, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr uint32_t NW = HIT_BUILD_T / 32;
    const uint32_t K = b.K;
    uint32_t *rt = reinterpret_cast<uint32_t *>(fem_hit_smem);  // times by rank [K][HIT_ROW]
    uint32_t *bits = rt + K * HIT_ROW;                          // [K][slab words]
    const uint32_t begin = b.begin[s], end = b.begin[s + 1], c = begin / CHUNK;
    const uint32_t p0 = begin % CHUNK, p1 = p0 + (end - begin);  // the slab's places in its chunk
    const uint32_t words = ((end - begin + 31) / 32) | 1u;  // (an odd stride: no bank conflicts)
    uint16_t *rp = reinterpret_cast<uint16_t *>(bits + K * (b.max_words | 1u));  // positions by rank [K][HIT_ROW]
    uint16_t *place = rp + K * HIT_ROW;                          // [K + 1]
    uint8_t *before = reinterpret_cast<uint8_t *>(place + K + 1);  // events before a word [K][words]
    uint8_t *hist = before + K * (b.max_words | 1u);                    // events before the slab [K]
    uint8_t *num = hist + K;                                     // events in the slab [K]
    const uint32_t origin = c * CHUNK - CHUNK;                   // index of position 0 (modulo 2^32)
    const uint16_t *off = b.boff + (uint64_t)c * b.offs;
    const uint2 *ev = b.bev + (uint64_t)c * CHUNK;
    for (uint32_t i = tid; i < K * words; i += T) bits[i] = 0;
    __syncthreads();
    for (uint32_t x = warp; x < K; x += NW) {
        const uint32_t g0 = off[x], g1 = off[x + 1];
        uint32_t a = g0, z = g0;  // the type's first event in the slab and past its last
        for (uint32_t j0 = g0; j0 < g1; j0 += 32) {
            const uint32_t j = j0 + lane, y = j < g1 ? ev[j].y : ~0u;
            a += __popc(__ballot_sync(0xffffffffu, y < p0));
            z += __popc(__ballot_sync(0xffffffffu, y < p1));
        }
        const uint32_t n = z - a, own = min(a - g0, 32u);
        if (lane < n) {
            const uint2 e = ev[a + lane];
            rt[x * HIT_ROW + 32 + lane] = e.x;
            rp[x * HIT_ROW + 32 + lane] = (uint16_t)(CHUNK + e.y);
            atomicOr(&bits[x * words + ((e.y - p0) >> 5)], 1u << ((e.y - p0) & 31));
        }
        uint32_t h = own;  // earlier ones: of this chunk, then of the chunk before
        if (lane < own) {
            const uint2 e = ev[a - 1 - lane];
            rt[x * HIT_ROW + 31 - lane] = e.x;
            rp[x * HIT_ROW + 31 - lane] = (uint16_t)(CHUNK + e.y);
        }
        if (own < 32 && c > 0) {
            const uint32_t f0 = off[(int)x - (int)b.offs], f1 = off[(int)x + 1 - (int)b.offs];
            const uint32_t more = min(f1 - f0, 32u - own);
            if (lane < more) {
                const uint2 e = *(ev - CHUNK + (f1 - 1 - lane));
                rt[x * HIT_ROW + 31 - own - lane] = e.x;
                rp[x * HIT_ROW + 31 - own - lane] = (uint16_t)e.y;
            }
            h += more;
        }
        if (lane == 0) hist[x] = (uint8_t)h, num[x] = (uint8_t)n, b.count[(uint64_t)s * b.types + x] = (uint8_t)n;
        __syncwarp();
        uint32_t sum = 0;
        for (uint32_t w0 = 0; w0 < words; w0 += 32) {
            const uint32_t v = w0 + lane < words ? __popc(bits[x * words + w0 + lane]) : 0u;
            uint32_t inc = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= (uint32_t)d) inc += y;
            }
            if (w0 + lane < words) before[x * words + w0 + lane] = (uint8_t)(sum + inc - v);
            sum += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();
    if (warp == 0) {  // where each type's events start in the slab's list
        uint32_t carry = 0;
        for (uint32_t x0 = 0; x0 < K; x0 += 32) {
            const uint32_t v = x0 + lane < K ? num[x0 + lane] : 0u;
            uint32_t inc = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= (uint32_t)d) inc += y;
            }
            if (x0 + lane < K) {
                place[x0 + lane] = (uint16_t)(carry + inc - v);
                b.place[(uint64_t)s * b.types + x0 + lane] = (uint16_t)(carry + inc - v);
            }
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();
    for (uint32_t x = warp; x < K && part == 0; x += NW)
        if (lane < num[x]) b.index[begin + place[x] + lane] = (uint16_t)(origin + rp[x * HIT_ROW + 32 + lane]);
    uint2 *const row = b.edge + (uint64_t)s * b.n_edges;
    // x's events before event r of type y: those of ranks below k0
    auto rank_of = [&](uint32_t x, uint32_t y, uint32_t r) {
        const uint32_t q = rp[y * HIT_ROW + 32 + r] - CHUNK - p0, w = q >> 5;
        return 32u + before[x * words + w] + __popc(bits[x * words + w] & ((1u << (q & 31)) - 1u));
    };
    const uint32_t groups = (K + 31) / 32;
    for (uint32_t u0 = 0; u0 < b.n_ivl; u0 += U) {
        // a gap lies in interval u iff gap - from[u] <= wide[u] (unsigned); the relaxed pass
        // takes any gap up to hi
        uint32_t from[U], wide[U], far = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint2 v = b.ivl[min(u0 + u, b.n_ivl - 1)];  // (past the set: one not looked at)
            from[u] = PASS == FEM_PASS_EXACT ? v.x + 1u : 0u;
            wide[u] = v.y - from[u];
            far = max(far, v.y);
        }
        for (uint32_t task = part * NW + warp; task < K * groups; task += NW * parts) {
            const uint32_t y = task / groups, x = (task % groups) * 32 + lane, n = num[y];
            uint32_t id[U], mask[U], any = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                id[u] = x < K && u0 + u < b.n_ivl ? __ldg(b.edge_id + (y * K + x) * b.n_ivl + u0 + u) : ~0u;
                any |= ~id[u];
                mask[u] = 0;
            }
            if (!__any_sync(0xffffffffu, any != 0)) continue;  // no edge in use
            const uint32_t *tx = rt + x * HIT_ROW, *ty = rt + y * HIT_ROW + 32;
            const uint32_t low = any ? 32u - hist[x] : ~0u;  // (no edge: no event is looked at)
            bool dense = false;
            for (uint32_t r = 0; r < n && any; ++r) {
                const uint32_t t = ty[r], k0 = rank_of(x, y, r);
                uint32_t k = k0;
                for (; k > low; --k) {
                    const uint32_t gap = t - tx[k - 1];
                    if (gap > far) break;
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (gap - from[u] <= wide[u]) mask[u] |= 1u << r;
                }
                // older events than the 32 kept may lie in an interval, or more than a range
                // can say
                dense = dense || (k == 0 && k0 > 0) || k0 - k > 32;
            }
            if (dense) atomicOr(b.err, ERR_DENSE), atomicMin(&b.dense[x], far);
            uint32_t c = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (id[u] == ~0u) mask[u] = 0;
                c += __popc(mask[u]);
            }
            uint32_t inc = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= (uint32_t)d) inc += v;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
            unsigned long long v = 0;
            if (total) {
                if (lane == 0) v = atomicAdd(b.used, (unsigned long long)total);
                v = __shfl_sync(0xffffffffu, v, 0);
            }
            const bool room = v + total <= b.capacity;
            uint32_t o = (uint32_t)v + inc - c, at = o;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (id[u] != ~0u) row[id[u]] = make_uint2(room ? mask[u] : 0u, at);
                at += __popc(mask[u]);
            }
            if (!room) continue;
            // the hits' ranges: where they are many for the events, event by event, with one
            // walk for all intervals
            if (__reduce_max_sync(0xffffffffu, c) > 2 * n) {
                if (c == 0) continue;
                uint32_t to[U];
#pragma unroll
                for (int u = 0; u < U; ++u) to[u] = o, o += __popc(mask[u]);
                for (uint32_t r = 0; r < n; ++r) {
                    const uint32_t t = ty[r], k0 = rank_of(x, y, r);
                    uint32_t in[U] = {};
                    uint32_t k = k0;
                    for (uint32_t bit = 1; k > low; --k, bit <<= 1) {
                        const uint32_t gap = t - tx[k - 1];
                        if (gap > far) break;
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (gap - from[u] <= wide[u]) in[u] |= bit;  // (rank k0 - 1 - bit)
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (!((mask[u] >> r) & 1u)) continue;
                        // (denser than a word, the tables are not counted with, but read they
                        // are: past 32 events the range is the latest one's)
                        const uint32_t w = in[u] ? in[u] : 1u;
                        const uint32_t m = __popc(w), last = k0 - __ffs(w);
                        b.range[to[u]++] = hit_pack(last + 1 - m, m, origin + rp[x * HIT_ROW + last]);
                    }
                }
                continue;
            }
            // else each lane its own, one after the other
            uint32_t u = 0, left = mask[0], f = from[0], wd = wide[0];
            for (; c; --c) {
                while (!left) {
                    ++u;
#pragma unroll
                    for (int j = 1; j < U; ++j)
                        if (u == (uint32_t)j) left = mask[j], f = from[j], wd = wide[j];
                }
                const uint32_t r = __ffs(left) - 1u;
                left &= left - 1u;
                const uint32_t t = ty[r];
                uint32_t k = rank_of(x, y, r), m = 0;
                if (PASS == FEM_PASS_EXACT)
                    while (t - tx[k - 1] - f > wd) --k;  // (too near; the mask says that one is not)
                const uint32_t last = k - 1;
                for (; k > low && t - tx[k - 1] - f <= wd; --k) ++m;
                m = min(m, 32u);  // (more only where denser than a word)
                b.range[o++] = hit_pack(last + 1 - m, m, origin + rp[x * HIT_ROW + last]);
            }
        }
    }
}

template <int PASS>
__global__ void __launch_bounds__(HIT_BUILD_T) k_hit_build(const HitBuild b) {
    hit_build_slab<PASS>(b, blockIdx.x, blockIdx.y, gridDim.y);
}

// The same for the streams of a batch: block i builds slab i - first[j] of stream j.
template <int PASS>
__global__ void __launch_bounds__(HIT_BUILD_T) k_hit_build_batch(const HitBuild *__restrict__ streams,
                                                                 const uint32_t *__restrict__ first,
                                                                 uint32_t n_streams) {
    __shared__ HitBuild b;
    uint32_t lo = 0, hi = n_streams;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (first[mid] <= blockIdx.x) lo = mid;
        else hi = mid;
    }
    if (threadIdx.x == 0) b = streams[lo];
    __syncthreads();
    hit_build_slab<PASS>(b, blockIdx.x - first[lo], 0, 1);
}

constexpr int kBuildSmem = 224 * 1024;
size_t build_smem(const HitBuild &b) {
    return (size_t)b.K * (HIT_ROW * 6 + (b.max_words | 1u) * 5 + 4) + 32;
}

// Launch kernel `k` over p.m candidates in blocks of 128.
template <int NMAX, typename Kernel, typename... Args>
cudaError_t run(Kernel k, cudaStream_t st, const CountParams &p, Args... args) {
    constexpr uint32_t T = 128;
    constexpr size_t sm = (size_t)hit_shared(NMAX) * 64 * T * 2;  // at most 48 KB: no opt-in
    static_assert(sm <= 48 * 1024, "dynamic shared memory without an attribute");
    k<<<dim3((p.m + T - 1) / T, p.P), T, sm, st>>>(p, args...);
    note_launch();
    return cudaGetLastError();
}

// (48 KB of starts and the shared parameters: past the default limit)
template <int NMAX>
cudaError_t run_batch(const CountParams *parts, const uint4 *list, uint32_t n_list, uint32_t n_items,
                      cudaStream_t st) {
    constexpr uint32_t T = 128;
    constexpr int sm = hit_shared(NMAX) * 64 * (int)T * 2;
    static std::atomic<uint64_t> set;
    const cudaError_t e = smem_limit(set, (const void *)k_hit_count_batch<NMAX>, sm);
    if (e != cudaSuccess) return e;
    k_hit_count_batch<NMAX><<<n_items, T, sm, st>>>(parts, list, n_list);
    note_launch();
    return cudaGetLastError();
}

// Per type: its pairs by slot, and where its events of a slab stand among all events by
// type and then time.
__global__ void __launch_bounds__(256) k_join_index(const HitTables h, const JoinTables g,
                                                    const uint32_t *__restrict__ hist, uint32_t K,
                                                    uint32_t n_ivl) {
    const uint32_t b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t slots = K * n_ivl;
    __shared__ uint32_t wsum[8];
    auto scan = [&](uint32_t v, uint32_t *before, uint32_t *all) {  // over the block's threads
        uint32_t inc = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (uint32_t)d) inc += y;
        }
        __syncthreads();
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        *before = inc - v, *all = 0;
        for (uint32_t w = 0; w < 8; ++w) {
            if (w < warp) *before += wsum[w];
            *all += wsum[w];
        }
    };
    for (int side = 0; side < 2; ++side) {
        uint32_t seen = 0;
        for (uint32_t l0 = 0; l0 < slots; l0 += 256) {
            const uint32_t l = l0 + tid;
            const uint32_t id = l < slots ? h.edge_id[side ? (l / n_ivl * K + b) * n_ivl + l % n_ivl : b * slots + l] : ~0u;
            uint32_t r, all;
            scan(id != ~0u, &r, &all);
            if (id != ~0u) (side ? g.begins : g.ends)[b * slots + seen + r] = make_uint2(id, l);
            seen += all;
        }
        if (tid == 0) (side ? g.n_begins : g.n_ends)[b] = seen;
    }
    uint32_t base, r;
    scan(tid < b ? hist[tid] : 0u, &r, &base);  // (at most 256 types)
    for (uint32_t s0 = 0; s0 < h.n_slabs; s0 += 256) {
        const uint32_t s = s0 + tid;
        uint32_t all;
        scan(s < h.n_slabs ? h.count[(uint64_t)s * h.types + b] : 0u, &r, &all);
        if (s < h.n_slabs) g.rank[(uint64_t)b * h.n_slabs + s] = base + r;
        base += all;
    }
}

// The lists of a slab's events of a type (a warp; lane r: event r): their lengths, or
// (FILL) their entries.
template <bool FILL>
__global__ void __launch_bounds__(256) k_join_list(const HitTables h, const JoinTables g, uint32_t K,
                                                   uint32_t slots, uint32_t *__restrict__ len) {
    const uint32_t lane = threadIdx.x & 31, unit = blockIdx.x * 8 + (threadIdx.x >> 5);
    const uint32_t s = unit / K, b = unit % K;
    if (s >= h.n_slabs) return;
    const uint32_t n = h.count[(uint64_t)s * h.types + b], n_first = g.n_ends[b];
    if (n == 0) return;
    const uint32_t at = g.rank[(uint64_t)b * h.n_slabs + s] + lane;
    const uint2 *row = h.edge + (uint64_t)s * h.n_edges;
    uint32_t o = FILL && lane < n ? g.off[at] : 0u;
    for (uint32_t i0 = 0; i0 < n_first; i0 += 32) {
        const uint2 e = i0 + lane < n_first ? row[g.ends[b * slots + i0 + lane].x] : make_uint2(0u, 0u);
#pragma unroll
        for (uint32_t k = 0; k < 32; ++k) {
            const uint32_t mask = __shfl_sync(0xffffffffu, e.x, k);
            if (FILL) {
                const uint32_t from = __shfl_sync(0xffffffffu, e.y, k);
                if ((mask >> lane) & 1u)
                    g.list[o++] = (i0 + k) << 16 | h.range[from + __popc(mask & ((1u << lane) - 1u))] >> 16;
            } else {
                o += (mask >> lane) & 1u;
            }
        }
    }
    if (!FILL && lane < n) len[at] = o;
}

// out[i] = the joined count of candidate i (three nodes)
__global__ void __launch_bounds__(256) k_join_gather(const uint32_t *cells, const fem_episode *cands,
                                                      const uint32_t *gather, uint32_t m, uint32_t K,
                                                      uint32_t n_ivl, uint32_t *out) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const fem_episode e = cands[gather ? gather[i] : i];
    const uint64_t slots = K * n_ivl;
    out[i] = cells[(e.types[1] * slots + e.types[2] * n_ivl + e.ivl[1]) * slots + e.types[0] * n_ivl + e.ivl[0]];
}

}  // namespace

uint32_t plan_bins(uint32_t K, uint32_t parts) { return PLAN_GROUPS * K * parts * parts * parts; }

cudaError_t launch_plan(const PlanArgs &a, const StreamDev &s, uint32_t *order, uint32_t *gather,
                        Publish pub, cudaStream_t st) {
    const uint32_t bins = plan_bins(a.K, a.parts), edges = a.K * a.K * a.n_ivl, blocks = (a.m + 255) / 256;
    cudaError_t e = cudaMemsetAsync(a.words, 0, (PLAN_WORDS + (size_t)bins + edges) * 4, st);
    if (e != cudaSuccess) return e;
    k_plan_bins<<<blocks, 256, 0, st>>>(a);
    k_hit_cuts<<<s.n_chunks, 256, 0, st>>>(s.bev, s.boff, s.offs, s.K, a.parts_of, a.max_hi, a.dense);
    k_plan_scan<<<1, 1024, 0, st>>>(a, bins, edges, pub);
    k_plan_place<<<blocks, 256, 0, st>>>(a, order, gather);
    note_launch(4);
    return cudaGetLastError();
}

cudaError_t launch_publish_info(const uint32_t *info, uint32_t n, Publish pub, cudaStream_t st) {
    if (n > PLAN_WORDS) return cudaErrorInvalidValue;
    k_publish_info<<<1, 1, 0, st>>>(info, n, pub);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_publish_count(const unsigned long long *src, Publish pub, cudaStream_t st) {
    k_publish_count<<<1, 1, 0, st>>>(src, pub);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_hit_build(int pass, uint32_t n_slabs, const HitBuild &b, int sm_count,
                             cudaStream_t st) {
    if (n_slabs == 0) return cudaSuccess;
    const size_t sm = build_smem(b);
    if (sm > kBuildSmem) return cudaErrorInvalidConfiguration;
    static std::atomic<uint64_t> set[2];
    const auto kernel = pass == FEM_PASS_RELAXED ? k_hit_build<FEM_PASS_RELAXED> : k_hit_build<FEM_PASS_EXACT>;
    const cudaError_t e = smem_limit(set[pass == FEM_PASS_RELAXED], (const void *)kernel, kBuildSmem);
    if (e != cudaSuccess) return e;
    // a few slabs: their types shared among several blocks, for about four per SM
    constexpr uint32_t NW = HIT_BUILD_T / 32;
    uint32_t split = 1;
    while (split < 8 && split * NW < b.K * ((b.K + 31) / 32) && split * n_slabs < 4 * (uint32_t)sm_count) split *= 2;
    kernel<<<dim3(n_slabs, split), HIT_BUILD_T, sm, st>>>(b);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_hit_build_batch(int pass, const HitBuild *host, const HitBuild *streams,
                                   const uint32_t *first, uint32_t n_streams, uint32_t n_slabs,
                                   cudaStream_t st) {
    if (n_slabs == 0) return cudaSuccess;
    size_t sm = 0;
    for (uint32_t j = 0; j < n_streams; ++j) sm = std::max(sm, build_smem(host[j]));
    if (sm > kBuildSmem) return cudaErrorInvalidConfiguration;
    static std::atomic<uint64_t> set[2];
    const auto kernel =
        pass == FEM_PASS_RELAXED ? k_hit_build_batch<FEM_PASS_RELAXED> : k_hit_build_batch<FEM_PASS_EXACT>;
    const cudaError_t e = smem_limit(set[pass == FEM_PASS_RELAXED], (const void *)kernel, kBuildSmem);
    if (e != cudaSuccess) return e;
    kernel<<<n_slabs, HIT_BUILD_T, sm, st>>>(streams, first, n_streams);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_hit_count_batch(uint32_t group, const CountParams *parts, const uint4 *list,
                                   uint32_t n_list, uint32_t n_items, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    switch (group) {
#define FEM_CASE(g, n) \
    case g: return run_batch<n>(parts, list, n_list, n_items, st);
        FEM_CASE(0, 2) FEM_CASE(1, 3) FEM_CASE(2, 4) FEM_CASE(3, 5) FEM_CASE(4, 8)
#undef FEM_CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_hit_count(uint32_t group, bool mc, const CountParams &p, cudaStream_t st) {
    if (p.m == 0) return cudaSuccess;
    switch (group) {
#define FEM_CASE(g, n) \
    case g: return mc ? run<n>(k_hit_count<n, true>, st, p) : run<n>(k_hit_count<n, false>, st, p);
        FEM_CASE(0, 2) FEM_CASE(1, 3) FEM_CASE(2, 4) FEM_CASE(3, 5) FEM_CASE(4, 8)
#undef FEM_CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_hit_windows(uint32_t group, const CountParams &p, const uint32_t *order, uint32_t w,
                               uint64_t *out, cudaStream_t st) {
    if (p.m == 0) return cudaSuccess;
    unsigned long long *o = reinterpret_cast<unsigned long long *>(out);
    switch (group) {
#define FEM_CASE(g, n) \
    case g: return run<n>(k_hit_windows<n>, st, p, order, w, o);
        FEM_CASE(0, 2) FEM_CASE(1, 3) FEM_CASE(2, 4) FEM_CASE(3, 5) FEM_CASE(4, 8)
#undef FEM_CASE
        default: return cudaErrorInvalidValue;
    }
}

size_t join_smem(uint32_t slots) { return JOIN_QUEUE * sizeof(uint4) + (size_t)slots * sizeof(uint2); }

cudaError_t launch_join(const HitTables &h, const JoinTables &g, const uint32_t *hist, uint32_t n, uint32_t K,
                        uint32_t n_ivl, uint32_t *len, uint32_t *scratch, uint32_t *out, cudaStream_t st) {
    static std::atomic<uint64_t> set;
    cudaError_t e = smem_limit(set, (const void *)k_join, 224 * 1024);
    if (e != cudaSuccess) return e;
    const uint32_t slots = K * n_ivl, units = h.n_slabs * K;
    k_join_index<<<K, 256, 0, st>>>(h, g, hist, K, n_ivl);
    note_launch();
    k_join_list<false><<<(units + 7) / 8, 256, 0, st>>>(h, g, K, slots, len);
    note_launch();
    if ((e = launch_exclusive_scan(len, n, g.off, g.off + n, scratch, st)) != cudaSuccess) return e;
    k_join_list<true><<<(units + 7) / 8, 256, 0, st>>>(h, g, K, slots, nullptr);
    note_launch();
    // blocks of up to eight warps in about 48 KB
    const uint32_t NW = (uint32_t)std::min<size_t>(8, std::max<size_t>(1, 48 * 1024 / join_smem(slots)));
    k_join<<<dim3(K, (slots + NW - 1) / NW), NW * 32, NW * join_smem(slots), st>>>(h, g, n, K, n_ivl, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_join_gather(const uint32_t *cells, const fem_episode *cands, const uint32_t *gather,
                                uint32_t m, uint32_t K, uint32_t n_ivl, uint32_t *out, cudaStream_t st) {
    if (m == 0) return cudaSuccess;
    k_join_gather<<<(m + 255) / 256, 256, 0, st>>>(cells, cands, gather, m, K, n_ivl, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace fem
