// fem_api.cu -- the C ABI of libfem.so (include/fem.h): contexts, resident
// streams, the counting driver (segment choice, capacity retries), Algorithm 4
// and the level-wise miner of Problem 1.  Every step of the method runs in the
// kernels of fem_stream.cu, fem_count.cu and fem_mine.cu; this file only
// allocates device memory, launches, and copies results.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "fem_internal.cuh"

using namespace fem;

namespace fem {
static std::atomic<uint64_t> g_launches{0};
void note_launch(uint32_t k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
}  // namespace fem

struct fem_result {
    std::vector<std::vector<fem_episode>> eps;    // [level-1]
    std::vector<std::vector<uint32_t>> counts;  // [level-1]
};

namespace {
struct DevBuf {
    void *p = nullptr;
    size_t cap = 0;
};
}  // namespace

struct fem_ctx {
    int device = 0;
    // device memory the context holds for streams, working buffers and batches, and
    // the caller's bound on it (0: none)
    size_t mem_budget = 0, mem_used = 0;
    size_t mem_device = 0;  // the device's memory
    cudaStream_t own = nullptr;
    fem_config cfg{};
    int sm_count = 152;
    std::map<int32_t, StreamDev> streams;
    // per loaded stream, its type histogram (the level-1 counts), read back in the
    // load's own round trip so that mining needs no wait for it
    std::map<int32_t, std::vector<uint32_t>> hist_h;
    int32_t next_id = 1;
    uint32_t *d_err = nullptr;    // device error word
    uint32_t *d_dense = nullptr;  // 256 device words: HitBuild::dense (2^32 - 1 between counts)
    uint32_t *d_small = nullptr;  // 64 device words for counters
    uint32_t *h_small = nullptr;  // kSmallWords pinned host words
    // device address of h_small[kPubWord..kPubWord+1], written by the compaction and scan
    // kernels (count and error word); null where pinned memory is not mapped
    uint32_t *d_pub = nullptr;
    uint32_t *d_plan = nullptr;  // the same of h_small[kPlanWord ..], written by the plan kernels
    uint32_t pub_seq = 0;  // sequence number of the last publishing launch
    // mapped pinned words a load's read-back is published to ([0] error word, [1] last
    // time, [2..258) type counts, [258] first time, [kLoadSeq] sequence number) and their
    // device address
    uint32_t *h_load = nullptr, *d_load = nullptr;
    // pinned staging of an interval set (so that its upload is asynchronous), and the
    // event after the last upload from it (the next one waits for that copy to leave)
    fem_interval *h_ivl = nullptr;
    cudaEvent_t ivl_ev = nullptr;
    std::vector<fem_interval> ivl_host;  // the interval set of the current call
    uint64_t next_gen = 1;  // stream contents' generations
    std::map<std::string, DevBuf> bufs;
    std::vector<fem_level_stats> stats;
    std::vector<StreamDev> pool;  // buffers of freed streams, reused by later loads
    // mining timings: [0,1] generation, [2,3] relaxed pass, [4,5] compaction, [6,7] exact
    cudaEvent_t ev[8] = {};
    // pinned host staging of each level's frequent set (copied out after the last sync)
    struct PinBuf {
        void *p = nullptr;
        size_t cap = 0;
    };
    PinBuf pin[FEM_MAX_LEN + 1];
    // around the counting kernel and stitch, two sets used in turn, so that a pass's
    // times can be read after the next pass has been queued
    cudaEvent_t kev[2][3] = {};
    int kev_flip = 0;
    // measured mapping choice: launch shape per (N, pass, distinct, log2 m,
    // log2 chunks, K) class, and whether the class goes over hit tables
    struct Shape {
        uint32_t P, T;
        float ms;
        uint32_t kernel;  // FEM_KERNEL_MACHINE or FEM_KERNEL_CHAIN; a choice: _HITS or _MACHINE
    };
    std::map<std::string, Shape> tune;
    bool tune_on = false, tuning = false;
    // the candidate set being counted comes in runs of shared prefixes (mining's sets
    // always do; count_any measures it): where it does not, the latest-chain kernels
    // would find few prefixes to share
    bool clustered = true;
    bool hits_busy = false;  // a count over hit tables is being planned or run
    cudaEvent_t tev[2] = {nullptr, nullptr};
};

namespace {

// FEM_DEBUG set: a failing CUDA call is reported on stderr with its line
void report_cuda(cudaError_t e, int line) {
    if (std::getenv("FEM_DEBUG"))
        std::fprintf(stderr, "fem: CUDA error %s at fem_api.cu:%d\n", cudaGetErrorString(e), line);
}
#define CK(x)                          \
    do {                               \
        cudaError_t e_ = (x);          \
        if (e_ != cudaSuccess) {       \
            report_cuda(e_, __LINE__); \
            return FEM_ECUDA;          \
        }                              \
    } while (0)
#define RET(x)                  \
    do {                        \
        int r_ = (x);           \
        if (r_ != FEM_OK) return r_; \
    } while (0)

// d_small word assignment
enum { W_COUNT0 = 0, W_COUNT1 = 1, W_COUNT2 = 2, W_INFO = 8 /* 11 words */ };
// first of the three pinned host words the kernels publish counts to
constexpr uint32_t kPubWord = 48;
constexpr uint32_t kLoadSeq = 2 + 256 + 1;  // the load read-back's sequence word
// first of the mapped host words a plan is published to (plan words, error word, sequence)
constexpr uint32_t kPlanWord = 64;
constexpr uint32_t kSmallWords = kPlanWord + PLAN_WORDS + 2;

size_t stream_bytes(const StreamDev &s) {
    if (!s.t) return 0;
    return s.cap_events * 5 + s.cap_chunks * CHUNK * 8 + (size_t)s.cap_offs * 2 +
           (s.cap_chunks + 1) * 4 + 256 * 4;
}

void free_stream_buffers(StreamDev &s);

// Gives the hit tables' memory back (cudaFree waits for the work that reads them); whether
// there was any.
bool release_hits(fem_ctx *c) {
    bool any = false;
    for (auto &kv : c->bufs) {
        if (kv.first.compare(0, 4, "hit_") != 0 || !kv.second.p) continue;
        cudaFree(kv.second.p);
        c->mem_used -= std::min(kv.second.cap, c->mem_used);
        kv.second = DevBuf{};
        any = true;
    }
    return any;
}

// Room for `bytes` more under the context's memory budget: over budget, the hit tables of
// earlier calls and the buffers kept from freed streams are released first; FEM_ENOMEM if
// it still does not fit.
int reserve(fem_ctx *c, size_t bytes) {
    if (!c->mem_budget) return FEM_OK;
    if (c->mem_used + bytes > c->mem_budget && !c->hits_busy) release_hits(c);
    while (c->mem_used + bytes > c->mem_budget && !c->pool.empty()) {
        c->mem_used -= std::min(stream_bytes(c->pool.front()), c->mem_used);
        free_stream_buffers(c->pool.front());
        c->pool.erase(c->pool.begin());
    }
    return c->mem_used + bytes > c->mem_budget ? FEM_ENOMEM : FEM_OK;
}

// Device allocation charged to the context's memory budget.
int cmalloc(fem_ctx *c, void **p, size_t bytes) {
    *p = nullptr;
    RET(reserve(c, bytes));
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        // (the device is full: once more without the hit tables of earlier calls)
        if (c->hits_busy || !release_hits(c) || cudaMalloc(p, bytes) != cudaSuccess) {
            cudaGetLastError();
            *p = nullptr;
            return FEM_ENOMEM;
        }
    }
    c->mem_used += bytes;
    return FEM_OK;
}

void cfree(fem_ctx *c, void *p, size_t bytes) {
    if (!p) return;
    cudaFree(p);
    c->mem_used -= std::min(bytes, c->mem_used);
}

template <typename T>
int dbuf(fem_ctx *c, const char *name, size_t count, T **out) {
    const size_t bytes = std::max<size_t>(count * sizeof(T), 256);
    DevBuf &b = c->bufs[name];
    if (b.cap < bytes) {
        size_t nb = std::max(bytes, (size_t)(b.cap * 3 / 2));
        cfree(c, b.p, b.cap);
        b.p = nullptr;
        b.cap = 0;
        nb = (nb + 4095) & ~(size_t)4095;
        RET(cmalloc(c, &b.p, nb));
        b.cap = nb;
    }
    *out = static_cast<T *>(b.p);
    return FEM_OK;
}

cudaStream_t pick(fem_ctx *c, void *s) { return s ? static_cast<cudaStream_t>(s) : c->own; }

// Pinned host buffer `slot` of at least `bytes` (contents are not kept on growth; the
// stream is drained first, so no copy into the old buffer is in flight).
int pinbuf(fem_ctx *c, uint32_t slot, size_t bytes, cudaStream_t st, void **out) {
    fem_ctx::PinBuf &b = c->pin[slot];
    if (b.cap < bytes) {
        CK(cudaStreamSynchronize(st));
        if (b.p) cudaFreeHost(b.p);
        b.p = nullptr;
        b.cap = 0;
        const size_t nb = (std::max(bytes, (size_t)4096) + 4095) & ~(size_t)4095;
        if (cudaMallocHost(&b.p, nb) != cudaSuccess) {
            cudaGetLastError();
            return FEM_ENOMEM;
        }
        b.cap = nb;
    }
    *out = b.p;
    return FEM_OK;
}

int read_words(fem_ctx *c, const uint32_t *d, uint32_t n, uint32_t *h, cudaStream_t st) {
    CK(cudaMemcpyAsync(c->h_small, d, n * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    std::memcpy(h, c->h_small, n * sizeof(uint32_t));
    return FEM_OK;
}

int read_err(fem_ctx *c, cudaStream_t st, uint32_t *err) {
    return read_words(c, c->d_err, 1, err, st);
}

// The count (and error word) the next compaction or scan publishes into the mapped host
// words, under a new sequence number.
Publish pub_of(fem_ctx *c) {
    if (!c->d_pub) return Publish{};
    return Publish{c->d_pub, c->d_err, ++c->pub_seq};
}

// Wait until the mapped word `w` holds `seq` (written by a kernel on st after what it
// publishes): the host watches the word rather than waiting for the stream, so it can
// queue the next launches while that kernel retires; after 2 s it waits for the stream.
int wait_seq(const volatile uint32_t *w, uint32_t seq, cudaStream_t st) {
    const auto t0 = std::chrono::steady_clock::now();
    for (uint32_t spin = 1; *w != seq; ++spin) {
        if ((spin & 1023u) == 0 && std::chrono::steady_clock::now() - t0 > std::chrono::seconds(2)) {
            CK(cudaStreamSynchronize(st));
            if (*w != seq) return FEM_ECUDA;
            break;
        }
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    return FEM_OK;
}

// A device count and the error word, in one round trip: read from the mapped words once
// the launch before has published them under its sequence number, else copied.
int read_count_err(fem_ctx *c, const uint32_t *d_count, uint32_t *count, uint32_t *err,
                   cudaStream_t st) {
    if (c->d_pub) {
        const volatile uint32_t *h = c->h_small + kPubWord;
        RET(wait_seq(h + 2, c->pub_seq, st));
        *count = h[0];
        *err = h[1];
        return FEM_OK;
    }
    CK(cudaMemcpyAsync(c->h_small, d_count, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(c->h_small + 1, c->d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    *count = c->h_small[0];
    *err = c->h_small[1];
    return FEM_OK;
}

int err_status(uint32_t e) {
    if (e & ERR_TIMEOUT) return FEM_ETIMEOUT;
    if (e & ERR_BADEP) return FEM_EINVAL;
    if (e & ERR_TYPE) return FEM_ETYPE;
    if (e & ERR_UNSORTED) return FEM_EUNSORTED;
    return FEM_OK;
}

const StreamDev *find_stream(fem_ctx *c, int32_t id) {
    auto it = c->streams.find(id);
    return it == c->streams.end() ? nullptr : &it->second;
}

int check_intervals(const StreamDev &s, const fem_interval *I, uint32_t nI) {
    if (nI > FEM_MAX_INTERVALS) return FEM_EINVAL;
    if (nI && !I) return FEM_EINVAL;
    uint64_t max_hi = 0;
    for (uint32_t i = 0; i < nI; ++i) {
        if (I[i].lo_us >= I[i].hi_us) return FEM_EINVAL;
        max_hi = std::max<uint64_t>(max_hi, I[i].hi_us);
    }
    // deadlines t + hi + 1 must fit in 32 bits
    if ((uint64_t)s.t_max + max_hi + 1 > 0xFFFFFFFFull) return FEM_ERANGE;
    return FEM_OK;
}

int upload_intervals(fem_ctx *c, const fem_interval *I, uint32_t nI, cudaStream_t st,
                     uint2 **d_ivl) {
    RET(dbuf(c, "ivl", std::max<uint32_t>(nI, 1), d_ivl));
    c->ivl_host.assign(I, I + nI);
    if (!nI) return FEM_OK;
    if (nI > FEM_MAX_INTERVALS + 1) {
        CK(cudaMemcpyAsync(*d_ivl, I, nI * sizeof(uint2), cudaMemcpyHostToDevice, st));
        return FEM_OK;
    }
    CK(cudaEventSynchronize(c->ivl_ev));  // the previous upload has left the staging
    std::memcpy(c->h_ivl, I, nI * sizeof(fem_interval));
    CK(cudaMemcpyAsync(*d_ivl, c->h_ivl, nI * sizeof(uint2), cudaMemcpyHostToDevice, st));
    CK(cudaEventRecord(c->ivl_ev, st));
    return FEM_OK;
}

// Capacity table of a resident stream for the given widths (host out[a * nh + j]);
// synchronous on st.  A width >= the stream's last time holds every event of a type.
// With dense_out (uint32[K * nh]): also the events of each type whose window of each width
// holds more than `over` events of the type.
int capacity(fem_ctx *c, const StreamDev &s, const uint32_t *widths, uint32_t nh,
             uint32_t *out, cudaStream_t st, uint32_t over = 0, uint32_t *dense_out = nullptr) {
    const uint32_t K = s.K;
    std::vector<uint32_t> hw, slot;
    for (uint32_t j = 0; j < nh; ++j)
        if (s.n && widths[j] < s.t_max) hw.push_back(widths[j]), slot.push_back(j);
    std::vector<uint32_t> hist(K, 0), part((size_t)K * hw.size(), 0), dpart(part.size(), 0);
    CK(cudaMemcpyAsync(hist.data(), s.hist, K * 4, cudaMemcpyDeviceToHost, st));
    if (!hw.empty()) {
        const uint32_t nk = (uint32_t)hw.size();
        uint32_t *d;
        RET(dbuf(c, "cap", (size_t)nk * (2 * K + 1), &d));
        uint32_t *d_dense = d + (size_t)K * nk, *d_h = d + (size_t)2 * K * nk;
        CK(cudaMemsetAsync(d, 0, (size_t)2 * K * nk * 4, st));
        CK(cudaMemcpyAsync(d_h, hw.data(), nk * 4, cudaMemcpyHostToDevice, st));
        CK(launch_capacity(s, d_h, nk, d, st, over, dense_out ? d_dense : nullptr));
        CK(cudaMemcpyAsync(part.data(), d, (size_t)K * nk * 4, cudaMemcpyDeviceToHost, st));
        if (dense_out)
            CK(cudaMemcpyAsync(dpart.data(), d_dense, (size_t)K * nk * 4, cudaMemcpyDeviceToHost, st));
    }
    CK(cudaStreamSynchronize(st));
    for (uint32_t a = 0; a < K; ++a) {
        for (uint32_t j = 0; j < nh; ++j) {
            out[(size_t)a * nh + j] = hist[a];
            if (dense_out) dense_out[(size_t)a * nh + j] = hist[a] > over ? hist[a] : 0u;
        }
        for (size_t q = 0; q < hw.size(); ++q) {
            out[(size_t)a * nh + slot[q]] = part[a * hw.size() + q];
            if (dense_out) dense_out[(size_t)a * nh + slot[q]] = dpart[a * hw.size() + q];
        }
    }
    return FEM_OK;
}

// Whether the per-thread exact kernel's lists should get rings of 32 entries instead of 8
// for the current interval set, from the capacity table: Algorithm 1's pruned list for
// node k holds type-E_k events within hi_k, as single times at most cap[E_k][hi_k] of
// them, as clusters at most ceil(hi / (hi - lo)) + 1.  Larger rings cost occupancy, so
// they are taken only where lists outgrow 8 often: more than one event in a thousand
// starts a window of length hi holding more than 8 events of its type (a bursting
// recording: 7% at 20 ms; an hour of 50 Hz Poisson trains: 0.001%, where the few
// episodes that overflow are recounted).  Kept with the stream for its contents and the
// last interval set.
constexpr uint32_t kRingSmall = 8, kRingLarge = 32;
int ring_choice(fem_ctx *c, const StreamDev &s, bool *large_singles, bool *large_clusters,
                cudaStream_t st) {
    const std::vector<fem_interval> &I = c->ivl_host;
    const std::string key(reinterpret_cast<const char *>(I.data()), I.size() * sizeof(fem_interval));
    if (s.ring_gen != s.gen || s.ring_ivl != key) {
        std::vector<uint32_t> w;
        for (const fem_interval &iv : I) w.push_back(iv.hi_us);
        std::vector<uint32_t> cap((size_t)s.K * w.size()), dense(cap.size());
        bool sg = false, cl = false;
        if (!w.empty() && s.n) {
            RET(capacity(c, s, w.data(), (uint32_t)w.size(), cap.data(), st, kRingSmall,
                         dense.data()));
            for (size_t j = 0; j < w.size(); ++j) {
                uint32_t mx = 0;
                uint64_t nd = 0;
                for (uint32_t a = 0; a < s.K; ++a) {
                    mx = std::max(mx, cap[(size_t)a * w.size() + j]);
                    nd += dense[(size_t)a * w.size() + j];
                }
                const bool often = nd * 1000 > s.n;
                const uint32_t span = I[j].hi_us - I[j].lo_us;
                const uint32_t ncl = (I[j].hi_us + span - 1) / span + 1;
                sg = sg || (often && mx > kRingSmall);
                cl = cl || (often && std::min(mx, ncl) > kRingSmall);
            }
        }
        s.ring_gen = s.gen;
        s.ring_ivl = key;
        s.ring_singles = sg;
        s.ring_clusters = cl;
    }
    *large_singles = s.ring_singles;
    *large_clusters = s.ring_clusters;
    return FEM_OK;
}

// Segments per episode for one pass.  One thread per (episode, segment); the aim is
// about 2048 threads per SM, and about 1024 for the two-node latest-chain kernel (one
// resident wave of its four 256-thread blocks per SM): the shapes the tuner keeps on
// the 64-type recording -- level-2 exact 29 segments (0.169 ms where 50 took 0.201),
// 13 on the deep variant -- while its longer episodes keep the larger aim (level-4
// exact of the deep variant: 6 segments 1.65 ms, 3 took 2.07).  Segments are whole
// chunks, so at most one per chunk.
uint32_t choose_segments(fem_ctx *c, const StreamDev &s, uint32_t m, bool distinct,
                         bool one_wave = false) {
    if (s.n_chunks == 0) return 1;
    const uint32_t maxP = std::min<uint32_t>(s.n_chunks, 65535);
    if (c->cfg.segments) return std::min<uint32_t>(c->cfg.segments, s.n_chunks);
    if (!distinct) return 1;
    const uint64_t target = (uint64_t)c->sm_count * (one_wave ? 1024 : 2048);
    uint64_t P = (target + m - 1) / m;
    if (P < 2) return 1;
    return (uint32_t)std::min<uint64_t>(P, maxP);
}

// Block size by shared memory (and, for few episodes, smaller blocks), ignoring any
// configured size.
uint32_t auto_threads(int N, int pass, bool mc, uint32_t R, uint32_t offs, uint32_t m,
                      uint32_t classes = S_MAX) {
    for (uint32_t T : {256u, 128u, 64u, 32u}) {
        if (T > 32 && m <= T / 2) continue;  // few episodes: small blocks, more of them
        if (T == 256 && N > 3) continue;  // register budget
        if (count_smem_bytes(N, pass, mc, R, T, offs, classes) <= 80 * 1024) return T;
    }
    for (uint32_t T : {32u, 16u, 8u}) {
        if (count_smem_bytes(N, pass, mc, R, T, offs, classes) <= 220 * 1024) return T;
    }
    return 8;
}

uint32_t choose_threads(fem_ctx *c, int N, int pass, bool mc, uint32_t R, uint32_t offs,
                        uint32_t m) {
    if (c->cfg.threads_per_block) return c->cfg.threads_per_block;
    return auto_threads(N, pass, mc, R, offs, m);
}

struct PassInfo {
    uint32_t segments = 1;
    uint32_t kernel = 0;  // FEM_KERNEL_MACHINE or FEM_KERNEL_CHAIN
    float ms_kernel = 0, ms_stitch = 0;
};

uint32_t ceil_log2(uint64_t v) {
    uint32_t r = 0;
    while ((1ull << r) < v) ++r;
    return r;
}

// The latest-chain kernels count distinct-type episodes of 2..8 nodes in sets that come
// in runs of shared prefixes (level-wise mining's candidates; fem_count_candidates
// measures the runs).  (Scattered candidates would be counted in parts, one per run of
// the node tables' capacity: slower than the per-thread machine.)
constexpr uint32_t kChainSmallSet = 64;
bool chain_eligible(const fem_ctx *c, int N, bool distinct, uint32_t m) {
    return distinct && N >= 2 && N <= FEM_MAX_LEN && m > 0 && c->clustered;
}

// The rule's kernel where no measurement says otherwise.  The latest-chain kernels for
// the exact pass, whose per-thread machine (sliding-window lists) costs the most per
// event, over at least a block of candidates, or over a small set (there a block's eight
// warps build the prefix lists together where the per-thread machine leaves a single
// warp per block: level-3 exact of 32 survivors 0.097 -> 0.063 ms).  For the relaxed pass,
// whose single slot per node makes the per-thread machine cheap, the latest-chain kernels
// only for longer episodes in large sets, where many candidates share each prefix list
// (the deep variant of the 64-type recording: level 3, 2.4M candidates, 55.5 -> 32.0 ms;
// level 4, 73k, 3.65 -> 1.60 ms), or in small sets; at the bench step's 13,657 level-3
// candidates, many of them in short prefix runs, the two measured level.
constexpr uint32_t kChainLargeSet = 32768;
uint32_t rule_kernel(const fem_ctx *c, int N, int pass, bool distinct, uint32_t m) {
    if (!chain_eligible(c, N, distinct, m)) return FEM_KERNEL_MACHINE;
    if (pass == FEM_PASS_EXACT)
        return m >= 256 || m <= kChainSmallSet ? FEM_KERNEL_CHAIN : FEM_KERNEL_MACHINE;
    return N >= 3 && (m >= kChainLargeSet || m <= kChainSmallSet) ? FEM_KERNEL_CHAIN
                                                                   : FEM_KERNEL_MACHINE;
}

// Block size of the latest-chain kernels: 256 threads, also for a few episodes (the
// block's warps share the prefix-list builds).
uint32_t chain_threads(uint32_t) { return 256u; }

// The class a measured launch shape is kept for: counts of the same length,
// pass and type structure, with m and the stream length in the same power-of-two
// range and the same type count, map alike.  Besides the shapes of the other kernels (distinct
// types or not), the choice between these and the hit tables is kept, for sets that do not
// come in runs (kind 2; N = 0: of several lengths) and for mining's levels (kind 3).
constexpr int kTuneSet = 2, kTuneLevel = 3;
std::string tune_key(int N, int pass, int kind, uint32_t m, uint32_t n_chunks, uint32_t K) {
    char b[96];
    std::snprintf(b, sizeof(b), "%d/%d/%d/%u/%u/%u", N, pass, kind, ceil_log2(m),
                  ceil_log2(n_chunks), K);
    return b;
}

int count_pass(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
               uint32_t m, int N, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
               bool distinct, cudaStream_t st, PassInfo *info);

// Mapping choice by measurement (it replaces the fixed crossover rule of
// Algorithm 2): time the rule's launch shape and its neighbours (half and twice
// the segments per episode, the other block size) on the real inputs and keep the
// fastest for the class.  Every trial is a complete, correct count.
int tune_pass(fem_ctx *c, const std::string &key, const StreamDev &s, const fem_episode *cands,
              const uint32_t *gather, uint32_t m, int N, const uint2 *d_ivl, uint32_t nI,
              int pass, uint32_t *out, bool distinct, cudaStream_t st) {
    // per kernel: its rule's segments, half and twice as many
    auto segment_choices = [&](bool chain_kind) {
        const uint32_t P0 = choose_segments(c, s, m, distinct, chain_kind && N == 2);
        std::vector<uint32_t> Ps{P0};
        if (distinct) {
            if (P0 > 1) Ps.push_back(std::max<uint32_t>(1, P0 / 2));
            if (P0 * 2 <= s.n_chunks) Ps.push_back(P0 * 2);
        }
        return Ps;
    };
    const uint32_t R0 = pass == FEM_PASS_EXACT ? (c->cfg.ring_capacity ? c->cfg.ring_capacity : 8) : 1;
    // the shapes to time: per segment count and kernel the rule's block size and its
    // neighbours; the rule's own shape first
    const bool chain = chain_eligible(c, N, distinct, m);
    const uint32_t k0 = c->cfg.kernel ? c->cfg.kernel : rule_kernel(c, N, pass, distinct, m);
    std::vector<fem_ctx::Shape> shapes;
    for (uint32_t kind : {k0, k0 == FEM_KERNEL_CHAIN ? (uint32_t)FEM_KERNEL_MACHINE : (uint32_t)FEM_KERNEL_CHAIN}) {
        if (kind == FEM_KERNEL_CHAIN && !chain) continue;
        if (c->cfg.kernel && kind != c->cfg.kernel) continue;
        for (uint32_t P : segment_choices(kind == FEM_KERNEL_CHAIN)) {
            if (kind == FEM_KERNEL_CHAIN) {
                const uint32_t T0 = chain_threads(m);
                shapes.push_back(fem_ctx::Shape{P, T0, -1.f, kind});
                for (uint32_t T : {128u, 256u})
                    if (T != T0 && m > T / 2 && chain_smem_bytes(N, P > 1, T, s.offs) <= 200 * 1024)
                        shapes.push_back(fem_ctx::Shape{P, T, -1.f, kind});
                continue;
            }
            const uint32_t R = (P > 1 && R0 > 32) ? 32 : R0;
            const uint32_t T0 = choose_threads(c, N, pass, P > 1, R, s.offs, m);
            shapes.push_back(fem_ctx::Shape{P, T0, -1.f, kind});
            for (uint32_t T : {128u, 256u})
                if (T != T0 && m > T / 2 && count_smem_bytes(N, pass, P > 1, R, T, s.offs) <= 100 * 1024)
                    shapes.push_back(fem_ctx::Shape{P, T, -1.f, kind});
        }
    }
    const fem_config saved = c->cfg;
    c->tuning = true;
    int rc = FEM_OK;
    // Two sweeps over all shapes, keeping each shape's faster time: interleaving keeps
    // a clock that is still rising at the first trials (or the first launch of a
    // kernel, which also loads it) from favouring the shapes timed last.
    for (int rep = 0; rep < 2 && rc == FEM_OK; ++rep) {
        for (fem_ctx::Shape &sh : shapes) {
            c->cfg.segments = sh.P;
            c->cfg.threads_per_block = sh.T;
            c->cfg.kernel = sh.kernel;
            cudaEventRecord(c->tev[0], st);
            rc = count_pass(c, s, cands, gather, m, N, d_ivl, nI, pass, out, distinct, st, nullptr);
            cudaEventRecord(c->tev[1], st);
            if (rc != FEM_OK) break;
            float t = 0;
            if (cudaEventSynchronize(c->tev[1]) != cudaSuccess ||
                cudaEventElapsedTime(&t, c->tev[0], c->tev[1]) != cudaSuccess) {
                rc = FEM_ECUDA;
                break;
            }
            if (sh.ms < 0 || t < sh.ms) sh.ms = t;
        }
    }
    // the rule's shape (the first) stays unless another is at least 2% faster
    fem_ctx::Shape best{0, 0, 0, 0};
    if (rc == FEM_OK && !shapes.empty()) {
        best = shapes[0];
        for (const fem_ctx::Shape &sh : shapes)
            if (sh.ms < 0.98f * best.ms) best = sh;
    }
    c->cfg = saved;
    c->tuning = false;
    if (rc == FEM_OK && best.P) c->tune[key] = best;
    return rc;
}

// A counting pass that has been launched: what its completion check needs.
struct PassLaunch {
    CountParams p{};
    int N = 0, pass = 0;
    bool distinct = true, chain = false;
    uint32_t R = 1;
    int evset = 0;  // the kernel event set recorded around it
    bool pairs = false;  // the level-2 pair kernel
    bool hits = false;   // over hit tables (finished when launched)
};

// Launch one counting pass over m candidates (all of length N) -> out[0..m)
// (kernel, then the stitch when segmented), without waiting for it.  The pass is
// complete only after count_finish has seen the error word.
int count_launch(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
                 uint32_t m, int N, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
                 bool distinct, cudaStream_t st, PassLaunch *pl) {
    pl->p = CountParams{};
    pl->N = N, pl->pass = pass, pl->distinct = distinct;
    if (m == 0) return FEM_OK;
    // a measured shape for this class, if any (explicit configuration wins)
    uint32_t P_t = 0, T_t = 0, K_t = 0;
    if (!c->cfg.segments && !c->cfg.threads_per_block && !c->cfg.kernel && !c->tuning) {
        const std::string key = tune_key(N, pass, distinct, m, s.n_chunks, s.K);
        auto it = c->tune.find(key);
        if (it == c->tune.end() && c->tune_on) {
            RET(tune_pass(c, key, s, cands, gather, m, N, d_ivl, nI, pass, out, distinct, st));
            it = c->tune.find(key);
        }
        if (it != c->tune.end()) P_t = it->second.P, T_t = it->second.T, K_t = it->second.kernel;
    }
    uint32_t kind = c->cfg.kernel ? c->cfg.kernel : K_t;
    if (!kind) kind = rule_kernel(c, N, pass, distinct, m);
    // (a configured or cached choice of the latest-chain kernels needs distinct types only)
    if (kind == FEM_KERNEL_CHAIN && !(distinct && N >= 2)) kind = FEM_KERNEL_MACHINE;
    CountParams p{};
    p.bev = s.bev;
    p.boff = s.boff;
    p.cfirst = s.cfirst;
    p.t = s.t;
    p.offs = s.offs;
    p.n_chunks = s.n_chunks;
    p.n = s.n;
    p.K = s.K;
    p.cands = cands;
    p.gather = gather;
    p.m = m;
    p.ivl = d_ivl;
    p.n_ivl = nI;
    p.out = out;
    p.err = c->d_err;
    uint8_t *redo;
    RET(dbuf(c, "redo", m, &redo));
    CK(cudaMemsetAsync(redo, 0, m, st));
    p.redo = redo;

    uint32_t P = P_t ? std::min<uint32_t>(P_t, std::max<uint32_t>(s.n_chunks, 1))
                     : choose_segments(c, s, m, distinct, kind == FEM_KERNEL_CHAIN && N == 2);
    if (!distinct) P = 1;
    uint32_t R = 1;
    if (pass == FEM_PASS_EXACT) R = c->cfg.ring_capacity ? c->cfg.ring_capacity : 8;
    if (pass == FEM_PASS_EXACT && !c->cfg.ring_capacity && kind == FEM_KERNEL_MACHINE) {
        // rings sized from the capacity table where lists outgrow the small rings often
        // (bursting recordings), so that the first count does not overflow
        bool sg, cl;
        RET(ring_choice(c, s, &sg, &cl, st));
        if (P > 1 ? sg : cl) R = kRingLarge;
    }
    if (P > 1 && pass == FEM_PASS_EXACT && R > 32) R = 32;
    if (!count_config_supported(N, pass, P > 1, R)) return FEM_EINVAL;
    const uint32_t cps = P > 1 ? (s.n_chunks + P - 1) / P : std::max<uint32_t>(s.n_chunks, 1);
    if (P > 1) P = (s.n_chunks + cps - 1) / cps;
    p.cps = cps;
    p.P = P;
    if (P > 1) {
        RET(dbuf(c, "tables", (size_t)P * m * S_MAX, &p.tables));
    }
    const int es = c->kev_flip ^= 1;
    pl->evset = es;
    cudaEvent_t *kev = c->kev[es];
    CK(cudaEventRecord(kev[0], st));
    pl->chain = kind == FEM_KERNEL_CHAIN;
    if (kind == FEM_KERNEL_CHAIN) {
        uint32_t T = c->cfg.threads_per_block ? c->cfg.threads_per_block : (T_t ? T_t : chain_threads(m));
        if (chain_smem_bytes(N, P > 1, T, s.offs) > 200 * 1024) T = 128;
        CK(launch_chain(N, pass, P > 1, T, p, st));
    } else {
        uint32_t T = choose_threads(c, N, pass, P > 1, R, s.offs, m);
        if (T_t && count_smem_bytes(N, pass, P > 1, R, T_t, s.offs) <= 100 * 1024) T = T_t;
        // a configured block size whose rings would not fit in shared memory is replaced
        if (count_smem_bytes(N, pass, P > 1, R, T, s.offs) > 200 * 1024)
            T = auto_threads(N, pass, P > 1, R, s.offs, m);
        CK(launch_count(N, pass, P > 1, R, T, p, st));
    }
    CK(cudaEventRecord(kev[1], st));
    if (P > 1) CK(launch_stitch(p.tables, m, P, out, redo, c->d_err, st));
    CK(cudaEventRecord(kev[2], st));
    pl->p = p;
    pl->R = R;
    return FEM_OK;
}

// The relaxed pass of fem_mine_levelwise's level 2 (f frequent types x nI <= 4 intervals,
// m = f (f - 1) nI candidates in canonical order) with every interval variant of an
// ordered type pair in one thread (fem_pairs.cu); segments for about three 256-thread
// blocks per SM (or the configured count), tables, stitch and completion as in
// count_launch.
int count_launch_pairs(fem_ctx *c, const StreamDev &s, const fem_episode *cands, uint32_t m,
                       uint32_t f, const uint2 *d_ivl, uint32_t nI, uint32_t *out, cudaStream_t st,
                       PassLaunch *pl) {
    pl->p = CountParams{};
    pl->N = 2, pl->pass = FEM_PASS_RELAXED, pl->distinct = true, pl->chain = false;
    pl->pairs = true;
    if (m == 0) return FEM_OK;
    CountParams p{};
    p.bev = s.bev;
    p.boff = s.boff;
    p.cfirst = s.cfirst;
    p.t = s.t;
    p.offs = s.offs;
    p.n_chunks = s.n_chunks;
    p.n = s.n;
    p.K = s.K;
    p.cands = cands;
    p.m = m;
    p.ivl = d_ivl;
    p.n_ivl = nI;
    p.out = out;
    p.err = c->d_err;
    p.pair_types = f;
    uint8_t *redo;
    RET(dbuf(c, "redo", m, &redo));
    CK(cudaMemsetAsync(redo, 0, m, st));
    p.redo = redo;
    const uint64_t pairs = (uint64_t)f * (f - 1);
    uint32_t P;
    if (c->cfg.segments) {
        P = std::min<uint32_t>(c->cfg.segments, std::max<uint32_t>(s.n_chunks, 1));
    } else {
        const uint64_t target = (uint64_t)c->sm_count * 3 * 256;
        P = (uint32_t)std::min<uint64_t>((target + pairs - 1) / pairs, std::max<uint32_t>(s.n_chunks, 1));
    }
    const uint32_t cps = P > 1 ? (s.n_chunks + P - 1) / P : std::max<uint32_t>(s.n_chunks, 1);
    if (P > 1) P = (s.n_chunks + cps - 1) / cps;
    p.cps = cps;
    p.P = P;
    if (P > 1) RET(dbuf(c, "tables", (size_t)P * m * S_MAX, &p.tables));
    const int es = c->kev_flip ^= 1;
    pl->evset = es;
    cudaEvent_t *kev = c->kev[es];
    CK(cudaEventRecord(kev[0], st));
    CK(launch_pairs_relaxed(p, 256, st));
    CK(cudaEventRecord(kev[1], st));
    if (P > 1) CK(launch_stitch(p.tables, m, P, out, redo, c->d_err, st));
    CK(cudaEventRecord(kev[2], st));
    pl->p = p;
    pl->R = 1;
    return FEM_OK;
}

// Kernel and stitch times of the last launched pass (its events have completed).
void pass_info(fem_ctx *c, const PassLaunch &pl, PassInfo *info) {
    info->segments = pl.p.m ? pl.p.P : 0;
    info->kernel = !pl.p.m    ? 0u
                   : pl.hits  ? FEM_KERNEL_HITS
                   : pl.pairs ? FEM_KERNEL_PAIRS
                   : pl.chain ? FEM_KERNEL_CHAIN
                              : FEM_KERNEL_MACHINE;
    info->ms_kernel = info->ms_stitch = 0;
    if (!pl.p.m) return;
    cudaEventElapsedTime(&info->ms_kernel, c->kev[pl.evset][0], c->kev[pl.evset][1]);
    cudaEventElapsedTime(&info->ms_stitch, c->kev[pl.evset][1], c->kev[pl.evset][2]);
}

// Complete a launched pass given the error word read after it: report hard errors,
// and recount the episodes whose rings or class tables overflowed.
int count_finish(fem_ctx *c, const StreamDev &s, const PassLaunch &pl, uint32_t e,
                 cudaStream_t st) {
    RET(err_status(e));
    if (!pl.p.m || !(e & ERR_CAP)) return FEM_OK;
    const CountParams &p = pl.p;
    const uint32_t m = p.m, P = p.P, R = pl.R;
    const int N = pl.N, pass = pl.pass;
    const bool distinct = pl.distinct;
    const uint32_t *gather = p.gather;
    uint32_t *out = p.out;
    uint8_t *redo = p.redo;

    // Recount the flagged episodes with one segment and larger rings.
    uint32_t *ridx, *rg, *rout, *scratch;
    RET(dbuf(c, "redo_idx", m, &ridx));
    RET(dbuf(c, "redo_scratch", compact_scratch_words(m), &scratch));
    CK(launch_compact(nullptr, redo, 0, m, ridx, c->d_small + W_COUNT2, scratch, st, pub_of(c)));
    uint32_t r, er;
    RET(read_count_err(c, c->d_small + W_COUNT2, &r, &er, st));
    if (std::getenv("FEM_DEBUG"))
        std::fprintf(stderr, "fem: pass %d N=%d m=%u P=%u R=%u: %u episodes recounted (err %#x)\n",
                     pass, N, m, P, R, r, e);
    if (r == 0) return FEM_OK;
    RET(dbuf(c, "redo_gather", r, &rg));
    RET(dbuf(c, "redo_out", r, &rout));
    CK(launch_compose_idx(gather, ridx, r, rg, st));
    // Episodes a latest-chain launch gave up on (its prefix tables or four class slots
    // were too small) go first to the per-thread kernels with the pass's own segments.
    // Then: the flagged episodes alone, one chunk per segment (short items, so the retry
    // costs about one chunk of work) with the largest segmented rings; last resort, one
    // segment per episode with the largest rings.
    struct Try {
        bool mc;
        uint32_t R;
        bool same_segments;
        uint32_t cls;  // entry-class slots of the segmented tables
    };
    std::vector<Try> tries;
    if (pl.pairs) tries.push_back({true, 8u, false, S_MAX});  // one chunk per segment
    if (pl.chain) {
        // a latest-chain launch that only ran out of its entry-class slots: the per-thread
        // kernel has twice the slots and merges classes before refusing one; one chunk per
        // segment, so that the few episodes spread over the GPU.  Other guards: the
        // per-thread kernel with the pass's own segments.
        if (e & ~ERR_CLASS & ERR_CAP) tries.push_back({P > 1, 8u, true, S_MAX});
        else tries.push_back({true, 8u, false, S_MAX});
    }
    tries.push_back({true, 32u, false, S_RECOUNT});  // four times the slots, larger rings
    tries.push_back({false, 32u, false, S_MAX});
    tries.push_back({false, 128u, false, S_MAX});
    for (const Try &tr : tries) {
        if (tr.mc && !distinct) continue;
        CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));
        CountParams q = p;
        q.gather = rg;
        q.m = r;
        q.out = rout;
        RET(dbuf(c, "redo2", r, &q.redo));
        CK(cudaMemsetAsync(q.redo, 0, r, st));
        const uint32_t Rq = pass == FEM_PASS_EXACT ? tr.R : 1;
        const uint32_t cls = tr.mc && s.n_chunks > 1 ? tr.cls : S_MAX;
        if (tr.same_segments) {
            if (q.P > 1) RET(dbuf(c, "redo_tables", (size_t)q.P * r * cls, &q.tables));
        } else if (tr.mc && s.n_chunks > 1) {
            q.P = s.n_chunks;
            q.cps = 1;
            RET(dbuf(c, "redo_tables", (size_t)q.P * r * cls, &q.tables));
        } else {
            q.P = 1;
            q.cps = std::max<uint32_t>(s.n_chunks, 1);
            q.tables = nullptr;
        }
        const bool mc2 = q.P > 1;
        // the recount's rings are larger: its block size is chosen for them, whatever
        // size is configured (or being tried) for the first count
        const uint32_t T2 = auto_threads(N, pass, mc2, Rq, s.offs, r, cls);
        CK(launch_count(N, pass, mc2, Rq, T2, q, st, cls));
        if (mc2) CK(launch_stitch(q.tables, r, q.P, rout, q.redo, c->d_err, st, cls));
        RET(read_err(c, st, &e));
        RET(err_status(e));
        if (std::getenv("FEM_DEBUG"))
            std::fprintf(stderr, "fem:   retry P=%u R=%u: err %#x\n", q.P, Rq, e);
        if (!(e & ERR_CAP)) {
            CK(launch_scatter_u32(rout, ridx, r, out, st));
            return FEM_OK;
        }
    }
    return FEM_EOVERFLOW;
}

// One counting pass, waited for and completed.
int count_pass(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
               uint32_t m, int N, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
               bool distinct, cudaStream_t st, PassInfo *info) {
    if (m == 0) return FEM_OK;
    PassLaunch pl;
    RET(count_launch(c, s, cands, gather, m, N, d_ivl, nI, pass, out, distinct, st, &pl));
    uint32_t e;
    RET(read_err(c, st, &e));
    if (info) pass_info(c, pl, info);
    return count_finish(c, s, pl, e, st);
}

// Segments of a hit-table pass over m candidates: about four 128-thread blocks for each
// place on the GPU (the episodes' hits differ, so blocks end at different times), but of
// eight slabs or more (a segment first goes through the window before it) unless that
// would leave SMs without a block.  And segments whose tables stay in a part of the L2
// cache while the blocks of all candidates, which run next to each other, read them (the
// hour-long recording, 481 KB a slab, with 240 segments 147 ms; while it took 168 so, with
// eight it took 300).
constexpr uint64_t kHitSegmentBytes = 24ull << 20;
uint32_t hit_segments(const fem_ctx *c, uint32_t n_slabs, uint32_t n_chunks, uint32_t m,
                      uint64_t slab_bytes) {
    if (n_slabs < 2) return 1;
    if (c->cfg.segments) return std::min(c->cfg.segments, std::max(n_chunks, 1u));
    const uint64_t tiles = (m + 127) / 128, wave = (uint64_t)c->sm_count * 6;
    const uint64_t P4 = (4 * wave + tiles - 1) / tiles, P1 = (wave + tiles - 1) / tiles;
    const uint64_t longest = std::max<uint64_t>(16, kHitSegmentBytes / std::max<uint64_t>(slab_bytes, 1));
    const uint64_t P = std::max(std::min<uint64_t>(P4, n_slabs / 8), std::min<uint64_t>(P1, n_slabs / 2));
    return (uint32_t)std::min<uint64_t>(std::max<uint64_t>({1, P, (n_slabs + longest - 1) / longest}), 65535);
}

int count_grouped(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
                  uint32_t m, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out, cudaStream_t st);

// Set a hit-table pass's segments.
void hits_segments(const fem_ctx *c, const StreamDev &s, CountParams &p) {
    const uint32_t P = hit_segments(c, p.hits.n_slabs, s.n_chunks, p.m, p.hits.slab_bytes);
    p.cps = (p.hits.n_slabs + P - 1) / P;
    p.P = (p.hits.n_slabs + p.cps - 1) / p.cps;
}

// Launch a hit-table pass over p.m candidates (and its stitch when segmented).  The transfer
// tables (30 KB a candidate on the hour-long recording) take at most a 64th of the device's
// memory: more candidates (145,000 there) are counted a part after the other, each with all
// segments.
int hits_launch(fem_ctx *c, const StreamDev &s, uint32_t group, CountParams &p, uint32_t classes,
                const char *tables, cudaStream_t st) {
    hits_segments(c, s, p);
    p.hit_classes = classes;
    uint32_t step = p.m;
    if (p.P > 1) {
        const size_t each = (size_t)p.P * classes;
        step = (uint32_t)std::min<size_t>(step, std::max<size_t>(128, c->mem_device / 64 / (each * sizeof(uint4)) / 128 * 128));
        RET(dbuf(c, tables, each * step, &p.tables));
    }
    for (uint64_t off = 0; off < p.m; off += step) {
        CountParams q = p;
        q.gather += off, q.out += off, q.redo += off;
        q.m = std::min(step, p.m - (uint32_t)off);
        CK(launch_hit_count(group, q.P > 1, q, st));
        if (q.P > 1) CK(launch_stitch(q.tables, q.m, q.P, q.out, q.redo, c->d_err, st, classes));
    }
    return FEM_OK;
}

// Recount what a hit-table pass flagged: with all the class slots the kernel can use, then
// by the per-thread kernels.
int hits_finish(fem_ctx *c, const StreamDev &s, uint32_t group, const CountParams &p, int pass,
                uint32_t e, cudaStream_t st) {
    uint32_t *ridx, *rg, *rout, *scratch, r, er;
    RET(dbuf(c, "hit_idx", p.m, &ridx));
    RET(dbuf(c, "redo_scratch", compact_scratch_words(p.m), &scratch));
    CK(launch_compact(nullptr, p.redo, 0, p.m, ridx, c->d_small + W_COUNT2, scratch, st, pub_of(c)));
    RET(read_count_err(c, c->d_small + W_COUNT2, &r, &er, st));
    if (r == 0) return FEM_OK;
    if (std::getenv("FEM_DEBUG"))
        std::fprintf(stderr, "fem: hit-table pass %d m=%u P=%u: %u episodes recounted (err %#x)\n", pass,
                     p.m, p.P, r, e);
    RET(dbuf(c, "hit_gather", r, &rg));
    RET(dbuf(c, "hit_out", r, &rout));
    CK(launch_compose_idx(p.gather, ridx, r, rg, st));
    CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));
    CountParams q = p;
    q.gather = rg;
    q.m = r;
    q.out = rout;
    RET(dbuf(c, "hit_redo", r, &q.redo));
    CK(cudaMemsetAsync(q.redo, 0, r, st));
    RET(hits_launch(c, s, group, q, S_RECOUNT, "hit_redo_tables", st));
    RET(read_err(c, st, &e));
    RET(err_status(e));
    if (e & ERR_CAP) {
        CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));
        RET(count_grouped(c, s, p.cands, rg, r, p.ivl, p.n_ivl, pass, rout, st));
    }
    CK(launch_scatter_u32(rout, ridx, r, p.out, st));
    return FEM_OK;
}

// A set planned for hit tables, and the tables.
struct HitPlan {
    uint32_t *order = nullptr, *gather = nullptr;  // slot -> place in the set, candidate record
    uint32_t group_m[PLAN_GROUPS] = {};            // candidates per launch, in slot order
    uint32_t len_m[FEM_MAX_LEN + 1] = {};          // candidates per length
    HitTables h{};
    HitBuild b{};
    uint64_t hits = 0;  // the range table's size
};

// A stream's types that a plan or build found too dense, kept with it.
int remember_dense(fem_ctx *c, const StreamDev &s, cudaStream_t st) {
    uint32_t found[256];
    CK(cudaMemcpyAsync(found, c->d_dense, sizeof(found), cudaMemcpyDeviceToHost, st));
    CK(cudaMemsetAsync(c->d_dense, 0xFF, sizeof(found), st));
    CK(cudaStreamSynchronize(st));
    s.dense_hi.resize(256, ~0u);
    for (uint32_t a = 0; a < 256; ++a) s.dense_hi[a] = std::min(s.dense_hi[a], found[a]);
    return FEM_OK;
}

// Whether tables over edges from these types (a bit each) are known to be too dense for the
// current interval set: plan, build and launches for nothing.  200 episodes on 3,000 events
// with bursts of a type: 1.02 ms when every call tried, 0.70 remembered, 0.71 before there
// were tables; 20,000 on 100,000 events 2.85, 1.67 and 1.68 ms.
bool known_dense(const fem_ctx *c, const StreamDev &s, const uint32_t *types) {
    uint32_t max_hi = 0;
    for (const fem_interval &iv : c->ivl_host) max_hi = std::max(max_hi, iv.hi_us);
    for (uint32_t a = 0; a < s.dense_hi.size(); ++a)
        if ((types[a >> 5] >> (a & 31) & 1u) && s.dense_hi[a] <= max_hi) return true;
    return false;
}

// Plan a set (checked and ordered, its edges numbered, the stream cut) and size its tables.
// *ok = false where tables do not apply: repeated types, or a stream whose chunks do not
// span the longest interval (the events before a slab are kept from its chunk and the one
// before).
// alloc(name, words, &pointer) gives the plan's device memory.  info: the words of a
// validation (three of them).
template <typename Alloc>
int hits_plan(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
              uint32_t m, bool fine, const uint2 *d_ivl, uint32_t nI, int pass, cudaStream_t st,
              HitPlan *pl, bool *ok, Alloc &&alloc, uint32_t *info = nullptr) {
    *ok = false;
    uint64_t max_hi = 0;
    for (const fem_interval &iv : c->ivl_host) max_hi = std::max<uint64_t>(max_hi, iv.hi_us);
    PlanArgs a{};
    a.cands = cands;
    a.gather = gather;
    a.m = m;
    a.K = s.K;
    a.n_ivl = nI;
    a.parts = std::min(nI, PLAN_PARTS);
    a.fine = fine;
    a.runs = info != nullptr;
    a.cfirst = s.cfirst;
    a.t = s.t;
    a.n_chunks = s.n_chunks;
    a.n = s.n;
    a.max_hi = (uint32_t)max_hi;
    a.dense = c->d_dense;
    a.err = c->d_err;
    const uint32_t bins = plan_bins(s.K, a.parts), tri = s.K * s.K * nI;
    const size_t max_slabs = (size_t)s.n_chunks * 64 + 1;
    RET(alloc("hit_plan", PLAN_WORDS + (size_t)bins + tri, &a.words));
    a.hist = a.words + PLAN_WORDS;
    a.edge_id = a.hist + bins;
    RET(alloc("hit_plan_slabs", s.n_chunks + 2 * max_slabs, &a.parts_of));
    a.begin = a.parts_of + s.n_chunks;
    a.t0 = a.begin + max_slabs;
    RET(alloc("hit_plan_bin", m, &a.bin));
    RET(alloc("hit_plan_rank", m, &a.rank));
    RET(alloc("hit_plan_order", m, &pl->order));
    RET(alloc("hit_plan_gather", m, &pl->gather));
    const uint32_t seq = ++c->pub_seq;
    CK(launch_plan(a, s, pl->order, pl->gather, Publish{c->d_plan, c->d_err, seq}, st));
    const volatile uint32_t *w = c->h_small + kPlanWord;
    RET(wait_seq(w + PLAN_WORDS + 1, seq, st));
    RET(err_status(w[PLAN_WORDS]));
    if (info) {
        info[0] = 0, info[1] = w[PLAN_REP], info[2] = w[PLAN_RUNS];
        for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N)
            if (w[N - 1]) info[0] |= 1u << N;
    }
    const uint64_t span = (uint32_t)~w[PLAN_SPAN];
    if (s.n_chunks > 1) s.least_span = std::min(s.least_span, span);
    if (w[PLAN_DENSE]) {
        if (std::getenv("FEM_DEBUG")) std::fprintf(stderr, "fem: hit tables of %u slabs: too dense\n", w[PLAN_SLABS]);
        return remember_dense(c, s, st);
    }
    if (w[PLAN_REP]) return FEM_OK;
    if (s.n_chunks > 1 && span <= max_hi) return FEM_OK;
    for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N) {
        pl->len_m[N] = w[N - 1];
        pl->group_m[plan_group(N, a.fine)] += w[N - 1];
    }
    HitTables &h = pl->h;
    h.n_slabs = w[PLAN_SLABS], h.n_edges = w[PLAN_EDGES];
    h.types = (s.K + 15) & ~15u;
    h.edge_id = a.edge_id, h.begin = a.begin, h.t0 = a.t0;
    HitBuild &b = pl->b;
    b.bev = s.bev, b.boff = s.boff, b.offs = s.offs, b.K = s.K, b.types = h.types;
    b.ivl = d_ivl, b.n_ivl = nI, b.n_edges = h.n_edges;
    b.max_words = CHUNK / 32 / w[PLAN_PARTS_MIN];
    b.edge_id = a.edge_id, b.begin = a.begin, b.err = c->d_err, b.dense = c->d_dense;
    // hits: as many as events lie in the intervals at the stream's mean rate, and a quarter
    // more (the table grows when that is too few), at most one per edge and event of its last type
    double per_event = 0;
    for (const fem_interval &iv : c->ivl_host)
        per_event += (double)(iv.hi_us - (pass == FEM_PASS_EXACT ? iv.lo_us : 0u)) * (double)s.n /
                     (double)std::max(s.t_max - s.t_min, 1u);
    per_event *= (double)h.n_edges / tri;
    pl->hits = std::min<uint64_t>((uint64_t)(1.25 * per_event * (double)s.n) + 65536,
                                  (uint64_t)s.n * (h.n_edges / s.K + 1));
    *ok = true;
    return FEM_OK;
}

// The tables' memory and their build.
int hits_build(fem_ctx *c, const StreamDev &s, int pass, HitPlan *pl, cudaStream_t st) {
    HitBuild &b = pl->b;
    HitTables &h = pl->h;
    RET(dbuf(c, "hit_edges", (size_t)h.n_slabs * h.n_edges, &b.edge));
    RET(dbuf(c, "hit_counts", (size_t)h.n_slabs * h.types, &b.count));
    RET(dbuf(c, "hit_places", (size_t)h.n_slabs * h.types, &b.place));
    RET(dbuf(c, "hit_index", s.n, &b.index));
    RET(dbuf(c, "hit_used", 1, &b.used));
    RET(dbuf(c, "hit_ranges", pl->hits, &b.range));
    b.capacity = std::min<uint64_t>(c->bufs["hit_ranges"].cap / sizeof(uint32_t), 0xFFFFFFF0ull);
    CK(cudaMemsetAsync(b.used, 0, 8, st));
    CK(launch_hit_build(pass, h.n_slabs, b, c->sm_count, st));
    h.slab_bytes = (uint64_t)h.n_edges * 8 + pl->hits * 4 / std::max(h.n_slabs, 1u);
    h.edge = b.edge, h.range = b.range, h.count = b.count, h.place = b.place, h.index = b.index;
    return FEM_OK;
}

// The kernel arguments of launch g (candidates from slot `off` on).
CountParams hits_params(fem_ctx *c, const StreamDev &s, const HitPlan &pl, const fem_episode *cands,
                        uint32_t g, uint32_t off) {
    CountParams p{};
    p.cfirst = s.cfirst;
    p.t = s.t;
    p.n_chunks = s.n_chunks;
    p.n = s.n;
    p.K = s.K;
    p.cands = cands;
    p.gather = pl.gather + off;
    p.m = pl.group_m[g];
    p.ivl = pl.b.ivl;
    p.n_ivl = pl.b.n_ivl;
    p.err = c->d_err;
    p.hits = pl.h;
    return p;
}

// What became of the launches over the tables: *e the error word (capacity guards), *again
// when the tables held too few hits (pl->hits is then what they need), *dense when events
// were too dense for them.  The error word is cleared where nothing was counted.
int hits_check(fem_ctx *c, const StreamDev &s, HitPlan *pl, uint32_t *e, bool *again, bool *dense,
               cudaStream_t st) {
    uint32_t used;
    CK(launch_publish_count(pl->b.used, pub_of(c), st));
    RET(read_count_err(c, nullptr, &used, e, st));
    RET(err_status(*e));
    *dense = (*e & ERR_DENSE) != 0 || used > 0xF0000000u;
    *again = !*dense && used > pl->b.capacity;
    if (*again) pl->hits = used + used / 16;
    if (std::getenv("FEM_DEBUG"))
        std::fprintf(stderr, "fem: hit tables of %u edges in %u slabs, %u hits: %s\n", pl->h.n_edges, pl->h.n_slabs,
                     used, *dense ? "too dense" : *again ? "too small" : "counted");
    if (*again || *dense) CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));
    if (*e & ERR_DENSE) RET(remember_dense(c, s, st));
    return FEM_OK;
}

// What a count takes in microseconds, over hit tables and by the other kernels.  The tables'
// cost is that of the edges a set may use (the plan numbers them), of events times types (the
// build, whose blocks share an SM as their rank rows leave room) and of hits (build and count);
// the other kernels' is that of a launch and a wait for each length, of events times nodes,
// and of an event's look-back for every length.  Fits to 3,680 counts of 100 to 60,000 episodes
// of one length (2 to 7) or several, on 500 to 3 million events of 8 to 200 types at 5 to 55
// Hz, both passes by both ways: half of the estimates within 12%, nine of ten within 33
// (tables) and 38%.  By the faster estimate 66 of those counts (and 19 of 400 others) take more
// than 5% longer than by the other kernels, 1.7 (1.2) times at most; over tables wherever they
// apply 1,604 would, up to 14 times (5,000 events of 128 types, 2,000 pairs, relaxed: 116 us
// and 270).  Over the 400 others the counts are 1.68 times as fast as without tables.
constexpr double kPlanEdgeUs = 1.05e-3;  // a plan, per type pair and interval
double events_in_interval(const fem_ctx *c, const StreamDev &s) {  // of a type, in the longest
    uint64_t max_hi = 0;
    for (const fem_interval &iv : c->ivl_host) max_hi = std::max<uint64_t>(max_hi, iv.hi_us);
    return (double)s.n * (double)max_hi / ((double)s.K * (double)std::max(s.t_max - s.t_min, 1u));
}

struct SetSize {  // candidates per length
    double len_m[FEM_MAX_LEN + 1] = {};
};
SetSize equal_parts(uint32_t lens, uint32_t m) {  // of the lengths in a mask
    SetSize z;
    for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N)
        if (lens >> N & 1u) z.len_m[N] = (double)m / __builtin_popcount(lens);
    return z;
}

double tables_us(const fem_ctx *c, const StreamDev &s, uint32_t nI, const SetSize &z, int pass) {
    const bool x = pass == FEM_PASS_EXACT;
    const double K = s.K, n = (double)s.n, pairs = K * K, in = events_in_interval(c, s);
    double m = 0, nodes = 0;
    for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N) m += z.len_m[N], nodes += N * z.len_m[N];
    const double edges = nodes - m;  // (of all episodes, some of them the same)
    const double used = std::min(1.0, edges / (pairs * nI)), groups = std::min(1.0, edges * std::min(K, 32.0) / pairs);
    // blocks of a build on an SM (at least four by registers): 719 bytes a type (build_smem)
    const double blocks = std::max(1.0, std::min(4.0, std::floor(232448.0 / (719 * K + 1024))));
    return (x ? 147 : 156) + kPlanEdgeUs * pairs * nI +
           4 / blocks * n * K * (3.1e-6 * groups + (x ? 1.65e-5 : 2.2e-5) * used * in) +
           (x ? 1.05e-6 : 1.6e-6) * nodes * n / K * in + 7e-4 * m;
}

double others_us(const fem_ctx *c, const StreamDev &s, const SetSize &z, int pass) {
    const bool x = pass == FEM_PASS_EXACT;
    const double each = (double)s.n / s.K;  // events of a type
    double us = 0;
    for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N) {
        const double m = z.len_m[N];
        if (m <= 0) continue;
        const double segments = std::max(1.0, std::min(c->sm_count * 2048.0 / m, (double)s.n / CHUNK));
        us += (x ? 38 + 13.0 * N : 52 + 6.0 * N) + (s.n_chunks > 1 ? (x ? 32 : 41) : 0) +
              (x ? 2.08e-6 : 5.95e-7) * m * N * N * each + (x ? 0.28 : 0.207) * N * each / segments;
    }
    return us;
}

// The same of window frequencies, whose other kernel has one thread per episode walk the whole
// stream, one length after the other (us by that kernel / over tables: 2,000 pairs on 1,000
// events of 64 types 110 / 137, of four nodes 160 / 144; pairs of 128 types on 1,000 events 93 /
// 183, on 3,400 139 / 204, on 20,000 431 / 224; 100 pairs of 16 types on 100 events 87 / 108, on
// 1,000 208 / 117).
bool windows_over_tables(const StreamDev &s, uint32_t nI, uint32_t lens, uint32_t m) {
    const double K = s.K, n = (double)s.n;
    double others = 52;
    uint32_t most = 1;
    for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N)
        if (lens >> N & 1u) others += 20 + (0.7 + 0.1 * N) * N * n / K + 10.0 * s.n_chunks, most = N;
    const double groups = std::min(1.0, (double)m * (most - 1) * std::min(K, 32.0) / (K * K));
    return 108 + 0.6e-3 * K * K * nI + 3e-3 * K * K * groups + 4e-3 * m < others;
}

// A set of fewer candidates is planned for the tables without a validation before (one wait
// less where they do count it), unless the plan, whose edges are scanned by one block, costs
// far more than that, or a mixed set of that size would not go over them.
constexpr uint32_t kPlanFirst = 256;
constexpr double kPlanUs = 20;  // a plan over a validation
bool plan_first(const fem_ctx *c, const StreamDev &s, uint32_t m, uint32_t nI, int pass) {
    const SetSize z = equal_parts(1u << 2 | 1u << 3 | 1u << 4, m);
    return m < kPlanFirst && kPlanEdgeUs * s.K * s.K * nI < 25 && tables_us(c, s, nI, z, pass) < others_us(c, s, z, pass);
}

// Count a candidate set over hit tables: all lengths, in an order of their own.  *done =
// false, with nothing counted, where they do not apply.
int count_hits(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
               uint32_t m, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
               cudaStream_t st, bool *done, uint32_t *segments = nullptr, uint32_t *info = nullptr) {
    *done = false;
    HitPlan pl;
    bool ok;
    RET(hits_plan(c, s, cands, gather, m, m >= PLAN_FINE, d_ivl, nI, pass, st, &pl, &ok,
                  [&](const char *n, size_t w, uint32_t **p) { return dbuf(c, n, w, p); }, info));
    if (!ok) return FEM_OK;
    if (info) {  // (nothing was known of the set; the plan is made now, whichever way it goes)
        SetSize z;
        for (uint32_t N = 1; N <= FEM_MAX_LEN; ++N) z.len_m[N] = pl.len_m[N];
        if (others_us(c, s, z, pass) + kPlanUs + kPlanEdgeUs * s.K * s.K * nI < tables_us(c, s, nI, z, pass)) return FEM_OK;
    }
    uint32_t *tmp;
    uint8_t *redo;
    RET(dbuf(c, "hit_plan_out", m, &tmp));
    RET(dbuf(c, "hit_plan_redo", m, &redo));
    for (;;) {
        CK(cudaMemsetAsync(redo, 0, m, st));
        RET(hits_build(c, s, pass, &pl, st));
        CountParams part[PLAN_GROUPS]{};
        uint32_t off = 0;
        for (uint32_t g = 0; g < PLAN_GROUPS; ++g) {
            if (!pl.group_m[g]) continue;
            part[g] = hits_params(c, s, pl, cands, g, off);
            part[g].out = tmp + off;
            part[g].redo = redo + off;
            RET(hits_launch(c, s, g, part[g], S_MAX, "hit_tables", st));
            off += part[g].m;
        }
        uint32_t e;
        bool again, dense;
        CK(launch_scatter_u32(tmp, pl.order, m, out, st));
        RET(hits_check(c, s, &pl, &e, &again, &dense, st));
        if (dense) return FEM_OK;
        if (again) continue;
        if (e & ERR_CAP) {
            for (uint32_t g = 0; g < PLAN_GROUPS; ++g)
                if (part[g].m) RET(hits_finish(c, s, g, part[g], pass, e, st));
            CK(launch_scatter_u32(tmp, pl.order, m, out, st));
            CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));  // nothing is flagged any more
            CK(cudaStreamSynchronize(st));
        }
        if (segments)
            for (const CountParams &q : part) *segments = std::max(*segments, q.P);
        *done = true;
        return FEM_OK;
    }
}

// The window-based frequency of a set over exact-pass hit tables (*done as above).
int windows_hits(fem_ctx *c, const StreamDev &s, const fem_episode *cands, uint32_t m,
                 const uint2 *d_ivl, uint32_t nI, uint32_t window_us, uint64_t *out,
                 cudaStream_t st, bool *done) {
    *done = false;
    HitPlan pl;
    bool ok;
    RET(hits_plan(c, s, cands, nullptr, m, m >= PLAN_FINE, d_ivl, nI, FEM_PASS_EXACT, st, &pl, &ok,
                  [&](const char *n, size_t w, uint32_t **p) { return dbuf(c, n, w, p); }));
    if (!ok) return FEM_OK;
    for (;;) {
        CK(cudaMemsetAsync(out, 0, (size_t)m * 8, st));
        RET(hits_build(c, s, FEM_PASS_EXACT, &pl, st));
        uint32_t off = 0;
        for (uint32_t g = 0; g < PLAN_GROUPS; ++g) {
            if (!pl.group_m[g]) continue;
            CountParams p = hits_params(c, s, pl, cands, g, off);
            hits_segments(c, s, p);
            CK(launch_hit_windows(g, p, pl.order + off, window_us, out, st));
            off += p.m;
        }
        uint32_t e;
        bool again, dense;
        RET(hits_check(c, s, &pl, &e, &again, &dense, st));
        if (again) continue;
        *done = !dense;
        return FEM_OK;
    }
}

// The status of work over hit tables; where there was no room for them beside the stream,
// their memory is given back and the other kernels count (nothing was).  So it is where they
// are more than a 16th of the device's memory: no more is kept for the next call (the
// hour-long recording's, 10 GB, are).
int or_no_room(fem_ctx *c, int rc, bool *done, cudaStream_t st) {
    c->hits_busy = false;
    if (c->mem_used > c->mem_device / 16) {
        size_t kept = 0;
        for (const auto &kv : c->bufs)
            if (kv.first.compare(0, 4, "hit_") == 0) kept += kv.second.cap;
        if (kept > c->mem_device / 16) release_hits(c);
    }
    if (rc != FEM_ENOMEM) return rc;
    *done = false;
    release_hits(c);
    CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));
    return FEM_OK;
}

// Whether a set may be counted over hit tables: no configured kernel or ring size, no more
// type pairs and intervals than are worth a table, and on average no more events of a type
// in an interval than a word is for; nor a stream known to have chunks shorter than an interval
// (hits_plan).
constexpr uint32_t kHitMaxEdges = 1u << 18;
bool hits_eligible(const fem_ctx *c, const StreamDev &s, uint32_t nI) {
    uint64_t max_hi = 0;
    for (const fem_interval &iv : c->ivl_host) max_hi = std::max<uint64_t>(max_hi, iv.hi_us);
    return !c->cfg.kernel && !c->cfg.ring_capacity && c->d_plan && s.n_chunks && nI &&
           (uint64_t)s.K * s.K * nI <= kHitMaxEdges && (s.n_chunks == 1 || s.least_span > max_hi) &&
           (double)s.n * (double)max_hi <= 8.0 * s.K * (double)std::max(s.t_max - s.t_min, 1u);
}

// Whether anything is or may be measured (else no key needs to be looked up).
bool tune_used(const fem_ctx *c) { return c->tune_on || !c->tune.empty(); }

// Whether a set that the rule sends over the hit tables goes there (*use): as measured for its
// class, or, with tuning on and nothing measured, as two counts of either kind tell, each of
// them complete (others(), tables(&done)).  The tables stay unless the other kernels are at
// least 2% faster.  A configured launch shape leaves the rule's choice.
template <typename Others, typename Tables>
int tuned_route(fem_ctx *c, const std::string &key, cudaStream_t st, bool *use, Others &&others,
                Tables &&tables) {
    if (c->cfg.segments || c->cfg.threads_per_block) return FEM_OK;
    auto it = c->tune.find(key);
    if (it == c->tune.end() && c->tune_on && !c->tuning) {
        float ms[2] = {-1.f, -1.f};  // (the first of the others also measures their shapes)
        for (int k : {0, 1, 0, 1}) {
            CK(cudaStreamSynchronize(st));
            const auto t0 = std::chrono::steady_clock::now();
            bool done = true;
            const int rc = k ? tables(&done) : others();
            if (rc == FEM_EOVERFLOW && !k) {  // (the others cannot count it at all)
                CK(cudaMemsetAsync(c->d_err, 0, sizeof(uint32_t), st));
                return FEM_OK;
            }
            RET(rc);
            if (!done) {
                *use = false;
                return FEM_OK;
            }
            CK(cudaStreamSynchronize(st));
            const float t = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
            if (ms[k] < 0 || t < ms[k]) ms[k] = t;
        }
        const bool hits = !(ms[0] < 0.98f * ms[1]);
        it = c->tune.emplace(key, fem_ctx::Shape{1, 32, ms[hits], hits ? (uint32_t)FEM_KERNEL_HITS
                                                                      : (uint32_t)FEM_KERNEL_MACHINE}).first;
        if (std::getenv("FEM_DEBUG"))
            std::fprintf(stderr, "fem: class %s: other kernels %.3f ms, tables %.3f ms\n", key.c_str(), ms[0], ms[1]);
    }
    if (it != c->tune.end()) *use = it->second.kernel == FEM_KERNEL_HITS;
    return FEM_OK;
}

// One pass of level 3 over m candidates of the frequent pairs F, all pairs at once (k_join):
// counts of cands[gather[i]] in out[i].  *done = false, with nothing counted, where the
// tables do not apply; a plan made before is used again if its tables are still there.
int join_pass(fem_ctx *c, const StreamDev &s, HitPlan *pl, bool planned, const fem_episode *F, uint32_t f,
              const fem_episode *cands, const uint32_t *gather, uint32_t m, const uint2 *d_ivl,
              uint32_t nI, int pass, uint32_t *out, cudaStream_t st, PassLaunch *pt, bool *done) {
    *done = false;
    *pt = PassLaunch{};
    pt->N = 3, pt->pass = pass, pt->hits = true;
    pt->p.m = m, pt->p.P = 1;
    if (!planned || !c->bufs["hit_plan"].p) {
        bool ok;
        *pl = HitPlan{};
        RET(hits_plan(c, s, F, nullptr, f, true, d_ivl, nI, pass, st, pl, &ok,
                      [&](const char *name, size_t w, uint32_t **p) { return dbuf(c, name, w, p); }));
        if (!ok) return FEM_OK;
    }
    const uint32_t slots = s.K * nI, n = (uint32_t)s.n;
    uint32_t *cells, *len, *scratch;
    JoinTables g{};
    g.err = c->d_err;
    RET(dbuf(c, "hit_join_cells", (size_t)s.K * slots * slots, &cells));
    RET(dbuf(c, "hit_join_ends", (size_t)s.K * slots, &g.ends));
    RET(dbuf(c, "hit_join_begins", (size_t)s.K * slots, &g.begins));
    RET(dbuf(c, "hit_join_sizes", (size_t)2 * s.K, &g.n_ends));
    g.n_begins = g.n_ends + s.K;
    RET(dbuf(c, "hit_join_rank", (size_t)s.K * pl->h.n_slabs, &g.rank));
    RET(dbuf(c, "hit_join_off", (size_t)n + 1, &g.off));
    RET(dbuf(c, "hit_join_len", n, &len));
    RET(dbuf(c, "hit_join_scan", compact_scratch_words(n), &scratch));
    pt->evset = c->kev_flip ^= 1;
    cudaEvent_t *kev = c->kev[pt->evset];
    for (;;) {
        CK(cudaEventRecord(kev[0], st));
        RET(hits_build(c, s, pass, pl, st));
        RET(dbuf(c, "hit_join_list", pl->b.capacity, &g.list));
        CK(launch_join(pl->h, g, s.hist, n, s.K, nI, len, scratch, cells, st));
        CK(cudaEventRecord(kev[1], st));
        CK(launch_join_gather(cells, cands, gather, m, s.K, nI, out, st));
        CK(cudaEventRecord(kev[2], st));
        uint32_t e;
        bool again, dense;
        RET(hits_check(c, s, pl, &e, &again, &dense, st));
        if (dense) return FEM_OK;
        if (again) continue;
        *done = true;
        return FEM_OK;
    }
}

// A mining level's pass over hit tables (count_hits).
int level_hits(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather, uint32_t m,
               int N, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out, cudaStream_t st,
               PassLaunch *pt, bool *done) {
    *pt = PassLaunch{};
    pt->N = N, pt->pass = pass, pt->hits = true;
    pt->p.m = m;
    pt->evset = c->kev_flip ^= 1;
    cudaEvent_t *kev = c->kev[pt->evset];
    CK(cudaEventRecord(kev[0], st));
    RET(count_hits(c, s, cands, gather, m, d_ivl, nI, pass, out, st, done, &pt->p.P));
    CK(cudaEventRecord(kev[1], st));
    CK(cudaEventRecord(kev[2], st));
    return FEM_OK;
}

// Whether a mining level's pass over m candidates of N nodes goes over hit tables.  Tables
// cost a plan, a build and their launches, about 100 us and 6 us for a million of (events x
// types); for a million of (candidates x events of their types) they then count in 1.2 us
// what the other kernels do in 1.9.  Those flag candidates with more than eight entry
// classes for a recount, which costs another 100 to 2,000 us when it comes.  Measured (us,
// before / over tables, recounts included): 22 candidates, 64 types, 406,000 events 86 /
// 131; 7,896 there 354 / 458 (the line is at 15,700); 44,544 there 3,316 / 1,304; 26,115 of 19 types, 64,000 events
// 643 / 340; 6,729 of 22 types, 147,000 events 1,614 / 328; 20 of 18 types, 6,200 events
// 340 / 127.  At level 2 (every type pair or most of them) the other kernels fill the device
// from about 1,000 candidates on: 239 pairs of 16 types, 4,000 events 290 / 96; 810 of 18,
// 6,200 events 155 / 112; 952 of 19, 64,000 events 155 / 146; 1,397 of 39, 101,000 events
// 95 / 172; 3,435 of 40, 20,000 events 104 / 144; 6,593 of 61, 179,000 events 145 / 192.  With a segment
// count configured, level 2 keeps its kernels.  (On recordings without structure the others
// need no recounts, and up to 64 candidates take 20 to 80 us there and 80 to 110 over tables; on
// those with embedded chains that choice made whole searches up to 1.6 times slower, 841 to 1,351
// us for one of 10 s.)  Large relaxed sets of four nodes and more, whose prefixes the
// latest-chain kernel shares: 4.9 million on 80,000 events of 48 types 17.2 ms / 53.1, 1.3
// million on 10,000 of 32 0.86 / 2.54, 57,000 on 406,000 of 64 1.28 / 2.10; from a thousand
// million (candidates x events) on the difference is more than the recounts.  Type pairs and
// intervals beyond 16,384 add a plan's time (548 episodes on 1,500 events of 200 types 88 / 285).
bool level_by_hits(const fem_ctx *c, const StreamDev &s, uint32_t N, int pass, uint32_t m, uint32_t nI) {
    if (!hits_eligible(c, s, nI) || m == 0) return false;
    const double cells = (double)s.n * s.K, work = (double)m * N * (double)s.n / s.K;
    if (N == 2) return !c->cfg.segments && m <= 1000 && cells <= 1.5e6;
    if (N >= 4 && pass == FEM_PASS_RELAXED && m >= kChainLargeSet && work >= 1e9) return false;
    const double edges = (double)s.K * s.K * nI;
    return 13 * cells + 2.3e3 * std::max(0.0, edges - 16384) <= 40e6 + work;
}

// Level 3 joins all pairs of frequent pairs from this many candidates on, with at most so
// many cells of (pair, pair) counts (512 MB).  Its cost is that of the pairs and their lists'
// entries; the candidates stand in for them here, since both grow with the frequent pairs.
// Over tables by candidate / joined, us: 9,800 candidates of 22 types and 147,000 events 456 /
// 899 (a few hundred warps that walk the whole stream); 31,000 of 29 types and 30,000 events 256
// / 210; 45,000 of 36 and 186,000 events 913 / 872; 76,000 of 46 and 159,000 events 1,081 / 696.
// On streams of a chunk or two the other kernels are as fast (74,500 of 64 types, 2,500 events
// 57 / joined 111).
constexpr uint32_t kJoinCandidates = 40000;
constexpr uint64_t kJoinCells = 1ull << 27;

// Validate a candidate set (optionally gathered): the words of launch_validate_cands, with the
// types where the stream is known to be too dense in some.
constexpr uint32_t kInfoWords = 11;
int validate(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
             uint32_t m, uint32_t nI, uint32_t *info, cudaStream_t st) {
    const bool types = !s.dense_hi.empty();
    const uint32_t n = types ? kInfoWords : 3;
    CK(cudaMemsetAsync(c->d_small + W_INFO, 0, n * sizeof(uint32_t), st));
    CK(launch_validate_cands(cands, gather, m, s.K, nI, c->d_small + W_INFO, c->d_err, st, types));
    uint32_t e;
    if (c->d_plan) {
        const uint32_t seq = ++c->pub_seq;
        CK(launch_publish_info(c->d_small + W_INFO, n, Publish{c->d_plan, c->d_err, seq}, st));
        const volatile uint32_t *w = c->h_small + kPlanWord;
        RET(wait_seq(w + PLAN_WORDS + 1, seq, st));
        for (uint32_t k = 0; k < n; ++k) info[k] = w[k];
        e = w[PLAN_WORDS];
    } else {
        RET(read_words(c, c->d_small + W_INFO, n, info, st));
        RET(read_err(c, st, &e));
    }
    return err_status(e);
}

// Sets in runs of shared prefixes (at least four candidates long on average) are for the
// latest-chain kernels.
bool in_runs(const uint32_t *info, uint32_t m) { return (uint64_t)m >= 4ull * ((uint64_t)info[2] + 1); }

// Most of all pairs, exact, on a long stream: the latest-chain kernel looks every last-node
// event up for each, the tables' cost is that of the stream.  Chain / tables, us: 16,128 pairs
// of 64 types over 383,000 events 570 / 481, over 1.5 million 1,904 / 1,171, over 128,000
// 240 / 269; 3,968 of 32 over 288,000 375 / 301; 2,208 of 24 over 864,000 476 / 411; 30% of
// the 64 types' pairs over 383,000 events 228 / 272.  (Relaxed, the machine is the faster.)
bool most_pairs(const StreamDev &s, const uint32_t *info, uint32_t m, uint32_t nI, int pass) {
    return pass == FEM_PASS_EXACT && info[0] == 1u << 2 && 4ull * m >= 3ull * s.K * (s.K - 1) * nI &&
           (double)m * (double)s.n >= 35e6 * s.K;
}

int count_validated(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
                    uint32_t m, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
                    const uint32_t *info, cudaStream_t st);

// Validate a candidate set (optionally gathered) and count it with `pass`,
// grouping candidates by length.  out[i] is the count of candidate i of the
// (gathered) set.
int count_any(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
              uint32_t m, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
              cudaStream_t st) {
    if (m == 0) return FEM_OK;
    uint32_t info[kInfoWords];
    bool hits = hits_eligible(c, s, nI), known = false;
    // a small set goes to the hit tables without a look at its runs (their plan validates
    // too, and saves it a wait); where they turn out not to apply, the plan's words are the
    // validation's (100 episodes with repeated types 338 us with a validation after the plan, 320
    // so, 315 without tables; 200 on a stream with chunks of 5 ms 513, 322 and 338)
    if (!hits || !plan_first(c, s, m, nI, pass) || !s.dense_hi.empty() || tune_used(c)) {
        RET(validate(c, s, cands, gather, m, nI, info, st));
        known = true;
        hits = hits && !info[1] && !known_dense(c, s, info + 3);
        if (hits && !most_pairs(s, info, m, nI, pass)) {
            const SetSize z = equal_parts(info[0], m);
            hits = (m < kPlanFirst || !in_runs(info, m)) && tables_us(c, s, nI, z, pass) < others_us(c, s, z, pass);
        }
    }
    auto tables = [&](bool *done) {
        c->hits_busy = true;
        const int rc = count_hits(c, s, cands, gather, m, d_ivl, nI, pass, out, st, done, nullptr,
                                  known ? nullptr : info);
        return or_no_room(c, rc, done, st);
    };
    if (hits && known && tune_used(c)) {
        const int N = __builtin_popcount(info[0]) == 1 ? __builtin_ctz(info[0]) : 0;
        RET(tuned_route(c, tune_key(N, pass, kTuneSet, m, s.n_chunks, s.K), st, &hits,
                        [&] { return count_validated(c, s, cands, gather, m, d_ivl, nI, pass, out, info, st); },
                        tables));
    }
    if (hits) {
        bool done = false;
        if (!known) info[0] = 0;
        RET(tables(&done));
        if (done) return FEM_OK;
        known = known || info[0];  // (no plan was made where there was no room for it)
    }
    if (!known) RET(validate(c, s, cands, gather, m, nI, info, st));
    return count_validated(c, s, cands, gather, m, d_ivl, nI, pass, out, info, st);
}

// The same by the other counting kernels, one length after the other.
int count_grouped(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
                  uint32_t m, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
                  cudaStream_t st) {
    if (m == 0) return FEM_OK;
    uint32_t info[kInfoWords];
    RET(validate(c, s, cands, gather, m, nI, info, st));
    return count_validated(c, s, cands, gather, m, d_ivl, nI, pass, out, info, st);
}

int count_validated(fem_ctx *c, const StreamDev &s, const fem_episode *cands, const uint32_t *gather,
                    uint32_t m, const uint2 *d_ivl, uint32_t nI, int pass, uint32_t *out,
                    const uint32_t *info, cudaStream_t st) {
    const uint32_t lens = info[0];
    struct Clustered {
        fem_ctx *c;
        bool saved;
        ~Clustered() { c->clustered = saved; }
    } restore{c, c->clustered};
    c->clustered = in_runs(info, m);
    if (info[1] && info[1] < m) {
        // distinct-type and repeated-type episodes mixed: count each part on its own
        // (repeated types run with one segment), then put the counts back in place
        uint8_t *rf;
        uint32_t *ridx, *rg, *rout, *scratch;
        RET(dbuf(c, "rep_flags", m, &rf));
        RET(dbuf(c, "rep_idx", m, &ridx));
        RET(dbuf(c, "rep_gather", m, &rg));
        RET(dbuf(c, "rep_out", m, &rout));
        RET(dbuf(c, "rep_scratch", compact_scratch_words(m), &scratch));
        for (bool rep : {false, true}) {
            CK(launch_repeat_flags(cands, gather, m, !rep, rf, st));
            CK(launch_compact(nullptr, rf, 0, m, ridx, c->d_small + W_COUNT2, scratch, st));
            uint32_t k;
            RET(read_words(c, c->d_small + W_COUNT2, 1, &k, st));
            if (!k) continue;
            CK(launch_compose_idx(gather, ridx, k, rg, st));
            RET(count_any(c, s, cands, rg, k, d_ivl, nI, pass, rout, st));
            CK(launch_scatter_u32(rout, ridx, k, out, st));
        }
        return FEM_OK;
    }
    const bool distinct = info[1] == 0;
    if (__builtin_popcount(lens) == 1) {
        const int N = __builtin_ctz(lens);
        return count_pass(c, s, cands, gather, m, N, d_ivl, nI, pass, out, distinct, st, nullptr);
    }
    uint8_t *flags;
    uint32_t *idx, *g2, *tmp, *scratch;
    RET(dbuf(c, "len_flags", m, &flags));
    RET(dbuf(c, "len_idx", m, &idx));
    RET(dbuf(c, "len_gather", m, &g2));
    RET(dbuf(c, "len_out", m, &tmp));
    RET(dbuf(c, "len_scratch", compact_scratch_words(m), &scratch));
    for (int N = 1; N <= FEM_MAX_LEN; ++N) {
        if (!(lens & (1u << N))) continue;
        CK(launch_len_flags(cands, gather, m, (uint32_t)N, flags, st));
        CK(launch_compact(nullptr, flags, 0, m, idx, c->d_small + W_COUNT1, scratch, st));
        uint32_t k;
        RET(read_words(c, c->d_small + W_COUNT1, 1, &k, st));
        if (!k) continue;
        CK(launch_compose_idx(gather, idx, k, g2, st));
        RET(count_pass(c, s, cands, g2, k, N, d_ivl, nI, pass, tmp, distinct, st, nullptr));
        CK(launch_scatter_u32(tmp, idx, k, out, st));
    }
    return FEM_OK;
}

void free_stream_buffers(StreamDev &s) {
    cudaFree(s.t);
    cudaFree(s.type);
    cudaFree(s.bev);
    cudaFree(s.boff);
    cudaFree(s.cfirst);
    cudaFree(s.hist);
    s = StreamDev{};
}

// Buffers for a stream of up to ne events in nc chunks (offs per chunk), charged to
// the context's budget as one block.  Where this fails, s holds no buffers and is
// otherwise as it was.
int alloc_stream(fem_ctx *c, StreamDev &s, size_t ne, size_t nc) {
    StreamDev q;
    q.cap_events = ne, q.cap_chunks = nc, q.cap_offs = (uint32_t)(nc * s.offs);
    q.t = reinterpret_cast<uint32_t *>(1);  // stream_bytes of the capacities
    const size_t bytes = stream_bytes(q);
    RET(reserve(c, bytes));
    auto take = [&] {
        q.t = nullptr;
        if (cudaMalloc(&q.t, ne * 4) == cudaSuccess && cudaMalloc(&q.type, ne) == cudaSuccess &&
            cudaMalloc(&q.bev, nc * CHUNK * 8) == cudaSuccess &&
            cudaMalloc(&q.boff, nc * s.offs * 2) == cudaSuccess &&
            cudaMalloc(&q.cfirst, (nc + 1) * 4) == cudaSuccess &&
            cudaMalloc(&q.hist, 256 * 4) == cudaSuccess)
            return true;
        cudaGetLastError();
        free_stream_buffers(q);
        return false;
    };
    // (the device is full: once more without the hit tables of earlier calls)
    if (!take() && (c->hits_busy || !release_hits(c) || !take())) return FEM_ENOMEM;
    s.t = q.t, s.type = q.type, s.bev = q.bev, s.boff = q.boff, s.cfirst = q.cfirst, s.hist = q.hist;
    s.cap_events = ne, s.cap_chunks = nc, s.cap_offs = (uint32_t)(nc * s.offs);
    c->mem_used += bytes;
    return FEM_OK;
}

}  // namespace

// ============================================================================ C ABI
extern "C" {

}  // extern "C"

namespace fem {
int fem_ctx_device(const fem_ctx *c) { return c->device; }
int fem_ctx_sms(const fem_ctx *c) { return c->sm_count; }
bool fem_ctx_release_hits(fem_ctx *c) { return release_hits(c); }
}  // namespace fem

extern "C" {

uint64_t fem_kernel_launches(void) { return g_launches.load(std::memory_order_relaxed); }

const char *fem_strerror(int s) {
    switch (s) {
        case FEM_OK: return "ok";
        case FEM_EINVAL: return "invalid argument";
        case FEM_EUNSORTED: return "stream times are not non-decreasing";
        case FEM_ETYPE: return "event type out of range";
        case FEM_ERANGE: return "time span plus interval bound exceeds 32 bits";
        case FEM_ENOMEM: return "out of memory";
        case FEM_EADMIT: return "request not admitted";
        case FEM_ETIMEOUT: return "bounded device wait timed out";
        case FEM_ECUDA: return "CUDA runtime error";
        case FEM_EOVERFLOW: return "internal capacity exceeded";
        case FEM_ENOSTREAM: return "unknown stream id";
        case FEM_EIO: return "file could not be opened, read or written";
        default: return "unknown status";
    }
}

int fem_create(fem_ctx **out, int device, size_t mem_budget_bytes) {
    if (!out) return FEM_EINVAL;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return FEM_ECUDA;
    }
    fem_ctx *c = new (std::nothrow) fem_ctx;
    if (!c) return FEM_ENOMEM;
    c->device = device;
    c->mem_budget = mem_budget_bytes;
    if (cudaSetDevice(device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device) !=
            cudaSuccess ||
        cudaStreamCreateWithFlags(&c->own, cudaStreamNonBlocking) != cudaSuccess ||
        cudaMalloc(&c->d_err, sizeof(uint32_t)) != cudaSuccess ||
        cudaMalloc(&c->d_dense, 256 * sizeof(uint32_t)) != cudaSuccess ||
        cudaMalloc(&c->d_small, 64 * sizeof(uint32_t)) != cudaSuccess ||
        cudaMallocHost(&c->h_small, kSmallWords * sizeof(uint32_t)) != cudaSuccess ||
        cudaMallocHost(&c->h_load, (kLoadSeq + 1) * sizeof(uint32_t)) != cudaSuccess ||
        cudaMallocHost(&c->h_ivl, (FEM_MAX_INTERVALS + 1) * sizeof(fem_interval)) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->ivl_ev, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreate(&c->tev[0]) != cudaSuccess ||
        cudaEventCreate(&c->tev[1]) != cudaSuccess) {
        cudaGetLastError();
        fem_destroy(c);
        return FEM_ECUDA;
    }
    for (auto &set : c->kev) {
        for (auto &e : set) {
            if (cudaEventCreate(&e) != cudaSuccess) {
                cudaGetLastError();
                fem_destroy(c);
                return FEM_ECUDA;
            }
        }
    }
    for (auto &e : c->ev) {
        if (cudaEventCreate(&e) != cudaSuccess) {
            cudaGetLastError();
            fem_destroy(c);
            return FEM_ECUDA;
        }
    }
    size_t mem_free = 0;
    if (cudaMemGetInfo(&mem_free, &c->mem_device) != cudaSuccess) {
        cudaGetLastError();
        fem_destroy(c);
        return FEM_ECUDA;
    }
    cudaMemset(c->d_err, 0, sizeof(uint32_t));
    cudaMemset(c->d_dense, 0xFF, 256 * sizeof(uint32_t));
    std::memset(c->h_small, 0, kSmallWords * sizeof(uint32_t));  // no stale sequence number
    std::memset(c->h_load, 0, (kLoadSeq + 1) * sizeof(uint32_t));
    {
        void *dp = nullptr, *dl = nullptr;
        if (cudaHostGetDevicePointer(&dp, c->h_small, 0) == cudaSuccess && dp &&
            cudaHostGetDevicePointer(&dl, c->h_load, 0) == cudaSuccess && dl) {
            c->d_pub = static_cast<uint32_t *>(dp) + kPubWord;
            c->d_plan = static_cast<uint32_t *>(dp) + kPlanWord;
            c->d_load = static_cast<uint32_t *>(dl);
        }
        cudaGetLastError();
    }
    *out = c;
    return FEM_OK;
}

int fem_destroy(fem_ctx *c) {
    if (!c) return FEM_EINVAL;
    cudaSetDevice(c->device);
    if (c->own) cudaStreamSynchronize(c->own);
    for (auto &kv : c->streams) free_stream_buffers(kv.second);
    for (auto &kv : c->bufs) cudaFree(kv.second.p);
    if (c->d_err) cudaFree(c->d_err);
    if (c->d_dense) cudaFree(c->d_dense);
    if (c->d_small) cudaFree(c->d_small);
    if (c->h_small) cudaFreeHost(c->h_small);
    if (c->h_load) cudaFreeHost(c->h_load);
    if (c->h_ivl) cudaFreeHost(c->h_ivl);
    if (c->ivl_ev) cudaEventDestroy(c->ivl_ev);
    for (auto &e : c->ev)
        if (e) cudaEventDestroy(e);
    for (auto &set : c->kev)
        for (auto &e : set)
            if (e) cudaEventDestroy(e);
    for (auto &e : c->tev)
        if (e) cudaEventDestroy(e);
    for (StreamDev &s : c->pool) free_stream_buffers(s);
    for (auto &b : c->pin)
        if (b.p) cudaFreeHost(b.p);
    if (c->own) cudaStreamDestroy(c->own);
    delete c;
    return FEM_OK;
}

int fem_set_config(fem_ctx *c, const fem_config *cfg) {
    if (!c) return FEM_EINVAL;
    if (!cfg) {
        c->cfg = fem_config{};
        return FEM_OK;
    }
    if (cfg->threads_per_block &&
        (cfg->threads_per_block % 32 || cfg->threads_per_block > 256))
        return FEM_EINVAL;
    if (cfg->ring_capacity && !count_config_supported(2, FEM_PASS_EXACT, false, cfg->ring_capacity))
        return FEM_EINVAL;
    if (cfg->kernel > FEM_KERNEL_CHAIN) return FEM_EINVAL;
    c->cfg = *cfg;
    return FEM_OK;
}

int fem_tune_enable(fem_ctx *c, int on) {
    if (!c) return FEM_EINVAL;
    c->tune_on = on != 0;
    return FEM_OK;
}

int fem_tune_size(fem_ctx *c, uint32_t *n_out) {
    if (!c || !n_out) return FEM_EINVAL;
    *n_out = (uint32_t)c->tune.size();
    return FEM_OK;
}

// One JSON object per line: {"key": "N/pass/distinct/log2m/log2chunks/K", "segments": P,
// "threads": T, "ms": t}
int fem_tune_save(fem_ctx *c, const char *path) {
    if (!c || !path) return FEM_EINVAL;
    FILE *f = std::fopen(path, "w");
    if (!f) return FEM_EIO;
    for (const auto &kv : c->tune)
        std::fprintf(f,
                     "{\"key\": \"%s\", \"segments\": %u, \"threads\": %u, \"ms\": %.6f, "
                     "\"kernel\": %u}\n",
                     kv.first.c_str(), kv.second.P, kv.second.T, kv.second.ms, kv.second.kernel);
    const bool ok = std::fclose(f) == 0;
    return ok ? FEM_OK : FEM_EIO;
}

int fem_tune_load(fem_ctx *c, const char *path) {
    if (!c || !path) return FEM_EINVAL;
    FILE *f = std::fopen(path, "r");
    if (!f) return FEM_EIO;
    std::map<std::string, fem_ctx::Shape> got;
    char line[512];
    int rc = FEM_OK;
    while (std::fgets(line, sizeof(line), f)) {
        if (line[0] == '\n' || line[0] == 0) continue;
        char key[96];
        unsigned P = 0, T = 0, K = FEM_KERNEL_MACHINE;
        float ms = 0;
        char close = 0;
        const int nf = std::sscanf(
            line, " {\"key\": \"%95[0-9/]\", \"segments\": %u, \"threads\": %u, \"ms\": %f%c",
            key, &P, &T, &ms, &close);
        bool good = nf == 5 && P != 0 && T != 0 && T <= 256 && T % 8 == 0;
        if (good && close == ',') {  // with the kernel field
            good = std::sscanf(std::strstr(line, "\"ms\""), "\"ms\": %*f, \"kernel\": %u}", &K) == 1 &&
                   (K == FEM_KERNEL_MACHINE || K == FEM_KERNEL_CHAIN || K == FEM_KERNEL_HITS);
            int kind = 0;  // (tables are a choice, not a shape)
            if (K == FEM_KERNEL_HITS) good = good && std::sscanf(key, "%*d/%*d/%d", &kind) == 1 && kind >= kTuneSet;
        } else if (good) {
            good = close == '}';
        }
        if (!good) {
            rc = FEM_EINVAL;
            break;
        }
        got[key] = fem_ctx::Shape{P, T, ms, K};
    }
    std::fclose(f);
    if (rc != FEM_OK) return rc;
    for (auto &kv : got) c->tune[kv.first] = kv.second;
    return FEM_OK;
}

int fem_load_stream(fem_ctx *c, const uint8_t *types, const uint32_t *t_us, uint64_t n,
                    uint32_t n_types, int on_device, void *cuda_stream, int32_t *id_out) {
    if (!c || !id_out || n_types == 0 || n_types > FEM_MAX_TYPES) return FEM_EINVAL;
    if (n && (!types || !t_us)) return FEM_EINVAL;
    if (n >= 0xFFFFFFF0ull) return FEM_EINVAL;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    StreamDev s;
    s.n = n;
    s.K = n_types;
    s.n_chunks = (uint32_t)((n + CHUNK - 1) / CHUNK);
    s.offs = offs_stride(n_types);
    const size_t nn = std::max<uint64_t>(n, 1);
    const size_t nc = std::max<uint32_t>(s.n_chunks, 1);
    bool okm = false;
    for (size_t i = 0; i < c->pool.size(); ++i) {
        StreamDev &q = c->pool[i];
        if (q.cap_events >= nn && q.cap_chunks >= nc && q.cap_offs >= nc * s.offs) {
            s.t = q.t, s.type = q.type, s.bev = q.bev, s.boff = q.boff, s.cfirst = q.cfirst,
            s.hist = q.hist;
            s.cap_events = q.cap_events, s.cap_chunks = q.cap_chunks, s.cap_offs = q.cap_offs;
            c->pool.erase(c->pool.begin() + i);
            okm = true;
            break;
        }
    }
    if (!okm) okm = alloc_stream(c, s, nn, nc) == FEM_OK;
    auto release = [&] {
        c->mem_used -= std::min(stream_bytes(s), c->mem_used);
        free_stream_buffers(s);
    };
    if (!okm) return FEM_ENOMEM;
    int rc = FEM_OK;
    std::vector<uint32_t> hist_host;
    do {
        // the histogram is cleared here (k_bucket accumulates into it); the chunk start
        // times are all written by k_bucket, and need filling only for an empty stream
        if (cudaMemsetAsync(c->d_err, 0, 4, st) != cudaSuccess ||
            cudaMemsetAsync(s.hist, 0, 256 * 4, st) != cudaSuccess ||
            (!n && cudaMemsetAsync(s.cfirst, 0xFF, (nc + 1) * 4, st) != cudaSuccess)) {
            rc = FEM_ECUDA;
            break;
        }
        if (n && on_device) {  // one kernel reads, checks, copies and groups the events
            if (launch_load_stream(s, st, c->d_err, t_us, types) != cudaSuccess) {
                rc = FEM_ECUDA;
                break;
            }
        } else if (n) {
            if (cudaMemcpyAsync(s.t, t_us, n * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaMemcpyAsync(s.type, types, n, cudaMemcpyHostToDevice, st) != cudaSuccess ||
                launch_load_stream(s, st, c->d_err) != cudaSuccess) {
                rc = FEM_ECUDA;
                break;
            }
        }
        // error word, last time and type histogram in one round trip: published by a
        // kernel into mapped words, else copied
        if (c->d_load) {
            const uint32_t seq = ++c->pub_seq;
            if (launch_publish_load(c->d_err, n ? s.t + (n - 1) : nullptr, s.hist, n_types,
                                    c->d_load, kLoadSeq, seq, s.t, st) != cudaSuccess) {
                rc = FEM_ECUDA;
                break;
            }
            if ((rc = wait_seq(c->h_load + kLoadSeq, seq, st)) != FEM_OK) break;
            const volatile uint32_t *hv = c->h_load;
            if ((rc = err_status(hv[0])) != FEM_OK) break;
            if (n) s.t_max = hv[1], s.t_min = hv[kLoadSeq - 1];
            hist_host.assign(n_types, 0);
            for (uint32_t a = 0; a < n_types; ++a) hist_host[a] = hv[2 + a];
            break;
        }
        void *hp;
        if ((rc = pinbuf(c, 0, (3 + 256) * sizeof(uint32_t), st, &hp)) != FEM_OK) break;
        uint32_t *hw = static_cast<uint32_t *>(hp);
        if (cudaMemcpyAsync(hw, c->d_err, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            (n && cudaMemcpyAsync(hw + 1, s.t + (n - 1), 4, cudaMemcpyDeviceToHost, st) !=
                      cudaSuccess) ||
            (n && cudaMemcpyAsync(hw + 258, s.t, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) ||
            cudaMemcpyAsync(hw + 2, s.hist, n_types * 4, cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = FEM_ECUDA;
            break;
        }
        if ((rc = err_status(hw[0])) != FEM_OK) break;
        if (n) s.t_max = hw[1], s.t_min = hw[258];
        hist_host.assign(hw + 2, hw + 2 + n_types);
    } while (0);
    if (rc != FEM_OK) {
        cudaGetLastError();
        cudaStreamSynchronize(st);
        release();
        return rc;
    }
    const int32_t id = c->next_id++;
    s.gen = c->next_gen++;
    c->streams[id] = s;
    c->hist_h[id] = std::move(hist_host);
    *id_out = id;
    return FEM_OK;
}

int fem_append_stream(fem_ctx *c, int32_t id, const uint8_t *types, const uint32_t *t_us,
                      uint64_t n, int on_device, void *cuda_stream) {
    if (!c || (n && (!types || !t_us))) return FEM_EINVAL;
    auto it = c->streams.find(id);
    if (it == c->streams.end()) return FEM_ENOSTREAM;
    if (n == 0) return FEM_OK;
    StreamDev &s = it->second;
    const uint64_t n_old = s.n, n_new = s.n + n;
    if (n_new >= 0xFFFFFFF0ull) return FEM_EINVAL;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    const uint32_t ch_old = s.n_chunks, K = s.K, t_min = s.t_min, t_max_old = s.t_max;
    const uint32_t ch_new = (uint32_t)((n_new + CHUNK - 1) / CHUNK);
    if (n_new > s.cap_events || ch_new > s.cap_chunks || (uint64_t)ch_new * s.offs > s.cap_offs) {
        // grow by half at least, keeping what is grouped already
        StreamDev g;
        g.offs = s.offs;
        RET(alloc_stream(c, g, std::max<uint64_t>(n_new, s.cap_events * 3 / 2),
                         std::max<uint64_t>(ch_new, s.cap_chunks * 3 / 2)));
        bool ok = true;
        if (n_old) {
            ok = cudaMemcpyAsync(g.t, s.t, n_old * 4, cudaMemcpyDeviceToDevice, st) == cudaSuccess &&
                 cudaMemcpyAsync(g.type, s.type, n_old, cudaMemcpyDeviceToDevice, st) == cudaSuccess &&
                 cudaMemcpyAsync(g.bev, s.bev, (size_t)ch_old * CHUNK * 8, cudaMemcpyDeviceToDevice,
                                 st) == cudaSuccess &&
                 cudaMemcpyAsync(g.boff, s.boff, (size_t)ch_old * s.offs * 2,
                                 cudaMemcpyDeviceToDevice, st) == cudaSuccess &&
                 cudaMemcpyAsync(g.cfirst, s.cfirst, ((size_t)ch_old + 1) * 4,
                                 cudaMemcpyDeviceToDevice, st) == cudaSuccess;
        }
        ok = ok && cudaMemcpyAsync(g.hist, s.hist, 256 * 4, cudaMemcpyDeviceToDevice, st) ==
                       cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            c->mem_used -= std::min(stream_bytes(g), c->mem_used);
            free_stream_buffers(g);
            return FEM_ECUDA;
        }
        c->mem_used -= std::min(stream_bytes(s), c->mem_used);
        g.dense_hi = std::move(s.dense_hi), g.least_span = s.least_span;
        free_stream_buffers(s);
        g.n = n_old, g.K = K, g.n_chunks = ch_old, g.t_min = t_min, g.t_max = t_max_old;
        s = g;
    }
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    CK(cudaMemcpyAsync(s.t + n_old, t_us, n * 4, kind, st));
    CK(cudaMemcpyAsync(s.type + n_old, types, n, kind, st));
    s.n = n_new;
    s.n_chunks = ch_new;
    // regroup from the chunk holding the old last event, so that the pair across the old
    // end is checked with the new events
    const uint32_t c0 = n_old ? (uint32_t)((n_old - 1) / CHUNK) : 0u;
    CK(launch_bucket_chunks(s, c0, ch_new, st, c->d_err));
    CK(launch_hist_add(s.type + n_old, n, s.K, +1, s.hist, st));
    void *hp;
    RET(pinbuf(c, 0, (3 + 256) * sizeof(uint32_t), st, &hp));
    uint32_t *hw = static_cast<uint32_t *>(hp);
    CK(cudaMemcpyAsync(hw, c->d_err, 4, cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(hw + 1, s.t + (n_new - 1), 4, cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(hw + 2, s.hist, s.K * 4, cudaMemcpyDeviceToHost, st));
    if (!n_old) CK(cudaMemcpyAsync(hw + 258, s.t, 4, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const int rc = err_status(hw[0]);
    if (rc != FEM_OK) {
        // undo: the old events' grouping, histogram and size
        CK(launch_hist_add(s.type + n_old, n, s.K, -1, s.hist, st));
        s.n = n_old;
        s.n_chunks = ch_old;
        if (n_old) CK(launch_bucket_chunks(s, c0, ch_old, st));
        else CK(cudaMemsetAsync(s.cfirst, 0xFF, 8, st));
        CK(cudaStreamSynchronize(st));
        s.t_max = t_max_old;
        return rc;
    }
    s.t_max = hw[1];
    if (!n_old) s.t_min = hw[258];
    s.gen = c->next_gen++;
    c->hist_h[id].assign(hw + 2, hw + 2 + s.K);
    return FEM_OK;
}

int fem_mem_usage(fem_ctx *c, size_t *used_out, size_t *budget_out) {
    if (!c) return FEM_EINVAL;
    if (used_out) *used_out = c->mem_used;
    if (budget_out) *budget_out = c->mem_budget;
    return FEM_OK;
}

int fem_free_stream(fem_ctx *c, int32_t id) {
    if (!c) return FEM_EINVAL;
    auto it = c->streams.find(id);
    if (it == c->streams.end()) return FEM_ENOSTREAM;
    cudaSetDevice(c->device);
    // Keep the buffers for the next load (work already queued that reads them runs
    // first: every stream of this context is synchronised before reuse).
    cudaDeviceSynchronize();
    c->pool.push_back(it->second);
    c->streams.erase(it);
    c->hist_h.erase(id);
    while (c->pool.size() > 4) {
        c->mem_used -= std::min(stream_bytes(c->pool.front()), c->mem_used);
        free_stream_buffers(c->pool.front());
        c->pool.erase(c->pool.begin());
    }
    return FEM_OK;
}

int fem_type_counts(fem_ctx *c, int32_t id, uint32_t *counts_out) {
    if (!c || !counts_out) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    cudaSetDevice(c->device);
    CK(cudaMemcpyAsync(counts_out, s->hist, s->K * 4, cudaMemcpyDeviceToHost, c->own));
    CK(cudaStreamSynchronize(c->own));
    return FEM_OK;
}

int fem_capacity_table(fem_ctx *c, int32_t id, const uint32_t *widths, uint32_t nh,
                       uint32_t *cap_out) {
    if (!c || !widths || !cap_out || nh == 0 || nh > FEM_MAX_CAP_WIDTHS) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    cudaSetDevice(c->device);
    return capacity(c, *s, widths, nh, cap_out, c->own);
}

int fem_count_pairs_relaxed(fem_ctx *c, int32_t id, const uint8_t *types, uint32_t f,
                            const fem_interval *I, uint32_t nI, uint32_t *counts_out) {
    if (!c || !types || !counts_out || f < 2 || f > 256 || nI == 0 || nI > 4) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    RET(check_intervals(*s, I, nI));
    bool seen[256] = {};
    for (uint32_t i = 0; i < f; ++i) {
        if (types[i] >= s->K || seen[types[i]]) return FEM_EINVAL;
        seen[types[i]] = true;
    }
    cudaSetDevice(c->device);
    cudaStream_t st = c->own;
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    uint2 *d_ivl;
    RET(upload_intervals(c, I, nI, st, &d_ivl));
    const uint32_t m = f * (f - 1) * nI;
    uint32_t *ft, *out;
    fem_episode *cands;
    RET(dbuf(c, "pair_types", f, &ft));
    RET(dbuf(c, "pair_cands", m, &cands));
    RET(dbuf(c, "pair_out", m, &out));
    std::vector<uint32_t> ftv(types, types + f);
    CK(cudaMemcpyAsync(ft, ftv.data(), f * 4, cudaMemcpyHostToDevice, st));
    CK(launch_level2(ft, f, nI, false, cands, st));
    PassLaunch pl;
    RET(count_launch_pairs(c, *s, cands, m, f, d_ivl, nI, out, st, &pl));
    uint32_t e;
    RET(read_err(c, st, &e));
    RET(count_finish(c, *s, pl, e, st));
    CK(cudaMemcpyAsync(counts_out, out, (size_t)m * 4, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    return FEM_OK;
}

int fem_count_candidates(fem_ctx *c, int32_t id, const fem_episode *cands, uint32_t m,
                         int cands_on_device, const fem_interval *I, uint32_t nI, int pass,
                         uint32_t *counts_out, int counts_on_device, void *cuda_stream) {
    if (!c || (m && (!cands || !counts_out))) return FEM_EINVAL;
    if (pass != FEM_PASS_RELAXED && pass != FEM_PASS_EXACT) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    RET(check_intervals(*s, I, nI));
    if (m == 0) return FEM_OK;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    uint2 *d_ivl;
    RET(upload_intervals(c, I, nI, st, &d_ivl));
    const fem_episode *dc = cands;
    if (!cands_on_device) {
        fem_episode *tmp;
        RET(dbuf(c, "cands_in", m, &tmp));
        CK(cudaMemcpyAsync(tmp, cands, (size_t)m * sizeof(fem_episode), cudaMemcpyHostToDevice, st));
        dc = tmp;
    }
    uint32_t *dout = counts_out;
    if (!counts_on_device) RET(dbuf(c, "counts_out", m, &dout));
    RET(count_any(c, *s, dc, nullptr, m, d_ivl, nI, pass, dout, st));
    if (!counts_on_device) {
        CK(cudaMemcpyAsync(counts_out, dout, (size_t)m * 4, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    return FEM_OK;
}

int fem_count_mapconcat_literal(fem_ctx *c, int32_t id, const fem_episode *cands, uint32_t m,
                                int cands_on_device, const fem_interval *I, uint32_t nI,
                                uint32_t segments, uint32_t *counts_out, int counts_on_device,
                                uint32_t *diag_out, void *cuda_stream) {
    if (!c || (m && (!cands || !counts_out))) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    RET(check_intervals(*s, I, nI));
    if (diag_out) diag_out[0] = diag_out[1] = 0;
    if (m == 0) return FEM_OK;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    uint2 *d_ivl;
    RET(upload_intervals(c, I, nI, st, &d_ivl));
    const fem_episode *dc = cands;
    if (!cands_on_device) {
        fem_episode *tmp;
        RET(dbuf(c, "cands_in", m, &tmp));
        CK(cudaMemcpyAsync(tmp, cands, (size_t)m * sizeof(fem_episode), cudaMemcpyHostToDevice, st));
        dc = tmp;
    }
    uint32_t *dout = counts_out;
    if (!counts_on_device) RET(dbuf(c, "counts_out", m, &dout));
    // the printed scheme needs distinct types (as the exact MapConcatenate does)
    CK(cudaMemsetAsync(c->d_small + W_INFO, 0, 3 * sizeof(uint32_t), st));
    CK(launch_validate_cands(dc, nullptr, m, s->K, nI, c->d_small + W_INFO, c->d_err, st));
    uint32_t info[3], e;
    RET(read_words(c, c->d_small + W_INFO, 3, info, st));
    RET(read_err(c, st, &e));
    RET(err_status(e));
    if (info[1]) return FEM_EINVAL;
    if (s->n == 0) {
        CK(cudaMemsetAsync(dout, 0, (size_t)m * 4, st));
    } else {
        // time cuts at the first event of every cps-th chunk (dropped where equal
        // times would make them non-increasing)
        std::vector<uint32_t> cf(s->n_chunks + 1);
        CK(cudaMemcpyAsync(cf.data(), s->cfirst, cf.size() * 4, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        const uint32_t P0 = std::max<uint32_t>(1, std::min<uint32_t>(segments ? segments : 1,
                                                                     s->n_chunks));
        const uint32_t cps = (s->n_chunks + P0 - 1) / P0;
        std::vector<int64_t> tau{(int64_t)cf[0] - 1};
        for (uint32_t c0 = cps; c0 < s->n_chunks; c0 += cps)
            if ((int64_t)cf[c0] - 1 > tau.back() && (int64_t)cf[c0] - 1 < (int64_t)s->t_max)
                tau.push_back((int64_t)cf[c0] - 1);
        tau.push_back((int64_t)s->t_max);
        const uint32_t P = (uint32_t)tau.size() - 1;
        int64_t *d_tau;
        uint4 *tuples;
        RET(dbuf(c, "lit_tau", tau.size(), &d_tau));
        RET(dbuf(c, "lit_tuples", (size_t)m * P * FEM_MAX_LEN, &tuples));
        CK(cudaMemcpyAsync(d_tau, tau.data(), tau.size() * sizeof(int64_t), cudaMemcpyHostToDevice,
                           st));
        CK(cudaMemsetAsync(c->d_small + W_INFO, 0, 2 * sizeof(uint32_t), st));
        LiteralParams p{};
        p.bev = s->bev;
        p.boff = s->boff;
        p.t = s->t;
        p.offs = s->offs;
        p.n = s->n;
        p.cands = dc;
        p.m = m;
        p.ivl = d_ivl;
        p.tau = d_tau;
        p.P = P;
        p.tuples = tuples;
        p.err = c->d_err;
        CK(launch_literal(p, info[0], dout, c->d_small + W_INFO, st));
        uint32_t dg[2];
        RET(read_words(c, c->d_small + W_INFO, 2, dg, st));
        RET(read_err(c, st, &e));
        if (e & ERR_RING) return FEM_EOVERFLOW;
        RET(err_status(e));
        if (diag_out) diag_out[0] = dg[0], diag_out[1] = dg[1];
    }
    if (!counts_on_device) {
        CK(cudaMemcpyAsync(counts_out, dout, (size_t)m * 4, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    return FEM_OK;
}

int fem_count_windows(fem_ctx *c, int32_t id, const fem_episode *cands, uint32_t m,
                      int cands_on_device, const fem_interval *I, uint32_t nI, uint32_t window_us,
                      uint64_t *counts_out, int counts_on_device, void *cuda_stream) {
    if (!c || (m && (!cands || !counts_out)) || window_us == 0) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    RET(check_intervals(*s, I, nI));
    if (m == 0) return FEM_OK;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    uint2 *d_ivl;
    RET(upload_intervals(c, I, nI, st, &d_ivl));
    const fem_episode *dc = cands;
    if (!cands_on_device) {
        fem_episode *tmp;
        RET(dbuf(c, "cands_in", m, &tmp));
        CK(cudaMemcpyAsync(tmp, cands, (size_t)m * sizeof(fem_episode), cudaMemcpyHostToDevice, st));
        dc = tmp;
    }
    uint64_t *dout = counts_out;
    if (!counts_on_device) RET(dbuf(c, "win_out", m, &dout));
    uint32_t info[kInfoWords], e;
    RET(validate(c, *s, dc, nullptr, m, nI, info, st));
    if (info[1]) return FEM_EINVAL;  // distinct types only
    bool done = false;
    auto tables = [&]() -> int {
        c->hits_busy = true;
        const int rc = windows_hits(c, *s, dc, m, d_ivl, nI, window_us, dout, st, &done);
        return or_no_room(c, rc, &done, st);
    };
    const bool eligible = hits_eligible(c, *s, nI) && !known_dense(c, *s, info + 3);
    const bool first = eligible && windows_over_tables(*s, nI, info[0], m);
    if (first) RET(tables());
    if (!done) {
        WindowParams p{};
        p.bev = s->bev;
        p.boff = s->boff;
        p.offs = s->offs;
        p.n = s->n;
        p.cands = dc;
        p.m = m;
        p.ivl = d_ivl;
        p.w = window_us;
        p.out = dout;
        p.err = c->d_err;
        CK(launch_count_windows(p, info[0], st));
        RET(read_err(c, st, &e));
        if (e & ERR_RING) {  // (its lists ran over: the tables, where they were not tried)
            if (!eligible || first) return FEM_EOVERFLOW;
            CK(cudaMemsetAsync(c->d_err, 0, 4, st));
            RET(tables());
            if (!done) return FEM_EOVERFLOW;
        } else {
            RET(err_status(e));
        }
    }
    if (!counts_on_device) {
        CK(cudaMemcpyAsync(counts_out, dout, (size_t)m * 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    return FEM_OK;
}

int fem_count_two_pass(fem_ctx *c, int32_t id, const fem_episode *cands, uint32_t m,
                       int cands_on_device, const fem_interval *I, uint32_t nI, uint32_t theta,
                       uint32_t *exact_out, uint8_t *survived_out, int outs_on_device,
                       void *cuda_stream) {
    if (!c || (m && !cands)) return FEM_EINVAL;
    const StreamDev *s = find_stream(c, id);
    if (!s) return FEM_ENOSTREAM;
    RET(check_intervals(*s, I, nI));
    if (m == 0) return FEM_OK;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    uint2 *d_ivl;
    RET(upload_intervals(c, I, nI, st, &d_ivl));
    const fem_episode *dc = cands;
    if (!cands_on_device) {
        fem_episode *tmp;
        RET(dbuf(c, "cands_in", m, &tmp));
        CK(cudaMemcpyAsync(tmp, cands, (size_t)m * sizeof(fem_episode), cudaMemcpyHostToDevice, st));
        dc = tmp;
    }
    uint32_t *rel, *idx, *ex, *exo, *scratch;
    uint8_t *sv;
    RET(dbuf(c, "tp_rel", m, &rel));
    RET(dbuf(c, "tp_idx", m, &idx));
    RET(dbuf(c, "tp_ex", m, &ex));
    RET(dbuf(c, "scratch", compact_scratch_words(m), &scratch));
    exo = (outs_on_device && exact_out) ? exact_out : nullptr;
    if (!exo) RET(dbuf(c, "tp_exo", m, &exo));
    sv = (outs_on_device && survived_out) ? survived_out : nullptr;
    if (!sv) RET(dbuf(c, "tp_sv", m, &sv));
    // first pass: relaxed counts, eliminate count < theta
    RET(count_any(c, *s, dc, nullptr, m, d_ivl, nI, FEM_PASS_RELAXED, rel, st));
    CK(launch_compact(rel, nullptr, theta, m, idx, c->d_small + W_COUNT0, scratch, st, pub_of(c)));
    uint32_t ms, e0;
    RET(read_count_err(c, c->d_small + W_COUNT0, &ms, &e0, st));
    RET(err_status(e0));
    // second pass: exact counts of the survivors
    RET(count_any(c, *s, dc, idx, ms, d_ivl, nI, FEM_PASS_EXACT, ex, st));
    CK(cudaMemsetAsync(exo, 0, (size_t)m * 4, st));
    CK(cudaMemsetAsync(sv, 0, m, st));
    CK(launch_scatter_u32(ex, idx, ms, exo, st));
    CK(launch_fill_flags(idx, ms, sv, st));
    if (!outs_on_device) {
        if (exact_out) CK(cudaMemcpyAsync(exact_out, exo, (size_t)m * 4, cudaMemcpyDeviceToHost, st));
        if (survived_out) CK(cudaMemcpyAsync(survived_out, sv, m, cudaMemcpyDeviceToHost, st));
    }
    CK(cudaStreamSynchronize(st));
    return FEM_OK;
}

int fem_mine_levelwise(fem_ctx *c, int32_t id, const fem_interval *I, uint32_t nI,
                       uint32_t theta, uint32_t max_len, void *cuda_stream, fem_result **out) {
    return fem_mine_levelwise_ex(c, id, I, nI, theta, max_len, 0u, cuda_stream, out);
}

int fem_mine_levelwise_ex(fem_ctx *c, int32_t id, const fem_interval *I, uint32_t nI,
                          uint32_t theta, uint32_t max_len, uint32_t flags, void *cuda_stream,
                          fem_result **out) {
    if (!c || !out || max_len < 1 || max_len > FEM_MAX_LEN) return FEM_EINVAL;
    if (flags & ~FEM_MINE_REPEATED_TYPES) return FEM_EINVAL;
    const bool repeats = (flags & FEM_MINE_REPEATED_TYPES) != 0;
    *out = nullptr;
    const StreamDev *sp = find_stream(c, id);
    if (!sp) return FEM_ENOSTREAM;
    const StreamDev &s = *sp;
    RET(check_intervals(s, I, nI));
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    c->stats.clear();
    fem_result *res = new (std::nothrow) fem_result;
    if (!res) return FEM_ENOMEM;
    res->eps.resize(max_len);
    res->counts.resize(max_len);
    auto fail = [&](int rc) {
        delete res;
        return rc;
    };
#define RETF(x)                         \
    do {                                \
        int r_ = (x);                   \
        if (r_ != FEM_OK) return fail(r_); \
    } while (0)
#define CKF(x)                                         \
    do {                                               \
        if ((x) != cudaSuccess) return fail(FEM_ECUDA); \
    } while (0)

    uint2 *d_ivl;
    RETF(upload_intervals(c, I, nI, st, &d_ivl));
    // per level, the (episode, event) pairs each pass visits (statistics only)
    unsigned long long *touched;
    RETF(dbuf(c, "touched", 2 * (FEM_MAX_LEN + 1), &touched));
    CKF(cudaMemsetAsync(touched, 0, 2 * (FEM_MAX_LEN + 1) * sizeof(unsigned long long), st));
    // level 1: the count of a one-node episode is the number of events of its type.
    // The device keeps the frequent types for generating level 2; the host takes the
    // same types (the same comparison) from the histogram the load read back, so it
    // needs no round trip to size level 2.
    uint32_t *ftypes;
    RETF(dbuf(c, "ftypes", 256, &ftypes));
    CKF(launch_type_filter(s.hist, s.K, theta, ftypes, c->d_small + W_COUNT0, st));
    const std::vector<uint32_t> &hist = c->hist_h[id];
    if (hist.size() != s.K) return fail(FEM_EINVAL);
    uint32_t f1 = 0, ftypes_h[8] = {};  // their number, a bit for each
    for (uint32_t a = 0; a < s.K; ++a) {
        if (!(hist[a] >= theta)) continue;
        ftypes_h[a >> 5] |= 1u << (a & 31);
        fem_episode e;
        std::memset(&e, 0, sizeof(e));
        e.types[0] = (uint8_t)a;
        e.len = 1;
        res->eps[0].push_back(e);
        res->counts[0].push_back(hist[a]);
        ++f1;
    }
    if (max_len < 2 || f1 < (repeats ? 1u : 2u) || nI == 0) {
        *out = res;
        return FEM_OK;
    }
    uint64_t m64 = (uint64_t)f1 * nI * (repeats ? f1 : f1 - 1);
    if (m64 > 0xFFFFFFF0ull) return fail(FEM_ENOMEM);
    uint32_t m = (uint32_t)m64;
    // level 2: ordered pairs of distinct frequent types x intervals.  Its relaxed pass
    // runs on the pair kernel (fem_pairs.cu) unless a kernel is configured or a shape
    // was measured or loaded for the pass's class: with two or more intervals a thread
    // shares one merge of a pair's events among its variants (on the 64-type
    // recording 0.26 ms against 0.29 for one thread per candidate)
    const bool pairs_level2 =
        !repeats && !c->cfg.kernel && nI >= 2 && nI <= 4 &&
        c->tune.find(tune_key(2, FEM_PASS_RELAXED, true, m, s.n_chunks, s.K)) == c->tune.end();
    const char *cname[2] = {"candsA", "candsB"};
    int cur = 0;
    fem_episode *cands;
    RETF(dbuf(c, cname[cur], m, &cands));
    cudaEventRecord(c->ev[0], st);
    CKF(launch_level2(ftypes, f1, nI, repeats, cands, st));
    cudaEventRecord(c->ev[1], st);
    // Per level the host waits three times: for the survivor count, the frequent
    // count and the next level's candidate count (each read together with the error
    // word; capacity recounts, when flagged, run before the count is used).
    // Timings are read from events after those waits; frequent sets are copied to
    // pinned staging and moved into the result after the last wait.
    uint32_t staged_f[FEM_MAX_LEN + 1] = {};
    auto compact_and_read = [&](const uint32_t *vals, uint32_t mm, uint32_t *idx, uint32_t word,
                                uint32_t *scratch, const PassLaunch &pl, uint32_t *kept,
                                cudaEvent_t done) -> int {
        CK(launch_compact(vals, nullptr, theta, mm, idx, c->d_small + word, scratch, st, pub_of(c)));
        if (done) CK(cudaEventRecord(done, st));
        uint32_t e;
        RET(read_count_err(c, c->d_small + word, kept, &e, st));
        if ((e & ERR_CAP) && !pl.hits) {  // (tables: no flags left)
            RET(count_finish(c, s, pl, e, st));
            CK(launch_compact(vals, nullptr, theta, mm, idx, c->d_small + word, scratch, st,
                              pub_of(c)));
            RET(read_count_err(c, c->d_small + word, kept, &e, st));
        }
        return err_status(e);
    };
    fem_episode *F = nullptr;  // the level's frequent episodes
    for (uint32_t N = 2; N <= max_len && m > 0; ++N) {
        fem_level_stats ls{};
        ls.level = N;
        ls.candidates = m;
        uint32_t *rel, *idx_s, *ex, *idx_f, *fcnt, *scratch;
        RETF(dbuf(c, "rel", m, &rel));
        RETF(dbuf(c, "idx_s", m, &idx_s));
        RETF(dbuf(c, "scratch", compact_scratch_words(m), &scratch));
        // first pass (Algorithm 3) on every candidate, then eliminate relaxed < theta
        PassLaunch plr;
        cudaEventRecord(c->ev[2], st);
        bool joined = false, counted = false;
        HitPlan hp;
        auto tables = [&] { return !repeats && !known_dense(c, s, ftypes_h); };
        // a pass over hit tables: the join of all pairs, or candidate by candidate
        auto over_tables = [&](bool join, bool planned, const uint32_t *g, uint32_t mm, int pass, uint32_t *o,
                               PassLaunch *pt, bool *done) {
            c->hits_busy = true;
            const int rc = join ? join_pass(c, s, &hp, planned, F, staged_f[2], cands, g, mm, d_ivl, nI, pass,
                                            o, st, pt, done)
                                : level_hits(c, s, cands, g, mm, (int)N, d_ivl, nI, pass, o, st, pt, done);
            return or_no_room(c, rc, done, st);
        };
        // whether it runs, where the rule says so: not if a shape of the other kernels is cached
        // for the class and no choice is; else as tuned_route finds
        auto chosen = [&](bool join, bool planned, const uint32_t *g, uint32_t mm, int pass, uint32_t *o,
                          bool *use) -> int {
            *use = true;
            if (!tune_used(c)) return FEM_OK;
            const std::string key = tune_key((int)N, pass, kTuneLevel, mm, s.n_chunks, s.K);
            if (!c->tune.count(key) && c->tune.count(tune_key((int)N, pass, 1, mm, s.n_chunks, s.K))) {
                *use = false;
                return FEM_OK;
            }
            return tuned_route(c, key, st, use,
                               [&] {
                                   return count_pass(c, s, cands, g, mm, (int)N, d_ivl, nI, pass, o, true, st,
                                                     nullptr);
                               },
                               [&](bool *done) {
                                   PassLaunch pt;
                                   return over_tables(join, planned, g, mm, pass, o, &pt, done);
                               });
        };
        bool use = false;
        const bool join = N == 3 && m >= kJoinCandidates && hits_eligible(c, s, nI) &&
                          (uint64_t)s.K * s.K * nI * s.K * nI <= kJoinCells;
        if (tables() && (join || (!(N == 2 && pairs_level2) && level_by_hits(c, s, N, FEM_PASS_RELAXED, m, nI)))) {
            RETF(chosen(join, false, nullptr, m, FEM_PASS_RELAXED, rel, &use));
            if (use) RETF(over_tables(join, false, nullptr, m, FEM_PASS_RELAXED, rel, &plr, &counted));
            joined = join && counted;
        }
        if (!counted) plr = PassLaunch{};
        if (counted) {
            // (over hit tables)
        } else if (repeats) {  // repeated types among the candidates: split and count (count_any)
            RETF(count_any(c, s, cands, nullptr, m, d_ivl, nI, FEM_PASS_RELAXED, rel, st));
        } else if (N == 2 && pairs_level2) {
            // every interval variant of an ordered type pair from one merge; the
            // candidates it gives up on go to the exact pass unfiltered when they are
            // at most 1/64 of the level, else to the recount
            uint32_t *work;
            RETF(dbuf(c, "pairs_work", 2, &work));
            CKF(cudaMemsetAsync(work, 0, 2 * sizeof(uint32_t), st));
            RETF(count_launch_pairs(c, s, cands, m, f1, d_ivl, nI, rel, st, &plr));
            CKF(launch_pairs_pass_flagged(rel, plr.p.redo, m, m / 64, work, c->d_err, st));
        } else {
            RETF(count_launch(c, s, cands, nullptr, m, (int)N, d_ivl, nI, FEM_PASS_RELAXED, rel,
                              true, st, &plr));
        }
        cudaEventRecord(c->ev[3], st);
        cudaEventRecord(c->ev[4], st);
        uint32_t ms;
        RETF(compact_and_read(rel, m, idx_s, W_COUNT0, scratch, plr, &ms, c->ev[5]));
        ls.survivors = ms;
        // second pass (Algorithm 1) on the survivors, then keep exact >= theta; the
        // relaxed pass's times are read and its statistics queued after this launch, so
        // that the device does not wait for the host's bookkeeping
        RETF(dbuf(c, "ex", ms, &ex));
        RETF(dbuf(c, "idx_f", ms, &idx_f));
        PassLaunch plx;
        cudaEventRecord(c->ev[6], st);
        counted = false;
        const bool again = joined && ms >= kJoinCandidates / 2;
        if (again || (tables() && level_by_hits(c, s, N, FEM_PASS_EXACT, ms, nI))) {
            RETF(chosen(again, true, idx_s, ms, FEM_PASS_EXACT, ex, &use));
            if (use) RETF(over_tables(again, true, idx_s, ms, FEM_PASS_EXACT, ex, &plx, &counted));
        }
        if (!counted) plx = PassLaunch{};
        if (counted)
            ;  // (over hit tables)
        else if (repeats)
            RETF(count_any(c, s, cands, idx_s, ms, d_ivl, nI, FEM_PASS_EXACT, ex, st));
        else
            RETF(count_launch(c, s, cands, idx_s, ms, (int)N, d_ivl, nI, FEM_PASS_EXACT, ex, true,
                              st, &plx));
        cudaEventRecord(c->ev[7], st);
        PassInfo pi;
        pass_info(c, plr, &pi);
        cudaEventElapsedTime(&ls.ms_generate, c->ev[0], c->ev[1]);
        cudaEventElapsedTime(&ls.ms_relaxed, c->ev[2], c->ev[3]);
        ls.segments = pi.segments;
        ls.kernel_relaxed = pi.kernel;
        ls.ms_relaxed_kernel = pi.ms_kernel;
        ls.ms_relaxed_stitch = pi.ms_stitch;
        uint32_t f = 0;
        if (ms) RETF(compact_and_read(ex, ms, idx_f, W_COUNT1, scratch, plx, &f, nullptr));
        // work statistics of both passes (idx_s and the candidates stay until the next
        // level): queued behind the next wait's publishing launch where there is one
        auto queue_touched = [&]() -> int {
            CK(launch_touched(cands, nullptr, m, s.hist, touched + 2 * N, st));
            CK(launch_touched(cands, idx_s, ms, s.hist, touched + 2 * N + 1, st));
            return FEM_OK;
        };
        PassInfo pe;
        pass_info(c, plx, &pe);
        cudaEventElapsedTime(&ls.ms_compact, c->ev[4], c->ev[5]);
        cudaEventElapsedTime(&ls.ms_exact, c->ev[6], c->ev[7]);
        ls.ms_exact_kernel = pe.ms_kernel;
        ls.exact_segments = ms ? pe.segments : 0;
        ls.kernel_exact = ms ? pe.kernel : 0;
        ls.frequent = f;
        c->stats.push_back(ls);
        if (f == 0) {
            RETF(queue_touched());
            break;
        }
        RETF(dbuf(c, "fcnt", f, &fcnt));
        RETF(dbuf(c, "F", f, &F));
        CKF(launch_gather_frequent(cands, idx_s, idx_f, f, ex, F, fcnt, st));
        void *h;
        RETF(pinbuf(c, N, (size_t)f * (sizeof(fem_episode) + 4), st, &h));
        CKF(cudaMemcpyAsync(h, F, (size_t)f * sizeof(fem_episode), cudaMemcpyDeviceToHost, st));
        CKF(cudaMemcpyAsync(static_cast<uint8_t *>(h) + (size_t)f * sizeof(fem_episode), fcnt,
                            (size_t)f * 4, cudaMemcpyDeviceToHost, st));
        staged_f[N] = f;
        if (N == max_len) {
            RETF(queue_touched());
            break;
        }
        // join level N -> N + 1
        uint32_t *jc, *joff;
        RETF(dbuf(c, "jc", f, &jc));
        RETF(dbuf(c, "joff", f, &joff));
        cudaEventRecord(c->ev[0], st);
        CKF(launch_join_count(F, f, N, repeats, jc, c->sm_count, st));
        CKF(launch_exclusive_scan(jc, f, joff, c->d_small + W_COUNT2, scratch, st, pub_of(c)));
        RETF(queue_touched());
        uint32_t mn, ej;
        RETF(read_count_err(c, c->d_small + W_COUNT2, &mn, &ej, st));
        RETF(err_status(ej));
        cur ^= 1;
        RETF(dbuf(c, cname[cur], std::max<uint32_t>(mn, 1), &cands));
        CKF(launch_join_emit(F, f, N, repeats, joff, cands, c->sm_count, st));
        cudaEventRecord(c->ev[1], st);
        m = mn;
    }
    // statistics and the error word in the last round trip (pinned words)
    constexpr size_t TB = 2 * (FEM_MAX_LEN + 1) * sizeof(unsigned long long);
    static_assert(TB + 4 <= 64 * sizeof(uint32_t), "pinned word buffer too small");
    CKF(cudaMemcpyAsync(c->h_small, touched, TB, cudaMemcpyDeviceToHost, st));
    CKF(cudaMemcpyAsync(c->h_small + TB / 4, c->d_err, 4, cudaMemcpyDeviceToHost, st));
    CKF(cudaStreamSynchronize(st));
    unsigned long long tv[2 * (FEM_MAX_LEN + 1)];
    std::memcpy(tv, c->h_small, TB);
    const uint32_t e = c->h_small[TB / 4];
    for (fem_level_stats &ls : c->stats) {
        ls.touched_relaxed = tv[2 * ls.level];
        ls.touched_exact = tv[2 * ls.level + 1];
    }
    for (uint32_t N = 2; N <= max_len; ++N) {
        const uint32_t f = staged_f[N];
        if (!f) continue;
        const uint8_t *h = static_cast<const uint8_t *>(c->pin[N].p);
        res->eps[N - 1].resize(f);
        res->counts[N - 1].resize(f);
        std::memcpy(res->eps[N - 1].data(), h, (size_t)f * sizeof(fem_episode));
        std::memcpy(res->counts[N - 1].data(), h + (size_t)f * sizeof(fem_episode), (size_t)f * 4);
    }
    RETF(err_status(e));
    *out = res;
    return FEM_OK;
#undef RETF
#undef CKF
}

int fem_result_level(const fem_result *r, uint32_t level, uint32_t *m_out,
                     const fem_episode **eps, const uint32_t **counts) {
    if (!r || !m_out || level < 1 || level > r->eps.size()) return FEM_EINVAL;
    *m_out = (uint32_t)r->eps[level - 1].size();
    if (eps) *eps = r->eps[level - 1].data();
    if (counts) *counts = r->counts[level - 1].data();
    return FEM_OK;
}

uint32_t fem_result_max_level(const fem_result *r) {
    if (!r) return 0;
    uint32_t L = 0;
    for (uint32_t i = 0; i < r->eps.size(); ++i)
        if (!r->eps[i].empty()) L = i + 1;
    return L;
}

void fem_result_free(fem_result *r) { delete r; }

int fem_last_mine_stats(fem_ctx *c, fem_level_stats *out, uint32_t cap) {
    if (!c || (cap && !out)) return FEM_EINVAL;
    const uint32_t k = std::min<uint32_t>(cap, (uint32_t)c->stats.size());
    for (uint32_t i = 0; i < k; ++i) out[i] = c->stats[i];
    return (int)k;
}

}  // extern "C"

// ============================================================================ batches
namespace {

constexpr uint32_t kBatchChunksPerItem = 16;  // segment length of batched work items (rule)
constexpr uint32_t kBatchMinChunksPerItem = 8;  // shortest segment length tried when tuning
constexpr uint32_t kBatchMinThreads = 64;       // smallest block size tried when tuning

struct BatchGroup {
    int N = 0;
    uint32_t n_jobs = 0, m = 0;
    std::vector<uint32_t> user_job;  // user job index of each group job
    std::vector<uint32_t> off;       // host copy of cand_off
    fem_episode *cands = nullptr;
    uint32_t *cand_off = nullptr, *theta = nullptr;
    CountParams *rjobs = nullptr, *xjobs = nullptr;
    BatchOut *outs = nullptr;
    uint32_t *rel = nullptr, *ex = nullptr, *idx = nullptr, *scratch = nullptr;
    uint8_t *flags = nullptr, *redo = nullptr, *xredo = nullptr;
    uint32_t *item_off_r = nullptr, *item_off_x = nullptr;
    uint4 *items_r = nullptr, *items_x = nullptr;
    uint32_t cap_r = 0, cap_x = 0;
    uint32_t *counters = nullptr;  // n_items_r, n_items_x, queue_r, queue_x, n_idx
    uint4 *tables = nullptr;
    uint32_t SB = 0, Tr = 128, Tx = 128, Rx = 16;
    uint32_t cpi = kBatchChunksPerItem;  // chunks per work item (segment length)
    std::vector<uint32_t> nch, mj;       // per group job: stream chunks, candidates
    std::vector<CountParams> rj, xj;     // host templates of the per-job parameters
};

}  // namespace

namespace {

// A batch counted over hit tables: its candidates by stream, each stream's planned once
// (order, edges, slabs), the tables built and the candidates counted in every run.  A part
// is a stream's candidates of one launch group; slots are in part order.
struct BatchHits {
    uint32_t n_jobs = 0, m = 0, n_streams = 0, n_parts = 0, n_slabs = 0;
    std::vector<HitBuild> build;            // per stream
    std::vector<CountParams> parts;         // per part, relaxed pass
    HitBuild *d_build = nullptr;
    uint32_t *first = nullptr;              // first slab block of each stream
    CountParams *rparts = nullptr, *xparts = nullptr;
    uint32_t *part_off = nullptr;           // first slot of each part
    struct Launch {
        uint4 *list = nullptr;
        uint32_t n_list = 0, n_items = 0;
    };
    Launch rel[PLAN_GROUPS], ex[PLAN_GROUPS];
    fem_episode *cands = nullptr;
    uint32_t *record = nullptr;             // slot -> candidate
    uint32_t *cand_off = nullptr, *theta = nullptr;  // per job
    BatchOut *outs = nullptr;
    uint32_t *r = nullptr, *x = nullptr, *idx = nullptr, *gx = nullptr, *scratch = nullptr, *n_idx = nullptr;
    uint8_t *flags = nullptr, *redo = nullptr, *xredo = nullptr;
    std::vector<uint32_t> job;              // the batch's job of each job here
    uint8_t *marks = nullptr;               // per job: to be recounted
    unsigned long long *used = nullptr;     // hits found by either pass
    uint64_t capacity = 0;
};

}  // namespace

struct fem_batch {
    fem_ctx *ctx = nullptr;
    std::vector<fem_job> jobs;
    bool over_hits = false;
    BatchHits hits;
    std::vector<BatchGroup> groups;
    std::vector<void *> allocs;
    std::vector<size_t> alloc_bytes;
    uint2 *ivl = nullptr;
    uint32_t nI = 0;
    cudaStream_t cap_stream = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint32_t graph_kernels = 0;  // kernel nodes of the captured graph (launch accounting)
};

namespace {

template <typename T>
int balloc(fem_batch *b, size_t count, T **out) {
    void *p = nullptr;
    const size_t bytes = std::max<size_t>(count * sizeof(T), 256);
    RET(cmalloc(b->ctx, &p, bytes));
    b->allocs.push_back(p);
    b->alloc_bytes.push_back(bytes);
    *out = static_cast<T *>(p);
    return FEM_OK;
}

void batch_free(fem_batch *b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    for (size_t i = 0; i < b->allocs.size(); ++i) cfree(b->ctx, b->allocs[i], b->alloc_bytes[i]);
    delete b;
}

// Set a group's launch shape: segment length (chunks per item) and block sizes of
// the two passes; rewrites the per-job segment counts and table slices.
int batch_shape(BatchGroup &g, uint32_t cpi, uint32_t Tr, uint32_t Tx, cudaStream_t st) {
    g.cpi = cpi, g.Tr = Tr, g.Tx = Tx;
    uint64_t toff = 0;
    for (uint32_t k = 0; k < g.n_jobs; ++k) {
        uint32_t P = (g.nch[k] + cpi - 1) / cpi;
        const uint32_t cps = (g.nch[k] + P - 1) / P;
        P = (g.nch[k] + cps - 1) / cps;
        for (CountParams *q : {&g.rj[k], &g.xj[k]}) {
            q->cps = cps;
            q->P = P;
            q->tables = g.tables + toff;
        }
        toff += (uint64_t)g.mj[k] * P * S_MAX;
    }
    CK(cudaMemcpyAsync(g.rjobs, g.rj.data(), g.n_jobs * sizeof(CountParams),
                       cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(g.xjobs, g.xj.data(), g.n_jobs * sizeof(CountParams),
                       cudaMemcpyHostToDevice, st));
    return FEM_OK;
}

// The two-pass count of one length group, enqueued on st without host round trips.
int batch_enqueue_group(fem_ctx *c, BatchGroup &g, cudaStream_t st) {
    {
        CK(cudaMemsetAsync(g.counters, 0, 8 * sizeof(uint32_t), st));
        CK(cudaMemsetAsync(g.redo, 0, g.m, st));
        CK(cudaMemsetAsync(g.xredo, 0, g.m, st));
        // first pass: relaxed counts of every candidate (Algorithm 3)
        CK(launch_batch_items(g.rjobs, g.n_jobs, g.Tr, g.item_off_r, g.counters + 0, g.cap_r,
                              g.items_r, st));
        CK(launch_count_batch(g.N, FEM_PASS_RELAXED, 1, g.Tr, g.rjobs, g.items_r, g.counters + 0,
                              g.counters + 2, g.SB, c->sm_count, st));
        CK(launch_stitch_batch(g.rjobs, g.cand_off, g.n_jobs, g.m, c->d_err, st));
        // elimination at each job's theta (Algorithm 4)
        CK(launch_batch_keep_flags(g.rel, g.cand_off, g.theta, g.n_jobs, g.m, g.flags, st));
        CK(launch_compact(nullptr, g.flags, 0, g.m, g.idx, g.counters + 4, g.scratch, st));
        // second pass: exact counts of the survivors (Algorithm 1)
        CK(launch_batch_exact_jobs(g.xjobs, g.cand_off, g.n_jobs, g.idx, g.counters + 4, g.ex, st));
        CK(launch_batch_items(g.xjobs, g.n_jobs, g.Tx, g.item_off_x, g.counters + 1, g.cap_x,
                              g.items_x, st));
        CK(launch_count_batch(g.N, FEM_PASS_EXACT, g.Rx, g.Tx, g.xjobs, g.items_x, g.counters + 1,
                              g.counters + 3, g.SB, c->sm_count, st));
        CK(launch_stitch_batch(g.xjobs, g.cand_off, g.n_jobs, g.m, c->d_err, st));
        CK(launch_batch_outputs(g.outs, g.cand_off, g.n_jobs, g.m, g.idx, g.counters + 4, g.ex, st));
    }
    return FEM_OK;
}

// The two-pass count of a batch over hit tables, enqueued without host round trips.
int batch_enqueue_hits(fem_ctx *c, BatchHits &h, cudaStream_t st) {
    CK(cudaMemsetAsync(h.used, 0, 16, st));
    CK(cudaMemsetAsync(h.redo, 0, h.m, st));
    CK(cudaMemsetAsync(h.xredo, 0, h.m, st));
    // first pass: relaxed counts of every candidate (Algorithm 3)
    CK(launch_hit_build_batch(FEM_PASS_RELAXED, h.build.data(), h.d_build, h.first, h.n_streams, h.n_slabs, st));
    for (uint32_t g = 0; g < PLAN_GROUPS; ++g)
        CK(launch_hit_count_batch(g, h.rparts, h.rel[g].list, h.rel[g].n_list, h.rel[g].n_items, st));
    CK(launch_stitch_batch(h.rparts, h.part_off, h.n_parts, h.m, c->d_err, st, S_RECOUNT));
    // elimination at each job's theta (Algorithm 4)
    CK(launch_batch_keep_slots(h.r, h.record, h.cand_off, h.theta, h.n_jobs, h.m, h.flags, st));
    CK(launch_compact(nullptr, h.flags, 0, h.m, h.idx, h.n_idx, h.scratch, st));
    CK(launch_batch_pick(h.idx, h.n_idx, h.m, h.record, h.gx, st));
    // second pass: exact counts of the survivors (Algorithm 1)
    CK(launch_batch_exact_jobs(h.xparts, h.part_off, h.n_parts, h.idx, h.n_idx, h.x, st, h.gx));
    CK(cudaMemcpyAsync(h.used + 1, h.used, 8, cudaMemcpyDeviceToDevice, st));
    CK(cudaMemsetAsync(h.used, 0, 8, st));
    CK(launch_hit_build_batch(FEM_PASS_EXACT, h.build.data(), h.d_build, h.first, h.n_streams, h.n_slabs, st));
    for (uint32_t g = 0; g < PLAN_GROUPS; ++g)
        CK(launch_hit_count_batch(g, h.xparts, h.ex[g].list, h.ex[g].n_list, h.ex[g].n_items, st));
    CK(launch_stitch_batch(h.xparts, h.part_off, h.n_parts, h.m, c->d_err, st, S_RECOUNT));
    CK(launch_batch_outputs(h.outs, h.cand_off, h.n_jobs, h.m, h.gx, h.n_idx, h.x, st));
    return FEM_OK;
}

// The whole two-pass count of the batch, enqueued on st without host round trips.
int batch_enqueue(fem_batch *b, cudaStream_t st) {
    if (b->over_hits) return batch_enqueue_hits(b->ctx, b->hits, st);
    for (BatchGroup &g : b->groups) RET(batch_enqueue_group(b->ctx, g, st));
    return FEM_OK;
}

// Batch launch shapes by measurement: for each length group, time every segment
// length (8, 16, 32 chunks per item) and block size pair, each a complete two-pass
// count, and keep the fastest.
int batch_tune(fem_batch *b, cudaStream_t st) {
    fem_ctx *c = b->ctx;
    for (BatchGroup &g : b->groups) {
        float best = -1;
        uint32_t bc = g.cpi, br = g.Tr, bx = g.Tx;
        for (uint32_t cpi : {8u, 16u, 32u}) {
            for (uint32_t Tr : {128u, 256u}) {
                if (Tr == 256 && g.N > 3) continue;
                for (uint32_t Tx : {64u, 128u}) {
                    RET(batch_shape(g, cpi, Tr, Tx, st));
                    float ms = -1;
                    for (int rep = 0; rep < 2; ++rep) {  // the faster of two (kernel loading)
                        CK(cudaMemsetAsync(c->d_err, 0, 4, st));
                        CK(cudaEventRecord(c->tev[0], st));
                        RET(batch_enqueue_group(c, g, st));
                        CK(cudaEventRecord(c->tev[1], st));
                        uint32_t e;
                        RET(read_err(c, st, &e));
                        RET(err_status(e));
                        float t = 0;
                        CK(cudaEventElapsedTime(&t, c->tev[0], c->tev[1]));
                        if (e & ERR_CAP) t *= 4;  // needs recounts
                        if (ms < 0 || t < ms) ms = t;
                    }
                    if (best < 0 || ms < best) best = ms, bc = cpi, br = Tr, bx = Tx;
                }
            }
        }
        RET(batch_shape(g, bc, br, bx, st));
        if (std::getenv("FEM_DEBUG"))
            std::fprintf(stderr, "fem: batch N=%d jobs=%u m=%u: %u chunks per item, T %u/%u, %.3f ms\n",
                         g.N, g.n_jobs, g.m, bc, br, bx, best);
    }
    return FEM_OK;
}

// Whether a batch of these jobs (and streams) is estimated to run faster over hit tables than by
// the other kernels, in microseconds a run: over tables, building them for both passes (the
// events times types of all streams, and a block's share where there are few slabs) and the
// hits; by the others, per length a launch of items whose longest goes through 16 chunks,
// and all events times nodes.  Fits to 260 batches of 1 to 48 jobs of 20 to 15,000
// candidates on streams of 4 to 128 types, 3 s to 10 min: half of the estimates within 18 and
// 28%, nine of ten within 55 and 95%; by them four batches take more than 5% longer than by the other
// kernels, 1.6 times at most, where over tables 76 did, up to 13 times (32 jobs of 1,000
// episodes of five nodes on 32 half-minutes of 128 types: 0.54 and 5.2 ms).
bool batch_over_tables(const fem_ctx *c, const std::vector<fem_job> &jobs, uint32_t nI) {
    struct Stream {
        const StreamDev *s = nullptr;
        double edges = 0;
    };
    std::map<int32_t, Stream> streams;
    double hits = 0, m = 0, work = 0, longest[FEM_MAX_LEN + 1] = {};
    for (const fem_job &jb : jobs) {
        if (!jb.m) continue;
        Stream &st = streams[jb.stream_id];
        st.s = &c->streams.at(jb.stream_id);
        const double each = (double)st.s->n / st.s->K, N = jb.len;
        st.edges += (double)jb.m * (N - 1);
        hits += jb.m * N * each * events_in_interval(c, *st.s);
        work += jb.m * N * N * each;
        m += jb.m;
        longest[jb.len] = std::max(longest[jb.len], N * std::min(each, 16.0 * CHUNK / st.s->K));
    }
    double tables = 105 + 2.5e-6 * hits + 1.6e-3 * m, block = 0, dense = 0;
    for (const auto &kv : streams) {
        const StreamDev &s = *kv.second.s;
        const double K = s.K, n = (double)s.n, in = events_in_interval(c, s);
        const double groups = std::min(1.0, kv.second.edges * std::min(K, 32.0) / (K * K));
        const double used = std::min(1.0, kv.second.edges / (K * K * std::max(nI, 1u)));
        tables += n * K * (8.1e-6 * groups + 3.5e-5 * used * in) + 2.7e-5 * s.n_chunks * K * K * groups;
        block = std::max(block, 0.05 * K * K * groups);
        dense = std::max(dense, 9.4e-3 * std::min<double>(n, CHUNK) * K * used * in);
    }
    double others = 3.1e-3 * m + 7.4e-7 * work;
    for (double l : longest)
        if (l > 0) others += 57 + 0.25 * l;
    return 0.9 * (tables + block + dense) < others;
}

// Plans a batch over hit tables and runs it once; *ok = false, with its memory given back,
// where tables do not apply to one of the streams or their memory would pass an eighth of
// the device's (or the context's budget).
int batch_plan_hits(fem_batch *b, cudaStream_t st, bool *ok) {
    *ok = false;
    fem_ctx *c = b->ctx;
    BatchHits &h = b->hits;
    const uint32_t nI = b->nI;
    if (!batch_over_tables(c, b->jobs, nI)) return FEM_OK;
    size_t free_bytes = 0, total_bytes = 0;
    CK(cudaMemGetInfo(&free_bytes, &total_bytes));
    const uint64_t most = std::min(total_bytes / 8, free_bytes / 2);
    // the jobs by stream
    std::vector<uint32_t> &job = h.job, off{0}, theta, iota, first{0}, part_off, part_group;
    std::vector<int32_t> streams;
    std::vector<BatchOut> outs;
    std::vector<CountParams> xp;
    std::vector<std::vector<uint4>> lists;
    // every upload goes in st's order, before the kernels that read it; what is uploaded
    // (declared above, or the batch's) lives until st has taken it
    struct Drain {
        cudaStream_t st;
        ~Drain() { cudaStreamSynchronize(st); }
    } drain{st};
    for (uint32_t j = 0; j < b->jobs.size(); ++j)
        if (b->jobs[j].m && std::find(streams.begin(), streams.end(), b->jobs[j].stream_id) == streams.end())
            streams.push_back(b->jobs[j].stream_id);
    std::vector<uint32_t> stream_off;
    uint64_t m = 0;
    for (int32_t id : streams) {
        if (!hits_eligible(c, *find_stream(c, id), nI)) return FEM_OK;
        stream_off.push_back((uint32_t)m);
        for (uint32_t j = 0; j < b->jobs.size(); ++j) {
            if (b->jobs[j].stream_id != id || !b->jobs[j].m) continue;
            job.push_back(j);
            m += b->jobs[j].m;
            off.push_back((uint32_t)m);
        }
        if (m > 0x7FFFFFFFull) return FEM_OK;
    }
    if (m == 0) return FEM_OK;
    h.m = (uint32_t)m, h.n_jobs = (uint32_t)job.size(), h.n_streams = (uint32_t)streams.size();
    RET(balloc(b, m, &h.cands));
    theta.resize(h.n_jobs), outs.resize(h.n_jobs);
    for (uint32_t k = 0; k < h.n_jobs; ++k) {
        const fem_job &jb = b->jobs[job[k]];
        CK(cudaMemcpyAsync(h.cands + off[k], jb.cands, (size_t)jb.m * sizeof(fem_episode),
                           cudaMemcpyDeviceToDevice, st));
        theta[k] = jb.theta;
        outs[k] = BatchOut{jb.exact_out, jb.survived_out};
    }
    // every candidate has its job's length (the counting kernels take any); in pieces, whatever
    // the batch's size is on the host
    uint32_t *d_iota;
    RET(balloc(b, m, &d_iota));
    {
        constexpr uint32_t PIECE = 1u << 16;
        std::vector<fem_episode> host(std::min<uint64_t>(m, PIECE));
        iota.resize(host.size());
        uint32_t k = 0;
        for (uint32_t i0 = 0; i0 < m; i0 += PIECE) {
            const uint32_t n = std::min<uint32_t>(PIECE, (uint32_t)m - i0);
            CK(cudaMemcpyAsync(host.data(), h.cands + i0, n * sizeof(fem_episode), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            for (uint32_t i = 0; i < n; ++i) {
                while (i0 + i >= off[k + 1]) ++k;
                if (host[i].len != b->jobs[job[k]].len) return FEM_EINVAL;
                iota[i] = i0 + i;
            }
            CK(cudaMemcpyAsync(d_iota + i0, iota.data(), n * 4, cudaMemcpyHostToDevice, st));
        }
    }
    RET(balloc(b, m, &h.record));
    RET(balloc(b, h.n_jobs + 1, &h.cand_off));
    RET(balloc(b, h.n_jobs, &h.theta));
    RET(balloc(b, h.n_jobs, &h.outs));
    RET(balloc(b, m, &h.r));
    RET(balloc(b, m, &h.x));
    RET(balloc(b, m, &h.idx));
    RET(balloc(b, m, &h.gx));
    RET(balloc(b, compact_scratch_words(h.m), &h.scratch));
    RET(balloc(b, 1, &h.n_idx));
    RET(balloc(b, m, &h.flags));
    RET(balloc(b, m, &h.redo));
    RET(balloc(b, m, &h.xredo));
    RET(balloc(b, 2, &h.used));
    RET(balloc(b, h.n_jobs, &h.marks));
    CK(cudaMemcpyAsync(h.cand_off, off.data(), off.size() * 4, cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(h.theta, theta.data(), theta.size() * 4, cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(h.outs, outs.data(), outs.size() * sizeof(BatchOut), cudaMemcpyHostToDevice, st));
    // per stream its plan; the bins and ranks are shared by the streams, one after the other
    uint32_t *bin, *rank, *order;
    RET(balloc(b, m, &bin));
    RET(balloc(b, m, &rank));
    RET(balloc(b, m, &order));
    uint64_t bytes = 0;
    h.capacity = 0;
    for (uint32_t k = 0; k < h.n_streams; ++k) {
        const StreamDev &s = *find_stream(c, streams[k]);
        const uint32_t s0 = stream_off[k], ms = (k + 1 < h.n_streams ? stream_off[k + 1] : h.m) - s0;
        HitPlan pl;
        bool fits;
        RET(hits_plan(c, s, h.cands, d_iota + s0, ms, true, b->ivl, nI, FEM_PASS_RELAXED, st, &pl, &fits,
                      [&](const char *n, size_t w, uint32_t **p) -> int {
                          if (!std::strcmp(n, "hit_plan_bin")) return *p = bin, FEM_OK;
                          if (!std::strcmp(n, "hit_plan_rank")) return *p = rank, FEM_OK;
                          if (!std::strcmp(n, "hit_plan_order")) return *p = order, FEM_OK;
                          if (!std::strcmp(n, "hit_plan_gather")) return *p = h.record + s0, FEM_OK;
                          return balloc(b, w, p);
                      }));
        if (!fits) return FEM_OK;
        bytes += (uint64_t)pl.h.n_slabs * (pl.h.n_edges * 8ull + pl.h.types * 3ull) + s.n * 2ull + pl.hits * 4ull;
        if (bytes > most || h.capacity + pl.hits > 0xF0000000ull) return FEM_OK;
        h.capacity += pl.hits;
        HitBuild &hb = pl.b;
        RET(balloc(b, (size_t)pl.h.n_slabs * pl.h.n_edges, &hb.edge));
        RET(balloc(b, (size_t)pl.h.n_slabs * pl.h.types, &hb.count));
        RET(balloc(b, (size_t)pl.h.n_slabs * pl.h.types, &hb.place));
        RET(balloc(b, s.n, &hb.index));
        hb.used = h.used;
        pl.h.edge = hb.edge, pl.h.count = hb.count, pl.h.place = hb.place, pl.h.index = hb.index;
        h.build.push_back(hb);
        first.push_back(first.back() + pl.h.n_slabs);
        uint32_t slot = s0;
        for (uint32_t g = 0; g < PLAN_GROUPS; ++g) {
            if (!pl.group_m[g]) continue;
            CountParams p = hits_params(c, s, pl, h.cands, g, 0);
            p.gather = h.record + slot;
            p.out = h.r + slot;
            p.redo = h.redo + slot;
            p.hit_classes = S_RECOUNT;
            part_off.push_back(slot);
            part_group.push_back(g);
            h.parts.push_back(p);
            slot += p.m;
        }
    }
    h.n_slabs = first.back();
    h.n_parts = (uint32_t)h.parts.size();
    part_off.push_back(h.m);
    // segments: the same number of slabs for every item of a launch, for about four blocks
    // for each place on the GPU (the exact pass, with fewer candidates, four times as many)
    xp = h.parts;
    uint64_t tab = 0;
    for (int pass = 0; pass < 2; ++pass) {
        uint64_t t = 0;
        for (uint32_t g = 0; g < PLAN_GROUPS; ++g) {
            uint64_t work = 0;
            for (uint32_t q = 0; q < h.n_parts; ++q)
                if (part_group[q] == g) work += (uint64_t)((h.parts[q].m + 127) / 128) * h.parts[q].hits.n_slabs;
            const uint64_t blocks = (uint64_t)c->sm_count * 24 * (pass ? 4 : 1);
            const uint32_t cps = (uint32_t)std::max<uint64_t>(8, (work + blocks - 1) / blocks);
            std::vector<uint4> list;
            uint32_t items = 0;
            for (uint32_t q = 0; q < h.n_parts; ++q) {
                if (part_group[q] != g) continue;
                CountParams &p = pass ? xp[q] : h.parts[q];
                const uint32_t P = (p.hits.n_slabs + cps - 1) / cps;
                p.cps = (p.hits.n_slabs + P - 1) / P;
                p.P = (p.hits.n_slabs + p.cps - 1) / p.cps;
                p.tables = reinterpret_cast<uint4 *>(t);  // (an offset until they are allocated)
                t += (uint64_t)p.P * p.m * S_RECOUNT;
                const uint32_t tiles = (p.m + 127) / 128;
                list.push_back(make_uint4(items, tiles, q, 0));
                items += tiles * p.P;
            }
            BatchHits::Launch &l = pass ? h.ex[g] : h.rel[g];
            l.n_list = (uint32_t)list.size(), l.n_items = items;
            if (list.empty()) continue;
            RET(balloc(b, list.size(), &l.list));
            CK(cudaMemcpyAsync(l.list, list.data(), list.size() * sizeof(uint4), cudaMemcpyHostToDevice, st));
            lists.push_back(std::move(list));
        }
        tab = std::max(tab, t);
    }
    if (bytes + tab * sizeof(uint4) > most) return FEM_OK;
    uint4 *tables;
    RET(balloc(b, tab, &tables));
    for (uint32_t q = 0; q < h.n_parts; ++q) {
        h.parts[q].tables = tables + reinterpret_cast<uint64_t>(h.parts[q].tables);
        xp[q].tables = tables + reinterpret_cast<uint64_t>(xp[q].tables);
        xp[q].redo = h.xredo + part_off[q];
        xp[q].m = 0;
    }
    RET(balloc(b, h.n_streams, &h.d_build));
    RET(balloc(b, first.size(), &h.first));
    RET(balloc(b, h.n_parts, &h.rparts));
    RET(balloc(b, h.n_parts, &h.xparts));
    RET(balloc(b, part_off.size(), &h.part_off));
    CK(cudaMemcpyAsync(h.first, first.data(), first.size() * 4, cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(h.part_off, part_off.data(), part_off.size() * 4, cudaMemcpyHostToDevice, st));
    // one run, in which the ranges may turn out to be more than estimated
    for (int attempt = 0; attempt < 2; ++attempt) {
        uint32_t *range;
        RET(balloc(b, h.capacity, &range));
        for (HitBuild &hb : h.build) hb.range = range, hb.capacity = h.capacity;
        for (uint32_t q = 0; q < h.n_parts; ++q) h.parts[q].hits.range = xp[q].hits.range = range;
        CK(cudaMemcpyAsync(h.d_build, h.build.data(), h.n_streams * sizeof(HitBuild), cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(h.rparts, h.parts.data(), h.n_parts * sizeof(CountParams), cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(h.xparts, xp.data(), h.n_parts * sizeof(CountParams), cudaMemcpyHostToDevice, st));
        CK(cudaMemsetAsync(c->d_err, 0, 4, st));
        RET(batch_enqueue_hits(c, h, st));
        unsigned long long used[2];
        uint32_t e;
        CK(cudaMemcpyAsync(used, h.used, 16, cudaMemcpyDeviceToHost, st));
        RET(read_err(c, st, &e));
        RET(err_status(e));
        const uint64_t need = std::max(used[0], used[1]);
        if (std::getenv("FEM_DEBUG"))
            std::fprintf(stderr, "fem: batch tables %.2f GB, transfer tables %.2f GB, hits %llu of %llu, err %#x\n",
                         bytes * 1e-9, tab * 16e-9, (unsigned long long)need, (unsigned long long)h.capacity, e);
        if (e & ERR_DENSE) {  // (of which stream, the words do not say)
            CK(cudaMemsetAsync(c->d_dense, 0xFF, 256 * sizeof(uint32_t), st));
            return FEM_OK;
        }
        if (need <= h.capacity) {
            *ok = true;
            return FEM_OK;
        }
        if (need > 0xF0000000ull || bytes + (tab * sizeof(uint4)) + need * 4 > most) return FEM_OK;
        cfree(c, range, b->alloc_bytes.back());
        b->allocs.pop_back(), b->alloc_bytes.pop_back();
        h.capacity = need + need / 16;
    }
    return FEM_OK;
}

}  // namespace

extern "C" {

int fem_batch_create(fem_ctx *c, const fem_job *jobs, uint32_t n_jobs, const fem_interval *I,
                     uint32_t nI, void *cuda_stream, fem_batch **out) {
    if (!c || !out || !jobs || n_jobs == 0) return FEM_EINVAL;
    *out = nullptr;
    for (uint32_t j = 0; j < n_jobs; ++j) {
        const StreamDev *s = find_stream(c, jobs[j].stream_id);
        if (!s) return FEM_ENOSTREAM;
        if (jobs[j].len < 1 || jobs[j].len > FEM_MAX_LEN) return FEM_EINVAL;
        if (jobs[j].m && (!jobs[j].cands || !jobs[j].exact_out || !jobs[j].survived_out))
            return FEM_EINVAL;
        RET(check_intervals(*s, I, nI));
    }
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    fem_batch *b = new (std::nothrow) fem_batch;
    if (!b) return FEM_ENOMEM;
    b->ctx = c;
    b->jobs.assign(jobs, jobs + n_jobs);
    b->nI = nI;
    auto fail = [&](int rc) {
        cudaStreamSynchronize(st);
        batch_free(b);
        return rc;
    };
#define BRET(x)                           \
    do {                                  \
        int r_ = (x);                     \
        if (r_ != FEM_OK) return fail(r_); \
    } while (0)
#define BCK(x)                                          \
    do {                                                \
        if ((x) != cudaSuccess) return fail(FEM_ECUDA); \
    } while (0)
    BRET(balloc(b, std::max<uint32_t>(nI, 1), &b->ivl));
    if (nI) BCK(cudaMemcpyAsync(b->ivl, I, nI * sizeof(uint2), cudaMemcpyHostToDevice, st));

    c->ivl_host.assign(I, I + nI);
    {
        const size_t kept = b->allocs.size();
        const int rch = batch_plan_hits(b, st, &b->over_hits);
        if (rch != FEM_OK && rch != FEM_ENOMEM) return fail(rch);
        if (std::getenv("FEM_DEBUG"))
            std::fprintf(stderr, "fem: batch of %u candidates, %u streams: %s (%u slabs, %llu hits' room)\n",
                         b->hits.m, b->hits.n_streams, b->over_hits ? "over hit tables" : "per-thread kernels",
                         b->hits.n_slabs, (unsigned long long)b->hits.capacity);
        if (!b->over_hits) {  // the per-thread kernels: give the tables' memory back
            cudaGetLastError();
            BCK(cudaStreamSynchronize(st));
            for (; b->allocs.size() > kept; b->allocs.pop_back(), b->alloc_bytes.pop_back())
                cfree(c, b->allocs.back(), b->alloc_bytes.back());
            b->hits = BatchHits{};
            BCK(cudaMemsetAsync(c->d_err, 0, 4, st));
        }
    }
    for (int N = 1; N <= FEM_MAX_LEN && !b->over_hits; ++N) {
        BatchGroup g;
        g.N = N;
        struct Ent {
            uint32_t j, nch;
        };
        std::vector<Ent> ents;
        for (uint32_t j = 0; j < n_jobs; ++j) {
            if ((int)jobs[j].len != N || jobs[j].m == 0) continue;
            const StreamDev &s = *find_stream(c, jobs[j].stream_id);
            ents.push_back({j, std::max<uint32_t>(s.n_chunks, 1)});
        }
        if (ents.empty()) continue;
        // longest streams first: with equal segment lengths their items are the
        // longest, and the persistent blocks then finish together
        std::stable_sort(ents.begin(), ents.end(),
                         [](const Ent &a, const Ent &b2) { return a.nch > b2.nch; });
        g.n_jobs = (uint32_t)ents.size();
        g.Tr = N <= 3 ? 256 : 128;
        g.Tx = 128;
        g.Rx = 16;
        // capacities for every shape batch_shape may set (shortest segments, smallest
        // blocks)
        uint64_t m = 0, tab = 0, cap = 0;
        uint32_t max_offs = 8;
        g.off.push_back(0);
        for (const Ent &e : ents) {
            const fem_job &jb = jobs[e.j];
            g.user_job.push_back(e.j);
            g.nch.push_back(e.nch);
            g.mj.push_back(jb.m);
            m += jb.m;
            g.off.push_back((uint32_t)m);
            const uint64_t Pmax = (e.nch + kBatchMinChunksPerItem - 1) / kBatchMinChunksPerItem;
            tab += (uint64_t)jb.m * Pmax * S_MAX;
            cap += (uint64_t)((jb.m + kBatchMinThreads - 1) / kBatchMinThreads) * Pmax;
            max_offs = std::max(max_offs, find_stream(c, jb.stream_id)->offs);
        }
        const uint64_t cap_r = cap, cap_x = cap;
        if (m > 0xFFFFFFF0ull || cap_r > 0xFFFFFFF0ull) return fail(FEM_ENOMEM);
        g.m = (uint32_t)m;
        g.cap_r = (uint32_t)cap_r;
        g.cap_x = (uint32_t)cap_x;
        g.SB = stage_bytes(max_offs);
        const uint32_t n = g.n_jobs;
        BRET(balloc(b, m, &g.cands));
        BRET(balloc(b, n + 1, &g.cand_off));
        BRET(balloc(b, n, &g.theta));
        BRET(balloc(b, n, &g.rjobs));
        BRET(balloc(b, n, &g.xjobs));
        BRET(balloc(b, n, &g.outs));
        BRET(balloc(b, m, &g.rel));
        BRET(balloc(b, m, &g.ex));
        BRET(balloc(b, m, &g.idx));
        BRET(balloc(b, compact_scratch_words(g.m), &g.scratch));
        BRET(balloc(b, m, &g.flags));
        BRET(balloc(b, m, &g.redo));
        BRET(balloc(b, m, &g.xredo));
        BRET(balloc(b, n + 1, &g.item_off_r));
        BRET(balloc(b, n + 1, &g.item_off_x));
        BRET(balloc(b, cap_r, &g.items_r));
        BRET(balloc(b, cap_x, &g.items_x));
        BRET(balloc(b, 8, &g.counters));
        BRET(balloc(b, tab, &g.tables));
        std::vector<CountParams> &rj = g.rj, &xj = g.xj;
        rj.resize(n);
        xj.resize(n);
        std::vector<uint32_t> th(n);
        std::vector<BatchOut> bo(n);
        for (uint32_t k = 0; k < n; ++k) {
            const fem_job &jb = jobs[ents[k].j];
            const StreamDev &s = *find_stream(c, jb.stream_id);
            BCK(cudaMemcpyAsync(g.cands + g.off[k], jb.cands, (size_t)jb.m * sizeof(fem_episode),
                                cudaMemcpyDeviceToDevice, st));
            CountParams p{};
            p.bev = s.bev;
            p.boff = s.boff;
            p.cfirst = s.cfirst;
            p.t = s.t;
            p.offs = s.offs;
            p.n_chunks = s.n_chunks;
            p.n = s.n;
            p.K = s.K;
            p.ivl = b->ivl;
            p.n_ivl = nI;
            p.err = c->d_err;  // segments and tables: batch_shape
            CountParams r = p, x = p;
            r.cands = g.cands + g.off[k];
            r.m = jb.m;
            r.out = g.rel + g.off[k];
            r.redo = g.redo + g.off[k];
            x.cands = g.cands;  // gathered through the survivor list at run time
            x.m = 0;
            x.redo = g.xredo + g.off[k];
            rj[k] = r;
            xj[k] = x;
            th[k] = jb.theta;
            bo[k] = BatchOut{jb.exact_out, jb.survived_out};
        }
        BRET(batch_shape(g, kBatchChunksPerItem, g.Tr, g.Tx, st));
        BCK(cudaMemcpyAsync(g.cand_off, g.off.data(), (n + 1) * 4, cudaMemcpyHostToDevice, st));
        BCK(cudaMemcpyAsync(g.theta, th.data(), n * 4, cudaMemcpyHostToDevice, st));
        BCK(cudaMemcpyAsync(g.outs, bo.data(), n * sizeof(BatchOut), cudaMemcpyHostToDevice, st));
        BCK(cudaStreamSynchronize(st));  // host staging vectors go out of scope
        b->groups.push_back(std::move(g));
    }
    // measured shapes when tuning is on; one eager run (sets kernel attributes, checks
    // the inputs); then capture
    if (c->tune_on && !b->over_hits) BRET(batch_tune(b, st));
    BRET(fem_batch_run(b, cuda_stream));
    BCK(cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking));
    BCK(cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
    const int rc = batch_enqueue(b, b->cap_stream);
    cudaGraph_t graph = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(b->cap_stream, &graph);
    if (rc != FEM_OK) return fail(rc);
    if (ce != cudaSuccess) return fail(FEM_ECUDA);
    b->graph = graph;
    BCK(cudaGraphInstantiate(&b->exec, graph, 0));
    size_t n_nodes = 0;
    BCK(cudaGraphGetNodes(graph, nullptr, &n_nodes));
    std::vector<cudaGraphNode_t> nodes(n_nodes);
    if (n_nodes) BCK(cudaGraphGetNodes(graph, nodes.data(), &n_nodes));
    for (cudaGraphNode_t nd : nodes) {
        cudaGraphNodeType ty;
        BCK(cudaGraphNodeGetType(nd, &ty));
        b->graph_kernels += ty == cudaGraphNodeTypeKernel;
    }
    *out = b;
    return FEM_OK;
#undef BRET
#undef BCK
}

int fem_batch_run(fem_batch *b, void *cuda_stream) {
    if (!b) return FEM_EINVAL;
    fem_ctx *c = b->ctx;
    cudaSetDevice(c->device);
    cudaStream_t st = pick(c, cuda_stream);
    CK(cudaMemsetAsync(c->d_err, 0, 4, st));
    if (b->exec) {
        CK(cudaGraphLaunch(b->exec, st));
        note_launch(b->graph_kernels);
    } else {
        RET(batch_enqueue(b, st));
    }
    uint32_t e;
    RET(read_err(c, st, &e));
    RET(err_status(e));
    if (!(e & (ERR_CAP | ERR_DENSE))) return FEM_OK;
    if (b->over_hits) {  // (more than 32 entry classes: seldom) the jobs with such candidates
        BatchHits &h = b->hits;
        std::vector<fem_interval> I(b->nI);
        std::vector<uint8_t> marks(h.n_jobs);
        if (b->nI) CK(cudaMemcpy(I.data(), b->ivl, b->nI * sizeof(uint2), cudaMemcpyDeviceToHost));
        CK(cudaMemsetAsync(h.marks, 0, h.n_jobs, st));
        CK(launch_batch_flagged_jobs(h.redo, h.xredo, h.record, h.idx, h.n_idx, h.m, h.part_off, h.n_parts,
                                     h.cand_off, h.n_jobs, h.marks, st));
        CK(cudaMemcpyAsync(marks.data(), h.marks, h.n_jobs, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        for (uint32_t k = 0; k < h.n_jobs; ++k) {
            if (!marks[k] && !(e & ERR_DENSE)) continue;
            const fem_job &jb = b->jobs[h.job[k]];
            RET(fem_count_two_pass(c, jb.stream_id, jb.cands, jb.m, 1, I.data(), b->nI, jb.theta,
                                   jb.exact_out, jb.survived_out, 1, st));
        }
        return FEM_OK;
    }
    // A capacity guard tripped somewhere: recount the affected jobs one at a time
    // with the single-recording path, which widens rings as needed.
    std::vector<fem_interval> I(b->nI);
    if (b->nI) CK(cudaMemcpy(I.data(), b->ivl, b->nI * sizeof(uint2), cudaMemcpyDeviceToHost));
    for (BatchGroup &g : b->groups) {
        std::vector<uint8_t> r(g.m), x(g.m);
        CK(cudaMemcpy(r.data(), g.redo, g.m, cudaMemcpyDeviceToHost));
        CK(cudaMemcpy(x.data(), g.xredo, g.m, cudaMemcpyDeviceToHost));
        for (uint32_t k = 0; k < g.n_jobs; ++k) {
            bool hit = false;
            for (uint32_t i = g.off[k]; i < g.off[k + 1] && !hit; ++i) hit = r[i] || x[i];
            if (!hit) continue;
            const fem_job &jb = b->jobs[g.user_job[k]];
            RET(fem_count_two_pass(c, jb.stream_id, jb.cands, jb.m, 1, I.data(), b->nI, jb.theta,
                                   jb.exact_out, jb.survived_out, 1, st));
        }
    }
    return FEM_OK;
}

int fem_batch_destroy(fem_batch *b) {
    if (!b) return FEM_EINVAL;
    cudaSetDevice(b->ctx->device);
    cudaDeviceSynchronize();
    batch_free(b);
    return FEM_OK;
}

}  // extern "C"
