/*
 * fem.h -- C ABI of libfem.so: frequent serial-episode counting and level-wise
 * mining on one NVIDIA GB300 (sm_103a).
 *
 * Method: Cao, Patnaik, Ponce, Archuleta, Butler, Feng, Ramakrishnan,
 * "Towards Chip-on-Chip Neuroscience: Fast Mining of Frequent Episodes Using
 * Graphics Processors" (arXiv 0905.2200).
 *
 * Conventions for every entry point
 *   - Return value: FEM_OK (0) or a negative fem_status.  No C++ exception
 *     crosses this boundary.  fem_strerror() names a status.
 *   - Pointers flagged "device" must be CUDA device pointers of the context's
 *     device; all others are host pointers.  Host inputs are copied before the
 *     call returns (or before the copy's stream position, for async calls);
 *     the caller keeps ownership of every buffer it passes.
 *   - cuda_stream is a cudaStream_t (NULL = the context's own stream).  Calls
 *     that write host outputs synchronise with that stream before returning.
 *     Calls whose outputs are all on the device are asynchronous.
 *   - A context is bound to one device and must not be used from two host
 *     threads at once.
 *   - Times are unsigned 32-bit microseconds; event types are 8-bit.
 */
#ifndef FEM_H
#define FEM_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

#define FEM_MAX_LEN 8        /* longest episode (nodes) */
#define FEM_MAX_TYPES 256    /* event types are uint8 */
#define FEM_MAX_INTERVALS 255

typedef enum {
    FEM_OK = 0,
    FEM_EINVAL = -1,     /* bad argument: size, NULL, lo >= hi, length out of 1..8, ... */
    FEM_EUNSORTED = -2,  /* stream times decrease somewhere */
    FEM_ETYPE = -3,      /* an event or episode type is >= n_types */
    FEM_ERANGE = -4,     /* t_max + max hi does not fit in 32 bits */
    FEM_ENOMEM = -5,     /* device or host allocation failed */
    FEM_EADMIT = -6,     /* serving: request not admitted (memory or slots) */
    FEM_ETIMEOUT = -7,   /* a bounded device wait gave up */
    FEM_ECUDA = -8,      /* a CUDA runtime call failed */
    FEM_EOVERFLOW = -9,  /* internal capacity guard tripped and could not be widened */
    FEM_ENOSTREAM = -10, /* unknown stream id */
    FEM_EIO = -11        /* a file could not be opened, read or written */
} fem_status;

/* Counting passes (Section 5.3): the relaxed upper-bound count of Algorithm 3
 * and the exact count of Algorithm 1. */
enum { FEM_PASS_RELAXED = 0, FEM_PASS_EXACT = 1 };

/* One inter-event interval (lo, hi] in microseconds (Section 2, temporal
 * constraints; Problem 1's set I).  Requires lo < hi. */
typedef struct {
    uint32_t lo_us, hi_us;
} fem_interval;

/* One serial episode (Def. 2.2 with the constraints of Problem 1), 16 bytes.
 * types[0..len-1] are the node types in order; ivl[k] (k < len-1) indexes the
 * interval table for the edge from node k to node k+1.  Unused tail bytes must
 * be 0.  Episodes generated by the miner have distinct types. */
typedef struct {
    uint8_t types[FEM_MAX_LEN];
    uint8_t ivl[FEM_MAX_LEN - 1];
    uint8_t len;
} fem_episode;

typedef struct fem_ctx fem_ctx;
typedef struct fem_result fem_result;

/* Launch-shape overrides; 0 in a field means "let the autotuner choose". */
typedef struct {
    uint32_t segments;          /* MapConcatenate segments per episode (1 = one thread per episode) */
    uint32_t threads_per_block; /* 32..256, multiple of 32 */
    uint32_t ring_capacity;     /* exact-pass list capacity per node (power of two) */
    uint32_t kernel;            /* FEM_KERNEL_AUTO, FEM_KERNEL_MACHINE or FEM_KERNEL_CHAIN */
} fem_config;
/* Counting kernels.  MACHINE: one thread per (episode, segment) runs the episode's
 * state machine over the events of its N types (the algorithms as printed).  CHAIN:
 * the same counts from the episodes' shared prefixes -- per chunk a block builds the
 * list of events each distinct prefix admits (with the start of the chain reaching
 * it), and a thread looks up only its last node's events (distinct types, lengths
 * 2..8).  PAIRS (not a configuration value): fem_count_pairs_relaxed's kernel, one
 * thread counting every interval variant of an ordered type pair from one merge of the
 * two types' events; with AUTO also fem_mine_levelwise's level-2 relaxed pass over two
 * to four intervals.  HITS (not a configuration value): tables of every edge's (type,
 * interval, next type) events with an event in the interval before them, built per slab of
 * the stream, and episodes counted over them in 64-bit words of events; with AUTO, where
 * they are estimated to be the faster way, the counts of sets that do not come in prefix
 * runs, batches, window frequencies, and the levels of fem_mine_levelwise whose work is large
 * for the stream's events times types (where a slab's words hold the events, K K n_intervals
 * <= 262,144, and the tables fit beside the stream; they have no segments or block sizes of
 * fem_config's beyond the number of segments); level 3 over 40,000 or more candidates joins them
 * all at once.  AUTO
 * otherwise: chosen by measurement when tuning is on; else CHAIN for the exact pass over
 * 256 or more candidates that come in runs of shared prefixes or over at most 64
 * candidates of three or more nodes, CHAIN for the relaxed pass over 32,768 or more such
 * candidates of three or more nodes (or at most 64), MACHINE otherwise. */
enum {
    FEM_KERNEL_AUTO = 0,
    FEM_KERNEL_MACHINE = 1,
    FEM_KERNEL_CHAIN = 2,
    FEM_KERNEL_PAIRS = 3,
    FEM_KERNEL_HITS = 4
};

/* Per-level record of the last fem_mine_levelwise call. */
typedef struct {
    uint32_t level;        /* episode length N */
    uint32_t candidates;   /* candidates counted at this level */
    uint32_t survivors;    /* candidates the exact pass counts (Algorithm 4): relaxed
                            * count >= theta, plus at level 2 the candidates whose
                            * relaxed count the pair kernel left unfinished when they
                            * are at most 1/64 of the level (their exact count decides) */
    uint32_t frequent;     /* exact count >= theta */
    uint32_t segments;     /* MapConcatenate segments used by the relaxed pass */
    float ms_generate, ms_relaxed, ms_compact, ms_exact;  /* device time per step */
    float ms_relaxed_kernel;   /* the relaxed counting kernel alone (CUDA events) */
    float ms_relaxed_stitch;   /* its MapConcatenate stitch (0 with one segment) */
    float ms_exact_kernel;     /* the exact counting kernel alone */
    uint32_t exact_segments;   /* segments used by the exact pass */
    /* (episode, event of one of its types) pairs each pass visits: the sum over
     * the counted candidates of the events of their N types (the machines' state
     * updates; the work measure of the counting kernels) */
    uint64_t touched_relaxed;
    uint64_t touched_exact;
    /* counting kernel of each pass: FEM_KERNEL_MACHINE, _CHAIN, _PAIRS or _HITS (0: none ran) */
    uint32_t kernel_relaxed, kernel_exact;
} fem_level_stats;

/* ------------------------------------------------------------------------ */
/*
 * Context.  One per device; allocates its own device working memory: resident
 * streams (about 13 bytes per event plus 2 (K + 1) bytes per chunk of 2048 events),
 * per-call working buffers (kept and reused), and batches.  mem_budget_bytes bounds
 * that memory (0: no bound).  A call that would need more first releases the hit tables
 * (FEM_KERNEL_HITS) of earlier calls and the buffers kept from freed streams, and otherwise
 * fails with FEM_ENOMEM, leaving the context usable; where the tables themselves find no
 * room, the other kernels count.  Between calls a context keeps tables of at most a 16th of
 * the device's memory (100,000 candidates on an hour of 64 types at 50 Hz: 10 GB); they are
 * given back where one of the context's own allocations or fem_server_create needs the
 * memory, and with fem_destroy.  fem_mem_usage tells what is held.  Serving (fem_server_*)
 * has its own budget in fem_server_config.
 */
int fem_create(fem_ctx **out, int device, size_t mem_budget_bytes);
/* Device bytes the context holds now (*used_out) and its budget (*budget_out, 0 = none);
 * either pointer may be NULL. */
int fem_mem_usage(fem_ctx *ctx, size_t *used_out, size_t *budget_out);
int fem_destroy(fem_ctx *ctx);
int fem_set_config(fem_ctx *ctx, const fem_config *cfg);   /* NULL restores autotuning */

/*
 * Mapping choice by measurement.  The paper picks between one thread per
 * episode and MapConcatenate with a fixed rule (Algorithm 2, crossovers of
 * Section 6.2); here every count picks its segments per episode and block size
 * from a per-context cache keyed by (N, pass, distinct types, ceil(log2 m),
 * ceil(log2 chunks), n_types).  With tuning on, a count whose class is not cached
 * first times the rule's shape and its neighbours (half and twice the segments,
 * the other block size), each a complete count with the same result, and caches
 * the fastest.  A class not cached and tuning off uses the rule.  An explicit
 * fem_set_config segment or block size overrides the cache.
 * Where the rule takes the hit tables (FEM_KERNEL_HITS; they have no shape to choose), the
 * count is timed over them and by the other kernels in their best shape, twice each, and the
 * choice is cached under "distinct" 2 for sets that do not come in prefix runs (N = 0: several
 * lengths) and 3 for fem_mine_levelwise's passes, "kernel" 4 for the tables.  A pass of
 * fem_mine_levelwise whose class has a shape but no choice (a file of an earlier version)
 * keeps that shape; other sets without a choice go by the rule.  Window frequencies are not
 * tuned; a batch is where it does not go over the tables, when it is created.
 * fem_tune_save writes the cache as JSON lines
 *   {"key": "N/pass/distinct/log2m/log2chunks/K", "segments": P, "threads": T, "ms": t,
 *    "kernel": k}
 * and fem_tune_load merges such a file (FEM_EIO: cannot open/write; FEM_EINVAL:
 * a malformed line, nothing merged).  Host only, not thread safe per context.
 */
int fem_tune_enable(fem_ctx *ctx, int on);
int fem_tune_size(fem_ctx *ctx, uint32_t *n_out);
int fem_tune_save(fem_ctx *ctx, const char *path);
int fem_tune_load(fem_ctx *ctx, const char *path);

/*
 * Event stream (Def. 2.1): n events (types[i], t_us[i]) ordered by time, ties in
 * the given order.  Validates (order, types < n_types <= 256), uploads, and
 * builds the device layouts the counters read (per-chunk type buckets).
 * types/t_us are device pointers if on_device, else host.  On success
 * *stream_id_out names the resident stream.  Errors: FEM_EINVAL, FEM_EUNSORTED,
 * FEM_ETYPE, FEM_ENOMEM, FEM_ECUDA.  Synchronous.
 */
int fem_load_stream(fem_ctx *ctx, const uint8_t *types, const uint32_t *t_us, uint64_t n,
                    uint32_t n_types, int on_device, void *cuda_stream, int32_t *stream_id_out);
/*
 * Append n events to a resident stream (Def. 2.1: the stream grows at its end, as a
 * live recording delivers it in chunks; Section 1's partitions of a live stream).
 * The new times must be >= the stream's last time and non-decreasing; types <
 * n_types.  types/t_us are device pointers if on_device, else host.  Only the last
 * partial chunk of 2048 events is regrouped; buffers grow by half when full.  The
 * type histogram (level-1 counts) is updated.  Every later count, mining call or
 * batch sees the grown stream.  On FEM_EUNSORTED or FEM_ETYPE nothing is appended.
 * Errors also: FEM_ENOSTREAM, FEM_EINVAL (n_total >= 2^32 - 16), FEM_ENOMEM
 * (budget), FEM_ECUDA.  Synchronous; work on other CUDA streams that reads this
 * stream must have completed (the last chunk is regrouped in place).
 */
int fem_append_stream(fem_ctx *ctx, int32_t stream_id, const uint8_t *types, const uint32_t *t_us,
                      uint64_t n, int on_device, void *cuda_stream);
int fem_free_stream(fem_ctx *ctx, int32_t stream_id);
/* Number of events of each type (the level-1 counts), uint32[n_types], host. */
int fem_type_counts(fem_ctx *ctx, int32_t stream_id, uint32_t *counts_out);

/*
 * Capacity table, the stream-side bound on the counters' state:
 * cap_out[a * n_widths + j] = the most events of type a inside one closed window
 * [x, x + widths_us[j]] of the stream, for every type a < n_types.  It bounds
 * Algorithm 1's lists (Section 5.1: once the entries older than hi are dropped, node
 * k holds at most cap[E_k][hi_k] events) and the entry classes of a MapConcatenate
 * segment (Section 5.2.2: at most 1 + cap[E_N][W], W the episode's sum of hi).
 * widths_us: host, 1 <= n_widths <= FEM_MAX_CAP_WIDTHS; cap_out: host,
 * uint32[n_types * n_widths].  One kernel over (chunk, type) pairs whose work grows
 * with the events inside each width (a width >= the stream's last time is answered
 * from the type counts).  Errors: FEM_EINVAL, FEM_ENOSTREAM, FEM_ENOMEM, FEM_ECUDA.
 * Synchronous.
 */
#define FEM_MAX_CAP_WIDTHS 64
int fem_capacity_table(fem_ctx *ctx, int32_t stream_id, const uint32_t *widths_us,
                       uint32_t n_widths, uint32_t *cap_out);

/*
 * Count m candidate episodes over a resident stream with one pass
 * (FEM_PASS_RELAXED: Algorithm 3, Section 5.3.1; FEM_PASS_EXACT: Algorithm 1,
 * Section 5.1).  cands: m fem_episode records (device if cands_on_device);
 * intervals: n_intervals (lo, hi] pairs, host.  counts_out: uint32[m] (device
 * if counts_on_device).  The launch shape (MapConcatenate segments per episode,
 * block size) comes from fem_set_config, the tuning cache or the occupancy rule.
 * Returns when the counts are final: the device error word is read after the
 * count, and episodes whose list rings or entry-class tables overflowed are
 * recounted with larger ones before returning.  Errors: FEM_EINVAL (bad episode,
 * len 0 or > 8, interval index out of range, lo >= hi), FEM_ETYPE, FEM_ERANGE,
 * FEM_ENOSTREAM, FEM_EOVERFLOW (still overflowing with the largest rings),
 * FEM_ETIMEOUT (a bounded device wait gave up), FEM_ECUDA.
 */
int fem_count_candidates(fem_ctx *ctx, int32_t stream_id, const fem_episode *cands, uint32_t m,
                         int cands_on_device, const fem_interval *intervals,
                         uint32_t n_intervals, int pass, uint32_t *counts_out,
                         int counts_on_device, void *cuda_stream);

/*
 * Relaxed counts (Algorithm 3, Section 5.3.1) of a complete level-2 candidate set: every
 * ordered pair (a, b) of distinct types from types[0..f) with every interval, in the
 * canonical order of fem_mine_levelwise's level 2 -- the count of (types[i], v,
 * types[j]) at counts_out[i * n_intervals * (f - 1) + v * (f - 1) + (j < i ? j : j - 1)]
 * (host, uint32[f (f - 1) n_intervals]).  One thread counts every interval variant of
 * a pair from one merge of the two types' events (FEM_KERNEL_PAIRS; n_intervals <= 4),
 * with MapConcatenate segments as configured or by the occupancy rule; episodes whose
 * entry-class tables (four per variant) overflowed are recounted before returning.  types: host, distinct, each < the
 * stream's n_types, 2 <= f <= 256.  Errors: FEM_EINVAL, FEM_ENOSTREAM, FEM_ERANGE,
 * FEM_EOVERFLOW, FEM_ETIMEOUT, FEM_ECUDA.  Synchronous.
 */
int fem_count_pairs_relaxed(fem_ctx *ctx, int32_t stream_id, const uint8_t *types, uint32_t f,
                            const fem_interval *intervals, uint32_t n_intervals,
                            uint32_t *counts_out);

/*
 * Two-pass elimination, Algorithm 4 (Section 5.3.2): relaxed count of every
 * candidate, drop those below theta, exact count of the rest.  exact_out[c] is
 * the exact count of candidate c if it survived, else 0; survived_out[c] is 1
 * or 0 (either may be NULL).  Outputs are device pointers if outs_on_device.
 */
int fem_count_two_pass(fem_ctx *ctx, int32_t stream_id, const fem_episode *cands, uint32_t m,
                       int cands_on_device, const fem_interval *intervals,
                       uint32_t n_intervals, uint32_t theta, uint32_t *exact_out,
                       uint8_t *survived_out, int outs_on_device, void *cuda_stream);

/*
 * Problem 1 (Section 2): every serial episode of 2..max_len distinct-type nodes
 * with edges from `intervals` whose non-overlapped count is >= theta, found
 * level by level (Section 5): level-2 candidates are all ordered pairs of
 * distinct frequent types times every interval; level N+1 joins level N's
 * frequent episodes (alpha without its first node == beta without its last);
 * each level is counted with Algorithm 4.  Every step runs on the device; only
 * each level's frequent set is copied to the host.  *out receives a result
 * owned by the library (free with fem_result_free).  Synchronous.
 */
int fem_mine_levelwise(fem_ctx *ctx, int32_t stream_id, const fem_interval *intervals,
                       uint32_t n_intervals, uint32_t theta, uint32_t max_len,
                       void *cuda_stream, fem_result **out);
/*
 * Level `level` (1..max_len) of a result: *m_out frequent episodes and their exact
 * counts, listed in canonical order (lexicographic on the interleaved tuple
 * E1, iv1, E2, iv2, ..., E_N).  Level 1 lists the frequent types as 1-node
 * episodes with their event counts.  Pointers stay valid until fem_result_free.
 */
int fem_result_level(const fem_result *res, uint32_t level, uint32_t *m_out,
                     const fem_episode **episodes, const uint32_t **counts);
uint32_t fem_result_max_level(const fem_result *res);
void fem_result_free(fem_result *res);
/*
 * Batched two-pass counting: many recordings, each with its own candidate set,
 * counted together.  Jobs of one episode length share one persistent launch per
 * pass (a device queue of (job, episode tile, segment) items, longest first);
 * the whole sequence (relaxed pass, per-job elimination at the job's theta,
 * exact pass on the survivors, scatter) runs without a host round trip and is
 * captured once in a CUDA graph that fem_batch_run replays.  Where that is estimated to be
 * faster, all lengths go over hit tables (FEM_KERNEL_HITS), built in every run.  Same results
 * as fem_count_two_pass on each job alone (Algorithm 4, Section 5.3.2).
 */
typedef struct {
    int32_t stream_id;          /* a resident stream of this context */
    uint32_t len;               /* episode length of every candidate of the job (2..8) */
    uint32_t m;                 /* number of candidates */
    const fem_episode *cands;   /* device, m records, distinct types */
    uint32_t theta;             /* elimination / frequency threshold of this job */
    uint32_t *exact_out;        /* device uint32[m]: exact count if survived, else 0 */
    uint8_t *survived_out;      /* device uint8[m]: 1 if relaxed count >= theta */
} fem_job;
typedef struct fem_batch fem_batch;

/* Builds the batch (allocates its working memory, copies the candidate records,
 * runs it once eagerly and captures the graph).  The job array is copied; the
 * candidate and output buffers must stay valid until fem_batch_destroy. */
int fem_batch_create(fem_ctx *ctx, const fem_job *jobs, uint32_t n_jobs,
                     const fem_interval *intervals, uint32_t n_intervals, void *cuda_stream,
                     fem_batch **out);
/* Replays the batch on cuda_stream (re-reading the candidate records given at
 * creation) and synchronises; outputs are then valid. */
int fem_batch_run(fem_batch *batch, void *cuda_stream);
int fem_batch_destroy(fem_batch *batch);

/*
 * Serving: near-real-time counting over streams that grow chunk by chunk (the
 * paper's "chip-on-chip" use, Section 1: partitions of a live recording processed
 * in turn), with continuous batching.  Requests are admitted while others run if
 * their device memory fits the server's budget and a slot is free (else
 * FEM_EADMIT); each admitted request's work is enqueued at once on one of the
 * server's CUDA streams, so requests overlap on the device.
 *   one-shot: Algorithm 4 over the last window_us of the stream at submission;
 *             result = exact count (0 if eliminated) and survived flag per episode.
 *   standing: exact counts (Algorithm 1) from submission on, advanced from a
 *             device-resident carried machine state whenever new events arrive;
 *             result = current counts and flag count >= theta.
 * Results are identical to counting the same event range alone.
 */
enum { FEM_REQ_ONESHOT = 0, FEM_REQ_STANDING = 1 };
typedef struct {
    size_t mem_budget_bytes;  /* device arena for admitted requests (0: 1 GiB) */
    uint32_t max_active;      /* requests active at once (0: 64) */
    uint32_t n_lanes;         /* CUDA streams requests are spread over (0: 8) */
} fem_server_config;
typedef struct fem_server fem_server;

int fem_server_create(fem_ctx *ctx, const fem_server_config *cfg, fem_server **out);
int fem_server_destroy(fem_server *srv);
/* A growing stream with room for capacity_events events. */
int fem_server_open_stream(fem_server *srv, uint32_t n_types, uint64_t capacity_events,
                           int32_t *stream_id_out);
/* Append n events (host arrays, times >= the stream's last time).  Asynchronous:
 * ordered before every later request on this stream.  Errors: FEM_EUNSORTED,
 * FEM_ETYPE (checked on the host), FEM_ENOMEM (capacity). */
int fem_server_append(fem_server *srv, int32_t stream_id, const uint8_t *types,
                      const uint32_t *t_us, uint32_t n);
/* Admit a request (candidates and intervals are host arrays, copied).  window_us
 * bounds a one-shot request's range (0: the whole stream).  *req_id_out names it. */
int fem_server_submit(fem_server *srv, int32_t stream_id, const fem_episode *cands, uint32_t m,
                      const fem_interval *intervals, uint32_t n_intervals, uint32_t theta,
                      int mode, uint32_t window_us, uint64_t *req_id_out);
/* Launch due standing updates, retire finished work; writes up to cap ids of
 * requests whose results changed since the last poll into done_ids. */
int fem_server_poll(fem_server *srv, uint64_t *done_ids, uint32_t cap, uint32_t *n_done);
/* Copy a request's latest result (host arrays of m entries; either may be NULL);
 * *events_out = number of events it covers.  Returns the request's status. */
int fem_server_result(fem_server *srv, uint64_t req_id, uint32_t *counts_out, uint8_t *flags_out,
                      uint64_t *events_out);
/* Release a request (a finished one-shot, or stop a standing one). */
int fem_server_release(fem_server *srv, uint64_t req_id);
/* Block until no work of the server is in flight, then poll. */
int fem_server_drain(fem_server *srv);

/*
 * MapConcatenate as Section 5.2.2 prints it, for comparison with the exact
 * counts of fem_count_candidates(FEM_PASS_EXACT) (same inputs and conventions).
 * The stream is cut in time at the first event of every ceil(n_chunks /
 * segments)-th chunk of 2048 events: tau[0] = t[0] - 1, tau[p] = (time of that
 * event) - 1 where that is above tau[p-1] and below t[n-1], tau[P] = t[n-1];
 * segment p holds the events with tau[p] < t <= tau[p+1].  Per segment, machine
 * k (0 <= k < N) runs Algorithm 1 on the events with t > tau[p] - (hi_1 + ... +
 * hi_k), counts its completions inside the segment, and records a (end time of
 * its first completion before tau[p] + W, W = sum of hi) and b (end time of the
 * completion of a partial occurrence it carries past tau[p+1], before
 * tau[p+1] + W; it starts no new one there).  Counts are the sums along the
 * chain of tuples joined where b equals a, from machine 0 of segment 0; where
 * several tuples match, the smallest k is taken, where none does, k = 0.  The
 * printed scheme can undercount (occurrences over more than two segments, an
 * occurrence ending exactly at tau + W, machines out of step with the serial
 * machine); the exact counts never differ from Algorithm 1.
 * diag_out (host uint32[2], may be NULL): boundaries, summed over candidates,
 * where no tuple matched / several did.  Candidates must have distinct types
 * (FEM_EINVAL otherwise); FEM_EOVERFLOW if a list outgrew 16 clusters.
 * Synchronous.
 */
int fem_count_mapconcat_literal(fem_ctx *ctx, int32_t stream_id, const fem_episode *cands,
                                uint32_t m, int cands_on_device, const fem_interval *intervals,
                                uint32_t n_intervals, uint32_t segments, uint32_t *counts_out,
                                int counts_on_device, uint32_t *diag_out, void *cuda_stream);

/*
 * fem_mine_levelwise with options.  FEM_MINE_REPEATED_TYPES: a type may appear at
 * several nodes of an episode (A -> B -> A; the paper's episodes are sets of types
 * and its future work names repeats): level 2 includes the pairs (a, a) and the
 * join keeps children whose new type already occurs (dropping the first or last
 * node of any episode cannot lower its count, so the level-wise search stays
 * complete).  Repeated-type episodes are counted with the node loop from last to
 * first (as Algorithms 1 and 3 print it) and one segment per episode.  Other flag
 * bits: FEM_EINVAL.
 */
#define FEM_MINE_REPEATED_TYPES 1u
int fem_mine_levelwise_ex(fem_ctx *ctx, int32_t stream_id, const fem_interval *intervals,
                          uint32_t n_intervals, uint32_t theta, uint32_t max_len, uint32_t flags,
                          void *cuda_stream, fem_result **out);

/*
 * Window-based frequency (the alternative measure Section 2 names, after Mannila
 * et al.), with each edge's interval constraint: counts_out[i] = the number of
 * integer window starts s (microseconds) such that the window [s, s + window_us)
 * holds every event of some occurrence of candidate i (first event at or after s,
 * last event before s + window_us).  Divide by (t[n-1] - t[0] + window_us) for the
 * fraction of windows.  One thread per episode, or per episode and segment over hit
 * tables (FEM_KERNEL_HITS); candidates must have distinct types (FEM_EINVAL otherwise);
 * window_us > 0.  counts_out: uint64[m], device if counts_on_device.  FEM_EOVERFLOW if an
 * edge held more than 32 pending entries where the tables do not apply.
 */
int fem_count_windows(fem_ctx *ctx, int32_t stream_id, const fem_episode *cands, uint32_t m,
                      int cands_on_device, const fem_interval *intervals, uint32_t n_intervals,
                      uint32_t window_us, uint64_t *counts_out, int counts_on_device,
                      void *cuda_stream);

/* Per-level statistics of the last fem_mine_levelwise call on this context;
 * returns the number of records written (at most cap). */
int fem_last_mine_stats(fem_ctx *ctx, fem_level_stats *out, uint32_t cap);

/*
 * Survivor selection that allocates nothing (the paper has no counterpart; it is
 * an interface for callers that may not call cudaMalloc, e.g. a real-time loop
 * with a fixed pre-reserved memory budget, or a thread that must not trigger the
 * implicit synchronisation of cudaMalloc/cudaFree).
 * values: device uint32[m]; idx_out: device uint32[m] receives, in increasing
 * order, every i with values[i] >= theta; count_out: device uint32 receives how
 * many.  Asynchronous on cuda_stream (NULL = legacy default stream), on the
 * current device.  Its per-block partial sums live in a fixed static device
 * array (about 256 KB, held on every GPU that loads the library until exit):
 * m > FEM_SELECT_NOALLOC_MAX returns FEM_EINVAL.  The first call on a device looks
 * up that array's address and must come before any stream capture on that
 * device.  All calls share the array, so calls that overlap on the GPU (on
 * different streams) race; serialise them.  No cudaMalloc, cudaFree or
 * allocating library routine is called.
 */
#define FEM_SELECT_NOALLOC_MAX (1u << 26)
int fem_select_noalloc(const uint32_t *values, uint32_t m, uint32_t theta, uint32_t *idx_out,
                       uint32_t *count_out, void *cuda_stream);

const char *fem_strerror(int status);
/* Number of CUDA kernels this library has launched in this process so far
 * (all contexts); a caller can difference it around a region of work. */
uint64_t fem_kernel_launches(void);

#ifdef __cplusplus
}
#endif
#endif /* FEM_H */
