/*
 * tim.h -- C ABI of libtim.so, a single-GPU (GB300, sm_103a) engine for the hot path
 * of TIM / TIM+ influence maximisation (Tang, Xiao, Shi, SIGMOD'14):
 *
 *   random RR sets by randomised reverse BFS under IC, LT and   (Section 3.1, 4.2, 6)
 *   general triggering models
 *   KptEstimation (Algorithm 2) and RefineKPT (Algorithm 3)     (Sections 3.2, 4.1)
 *   greedy maximum coverage node selection (Algorithm 1)        (Section 3.1)
 *
 * Conventions shared by every call
 *   - Every call returns an int status: TIM_OK (0) or a negative TIM_ERR_* code;
 *     tim_strerror() names it and tim_last_error_message() gives detail for the
 *     context's last failing call. A failing call leaves previously loaded state
 *     usable unless stated.
 *   - Pointers named host_* or documented as host memory are read/written with
 *     synchronous copies before the call returns; the caller keeps ownership. Pointers
 *     documented as device memory must be allocations on the context's device; the
 *     library reads them on the context's stream and never frees them.
 *   - The context owns every device buffer it allocates (graph, RR-set store, index,
 *     scratch) and frees them in tim_destroy. All work is ordered on one CUDA stream:
 *     the one passed to tim_create, or a stream the context creates when NULL.
 *   - Node ids are int32 in [0, n); n >= 2, m < 2^32. Graphs are directed, without
 *     self-loops or duplicate edges (rejected with TIM_ERR_ARG).
 *   - Randomness is counter-based: every RR set is a pure function of (seed, set id),
 *     so results do not depend on launch shapes, scheduling or the GPU.
 *     Set ids: sid = (phase << 56) | (round << 48) | j with phase 1 = KptEstimation
 *     round `round`, 2 = RefineKPT's theta' sets, 3 = NodeSelection; tim_sample_rr
 *     takes the first id from the caller.
 *   - Not thread-safe per context: one host thread at a time per tim_ctx.
 */
#ifndef TIM_H
#define TIM_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

#define TIM_OK 0
#define TIM_ERR_ARG (-1)      /* invalid argument or graph */
#define TIM_ERR_OOM (-2)      /* device allocation failed */
#define TIM_ERR_OVERFLOW (-3) /* an output buffer given by the caller is too small */
#define TIM_ERR_TIMEOUT (-4)  /* a bounded device wait gave up */
#define TIM_ERR_CUDA (-5)     /* a CUDA runtime call failed */
#define TIM_ERR_STATE (-6)    /* call out of order (e.g. no graph loaded) */

#define TIM_IC 0 /* independent cascade, Section 2.1 */
#define TIM_LT 1 /* linear threshold, Section 6 (triggering model of Section 4.2) */
#define TIM_TRIG 2 /* a general triggering model, Section 4.2 (tim_load_graph_triggering) */

typedef struct tim_ctx tim_ctx;

/* Per-run report of tim_run / tim_run_tim. Times are device times (CUDA events). */
typedef struct tim_stats {
    int kpt_round;            /* round of Algorithm 2 that stopped; 0 = none (KPT* = 1) */
    int kpt_last_round;       /* round whose RR sets form R' of Algorithm 3 */
    double kpt_star;          /* Algorithm 2 output */
    double kpt_prime;         /* KPT' of Algorithm 3 (0 for plain TIM) */
    double kpt_plus;          /* Algorithm 3 output (= kpt_star for plain TIM) */
    double eps_prime;         /* Section 4.1 (0 for plain TIM) */
    double lambda;            /* Eq. 4 */
    uint64_t theta_prime;     /* theta' of Algorithm 3 (0 for plain TIM) */
    uint64_t covered_prime;   /* RR sets of Algorithm 3's theta' covered by S'_k */
    uint64_t theta;           /* RR sets of Algorithm 1 */
    uint64_t covered;         /* of those, covered by the returned seeds */
    uint64_t sets_total;      /* RR sets generated by the call, all phases */
    uint64_t members_select;  /* sum |R| over Algorithm 1's sets */
    uint64_t width_total;     /* sum of w(R) (Eq. 1) over the sets of Algorithms 1 and 2
                                 (Algorithm 3's coverage test stops a set at its first
                                 seed, so those sets have no width) */
    uint64_t width_select;    /* sum of w(R) over Algorithm 1's sets */
    double ms_kpt;            /* Algorithm 2 */
    double ms_refine;         /* Algorithm 3 */
    double ms_select_sample;  /* Algorithm 1, sampling */
    double ms_select_greedy;  /* Algorithm 1, selection (index build + k rounds) */
    double ms_total;
    uint64_t kpt_sets;        /* RR sets Algorithm 2 generated (learned start included) */
    int kpt_predicted_round;  /* learned start round i0; 0 when no predictor was used */
    int kpt_accepted;         /* 1: the start round was accepted; 0: plain sweep ran */
} tim_stats;

/* Device-time account of the RR sampler, accumulated over every sampling call of a
 * context (Algorithms 1-3 all sample through it). Pass 1: one warp per set, shared
 * memory, IC in-edge budget. Pass 2: one warp per set with a larger queue in global
 * memory, for the sets pass 1 gave up on. Pass 3: the sets beyond pass 2's queue
 * (IC: batched level-synchronous BFS; LT: chain walk with a visited bitmap; triggering
 * models: one block per set, level by level, with a visited bitmap).
 * width = sum of w(R) (Eq. 1) over completed sets, live = live in-edges followed,
 * members = sum of |R| of completed sets, examined = IC in-edges examined: every
 * in-edge of a list outside the geometric-skip rule plus the live in-edges the rule
 * finds (not counted in pass 3). Times come from CUDA events recorded around each
 * pass. */
typedef struct tim_profile {
    uint64_t pass1_launches;
    double pass1_ms;
    uint64_t pass1_sets, pass1_width, pass1_live, pass1_members;
    uint64_t pass2_launches;
    double pass2_ms;
    uint64_t pass2_sets, pass2_width, pass2_live, pass2_members;
    uint64_t pass3_launches;
    double pass3_ms;
    uint64_t pass3_sets, pass3_width, pass3_live, pass3_members;
    uint64_t pass1_examined, pass2_examined, pass3_examined;
    /* heavy-set pass, persistent launch: batches, BFS levels, and block 0's time in the
     * group-count and offset phases, in the expand phase, and waiting at barriers */
    uint64_t pass3_batches, pass3_levels;
    double pass3_ms_offsets, pass3_ms_expand, pass3_ms_wait;
    double pass3_ms_kernel;  /* device time of the persistent launches alone (events) */
} tim_profile;

/* Create a context on CUDA device `device`. `cuda_stream` is a cudaStream_t (may be
 * NULL: the context then creates and owns a non-blocking stream, which is not ordered
 * against the legacy default stream; pass cudaStreamLegacy to run on that stream). */
int tim_create(tim_ctx** out, int device, void* cuda_stream);

/* Free every device buffer of the context and the context itself. NULL is a no-op. */
int tim_destroy(tim_ctx* ctx);

/* Static name of a status code. */
const char* tim_strerror(int code);

/* Detail of the context's last failing call (static storage inside the context). */
const char* tim_last_error_message(tim_ctx* ctx);

/* Load G and its diffusion model (Section 2.1 / Section 6), replacing any previous
 * graph and RR-set store. Builds G^T (Table 1) on the device: the in-CSR with the
 * in-edges of each node ascending by source, and per-edge thresholds.
 *   n           number of nodes, >= 2
 *   m           number of edges, 0 <= m < 2^32
 *   out_rowptr  host int64[n+1], out-edge offsets of G (rowptr[0] = 0, rowptr[n] = m)
 *   out_dst     host int32[m], destination of each edge
 *   edge_w      host float32[m]: IC p(e) in [0, 1]; LT in-weight b(e) in [0, 1] with
 *               the weights into every node summing to at most 1 (+1e-5)
 *   model       TIM_IC or TIM_LT
 * The arrays are copied to device buffers that the context keeps for the next load
 * (freed by tim_destroy), then read as by tim_load_graph_device; the host arrays may be
 * reused when the call returns.
 * Errors: TIM_ERR_ARG for an invalid graph or weights, TIM_ERR_OOM, TIM_ERR_CUDA. */
int tim_load_graph(tim_ctx* ctx, int64_t n, int64_t m, const int64_t* out_rowptr,
                   const int32_t* out_dst, const float* edge_w, int model);

/* Same as tim_load_graph, but the three arrays are device memory on the context's
 * device, read on the context's stream (work that writes them on another stream must
 * be complete, or ordered before the call); not retained after the call. */
int tim_load_graph_device(tim_ctx* ctx, int64_t n, int64_t m, const int64_t* d_out_rowptr,
                          const int32_t* d_out_dst, const float* d_edge_w, int model);

/* Load G under a general triggering model (Section 4.2): every node v has a
 * distribution over subsets of its in-edges (its options), each taken with its
 * probability, none with the remainder. A node reached by an RR set's BFS picks the
 * first option whose inclusive cumulative threshold sum floor(p * 2^32) (saturated at
 * 2^32 - 1) exceeds word 0 of Philox(seed; set id, v, TAG_LT) -- the LT draw, so the LT
 * model written as singleton options gives LT's sets -- and the BFS follows the
 * option's in-edges. All arrays are host memory, not retained:
 *   n, m, out_rowptr, out_dst   G as for tim_load_graph
 *   opt_rowptr       int64[n+1]: node v's options are opt_rowptr[v] .. opt_rowptr[v+1]
 *   opt_prob         float32[n_opts], n_opts = opt_rowptr[n]: probability of each option,
 *                    in [0, 1], summing to at most 1 (+1e-5) per node
 *   opt_edge_rowptr  int64[n_opts+1]: option o lists opt_edges[opt_edge_rowptr[o] ..
 *                    opt_edge_rowptr[o+1])
 *   opt_edges        int64[]: out-CSR edge ids (indices into out_dst) that end in the
 *                    option's node, each at most once per option
 * RR sampling, Algorithms 1-3 (tim_run, tim_run_tim, the stepwise calls),
 * tim_run_sharded and tim_spread_mc take such a graph; tim_run_batch and the learned
 * start round answer TIM_ERR_ARG. tim_get_graph reports thr as 0. Errors: TIM_ERR_ARG
 * for an invalid graph or distribution, TIM_ERR_OOM, TIM_ERR_CUDA. */
int tim_load_graph_triggering(tim_ctx* ctx, int64_t n, int64_t m, const int64_t* out_rowptr,
                              const int32_t* out_dst, const int64_t* opt_rowptr,
                              const float* opt_prob, const int64_t* opt_edge_rowptr,
                              const int64_t* opt_edges);

/* Copy G^T of the loaded graph (Table 1) to host memory: rowptr[n+1] (in-list of v at
 * rowptr[v] .. rowptr[v+1]), src[m] (sources, ascending within each in-list) and thr[m]
 * (IC: live iff a coin word < thr, 0xFFFFFFFF = always live; LT: inclusive prefix of
 * floor(b * 2^32) over the in-list, saturated). Any output may be NULL. Errors:
 * TIM_ERR_STATE without a graph. */
int tim_get_graph(tim_ctx* ctx, uint64_t* rowptr, uint32_t* src, uint32_t* thr);

/* Generate RR sets with ids first_set_id + j, j in [0, theta) (the sampling step of
 * Algorithm 1, Section 3.1 "Implementation"; Section 4.2 for LT) into the context's RR-set store,
 * replacing its previous contents. *total_members (may be NULL) receives sum |R|.
 * theta = 0 empties the store. Errors: TIM_ERR_STATE without a graph, TIM_ERR_OOM. */
int tim_sample_rr(tim_ctx* ctx, uint64_t theta, uint64_t seed, uint64_t first_set_id,
                  uint64_t* total_members);

/* Copy the RR-set store to the host as a CSR of sets in set-id order:
 *   off     host int64[theta+1]
 *   mem     host int32[mem_cap]; the members of set j are mem[off[j] .. off[j+1]),
 *           in no particular order
 *   widths  host int64[theta] (may be NULL): w(R) of each set (Eq. 1)
 * TIM_ERR_OVERFLOW if mem_cap < sum |R| (off is still filled). */
int tim_get_rr(tim_ctx* ctx, int64_t* off, int32_t* mem, uint64_t mem_cap, int64_t* widths);

/* Number of RR sets in the store and sum |R|. */
int tim_rr_size(tim_ctx* ctx, uint64_t* n_sets, uint64_t* total_members);

/* Sum of kappa(R) = 1 - (1 - w(R)/m)^k (Eq. 6) over RR sets first_set_id + j,
 * j in [0, count), in 2^-63 fixed point: each kappa is evaluated in FP64 as
 * (w/m) * sum_{i<k} (1 - w/m)^i and truncated once; the 128-bit total is exact and
 * returned as (*sum_hi << 64) | *sum_lo. *width_sum (may be NULL) = sum of w(R).
 * This is one round's sum in Algorithm 2; the sets are not stored. */
int tim_kappa_sum(tim_ctx* ctx, int k, uint64_t seed, uint64_t first_set_id, uint64_t count,
                  uint64_t* sum_hi, uint64_t* sum_lo, uint64_t* width_sum);

/* Algorithm 2 (KptEstimation): rounds i = 1 .. floor(log2 n) - 1 with
 * c_i = ceil((6 l ln n + 6 ln log2 n) 2^i) fresh RR sets each (Eq. 7); stops at the
 * first round whose kappa mean exceeds 2^-i and returns KPT* = n sum / (2 c_i), else
 * KPT* = 1 (*round = 0). The stop test compares the exact fixed-point sum in
 * integers. The last round's RR sets stay in the store (R' of Algorithm 3). */
int tim_kpt_estimate(tim_ctx* ctx, int k, double ell, uint64_t seed, double* kpt_star,
                     int* round);

/* Algorithm 3 (RefineKPT) after tim_kpt_estimate on the same context: greedy on R',
 * eps' = 5 (l eps^2 / (k + l))^(1/3) (Section 4.1), theta' = ceil(lambda' / KPT*)
 * fresh RR sets, f = covered fraction, KPT' = f n / (1 + eps'), KPT+ = max(KPT', KPT*).
 * Outputs may be NULL. TIM_ERR_STATE without a preceding tim_kpt_estimate. */
int tim_refine_kpt(tim_ctx* ctx, int k, double ell, double eps, uint64_t seed,
                   double* kpt_plus, double* eps_prime, uint64_t* theta_prime);

/* The selection of Algorithm 1 on the RR-set store: k greedy rounds, each picking the node
 * that covers the most uncovered sets (ties: smallest id; chosen nodes excluded) and
 * removing the sets it covers.
 *   seeds              host int32[k]
 *   covered_fraction   F_R(S_k) (may be NULL)
 *   covered_count      number of covered sets (may be NULL)
 * 1 <= k <= n. */
int tim_node_select(tim_ctx* ctx, int k, int32_t* seeds, double* covered_fraction,
                    uint64_t* covered_count);

/* Coverage count of every node over the RR-set store (the first greedy round's
 * counts): host int32[n]. */
int tim_coverage_counts(tim_ctx* ctx, int32_t* counts);

/* The greedy of Algorithm 1 one step at a time, with the node of each step chosen by
 * the caller (for example from counts summed over the stores of several contexts):
 * tim_select_begin builds the node -> RR-set index of the store and marks every set
 * uncovered; tim_select_counts copies the current coverage count of every node (host
 * int32[n]: the sets that contain it and are not covered yet); tim_select_take covers
 * the sets that contain `node` and lowers the counts of their members accordingly,
 * *newly_covered (may be NULL) = sets covered by this step. Sampling into the store or
 * loading a graph ends the open selection (TIM_ERR_STATE until the next begin). */
int tim_select_begin(tim_ctx* ctx);
int tim_select_counts(tim_ctx* ctx, int32_t* counts);
int tim_select_take(tim_ctx* ctx, int32_t node, uint64_t* newly_covered);

/* All-reduce supplied by the caller for tim_run_sharded: replace data[0 .. count) by its
 * element-wise sum over all ranks (every rank calls it with the same count, in the same
 * order). Return 0 on success. */
typedef int (*tim_allreduce_fn)(void* user, int64_t* data, uint64_t count);

/* TIM+ (Section 4.1) for one query split over `world` ranks by set id: every rank has
 * the same graph loaded and generates only its share [c r / W, c (r+1) / W) of each
 * phase's c RR sets (RR sets are independent given their ids, Section 3). Per round of
 * Algorithm 2 the exact 2^-63 fixed-point kappa sum is all-reduced (four 32-bit limbs);
 * Algorithm 3 all-reduces the covered count of its theta' sets; in both greedy
 * selections (on R' and on the theta sets) each round all-reduces the n coverage
 * counts and every rank covers the chosen node in its own store. Seeds, KPT*, KPT+,
 * theta and the covered count equal tim_run's on one context with the same seed and
 * tag. stats->sets_total counts all ranks' sets; the phase times are not filled
 * (ms_total is this rank's wall time). */
int tim_run_sharded(tim_ctx* ctx, int k, double eps, double ell, uint64_t seed, int rank,
                    int world, tim_allreduce_fn allreduce, void* user, int32_t* seeds,
                    double* covered_fraction, tim_stats* stats);

/* Number of RR sets first_set_id + j, j in [0, count), that contain at least one of
 * the host int32[n_seeds] nodes (the coverage test of Algorithm 3). Sets are not stored. */
int tim_covered_count(tim_ctx* ctx, const int32_t* seeds, int n_seeds, uint64_t seed,
                      uint64_t first_set_id, uint64_t count, uint64_t* covered);

/* TIM+ end to end (Section 4.1): Algorithm 2 -> Algorithm 3 -> theta = ceil(lambda /
 * KPT+) with lambda of Eq. 4 -> Algorithm 1. seeds: host int32[k]; covered_fraction
 * and stats may be NULL. theta_override > 0 replaces the computed theta. */
int tim_run(tim_ctx* ctx, int k, double eps, double ell, uint64_t seed, int32_t* seeds,
            double* covered_fraction, tim_stats* stats, uint64_t theta_override);

/* Plain TIM (Section 3.3): Algorithm 2 -> theta = ceil(lambda / KPT*) -> Algorithm 1. */
int tim_run_tim(tim_ctx* ctx, int k, double eps, double ell, uint64_t seed, int32_t* seeds,
                double* covered_fraction, tim_stats* stats);

/* IC sampler tuning: pass 1 (one warp per RR set, shared memory) hands a set to pass 2
 * once the in-edges it would examine exceed `budget` (default 16384). 0 sends every
 * set that has in-edges to pass 2. Results do not change. */
int tim_set_width_budget(tim_ctx* ctx, uint64_t budget);

/* Set-id tag of the context's runs (tim_kpt_estimate, tim_refine_kpt, tim_run,
 * tim_run_tim): set ids become (phase << 56) | (round << 48) | (tag << 32) | j, so
 * queries that share a seed draw independent RR sets. Default 0; tag < 65536. */
int tim_set_query_tag(tim_ctx* ctx, uint32_t tag);

/* Sampler tuning: RR sets a warp (or team) claims per work-counter increment, 1..64
 * (default 2). Results do not change. */
int tim_set_chunk(tim_ctx* ctx, int sets);

/* IC sampler tuning: warps that expand one RR set together in pass 2 (1, 2, 4 or 8;
 * 0 = chosen per call from the number of sets pass 1 handed over). Results do not
 * change. */
int tim_set_team_size(tim_ctx* ctx, int warps);

/* IC sampler tuning: the rule that chooses pass 2's warps per set when team_size is 0
 * takes the smallest T in {1, 2, 4, 8} with listed * factor >= resident warps / T
 * (listed = sets pass 1 handed over); factor in [1, 64], default 2. Results do not
 * change. */
int tim_set_team_factor(tim_ctx* ctx, int factor);

/* IC sampler tuning: pass 1's queue capacity per RR set, 128, 256 (default) or 512
 * members per warp, of which each of its eight sets has an eighth (the visited hash has
 * twice as many slots; both sit in shared memory); in a call of no more sets than warps a
 * set has 16 members whatever the capacity. Larger sets move on to pass 2. Results do not
 * change. */
int tim_set_pass1_capacity(tim_ctx* ctx, int members);

/* IC sampler tuning: pass 2 (a team of warps per RR set, queue of 8192 members) hands a
 * set to the heavy-set pass, whose warps spread each in-list over the whole GPU, once
 * the in-edges the team would examine exceed `budget` (default 2^64 - 1). Sets that outgrow
 * the queue, or whose coins in long in-lists (512 in-edges or more, outside the
 * geometric-skip rule) would pass a number that depends on the call's sets and the graph's
 * edges, go there whatever the budget. Results do not change. */
int tim_set_pass2_budget(tim_ctx* ctx, uint64_t budget);

/* Polls a block makes at a grid barrier of a persistent kernel (the heavy-set pass of
 * the IC sampler, the greedy of Algorithm 1) before it gives up; default 2^24 (about a
 * second). A training run waits at least the default. When one block gives up, every block
 * of the launch stops and the call returns TIM_ERR_TIMEOUT; the context stays usable.
 * Results do not change. */
int tim_set_wait_limit(tim_ctx* ctx, uint32_t polls);

/* Device memory that the context's buffers may take in all (default: no limit); an
 * allocation beyond it fails as one that the device has no room for: TIM_ERR_OOM, after
 * which the context stays usable (a call that was storing RR sets leaves an empty store).
 * tim_memory_held: the bytes they take now. */
int tim_set_memory_limit(tim_ctx* ctx, uint64_t bytes);
uint64_t tim_memory_held(tim_ctx* ctx);

/* IC sampler: stepped = 0 (default) runs the levels of the heavy-set pass (sets beyond
 * pass 2's capacity) in one persistent launch per batch; stepped = 1 steps them from the
 * host, a launch sequence per level. Results do not change. */
int tim_set_heavy_pass(tim_ctx* ctx, int stepped);

/* Result of tim_autotune. */
typedef struct tim_tuning {
    uint64_t width_budget;  /* chosen pass-1 in-edge budget (IC) */
    int team_size;          /* pass-2 warps per set: 0 = chosen per call (the rule below) */
    int chunk;              /* chosen sets per work claim */
    int trials;             /* settings timed */
    double best_ms;         /* calibration time of the chosen setting */
    double default_ms;      /* calibration time of the defaults (16384, 2, factor 2, 256) */
    int team_factor;        /* chosen factor of the pass-2 team-size rule (IC) */
    int pass1_capacity;     /* chosen pass-1 queue capacity in members (IC) */
} tim_tuning;

/* Choose the sampler settings for the loaded graph by timing tim_sample_rr of
 * `sample_sets` RR sets (set ids of phase 4, so no algorithm's sets are reused) and
 * keeping the fastest: first the pass-1 in-edge budget (IC: 512 .. 16384) with the sets
 * per work claim (1, 2, 4); then, for IC, the factor of the pass-2 team-size rule (1, 2,
 * 4, 8: the warps per set stay chosen per call from the number of sets pass 1 hands
 * over) and the pass-1 queue capacity (128, 256, 512 members). 20 settings for IC, 3
 * for LT; the context keeps the winner. The settings never change results, only
 * speed. The RR-set store is left holding the last calibration sample. */
int tim_autotune(tim_ctx* ctx, uint64_t sample_sets, uint64_t seed, tim_tuning* out);

/* Copy the sampler account into *out; reset != 0 zeroes it afterwards. */
int tim_get_profile(tim_ctx* ctx, tim_profile* out, int reset);

/* Greedy node selection that allocates nothing. The paper has no counterpart: this is
 * the greedy of tim_node_select (k rounds of "take the node that covers the most
 * uncovered RR sets, ties to the smallest id") for callers that cannot let the
 * library allocate device memory -- code whose device memory belongs to another
 * allocator or a fixed budget, and code that must not trigger the device-wide
 * synchronisation of cudaMalloc/cudaFree. It needs no context and no loaded graph.
 *   device      CUDA device of all pointers
 *   cuda_stream cudaStream_t to run on (NULL: the default stream)
 *   n           number of nodes, 1 <= n <= 262144
 *   n_sets      number of RR sets, <= 1048576
 *   d_off       device int64[n_sets + 1], d_off[0] = 0, d_off[n_sets] <= 2097152
 *   d_mem       device int32[d_off[n_sets]]: members of set j at d_off[j] .. d_off[j+1],
 *               distinct within a set, in [0, n) (a member listed twice in one set is
 *               not detected: the seeds and the covered count are then undefined)
 *   k           1 <= k <= min(n, 1024)
 *   d_seeds     device int32[k] (output)
 *   d_covered   device uint64[1] (output): number of sets the seeds cover
 * Returns TIM_ERR_ARG, without running anything, for sizes beyond these limits, and
 * after the run if a member or an offset was out of range; TIM_ERR_TIMEOUT if the blocks
 * of its one cooperative launch waited too long for each other. That launch starts when all
 * of its blocks (at most one per SM, 512 threads and 33 KB of shared memory each) find room at
 * once: beside other streams' kernels that fill every SM it waits for theirs to end (an
 * 8192^3 GEMM after another beside it: 1.2 ms instead of 0.7). Every call copies d_off[0]
 * and d_off[n_sets] to the host and waits for the stream before its kernels, and
 * waits again before it returns. Scratch is one __device__ array of about 13.3 MiB
 * that every GPU holds once the library is loaded; the first call on a device also
 * looks up the array's device address, so make that first call before any stream
 * capture. All calls share the array: calls that overlap on the GPU race. */
int tim_node_select_noalloc(int device, void* cuda_stream, int64_t n, uint64_t n_sets,
                            const int64_t* d_off, const int32_t* d_mem, int k,
                            int32_t* d_seeds, uint64_t* d_covered);

/* One query of a batch: a context holding the query's graph (one context per query,
 * all on one device), its parameters, and its outputs. */
typedef struct tim_query {
    tim_ctx* ctx;
    int k;
    double eps, ell;
    uint32_t tag;             /* set-id tag, distinct per query; < 65536 */
    int32_t* seeds;           /* host int32[k], output */
    double covered_fraction;  /* output */
    tim_stats stats;          /* output; the phase times of a batch are in tim_batch_stats */
} tim_query;

typedef struct tim_batch_stats {
    int queries;
    int kpt_launch_rounds;    /* multi-query launches of Algorithm 2 */
    uint64_t sets_total;      /* RR sets of all queries, all phases */
    double ms_kpt, ms_refine, ms_select_sample, ms_select_greedy, ms_total;
    int learned_accepted;     /* queries whose learned start round was accepted */
    double ms_predict;        /* features + network (inside ms_kpt) */
} tim_batch_stats;

/* TIM+ (plus != 0) or TIM (plus = 0) for nq <= 256 independent queries at once
 * (Sections 3.3 and 4.1 for each query). Each phase samples every active query in one
 * multi-query launch per sampler tier: the rounds of Algorithm 2 run in lockstep and a
 * query leaves when its own stop test passes; the greedy rounds of all queries share
 * launches captured in one CUDA graph. All queries draw from the key of `seed`;
 * query q's sets carry tag queries[q].tag, so its result equals tim_run (or tim_run_tim)
 * on its context after tim_set_query_tag(ctx, tag) with the same seed. Runs on the
 * first query's stream; the other contexts' streams must be idle. */
int tim_run_batch(tim_query* queries, int nq, uint64_t seed, int plus, tim_batch_stats* stats);

/* ------------------------------------------- learned start round of Algorithm 2
 *
 * The paper has no predictor: Algorithm 2 always starts at round 1 and doubles the
 * number of RR sets per round until the stop test passes. These calls add a small
 * network that predicts the stopping round from graph statistics, and a form of
 * Algorithm 2 that starts there. A prediction i0 is accepted only when round i0 - 1
 * fails the stop test and round i0 passes it (i0 = 1: when round 1 passes); the two
 * rounds run in one multi-query launch. Otherwise the plain sweep of Algorithm 2 runs
 * from round 1 (skipping rounds already seen to fail), so a rejected prediction
 * returns exactly the plain result. An accepted prediction returns the plain result
 * whenever no round before i0 - 1 would have passed.
 *
 * Graph features (TIM_GRAPH_FEATURES floats, mean and max over all nodes, in order):
 *   log(1 + indeg v), log(1 + outdeg v), sum of p(u, v) over the in-edges of v (LT:
 *   the node's total in-weight), log(1 + sum over in-edges (u, v) of indeg u).
 * Query features (TIM_START_FEATURES floats): the graph features, then ln n,
 *   ln max(m, 1), ln k, model (0 IC, 1 LT).
 * Prediction target (the network's scaled output): rho = log2(n / (2 KPT*)) -
 *   log2(max(m, 1) / k); i0 = floor(rho + log2(max(m, 1) / k)) + 1, clamped to the
 *   rounds 1 .. floor(log2 n) - 1 of Algorithm 2. */
#define TIM_GRAPH_FEATURES 8
#define TIM_START_FEATURES 12
#define TIM_MLP_HIDDEN 64
#define TIM_MLP_MAX_IN 32

/* Pooled features of the context's graph, computed by kernels on the device at the
 * first call after a load and cached: host float[TIM_GRAPH_FEATURES]. */
int tim_graph_features(tim_ctx* ctx, float* host_out);

/* The network: x (d_in floats) -> xn = (x - in_mu) * in_isd -> h1 = gelu(W1 xn + b1)
 * -> h2 = gelu(W2 h1 + b2) -> z = W3 h2 + b3 (one output) -> y = out_mu + out_sd z,
 * with TIM_MLP_HIDDEN hidden units, gelu(t) = t Phi(t). The weight matrices are used
 * rounded to bfloat16 (nearest, ties to even); activations, biases and every sum are
 * fp32. Parameters are one flat fp32 vector, W1[64][d_in] b1[64] W2[64][64] b2[64]
 * W3[1][64] b3[1] (row-major), zero at creation; scaling defaults to the identity.
 * The network lives on the device of `ctx`, runs on its stream and reports errors
 * through it (tim_last_error_message(ctx)); ctx must outlive it. 1 <= d_in <=
 * TIM_MLP_MAX_IN. Not thread-safe. */
typedef struct tim_mlp tim_mlp;
int tim_mlp_create(tim_mlp** out, tim_ctx* ctx, int d_in);
int tim_mlp_destroy(tim_mlp* mlp);
/* Number of parameters: 64 d_in + 64 + 64*64 + 64 + 64 + 1. */
uint64_t tim_mlp_param_count(const tim_mlp* mlp);
/* Host fp32 params[count]; count must equal tim_mlp_param_count. Setting the
 * parameters resets the Adam moments and step. */
int tim_mlp_set_params(tim_mlp* mlp, const float* params, uint64_t count);
int tim_mlp_get_params(tim_mlp* mlp, float* params, uint64_t count);
/* Host in_mu[d_in], in_isd[d_in]; out_sd != 0. */
int tim_mlp_set_scaling(tim_mlp* mlp, const float* in_mu, const float* in_isd, float out_mu,
                        float out_sd);
/* Loss (1 / 2N) sum_b (z_b - (y_b - out_mu) / out_sd)^2 over host x[N][d_in],
 * y[N] and its gradient w.r.t. the flat parameters (host grad[count], may be NULL),
 * both from the forward and backward kernels; sums over samples run in a fixed
 * order, so results are reproducible. 1 <= N <= 2^24. */
int tim_mlp_grad(tim_mlp* mlp, const float* x, const float* y, uint64_t n_samples,
                 float* loss, float* grad);
/* `steps` full-batch Adam steps (beta1 0.9, beta2 0.999, eps 1e-8, learning rate
 * lr) on host x[N][d_in], y[N], entirely on the device; loss_history (host
 * float[steps], may be NULL) receives the loss before each step. The Adam moments and
 * step count carry over between calls. */
int tim_mlp_train(tim_mlp* mlp, const float* x, const float* y, uint64_t n_samples,
                  int steps, float lr, float* loss_history);
/* Network outputs y (scaled) for host x[N][d_in] into host out[N]. */
int tim_mlp_predict(tim_mlp* mlp, const float* x, uint64_t n_samples, float* out);

/* Algorithm 2 from a learned start round: features of ctx's graph (cached) and k go
 * through `mlp` (d_in = TIM_START_FEATURES) to give i0; then the accept-or-sweep rule
 * above. Outputs as tim_kpt_estimate (may be NULL); *predicted = i0, *accepted = 1
 * when i0 was accepted. The store holds the stopping round's (or the last round's)
 * RR sets, as after tim_kpt_estimate. */
int tim_kpt_estimate_learned(tim_ctx* ctx, tim_mlp* mlp, int k, double ell, uint64_t seed,
                             double* kpt_star, int* round, int* predicted, int* accepted);

/* tim_run (TIM+) with Algorithm 2 started from the learned round. */
int tim_run_learned(tim_ctx* ctx, tim_mlp* mlp, int k, double eps, double ell, uint64_t seed,
                    int32_t* seeds, double* covered_fraction, tim_stats* stats);

/* tim_run_batch with Algorithm 2 started from learned rounds: one network launch
 * predicts every query's i0, one multi-query launch runs rounds i0 - 1 and i0 of all
 * queries, and the queries whose prediction is rejected continue with the lockstep
 * plain sweep. Per-query predictions and acceptance are in queries[q].stats. */
int tim_run_batch_learned(tim_query* queries, int nq, uint64_t seed, int plus, tim_mlp* mlp,
                          tim_batch_stats* stats);

/* Number of kernel launches the context has issued since creation. */
uint64_t tim_launch_count(tim_ctx* ctx);

/* ---------------------------------------------------- forward Monte-Carlo spread
 *
 * The Monte Carlo estimate of E[I(S)] of Section 2.1 (the average number of nodes
 * reachable from S in random graphs g in which every edge is kept with its propagation
 * probability; under LT, Section 4.2, every node keeps the in-edge of its sampled
 * triggering set), as Section 7 uses it to compare seed sets (10^5 cascades there).
 *
 * seeds: host int32[k], node ids in [0, n) (repeats count once; k = 0 activates
 * nothing). Cascade c (c < count < 2^32) walks the world of set id first_set_id + c
 * drawn with the RR sets' keys: IC in-edge at in-CSR position j kept iff word (j & 3)
 * of Philox(seed; sid, j >> 2, TAG_IC) is below its threshold (one coin per in-edge,
 * also in in-lists that RR sampling skips geometrically); LT node v keeps the in-edge
 * picked by word 0 of Philox(seed; sid, v, TAG_LT), and under a general triggering
 * model (tim_load_graph_triggering) the in-edges of the option that word picks. Where
 * no in-list is skipped (LT, triggering models, or IC lists outside the skip rule) the RR
 * set of sid is the set of nodes that reach its root in that world, so root in cascade(S) <=> RR set meets S, world by world.
 * Outputs (each may be NULL): *total = sum over cascades of the activated nodes
 * (seeds included; exact), *mean = total / count in FP64, counts_out = host
 * uint32[count] of per-cascade counts. G as out-records (8 B per node and per edge,
 * and 4 B per edge more once whole worlds are drawn, which they are where the device has
 * room) is built from G^T on the first call after a load and kept. Errors: TIM_ERR_STATE without a graph,
 * TIM_ERR_ARG for a seed out of range or count >= 2^32, TIM_ERR_OOM. */
int tim_spread_mc(tim_ctx* ctx, const int32_t* seeds, int k, uint64_t count, uint64_t seed,
                  uint64_t first_set_id, uint64_t* total, double* mean, uint32_t* counts_out);

#ifdef __cplusplus
}
#endif

#endif /* TIM_H */
