// sample.cu -- random RR sets on the GPU (Definitions 1-2; randomised BFS of Section
// 3.1 "Implementation" for IC; the triggering-model BFS of Section 4.2 with the LT
// triggering distribution of Section 6).
//
// Every coin is keyed on (seed, set id, in-CSR position) and every LT draw on (seed,
// set id, node), so a set does not depend on which kernel expands it, in what order,
// or on how many threads: the three tiers below give identical sets.
//
// Tier 1: a persistent kernel. IC: a warp keeps eight RR sets in flight (rr_pack_kernel),
//   triggering: one (rr_team_kernel), LT: each thread one (rr_lt_lane_kernel). A set's BFS
//   queue (which is also its member list) and a visited hash live in shared memory. Up to 32
//   frontier nodes are expanded at once: their in-lists are cut into 4-aligned groups of
//   in-CSR positions, spread over the lanes, and each lane draws one Philox block (4
//   coin words) and, where the list's thresholds differ, loads 4 of them with one 16-byte
//   load. A set whose members outgrow the queue, or (IC) whose examined in-edges would pass
//   a budget, is listed for tier 2. This keeps the kernel's tail short: light sets are most
//   sets. An IC set that tier 1 gives up on is handed over with its state (the queue so far,
//   the frontier batch to redo, the width before it), and tier 2 goes on from there
//   instead of starting again from the root (the coins are keyed, so the set is the same).
// Tier 2: a queue of 8192 members and a visited hash or bitmap per team of T warps (rr_team_kernel;
//   one arena slot per team in global memory; the queue tail and status stay in shared memory,
//   since every new member takes a tail atomic): T = 1 when the listed sets are many
//   (parallelism across sets fills the GPU), up to 8 when they are few (the team splits each
//   batch, so one heavy set does not leave the GPU idle).
// In all of them in-lists of at least 512 edges (hubs) go by the skip rule, or, with thresholds of
// their own, are streamed one at a time; the rest of a frontier is flattened.
// Tier 3: sets beyond tier 2's queue: IC goes to the batched level-synchronous pass of
//   sample_bulk.cu; LT (a chain) is walked by one warp per set with a visited bitmap; a
//   general triggering model's set is expanded level by level by one block per set.
//
// Per set the kernels can (flags): EMIT the members into the RR-set store, sum KAPPA
// (Eq. 6) in 2^-63 fixed point, and test COVER (does the set meet a given seed set;
// the coverage test of Algorithm 3; the BFS stops at the first member in the seed set).
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

constexpr uint32_t EMPTY = 0xFFFFFFFFu;
constexpr int ST_OVERFLOW = 1;
constexpr int ST_COVERED = 2;
constexpr int WARPS = 8;          // warps per CTA (tiers 1 and 2)
constexpr int BIG_THREADS = 256;  // tier 3 LT CTA size
// IC, tier 2 hands a set to the heavy-set pass once it would have drawn this many coins in
// lists of TIM_SKIP_MIN_INDEG in-edges or more (lists under the skip rule draw none): one
// team streams such a list while the rest of the GPU waits for it, the heavy-set pass
// spreads it over every SM. TIM+ at 1024, 2048, 4096, 8192, 16384, 65536 and no limit:
// trivalency on Chung-Lu graphs of 100,001 nodes 9.4 9.4 9.1 9.4 9.8 10.9 12.0 ms, 700,001
// nodes 18.9 19.1 19.5 20.4 22.1 29.5 44.7, 4.16M nodes 38.1 38.5 38.8 40.2 42.4 59.4 83.5,
// 41.6M nodes - 225.9 224.0 220.3 220.1 229.6 247.3.
// A call of few sets, or on a graph of few edges, has a larger one: a launch of the heavy-set pass
// takes 0.2 ms or more, a set waits for at most its graph's edges, and where many sets are heavy
// the teams have enough of them (trivalency, 6144 -> 24576: 1000 sets of the 100,001 nodes 0.37 ->
// 0.17 ms; 10,000 of 20,001 nodes, 378K edges, 0.37 -> 0.17, TIM+ 3.3 -> 2.5; 200,000 of R-MAT 14,
// 228K edges, 30.0 -> 13.9, TIM+ 121 -> 60; but 1000 of R-MAT 14 0.53 -> 0.67; R-MAT 16, 956K
// edges, the same within 3 %).
constexpr unsigned long long LONG_BUDGET2 = 6144, LONG_BUDGET2_FEW = 24576;
constexpr uint64_t LONG_FEW_SETS = 2048, LONG_FEW_EDGES = 400'000;

// Queue capacity Q and hash size 2^LOG2H (>= 2Q) of one warp's set. With BM the visited set is
// a bitmap (bit 0: a member) instead of the hash, in the hash's place or in shared memory; like
// the hash it holds only EMPTY words between sets.
template <int QQ, int LG, bool BM = false>
struct Cap {
    static constexpr bool BITMAP = BM;
    static constexpr int Q = QQ;
    static constexpr int LOG2H = LG;
    static constexpr int H = 1 << LG;
    // hash[H] u32, queue[Q] u32, slot[Q] u16, ctl[4] int
    static constexpr int WORDS = (1 << LG) + QQ + QQ / 2 + 4;
};
using Tier1 = Cap<256, 9>;
// IC: a warp's eight sets in flight take an eighth of the first-pass capacity (128, 256 or 512
// members) each
using PackS = Cap<16, 5>;
using PackM = Cap<32, 6>;
using PackL = Cap<64, 7>;
using Tier2 = Cap<8192, 14>;
// Second pass of IC, triggering and batched queries on graphs whose bitmap is no larger than the
// hash: one atomic tells whether a node is new, nothing is probed, and a bitmap of n / 8 bytes per
// team stays in L2 where 64 KB per team do not. (Triggering sets of R-MAT 13, 15, 16, 17, 60,001 of
// them: 5.6, 15.9, 28.6, 91.6 ms with the hash, 2.5, 7.1, 13.0, 79.5 ms with the bitmap; weighted
// cascade queries on R-MAT 14 to 18 2-3 % faster.)
using Tier2B = Cap<8192, 14, true>;
constexpr uint32_t BITMAP_GLOBAL = Tier2::H;  // words
// The bitmaps go to shared memory where they leave the blocks resident (the first figure), and
// with teams of a whole block, that is for few sets, up to what a block may have: there also on
// graphs past the line above. (Queries: R-MAT 14 1.63 -> 1.57 ms, R-MAT 20 weighted cascade
// 12.88 -> 12.65 ms. Triggering with 36 KB a block, R-MAT 15, loses: 7.1 -> 11.7 ms, four blocks
// per SM instead of six.)
constexpr size_t BITMAP_SMEM = 16 * 1024, BITMAP_SMEM_FEW = 200 * 1024;

struct SampleArgs {
    const uint4* node;  // node records
    const uint32_t* src;
    const uint32_t* thr;
    const unsigned long long* qtab;      // IC: gap tables of skip-rule nodes
    uint64_t n, m;
    PhiloxKeys K;
    SidMap ids;
    uint64_t count;
    int flags, k;
    const uint32_t* seed_mark;
    uint32_t* pool;
    uint32_t* pool_sid;
    uint64_t pool_cap;
    uint64_t* set_start;
    uint32_t* set_len;
    uint64_t* set_width;
    DevScalars* ds;
    uint32_t* list1;   // tier 1 -> tier 2
    uint32_t* list2;   // tier 2 -> tier 3
    uint32_t list_cap;
    uint32_t* arena;   // tier 2 per-warp storage
    uint32_t bm_words;   // tier 2 with bitmaps: words of each
    uint32_t bm_shared;  // they are in shared memory (otherwise in the hash regions)
    uint32_t* big_bitmap;  // tier 3 LT
    uint32_t* big_queue;
    uint64_t big_words;
    unsigned long long width_budget;  // tier 1 IC: in-edges one warp may examine per set
    unsigned long long width_budget2; // tier 2 IC: in-edges one team may examine per set
    unsigned long long long_budget2;  // tier 2 IC: and in lists of 512 or more
    int chunk;                        // sets claimed per work-counter increment
    int inflight;                     // tier 1 IC: sets in flight per warp
    uint32_t* lt_col;                 // tier 1 LT: per-thread member columns
    // IC: the state pass 1 hands to pass 2 for the set at list1 position i < hcap, hw
    // words at hand + i hw: queue length, resume position, width so far (2 words), queue
    uint32_t* hand;
    uint32_t hcap, hw;
    // IC: the state pass 2 hands to the heavy pass for the set at list2 position i < h2cap,
    // h2w words at hand2 + i h2w: queue length, resume position, width before it (2
    // words), queue
    uint32_t* hand2;
    uint32_t h2cap, h2w;
    // triggering model: options of each node, their cumulative thresholds, their in-edges
    const uint64_t* node_opt;
    const uint32_t* opt_cum;
    const uint64_t* opt_off;
    const uint32_t* opt_pos;
};

__device__ __forceinline__ uint4 draw(const SampleArgs& a, uint64_t sid, uint32_t elem,
                                      uint32_t tag) {
    return philox4x32_10((uint32_t)sid, (uint32_t)(sid >> 32), elem, tag, a.K);
}

__device__ __forceinline__ bool marked(const uint32_t* mark, uint32_t u) {
    return (__ldg(mark + (u >> 5)) >> (u & 31)) & 1u;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Visited set of one RR set: insert u. Returns INS_NEW, INS_OLD, or INS_FULL when the
// queue or the hash is full (the set then moves to the next tier). Bounded probing.
constexpr int INS_OLD = 0, INS_NEW = 1, INS_FULL = 2;

template <class C>
__device__ __forceinline__ int set_insert(uint32_t* hash, uint32_t* queue, uint16_t* slot,
                                          int* ctl, uint32_t u) {
    if constexpr (C::BITMAP) {
        const uint32_t bit = 1u << (u & 31);
        if (!(atomicAnd(&hash[u >> 5], ~bit) & bit)) return INS_OLD;
        const int pos = atomicAdd(&ctl[0], 1);
        if (pos < C::Q) {
            queue[pos] = u;
            return INS_NEW;
        }
        atomicOr(&ctl[1], ST_OVERFLOW);
        return INS_FULL;
    }
    uint32_t h = (u * 0x9E3779B1u) >> (32 - C::LOG2H);
    for (int probe = 0; probe < C::H; probe++) {
        uint32_t old = atomicCAS(&hash[h], EMPTY, u);
        if (old == EMPTY) {
            int pos = atomicAdd(&ctl[0], 1);
            if (pos < C::Q) {
                queue[pos] = u;
                slot[pos] = (uint16_t)h;
                return INS_NEW;
            }
            atomicOr(&ctl[1], ST_OVERFLOW);
            return INS_FULL;
        }
        if (old == u) return INS_OLD;
        h = (h + 1) & (C::H - 1);
    }
    atomicOr(&ctl[1], ST_OVERFLOW);
    return INS_FULL;
}

// Member queue[i] = u of a handed-over set (members are distinct): into the visited set.
template <class C>
__device__ __forceinline__ void set_restore(uint32_t* hash, uint16_t* slot, uint32_t i,
                                            uint32_t u) {
    if constexpr (C::BITMAP) {
        atomicAnd(&hash[u >> 5], ~(1u << (u & 31)));
    } else {
        uint32_t h = (u * 0x9E3779B1u) >> (32 - C::LOG2H);  // the first empty slot it finds
        for (int probe = 0; probe < C::H; probe++) {
            if (atomicCAS(&hash[h], EMPTY, u) == EMPTY) break;
            h = (h + 1) & (C::H - 1);
        }
        slot[i] = (uint16_t)h;
    }
}

// The visited set empty again: of its members, or of everything (words: the bitmap's).
template <class C>
__device__ __forceinline__ void set_clear(uint32_t* hash, const uint32_t* queue,
                                          const uint16_t* slot, int tail, int tl, int step) {
    for (int i = tl; i < tail; i += step) {
        if constexpr (C::BITMAP)
            hash[queue[i] >> 5] = EMPTY;
        else
            hash[slot[i]] = EMPTY;
    }
}

template <class C>
__device__ __forceinline__ void set_clear_all(uint32_t* hash, uint32_t words, int tl, int step) {
    if constexpr (C::BITMAP)
        for (uint32_t i = tl; i < words; i += step) hash[i] = EMPTY;
    else
        for (int i = tl; i < C::H; i += step) hash[i] = EMPTY;
}

// First position j in [lo, hi) with thr[j] > x (thr non-decreasing), or hi.
// 32-ary search by the whole warp.
__device__ __forceinline__ uint64_t warp_lt_search(const uint32_t* __restrict__ thr, uint64_t lo,
                                                   uint64_t hi, uint32_t x, int lane) {
    for (int it = 0; it < 16 && hi - lo > 32; it++) {
        uint64_t stride = (hi - lo + 31) >> 5;
        uint64_t p = lo + (uint64_t)(lane + 1) * stride - 1;
        bool valid = p < hi;
        bool pred = valid && __ldg(thr + p) > x;
        uint32_t b = __ballot_sync(0xffffffffu, pred);
        if (b) {
            int f = __ffs(b) - 1;
            uint64_t nlo = lo + (uint64_t)f * stride;
            hi = nlo + stride;
            lo = nlo;
        } else {
            lo += (uint64_t)__popc(__ballot_sync(0xffffffffu, valid)) * stride;
        }
    }
    uint64_t p = lo + lane;
    bool pred = p < hi && __ldg(thr + p) > x;
    uint32_t b = __ballot_sync(0xffffffffu, pred);
    return b ? lo + (uint64_t)(__ffs(b) - 1) : hi;
}

// ------------------------------------------------------------ tiers 1 and 2

// Barrier over the T warps of a team (T = 1: the warp itself). Named barrier ids
// 1..8 are one per team of the block; 0 stays free for __syncthreads.
template <int T>
__device__ __forceinline__ void team_sync(int team) {
    if (T == 1)
        __syncwarp();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(T * 32) : "memory");
}

// Which of the in-CSR positions 4g .. 4g+3 lie in [beg, end) (bit c = position 4g+c).
// Positions are 32-bit: the graph loader rejects m >= 2^32.
__device__ __forceinline__ uint32_t range_mask(uint32_t g, uint32_t beg, uint32_t end) {
    const uint32_t p0 = g << 2;
    if (p0 >= beg && p0 + 4u <= end) return 0xFu;
    const uint32_t lo = beg > p0 ? beg - p0 : 0u;
    const uint32_t hi = end < p0 + 4u ? end - p0 : 4u;
    return ((1u << hi) - 1u) & ~((1u << lo) - 1u);
}

// Live coins of one group whose 4 in-edges share threshold t (0 < t < 0xFFFFFFFF).
__device__ __forceinline__ uint32_t live_mask_shared(uint4 x, uint32_t t) {
    return (x.x < t ? 1u : 0u) | (x.y < t ? 2u : 0u) | (x.z < t ? 4u : 0u) |
           (x.w < t ? 8u : 0u);
}

// Live coins of one group: bit c set iff word c < thr c, or thr c marks p >= 1.
__device__ __forceinline__ uint32_t live_mask(uint4 x, uint4 t) {
    return ((x.x < t.x) | (t.x == 0xFFFFFFFFu) ? 1u : 0u) |
           ((x.y < t.y) | (t.y == 0xFFFFFFFFu) ? 2u : 0u) |
           ((x.z < t.z) | (t.z == 0xFFFFFFFFu) ? 4u : 0u) |
           ((x.w < t.w) | (t.w == 0xFFFFFFFFu) ? 8u : 0u);
}

// Shared memory of one warp of the IC passes: the in-lists of a frontier batch that the warp
// flattens over its lanes ({begin, end, first group | own thresholds << 31, threshold}), and
// the live in-CSR positions it has found and not inserted yet (fewer than 32, plus a step's 32).
struct alignas(16) WarpScratch {
    uint4 info[32];
    uint32_t stage[64];
};

// Where an IC expansion stopped: the queue position of the frontier batch to process
// next and the width of the members before it.
struct Resume {
    int head;
    unsigned long long width;
};

// Expand one RR set with a team of T warps (wt = warp index in the team, team = team
// index in the block). IC only: with `in` the queue, hash and ctl already hold a set
// that an earlier pass stopped (queue[0 .. ctl[0])), and the expansion goes on from
// in->head with width in->width; with `out`, an expansion that stops records where; wsp is
// the warp's scratch and tot the team's (T > 1). Returns the status bits; *width_out = w(R)
// (Eq. 1); *live_out counts live in-edges followed (per lane).
//
// An IC batch holds up to 32 T frontier nodes, dealt to the warps of the team. A warp lays
// the groups of its nodes' in-lists out over its lanes: the lanes whose list starts within
// the next 32 groups set a bit each (one OR-reduction), popcounts give every lane its list,
// one 16-byte shared load its bounds. Live positions are staged in shared memory and
// inserted 32 at a time, so that the loads of their sources and the hash probes run with
// full lanes and overlap, instead of one by one as each group or gap finds them. Against a
// shuffle search per group, five shuffles for the list's bounds, insertion by the finding
// lane and one batch of 32 nodes per team: R-MAT 20, weighted cascade, pass 1 19.6 -> 16.9 ms
// and pass 2 17.5 -> 12.6 ms per TIM+ run, Algorithm 2 3.3 -> 1.6 ms. Both passes are now
// bound by issue (67 to 73 % active).
template <int MODEL, class C, int T, class A>
__device__ __forceinline__ int team_rr(const A& a, const PhiloxKeys& K, uint64_t sid, uint32_t* hash,
                                       uint32_t* queue, uint16_t* slot, int* ctl,
                                       unsigned long long budget,
                                       unsigned long long long_budget, int wt, int team,
                                       unsigned long long* width_out,
                                       unsigned long long* live_out,
                                       unsigned long long* exam_out,
                                       WarpScratch* wsp, uint32_t* tot,
                                       const Resume* in = nullptr, Resume* out = nullptr) {
    const int lane = threadIdx.x & 31;
    volatile int* vctl = ctl;
    const bool cover = a.flags & SAMPLE_COVER;
    const uint32_t root = rr_root(sid, a.n, K);
    if (!in && wt == 0 && lane == 0) {
        if constexpr (C::BITMAP) {
            hash[root >> 5] = ~(1u << (root & 31));
        } else {
            const uint32_t h = (root * 0x9E3779B1u) >> (32 - C::LOG2H);
            hash[h] = root;
            slot[0] = (uint16_t)h;
        }
        queue[0] = root;
        ctl[0] = 1;
        ctl[1] = (cover && marked(a.seed_mark, root)) ? ST_COVERED : 0;
    }
    if (MODEL == TIM_IC && T > 1 && wt == 0 && lane < 4) tot[lane] = 0u;
    team_sync<T>(team);
    // a set's members are distinct nodes, so every sum of in-degrees stays below m < 2^32
    uint32_t width = in ? (uint32_t)in->width : 0u, live = 0, work = 0, longs = 0, exam = 0;
    if constexpr (MODEL == TIM_IC) {
        const uint32_t s0 = (uint32_t)sid, s1 = (uint32_t)(sid >> 32);
        const uint4* thr4 = reinterpret_cast<const uint4*>(a.thr);
        int head = in ? in->head : 0;
        int bh = head;                // the batch being processed and the width before it
        uint32_t bw = width;
        const uint32_t cap1 = (uint32_t)min(budget, 0xFFFFFFFFull);
        const uint32_t cap2 = (uint32_t)min(long_budget, 0xFFFFFFFFull);
        for (int guard = 0; guard < C::Q + 1; guard++) {
            // a consistent snapshot of (tail, status) for the whole team
            int tail, stat;
            if (T == 1) {
                tail = __shfl_sync(0xffffffffu, vctl[0], 0);
                stat = __shfl_sync(0xffffffffu, vctl[1], 0);
            } else {
                tail = vctl[0];
                stat = vctl[1];
                team_sync<T>(team);
            }
            if (stat || head >= tail) break;
            bh = head;
            bw = width;
            const int nb = min(32 * T, tail - head);
            uint32_t beg = 0, end = 0, t = 0, word = 0;
            // a node's in-edges often share one threshold (weighted cascade: p = 1/indeg);
            // then no threshold is loaded, t = 0 needs no coins, t = 2^32-1 (p >= 1)
            // makes every in-edge live without a draw, and a long list is sampled by
            // geometric skipping
            if (wt + T * lane < nb) {
                const uint4 r = __ldg(a.node + queue[head + wt + T * lane]);
                beg = r.x;
                end = r.y;
                t = r.z;
                word = r.w;
            }
            const bool shared = word & 1u, skip_list = (word >> 1) != 0u;
            const uint32_t deg = end - beg;
            const uint32_t ng = deg ? ((end - 1) >> 2) - (beg >> 2) + 1 : 0u;
            const bool big = !skip_list && deg >= TIM_SKIP_MIN_INDEG;
            const uint32_t skips = __ballot_sync(0xffffffffu, skip_list);
            uint32_t bigs = __ballot_sync(0xffffffffu, big);
            // width of the batch; in-edges that take a coin each (a list under the skip rule
            // counts as 64 against the budget and as the live ones it finds among the
            // examined); those of them in long lists. The frontier's nodes are distinct, so
            // these sums stay below m < 2^32
            const uint32_t dt = __reduce_add_sync(0xffffffffu, skip_list ? 0u : deg);
            uint32_t dw = dt, dx = dt + 64u * __popc(skips), dl = 0;
            if (skips) dw += __reduce_add_sync(0xffffffffu, skip_list ? deg : 0u);
            if (bigs) dl = __reduce_add_sync(0xffffffffu, big ? deg : 0u);
            if (T > 1) {
                if (lane == 0) {
                    if (dw) atomicAdd(&tot[0], dw);
                    if (dx) atomicAdd(&tot[1], dx);
                    if (dl) atomicAdd(&tot[2], dl);
                }
                team_sync<T>(team);
                dw = ((volatile uint32_t*)tot)[0] + (in ? (uint32_t)in->width : 0u) - width;
                dx = ((volatile uint32_t*)tot)[1] - work;
                dl = ((volatile uint32_t*)tot)[2] - longs;
            }
            if (work + dx > cap1 || longs + dl > cap2) {
                // too heavy for this tier: list the set for the next one
                if (wt == 0 && lane == 0) ctl[1] |= ST_OVERFLOW;
                break;
            }
            work += dx;
            longs += dl;
            width += dw;
            if (lane == 0) exam += dt;
            uint32_t held = 0;  // staged positions
            // insert the sources of stage[from .. from + cnt); true: the set stops
            auto take = [&](uint32_t from, uint32_t cnt) {
                __syncwarp();
                bool stop = false;
                if ((uint32_t)lane < cnt) {
                    const uint32_t u = __ldg(a.src + wsp->stage[from + lane]);
                    const int r = set_insert<C>(hash, queue, slot, ctl, u);
                    stop = r == INS_FULL;
                    if (r == INS_NEW && cover && marked(a.seed_mark, u)) {
                        atomicOr(&ctl[1], ST_COVERED);
                        stop = true;
                    }
                }
                return __any_sync(0xffffffffu, stop) != 0;
            };
            // stage the live positions 4 g + c of each lane's mask, one of every lane per turn
            // (few groups have more than one); true: the set stops
            auto append = [&](uint32_t m, uint32_t g) {
                for (uint32_t b; (b = __ballot_sync(0xffffffffu, m != 0u)) != 0u;) {
                    if (m) {
                        wsp->stage[held + __popc(b & ((1u << lane) - 1u))] = (g << 2) + (__ffs(m) - 1);
                        m &= m - 1;
                    }
                    const uint32_t cnt = __popc(b);
                    held += cnt;
                    if (lane == 0) live += cnt;
                    if (held >= 32) {
                        held -= 32;
                        if (take(held, 32)) return true;
                        __syncwarp();
                    }
                }
                return false;
            };
            bool stop = false;
            // lists under the skip rule: one step per live in-edge, two lists at a time but for
            // the longest
            const uint32_t halves = __ballot_sync(0xffffffffu, skip_list && deg < SKIP_HALF);
            for (uint32_t todo = halves; todo && !stop;) {
                const int b0 = __ffs(todo) - 1;
                todo &= todo - 1;
                const int b1 = todo ? __ffs(todo) - 1 : -1;
                todo &= todo - 1;
                const int b = lane < 16 ? b0 : b1;
                const uint32_t bb = __shfl_sync(0xffffffffu, beg, b & 31);
                uint32_t bd = __shfl_sync(0xffffffffu, deg, b & 31);
                const uint32_t bw2 = __shfl_sync(0xffffffffu, word, b & 31);
                if (b < 0) bd = 0u;
                skip_live_half(s0, s1, K, bb, bd, a.qtab + (uint64_t)((bw2 >> 1) - 1) * SKIP_TABLE,
                               lane, [&](bool found, uint32_t j) {
                    const uint32_t f = __ballot_sync(0xffffffffu, found && (lane & 15) == 0);
                    if (found && (lane & 15) == 0)
                        wsp->stage[held + __popc(f & ((1u << lane) - 1u))] = j;
                    if (lane == 0) {
                        live += __popc(f);
                        exam += __popc(f);
                    }
                    held += __popc(f);
                    if (held < 32) return false;
                    held -= 32;
                    stop = take(held, 32);
                    __syncwarp();
                    return stop;
                });
            }
            for (uint32_t todo = skips & ~halves; todo && !stop; todo &= todo - 1) {
                const int b = __ffs(todo) - 1;
                const uint32_t bb = __shfl_sync(0xffffffffu, beg, b);
                const uint32_t be = __shfl_sync(0xffffffffu, end, b);
                const uint32_t bw2 = __shfl_sync(0xffffffffu, word, b);
                skip_live_warp(s0, s1, K, bb, be - bb, a.qtab + (uint64_t)((bw2 >> 1) - 1) * SKIP_TABLE,
                               lane, [&](uint32_t j) {
                    if (lane == 0) {
                        live++;
                        exam++;
                        wsp->stage[held] = j;
                    }
                    if (++held < 32) return false;
                    held = 0;
                    stop = take(0, 32);
                    __syncwarp();
                    return stop;
                });
            }
            // long lists with their own coins; only a list's first and last group need a
            // range mask
            for (; bigs && !stop; bigs &= bigs - 1) {
                const int b = __ffs(bigs) - 1;
                const uint32_t bb = __shfl_sync(0xffffffffu, beg, b);
                const uint32_t be = __shfl_sync(0xffffffffu, end, b);
                const uint32_t bt = __shfl_sync(0xffffffffu, t, b);
                const bool bs = __shfl_sync(0xffffffffu, word, b) & 1u;
                if (bs && bt == 0u) continue;
                const uint32_t gfirst = bb >> 2, glast = (be - 1) >> 2;
                for (uint32_t gb = gfirst; gb <= glast && !stop; gb += 64u) {
                    uint32_t m[2], g[2] = {gb + lane, gb + 32u + lane};
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        m[i] = 0;
                        if (g[i] > glast) continue;
                        if (bs && bt == 0xFFFFFFFFu) {
                            m[i] = 0xFu;
                        } else {
                            const uint4 th = bs ? make_uint4(bt, bt, bt, bt) : __ldg(thr4 + g[i]);
                            m[i] = live_mask(philox4x32_10(s0, s1, g[i], TIM_TAG_IC, K), th);
                        }
                        if (m[i] && (g[i] == gfirst || g[i] == glast)) m[i] &= range_mask(g[i], bb, be);
                    }
                    stop = append(m[0], g[0]) || append(m[1], g[1]);
                }
            }
            // the rest, flattened over the lanes
            const uint32_t ngs = skip_list || big || (shared && t == 0u) ? 0u : ng;
            uint32_t incl = ngs;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            const uint32_t excl = ngs ? incl - ngs : ~0u;
            const uint32_t lists = __ballot_sync(0xffffffffu, ngs != 0u);
            if (ngs)
                wsp->info[__popc(lists & ((1u << lane) - 1u))] =
                    make_uint4(beg, end, excl | (shared ? 0u : 0x80000000u), t);
            __syncwarp();
            for (uint32_t base = 0; base < total && !stop; base += 32) {
                // lists that start before these 32 groups, and at which of them others do
                const uint32_t before = base ? __popc(__ballot_sync(0xffffffffu, excl < base)) : 0u;
                const uint32_t starts = __reduce_or_sync(
                    0xffffffffu, excl - base < 32u ? 1u << (excl - base) : 0u);
                const uint32_t own =
                    before + __popc(starts & (0xFFFFFFFFu >> (31 - lane))) - 1u;
                uint32_t m = 0, g = 0;
                if (base + lane < total) {
                    const uint4 f = wsp->info[own];
                    g = (f.x >> 2) + (base + lane - (f.z & 0x7FFFFFFFu));
                    if (f.z >> 31)
                        m = live_mask(philox4x32_10(s0, s1, g, TIM_TAG_IC, K), __ldg(thr4 + g));
                    else if (f.w == 0xFFFFFFFFu)
                        m = 0xFu;
                    else
                        m = live_mask_shared(philox4x32_10(s0, s1, g, TIM_TAG_IC, K), f.w);
                    if (m) m &= range_mask(g, f.x, f.y);
                }
                stop = append(m, g);
            }
            if (held && !stop) take(0, held);
            team_sync<T>(team);
            head += nb;
        }
        if (out) {  // meaningful when the set stopped: the batch to (re)process
            out->head = bh;
            out->width = bw;
        }
    } else if constexpr (MODEL == TIM_TRIG) {
        // a general triggering model (Section 4.2): every reached node picks one option
        // with the LT draw (the first whose cumulative threshold exceeds it) and the
        // option's in-edges are followed, flattened over the lanes
        const uint32_t s0 = (uint32_t)sid, s1 = (uint32_t)(sid >> 32);
        int head = 0;
        for (int guard = 0; guard < C::Q + 1; guard++) {
            int tail, stat;
            if (T == 1) {
                tail = __shfl_sync(0xffffffffu, vctl[0], 0);
                stat = __shfl_sync(0xffffffffu, vctl[1], 0);
            } else {
                tail = vctl[0];
                stat = vctl[1];
                team_sync<T>(team);
            }
            if (stat || head >= tail) break;
            const int nb = min(32, tail - head);
            uint64_t beg = 0, end = 0, ob = 0, oe = 0;
            if (lane < nb) {
                const uint32_t v = queue[head + lane];
                const uint4 r = __ldg(a.node + v);
                beg = r.x;
                end = r.y;
                const uint64_t o0 = __ldg(a.node_opt + v), o1 = __ldg(a.node_opt + v + 1);
                if (o1 > o0) {
                    const uint32_t x = philox4x32_10(s0, s1, v, TIM_TAG_LT, K).x;
                    const uint64_t o = lane_lt_search(a.opt_cum, o0, o1, x);
                    if (o < o1) {
                        ob = __ldg(a.opt_off + o);
                        oe = __ldg(a.opt_off + o + 1);
                    }
                }
            }
            width += __reduce_add_sync(0xffffffffu, (unsigned)(end - beg));
            const uint32_t ne = (uint32_t)(oe - ob);
            uint32_t incl = ne;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            const uint32_t excl = incl - ne;
            if (wt == 0 && lane == 0) exam += total;
            int flags = 0;
            for (uint32_t base = wt * 32; base < total && !(flags & 3); base += 32 * T) {
                const uint32_t t = base + lane;
                int own = 0;  // number of lanes whose inclusive count is <= t
#pragma unroll
                for (int sft = 16; sft > 0; sft >>= 1) {
                    const uint32_t ic = __shfl_sync(0xffffffffu, incl, own + sft - 1);
                    if (ic <= t) own += sft;
                }
                const uint64_t o_b = __shfl_sync(0xffffffffu, ob, own);
                const uint32_t o_x = __shfl_sync(0xffffffffu, excl, own);
                if (t < total) {
                    live++;
                    const uint32_t u = __ldg(a.src + __ldg(a.opt_pos + o_b + (t - o_x)));
                    const int r = set_insert<C>(hash, queue, slot, ctl, u);
                    if (r == INS_FULL) {
                        flags |= 1;
                    } else if (r == INS_NEW && cover && marked(a.seed_mark, u)) {
                        atomicOr(&ctl[1], ST_COVERED);
                        flags |= 2;
                    }
                }
                flags = __reduce_or_sync(0xffffffffu, flags);
            }
            team_sync<T>(team);
            head += nb;
        }
    } else if (wt == 0) {
        // an LT set is a chain: one warp walks it, the team's other warps wait
        uint32_t v = root;
        for (int guard = 0; guard < C::Q + 1; guard++) {
            if (__shfl_sync(0xffffffffu, vctl[1], 0)) break;
            const uint4 rec = __ldg(a.node + v);
            const uint64_t beg = rec.x, end = rec.y;
            width += end - beg;
            if (beg == end) break;
            const uint32_t x =
                philox4x32_10((uint32_t)sid, (uint32_t)(sid >> 32), v, TIM_TAG_LT, K).x;
            const unsigned long long nt = node_nt(rec);
            const uint64_t j = (nt >> 32) ? lt_uniform_pick(nt, beg, end, x)
                                          : warp_lt_search(a.thr, beg, end, x, lane);
            if (j >= end) break;
            const uint32_t u = __ldg(a.src + j);
            int fresh = 0;
            if (lane == 0) {
                live++;
                fresh = set_insert<C>(hash, queue, slot, ctl, u) == INS_NEW ? 1 : 0;
                if (fresh && cover && marked(a.seed_mark, u)) atomicOr(&ctl[1], ST_COVERED);
            }
            fresh = __shfl_sync(0xffffffffu, fresh, 0);
            __syncwarp();
            if (!fresh) break;
            v = u;
        }
    }
    team_sync<T>(team);
    *width_out = width;
    *live_out += live;
    *exam_out += exam;
    return T == 1 ? __shfl_sync(0xffffffffu, vctl[1], 0) : vctl[1];
}

// kappa (Eq. 6) of the sets whose widths lanes 0 .. cnt-1 hold, one set per lane: the
// FP64 operations of 32 sets share one warp instruction each (GB300's FP64 rate is a
// small fraction of its FP32 rate, and one set per warp instruction cost several ms per
// run of Algorithm 2 on the largest graphs). Each lane adds into its own 128-bit sum.
__device__ __forceinline__ void kappa_lanes(unsigned long long w, unsigned cnt, int lane,
                                            unsigned long long m, int k, unsigned long long& lo,
                                            unsigned long long& hi) {
    if ((unsigned)lane < cnt) {
        const unsigned long long kf = kappa_fixed(kappa_fp64(w, m, k));
        lo += kf;
        if (lo < kf) hi++;
    }
}

// TIER 1 (triggering): teams of one warp, storage in shared memory, every set index of
// [0, count); listed sets go to list1. TIER 2: teams of T warps, storage in
// the global arena, the sets of list1; listed sets go to list2.
// Four blocks of 64 registers per SM for IC: it is bound by issue (six blocks of 40 registers
// spill and are no faster).
template <int MODEL, class C, int TIER, int T>
__global__ void __launch_bounds__(WARPS * 32, TIER == 1 || MODEL == TIM_IC ? 4 : 6) rr_team_kernel(SampleArgs a) {
    extern __shared__ uint32_t smem[];
    __shared__ unsigned long long s_claim[WARPS];
    __shared__ int s_ctl[WARPS][4];  // tier 2: a team's tail and status (shared atomics)
    __shared__ WarpScratch s_scratch[MODEL == TIM_IC ? WARPS : 1];
    __shared__ uint32_t s_tot[WARPS][4];  // a team's batch sums
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int wt = wid % T, team = wid / T;
    const int tl = wt * 32 + lane;  // thread index inside the team
    uint32_t* hash;
    uint32_t* queue;
    if (TIER == 1) {
        hash = smem + team * C::WORDS;
        queue = hash + C::H;
        for (int i = tl; i < C::H; i += 32 * T) hash[i] = EMPTY;
    } else {
        // the arena's hash regions are all EMPTY between sets
        const uint64_t slot_id = (uint64_t)blockIdx.x * (WARPS / T) + team;
        hash = a.arena + slot_id * C::WORDS;
        queue = hash + C::H;
        if (C::BITMAP && a.bm_shared) {
            hash = smem + team * a.bm_words;
            set_clear_all<C>(hash, a.bm_words, tl, 32 * T);
        }
    }
    team_sync<T>(team);
    uint16_t* slot = reinterpret_cast<uint16_t*>(queue + C::Q);
    int* ctl = TIER == 1 ? reinterpret_cast<int*>(queue + C::Q + C::Q / 2) : s_ctl[team];
    const unsigned long long budget = MODEL == TIM_IC ? a.width_budget2 : ~0ull;
    const unsigned long long long_budget = MODEL == TIM_IC ? a.long_budget2 : ~0ull;
    unsigned long long* counter = TIER == 1 ? &a.ds->next_set : &a.ds->next2;
    const uint64_t items =
        TIER == 1 ? a.count : (uint64_t)min(((volatile unsigned*)&a.ds->cnt1)[0], a.list_cap);
    uint32_t* out_list = TIER == 1 ? a.list1 : a.list2;
    unsigned* out_cnt = TIER == 1 ? &a.ds->cnt1 : &a.ds->cnt2;
    unsigned long long k_lo = 0, k_hi = 0, wsum = 0, cov = 0, live = 0, memb = 0, exam = 0;
    const bool emit = a.flags & SAMPLE_EMIT, kap = a.flags & SAMPLE_KAPPA;
    const bool leader = wt == 0 && lane == 0;
    // widths of completed sets waiting for their kappa (warp 0 of the team; lane i holds
    // the i-th, kcnt is the same on every lane)
    unsigned long long kw = 0;
    unsigned kcnt = 0;
    for (;;) {
        unsigned long long i0 = 0;
        if (leader) i0 = atomicAdd(counter, (unsigned long long)a.chunk);
        if (T == 1) {
            i0 = __shfl_sync(0xffffffffu, i0, 0);
        } else {
            if (leader) s_claim[team] = i0;
            team_sync<T>(team);
            i0 = s_claim[team];
            team_sync<T>(team);
        }
        if (i0 >= items) break;
        const unsigned long long i1 = min(i0 + (unsigned long long)a.chunk, (unsigned long long)items);
        for (unsigned long long it = i0; it < i1; it++) {
            const uint64_t j = TIER == 1 ? it : a.list1[it];
            unsigned long long width;
            // IC: pass 2 goes on with a set where pass 1 stopped, from the state pass 1
            // handed over (its queue, the batch to redo, the width before it)
            constexpr bool HAND = MODEL == TIM_IC;
            Resume rin{0, 0ull}, rout{0, 0ull};
            bool resumed = false;
            if (HAND && a.hand && it < a.hcap) {
                const uint32_t* hs = a.hand + it * (uint64_t)a.hw;
                const uint32_t t0 = hs[0];
                if (t0 > 0 && t0 <= (uint32_t)C::Q) {
                    if (leader) {
                        ctl[0] = (int)t0;
                        ctl[1] = 0;
                    }
                    team_sync<T>(team);
                    for (uint32_t i = tl; i < t0; i += 32 * T) {
                        const uint32_t u = hs[4 + i];
                        queue[i] = u;
                        set_restore<C>(hash, slot, i, u);
                        // a member in the seed set found in the batch that overflowed pass
                        // 1's queue: the set is covered (as a fresh expansion would find)
                        if ((a.flags & SAMPLE_COVER) && marked(a.seed_mark, u))
                            atomicOr(&ctl[1], ST_COVERED);
                    }
                    rin.head = (int)min(hs[1], t0);
                    rin.width = (unsigned long long)hs[2] | ((unsigned long long)hs[3] << 32);
                    resumed = true;
                }
                team_sync<T>(team);
            }
            const int st = team_rr<MODEL, C, T, SampleArgs>(
                a, a.K, sid_of(a.ids, j), hash, queue, slot, ctl, budget, long_budget, wt, team, &width, &live,
                &exam, &s_scratch[MODEL == TIM_IC ? wid : 0], s_tot[team],
                resumed ? &rin : nullptr,
                (HAND && a.hand2) ? &rout : nullptr);
            const int tail = min(T == 1 ? __shfl_sync(0xffffffffu, ((volatile int*)ctl)[0], 0)
                                        : ((volatile int*)ctl)[0],
                                 C::Q);
            team_sync<T>(team);
            if (st & ST_OVERFLOW) {
                unsigned idx = 0;
                if (leader) {
                    idx = atomicAdd(out_cnt, 1u);
                    if (idx < a.list_cap)
                        out_list[idx] = (uint32_t)j;
                    else
                        atomicOr(&a.ds->err, TIM_DEV_ERR_OVF_LIST);
                }
                if (HAND && a.hand2) {  // hand the state to the heavy pass
                    if (T == 1) {
                        idx = __shfl_sync(0xffffffffu, idx, 0);
                    } else {
                        if (leader) s_claim[team] = idx;
                        team_sync<T>(team);
                        idx = (unsigned)s_claim[team];
                    }
                    if (idx < a.h2cap) {
                        uint32_t* hs = a.hand2 + idx * (uint64_t)a.h2w;
                        for (int i = tl; i < tail; i += 32 * T) hs[4 + i] = queue[i];
                        if (leader) {
                            hs[0] = (uint32_t)tail;
                            hs[1] = (uint32_t)min(rout.head, tail);
                            hs[2] = (uint32_t)rout.width;  // in-degrees of queue[0 .. hs[1])
                            hs[3] = (uint32_t)(rout.width >> 32);
                        }
                    }
                    team_sync<T>(team);
                }
                set_clear_all<C>(hash, a.bm_words, tl, 32 * T);
                team_sync<T>(team);
                continue;
            }
            if (leader) {
                wsum += width;
                memb += tail;
                if (st & ST_COVERED) cov++;
            }
            if (kap && wt == 0) {  // width is the same on every lane
                if ((unsigned)lane == kcnt) kw = width;
                if (++kcnt == 32) {
                    kappa_lanes(kw, kcnt, lane, a.m, a.k, k_lo, k_hi);
                    kcnt = 0;
                }
            }
            if (emit) {
                unsigned long long base = 0;
                if (leader) base = atomicAdd(&a.ds->pool_used, (unsigned long long)tail);
                if (T == 1) {
                    base = __shfl_sync(0xffffffffu, base, 0);
                } else {
                    if (leader) s_claim[team] = base;
                    team_sync<T>(team);
                    base = s_claim[team];
                }
                if (base + tail <= a.pool_cap) {
                    for (int i = tl; i < tail; i += 32 * T) {
                        a.pool[base + i] = queue[i];
                        a.pool_sid[base + i] = (uint32_t)j;
                    }
                    if (leader) {
                        a.set_start[j] = base;
                        a.set_len[j] = (uint32_t)tail;
                        a.set_width[j] = width;
                    }
                } else if (leader) {
                    atomicOr(&a.ds->err, TIM_DEV_ERR_POOL);
                }
            }
            set_clear<C>(hash, queue, slot, tail, tl, 32 * T);
            team_sync<T>(team);
        }
    }
    live = warp_sum_u64(live);
    if (lane == 0 && live) atomicAdd(&a.ds->live[TIER - 1], live);
    if (lane == 0 && exam) atomicAdd(&a.ds->exam[TIER - 1], exam);
    if (kap && wt == 0) {
        kappa_lanes(kw, kcnt, lane, a.m, a.k, k_lo, k_hi);
        if (k_lo || k_hi) atomic_add_u128(&a.ds->ksum_lo, &a.ds->ksum_hi, k_lo, k_hi);
    }
    if (leader) {
        if (wsum) {
            atomicAdd(&a.ds->wsum, wsum);
            atomicAdd(&a.ds->width[TIER - 1], wsum);
        }
        if (cov) atomicAdd(&a.ds->covered, cov);
        if (memb) atomicAdd(&a.ds->memb[TIER - 1], memb);
    }
}

// What team_rr and pack_run read of one query: its graph and flags, plus the launch's keys.
struct QArgs {
    const uint4* node;
    const uint32_t* src;
    const uint32_t* thr;
    const unsigned long long* qtab;
    uint64_t n, m;
    int flags, k;
    const uint32_t* seed_mark;
};

// ------------------------------------------- tier 1 for IC: several sets per warp
//
// Most RR sets are small (R-MAT 20, weighted cascade: 93 % of 4.9M have at most 32 members), and
// a batch of their frontier is a node or two: a warp that expands one set at a time spends its
// instructions on the batch's bookkeeping with most lanes idle. Here a warp holds eight sets. A
// batch takes up to 32 frontier nodes from all of them, the groups of all their lists are laid
// out over the lanes together (each group draws with its own set's id), and live positions are
// staged with their set and inserted 32 at a time. Lane s keeps set s's queue position; tails,
// widths and work are shared-memory atomics. Finished sets are stored, and new ones claimed,
// two or more at a time.
// A set has room for an eighth of the first-pass capacity, 32 members of 256: small enough for
// four blocks per SM, and a larger set fills a warp's lanes by itself, which is what the second
// pass gives it (rr_team_kernel, from the state that it had here). Bound by issue, as the second
// pass. Queries, weighted cascade, one set per warp with room for 256 -> this:
// R-MAT 20 (eps 0.1) 33.9 -> 28.3 ms, R-MAT 18 8.1 -> 7.3, R-MAT 16 5.6 -> 5.0 (eps 0.2),
// 24 mixed queries 33.1 -> 28.4, 4.16M nodes trivalency 32.5 -> 29.2 ms; R-MAT 14 1.57 -> 1.56.
// With room for 256 / 4 sets: 34.0 ms on R-MAT 20; 128 / 4: 30.7; 64 / 8: 29.2 (before lists under
// the skip rule were taken in pairs); 16 or 64 members in place of 32: within 2 %.
constexpr int PACK_SETS = 8;  // in flight per warp
template <class C>
struct Pack {
    static constexpr int WORDS = PACK_SETS * (C::H + C::Q);  // of a warp: its hashes, then its queues
};
// finished sets wait until 1 / PACK_WAIT of the warp's sets have finished
constexpr int PACK_WAIT = 4;

// Shared memory of one warp: as in WarpScratch, with the set of each list (info.z bits 24 ..) and
// of each staged position, and every set's state.
struct alignas(16) PackScratch {
    uint4 info[32];
    uint32_t stage[64];
    uint8_t stage_set[64];
    int tail[PACK_SETS], stat[PACK_SETS];
    uint32_t width[PACK_SETS], work[PACK_SETS];
    uint32_t s0[PACK_SETS], s1[PACK_SETS];  // the set id
    uint32_t kw[32];                      // widths that wait for their kappa
};

template <class C>
__device__ __forceinline__ int pack_insert(uint32_t* hash, uint32_t* queue, int* tail,
                                           uint32_t u) {
    uint32_t h = (u * 0x9E3779B1u) >> (32 - C::LOG2H);
    for (int probe = 0; probe < C::H; probe++) {
        const uint32_t old = atomicCAS(&hash[h], EMPTY, u);
        if (old == u) return INS_OLD;
        if (old == EMPTY) {
            const int pos = atomicAdd(tail, 1);
            if (pos >= C::Q) return INS_FULL;
            queue[pos] = u;
            return INS_NEW;
        }
        h = (h + 1) & (C::H - 1);
    }
    return INS_FULL;
}

// The sets that next(want, &first) hands to this warp (indexes first .. first + returned, 0 when
// there are no more), up to `inflight` of them at a time. d: where the results go; list(j) puts
// set j on the list for pass 2 and returns its position there.
template <class C, class D, class SidOf, class Next, class List>
__device__ __forceinline__ void pack_run(const QArgs& a, const D& d, const PhiloxKeys& K,
                                         unsigned long long budget, int inflight, uint32_t* mem,
                                         PackScratch* w, uint32_t* hand, uint32_t hcap,
                                         uint32_t hw, SidOf&& sid_at, Next&& next, List&& list) {
    constexpr int S = PACK_SETS, Q = C::Q, H = C::H;
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    uint32_t* hash = mem;
    uint32_t* queue = mem + S * H;
    const bool cover = a.flags & SAMPLE_COVER, emit = a.flags & SAMPLE_EMIT,
               kap = a.flags & SAMPLE_KAPPA;
    const uint4* thr4 = reinterpret_cast<const uint4*>(a.thr);
    const uint32_t cap1 = (uint32_t)min(budget, 0xFFFFFFFFull);
    const int wait = max(1, inflight / PACK_WAIT);
    // lane s: the state of set s; the frontier batch being processed starts at bh, its width
    // before it is bw
    int head = 0, bh = 0;
    uint32_t bw = 0, item = 0;
    bool alive = false;
    unsigned long long wsum = 0, memb = 0, cov = 0, live = 0, exam = 0, k_lo = 0, k_hi = 0;
    unsigned kcnt = 0;
    auto kflush = [&]() {
        __syncwarp();
        kappa_lanes(w->kw[lane], kcnt, lane, a.m, a.k, k_lo, k_hi);
        kcnt = 0;
        __syncwarp();
    };
    for (;;) {
        __syncwarp();
        int tail = 0, stat = 0;
        if (alive) {
            tail = ((volatile int*)w->tail)[lane];
            stat = ((volatile int*)w->stat)[lane];
        }
        const bool done = alive && (stat || head >= tail);
        const uint32_t fin = __ballot_sync(0xffffffffu, done);
        const bool running = __any_sync(0xffffffffu, alive && !done);
        if (__popc(fin) >= wait || !running) {
            if (fin) {
                tail = min(tail, Q);
                const bool over = done && (stat & ST_OVERFLOW), good = done && !over;
                const uint32_t overs = __ballot_sync(0xffffffffu, over);
                const uint32_t goods = __ballot_sync(0xffffffffu, good);
                uint32_t idx = 0;
                if (over) idx = list(item);
                for (uint32_t o = overs; o && hand; o &= o - 1) {
                    const int s = __ffs(o) - 1;
                    const uint32_t at = __shfl_sync(0xffffffffu, idx, s);
                    const int cnt = __shfl_sync(0xffffffffu, tail, s);
                    if (at >= hcap) continue;
                    uint32_t* hs = hand + at * (uint64_t)hw;
                    for (int i = lane; i < cnt; i += 32) hs[4 + i] = queue[s * Q + i];
                    if (lane == s) {
                        hs[0] = (uint32_t)tail;
                        hs[1] = (uint32_t)bh;
                        hs[2] = bw;
                        hs[3] = 0u;
                    }
                }
                const uint32_t width = good ? ((volatile uint32_t*)w->width)[lane] : 0u;
                if (good) {
                    wsum += width;
                    memb += tail;
                    if (stat & ST_COVERED) cov++;
                }
                if (kap) {
                    if (kcnt + __popc(goods) > 32) kflush();
                    if (good) w->kw[kcnt + __popc(goods & below)] = width;
                    kcnt += __popc(goods);
                }
                if (emit && goods) {
                    const uint32_t mine = good ? (uint32_t)tail : 0u;
                    uint32_t incl = mine;
#pragma unroll
                    for (int o = 1; o < S; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    unsigned long long base = 0;
                    if (lane == S - 1) base = atomicAdd(&d.ds->pool_used, (unsigned long long)incl);
                    base = __shfl_sync(0xffffffffu, base, S - 1) + (incl - mine);
                    const bool fits = base + mine <= d.pool_cap;
                    if (good && fits) {
                        d.set_start[item] = base;
                        d.set_len[item] = mine;
                        d.set_width[item] = width;
                    } else if (good) {
                        atomicOr(&d.ds->err, TIM_DEV_ERR_POOL);
                    }
                    for (uint32_t o = __ballot_sync(0xffffffffu, good && fits); o; o &= o - 1) {
                        const int s = __ffs(o) - 1;
                        const int cnt = __shfl_sync(0xffffffffu, tail, s);
                        const unsigned long long to = __shfl_sync(0xffffffffu, base, s);
                        const uint32_t j = __shfl_sync(0xffffffffu, item, s);
                        for (int i = lane; i < cnt; i += 32) {
                            d.pool[to + i] = queue[s * Q + i];
                            d.pool_sid[to + i] = j;
                        }
                    }
                }
                // the hashes empty again: member by member, or all of it
                for (uint32_t o = fin; o; o &= o - 1) {
                    const int s = __ffs(o) - 1;
                    const int cnt = __shfl_sync(0xffffffffu, tail, s);
                    uint32_t* hs = hash + s * H;
                    if (cnt <= 32 && !((overs >> s) & 1u)) {
                        if (lane < cnt) {
                            const uint32_t u = queue[s * Q + lane];
                            uint32_t h = (u * 0x9E3779B1u) >> (32 - C::LOG2H);
                            for (int probe = 0; probe < H; probe++) {
                                if (((volatile uint32_t*)hs)[h] == u) break;
                                h = (h + 1) & (H - 1);
                            }
                            hs[h] = EMPTY;
                        }
                    } else {
                        for (int i = lane; i < H / 4; i += 32)
                            reinterpret_cast<uint4*>(hs)[i] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
                    }
                }
                if (done) alive = false;
                __syncwarp();
            }
            const uint32_t idle = __ballot_sync(0xffffffffu, lane < inflight && !alive);
            if (idle) {
                unsigned long long first = 0;
                const unsigned got = next(__popc(idle), &first);
                const unsigned rank = __popc(idle & below);
                if (((idle >> lane) & 1u) && rank < got) {
                    item = (uint32_t)(first + rank);
                    const uint64_t sid = sid_at(item);
                    const uint32_t root = rr_root(sid, a.n, K);
                    hash[lane * H + ((root * 0x9E3779B1u) >> (32 - C::LOG2H))] = root;
                    queue[lane * Q] = root;
                    tail = 1;
                    stat = (cover && marked(a.seed_mark, root)) ? ST_COVERED : 0;
                    w->tail[lane] = tail;
                    w->stat[lane] = stat;
                    w->width[lane] = 0u;
                    w->work[lane] = 0u;
                    w->s0[lane] = (uint32_t)sid;
                    w->s1[lane] = (uint32_t)(sid >> 32);
                    head = bh = 0;
                    bw = 0;
                    alive = true;
                }
                if (!__any_sync(0xffffffffu, alive)) break;
                __syncwarp();
            }
        }
        // the batch: up to 32 frontier nodes, set by set
        const int av = alive && !stat ? min(tail - head, 32) : 0;
        int incl_n = av;
#pragma unroll
        for (int o = 1; o < S; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl_n, o);
            if (lane >= o) incl_n += y;
        }
        const int nb = min(__shfl_sync(0xffffffffu, incl_n, S - 1), 32);
        int set = 0;  // this lane's node's
#pragma unroll
        for (int s = 0; s + 1 < S; s++)
            if (lane >= __shfl_sync(0xffffffffu, incl_n, s)) set++;
        const int at = __shfl_sync(0xffffffffu, head - (incl_n - av), set) + lane;
        const int mine = min(av, 32 - (incl_n - av));  // nodes that the batch takes from set `lane`
        uint32_t beg = 0, end = 0, t = 0, word = 0;
        if (lane < nb) {
            const uint4 r = __ldg(a.node + queue[set * Q + at]);
            beg = r.x;
            end = r.y;
            t = r.z;
            word = r.w;
        }
        if (mine > 0) {
            bh = head;
            bw = w->width[lane];
        }
        __syncwarp();
        const bool shared = word & 1u;
        bool skip_list = (word >> 1) != 0u;
        uint32_t deg = end - beg;
        // widths; in-edges that take a coin each (a list under the skip rule counts as 64 against
        // the budget and as the live ones it finds among the examined). A set's members are
        // distinct, so its sums stay below m < 2^32
        if (deg) {
            atomicAdd(&w->width[set], deg);
            atomicAdd(&w->work[set], skip_list ? 64u : deg);
        }
        __syncwarp();
        const bool heavy = mine > 0 && w->work[lane] > cap1;
        if (heavy) w->stat[lane] |= ST_OVERFLOW;  // too heavy for this tier: on to the next
        const uint32_t heavies = __ballot_sync(0xffffffffu, heavy);
        if ((heavies >> set) & 1u) {
            deg = 0;
            skip_list = false;
        }
        if (!skip_list) exam += deg;
        const bool big = !skip_list && deg >= TIM_SKIP_MIN_INDEG;
        uint32_t held = 0;  // staged positions
        // insert the sources of stage[from .. from + cnt) into their sets
        auto take = [&](uint32_t from, uint32_t cnt) {
            __syncwarp();
            if ((uint32_t)lane < cnt) {
                const int s = w->stage_set[from + lane];
                const uint32_t u = __ldg(a.src + w->stage[from + lane]);
                if (!((volatile int*)w->stat)[s]) {
                    const int r = pack_insert<C>(hash + s * H, queue + s * Q, &w->tail[s], u);
                    if (r == INS_FULL)
                        atomicOr(&w->stat[s], ST_OVERFLOW);
                    else if (r == INS_NEW && cover && marked(a.seed_mark, u))
                        atomicOr(&w->stat[s], ST_COVERED);
                }
            }
            __syncwarp();
        };
        // stage the live positions 4 g + c of each lane's mask, of set s: one of every lane per
        // turn (few groups have more than one)
        auto append = [&](uint32_t m, uint32_t g, int s) {
            for (uint32_t b; (b = __ballot_sync(0xffffffffu, m != 0u)) != 0u;) {
                if (m) {
                    const uint32_t i = held + __popc(b & below);
                    w->stage[i] = (g << 2) + (__ffs(m) - 1);
                    w->stage_set[i] = (uint8_t)s;
                    m &= m - 1;
                }
                const uint32_t cnt = __popc(b);
                held += cnt;
                if (lane == 0) live += cnt;
                if (held >= 32) {
                    held -= 32;
                    take(held, 32);
                }
            }
        };
        // lists under the skip rule: one step per live in-edge, two lists at a time but for the
        // longest
        const uint32_t skips = __ballot_sync(0xffffffffu, skip_list);
        const uint32_t halves = __ballot_sync(0xffffffffu, skip_list && deg < SKIP_HALF);
        for (uint32_t todo = halves; todo;) {
            const int b0 = __ffs(todo) - 1;
            todo &= todo - 1;
            const int b1 = todo ? __ffs(todo) - 1 : -1;
            todo &= todo - 1;
            const int b = lane < 16 ? b0 : b1;
            const uint32_t bb = __shfl_sync(0xffffffffu, beg, b & 31);
            uint32_t bd = __shfl_sync(0xffffffffu, deg, b & 31);
            if (b < 0) bd = 0u;
            const uint32_t wd = __shfl_sync(0xffffffffu, word, b & 31);
            const int s = __shfl_sync(0xffffffffu, set, b & 31);
            skip_live_half(w->s0[s], w->s1[s], K, bb, bd,
                           a.qtab + (uint64_t)((wd >> 1) - 1) * SKIP_TABLE, lane,
                           [&](bool found, uint32_t j) {
                const uint32_t f = __ballot_sync(0xffffffffu, found && (lane & 15) == 0);
                if (found && (lane & 15) == 0) {
                    live++;
                    exam++;
                    const uint32_t i = held + __popc(f & below);
                    w->stage[i] = j;
                    w->stage_set[i] = (uint8_t)s;
                }
                held += __popc(f);
                if (held < 32) return false;
                held -= 32;
                take(held, 32);
                return ((volatile int*)w->stat)[s] != 0;
            });
        }
        for (uint32_t todo = skips & ~halves; todo; todo &= todo - 1) {
            const int b = __ffs(todo) - 1;
            const uint32_t bb = __shfl_sync(0xffffffffu, beg, b);
            const uint32_t bd = __shfl_sync(0xffffffffu, deg, b);
            const uint32_t wd = __shfl_sync(0xffffffffu, word, b);
            const int s = __shfl_sync(0xffffffffu, set, b);
            skip_live_warp(w->s0[s], w->s1[s], K, bb, bd,
                           a.qtab + (uint64_t)((wd >> 1) - 1) * SKIP_TABLE, lane, [&](uint32_t j) {
                if (lane == 0) {
                    live++;
                    exam++;
                    w->stage[held] = j;
                    w->stage_set[held] = (uint8_t)s;
                }
                if (++held < 32) return false;
                held = 0;
                take(0, 32);
                return __shfl_sync(0xffffffffu, ((volatile int*)w->stat)[s], 0) != 0;
            });
        }
        // long lists with their own coins; only a list's first and last group need a range mask
        for (uint32_t todo = __ballot_sync(0xffffffffu, big); todo; todo &= todo - 1) {
            const int b = __ffs(todo) - 1;
            const uint32_t bb = __shfl_sync(0xffffffffu, beg, b);
            const uint32_t be = __shfl_sync(0xffffffffu, end, b);
            const uint32_t bt = __shfl_sync(0xffffffffu, t, b);
            const bool bs = __shfl_sync(0xffffffffu, word, b) & 1u;
            const int s = __shfl_sync(0xffffffffu, set, b);
            if (bs && bt == 0u) continue;
            const uint32_t z0 = w->s0[s], z1 = w->s1[s];
            const uint32_t gfirst = bb >> 2, glast = (be - 1) >> 2;
            for (uint32_t gb = gfirst; gb <= glast; gb += 64u) {
                uint32_t m[2], g[2] = {gb + lane, gb + 32u + lane};
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    m[i] = 0;
                    if (g[i] > glast) continue;
                    if (bs && bt == 0xFFFFFFFFu) {
                        m[i] = 0xFu;
                    } else {
                        const uint4 th = bs ? make_uint4(bt, bt, bt, bt) : __ldg(thr4 + g[i]);
                        m[i] = live_mask(philox4x32_10(z0, z1, g[i], TIM_TAG_IC, K), th);
                    }
                    if (m[i] && (g[i] == gfirst || g[i] == glast)) m[i] &= range_mask(g[i], bb, be);
                }
                append(m[0], g[0], s);
                append(m[1], g[1], s);
                if (__shfl_sync(0xffffffffu, ((volatile int*)w->stat)[s], 0)) break;
            }
        }
        // the rest, flattened over the lanes
        const uint32_t ngs = skip_list || big || deg == 0u || (shared && t == 0u)
                                 ? 0u
                                 : ((end - 1) >> 2) - (beg >> 2) + 1;
        uint32_t incl = ngs;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);  // at most 32 x 129
        const uint32_t excl = ngs ? incl - ngs : ~0u;
        const uint32_t lists = __ballot_sync(0xffffffffu, ngs != 0u);
        if (ngs)
            w->info[__popc(lists & below)] =
                make_uint4(beg, end, excl | ((uint32_t)set << 24) | (shared ? 0u : 0x80000000u), t);
        __syncwarp();
        for (uint32_t base = 0; base < total; base += 32) {
            // lists that start before these 32 groups, and at which of them others do
            const uint32_t before = base ? __popc(__ballot_sync(0xffffffffu, excl < base)) : 0u;
            const uint32_t starts = __reduce_or_sync(
                0xffffffffu, excl - base < 32u ? 1u << (excl - base) : 0u);
            const uint32_t own = before + __popc(starts & (0xFFFFFFFFu >> (31 - lane))) - 1u;
            uint32_t m = 0, g = 0;
            int s = 0;
            if (base + lane < total) {
                const uint4 f = w->info[own];
                s = (f.z >> 24) & (PACK_SETS - 1);
                g = (f.x >> 2) + (base + lane - (f.z & 0xFFFFFFu));
                if (!(f.z >> 31) && f.w == 0xFFFFFFFFu) {
                    m = 0xFu;
                } else {
                    const uint4 x = philox4x32_10(w->s0[s], w->s1[s], g, TIM_TAG_IC, K);
                    m = f.z >> 31 ? live_mask(x, __ldg(thr4 + g)) : live_mask_shared(x, f.w);
                }
                if (m) m &= range_mask(g, f.x, f.y);
            }
            append(m, g, s);
        }
        if (held) take(0, held);
        if (mine > 0) head += mine;
    }
    if (kap) {
        kflush();
        if (k_lo || k_hi) atomic_add_u128(&d.ds->ksum_lo, &d.ds->ksum_hi, k_lo, k_hi);
    }
    wsum = warp_sum_u64(wsum);
    memb = warp_sum_u64(memb);
    cov = warp_sum_u64(cov);
    live = warp_sum_u64(live);
    exam = warp_sum_u64(exam);
    if (lane == 0) {
        if (wsum) {
            atomicAdd(&d.ds->wsum, wsum);
            atomicAdd(&d.ds->width[0], wsum);
        }
        if (cov) atomicAdd(&d.ds->covered, cov);
        if (memb) atomicAdd(&d.ds->memb[0], memb);
        if (live) atomicAdd(&d.ds->live[0], live);
        if (exam) atomicAdd(&d.ds->exam[0], exam);
    }
}

template <class C>
__global__ void __launch_bounds__(WARPS * 32, 4) rr_pack_kernel(SampleArgs a) {
    extern __shared__ uint4 smem4[];
    __shared__ PackScratch s_scratch[WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t* mem = reinterpret_cast<uint32_t*>(smem4) + wid * Pack<C>::WORDS;
    for (int i = lane; i < PACK_SETS * C::H; i += 32) mem[i] = EMPTY;
    __syncwarp();
    const QArgs qa{a.node, a.src, a.thr, a.qtab, a.n, a.m, a.flags, a.k, a.seed_mark};
    unsigned long long ci = 0, ce = 0;  // claimed
    bool more = true;
    pack_run<C>(
        qa, a, a.K, a.width_budget, a.inflight, mem, &s_scratch[wid], a.hand, a.hcap, a.hw,
        [&](uint32_t j) { return sid_of(a.ids, j); },
        [&](int want, unsigned long long* first) -> unsigned {
            if (ci == ce && more) {
                const int step = max(a.chunk, want);
                if (lane == 0) ci = atomicAdd(&a.ds->next_set, (unsigned long long)step);
                ci = __shfl_sync(0xffffffffu, ci, 0);
                more = ci < a.count;
                if (!more) ci = a.count;
                ce = min(ci + step, (unsigned long long)a.count);
            }
            *first = ci;
            const unsigned got = (unsigned)min((unsigned long long)want, ce - ci);
            ci += got;
            return got;
        },
        [&](uint32_t j) {
            const uint32_t at = atomicAdd(&a.ds->cnt1, 1u);
            if (at < a.list_cap)
                a.list1[at] = j;
            else
                atomicOr(&a.ds->err, TIM_DEV_ERR_OVF_LIST);
            return at;
        });
}

// ------------------------------------------------- tier 1 for LT: a chain per lane
//
// An LT RR set is a chain (Section 4.2: each node keeps at most one live in-edge), so
// its walk has no parallelism of its own: every thread walks one chain. The members go
// to the thread's column of a global array (contiguous per thread: a warp that reads one
// column, to test a revisit or to store the set, reads whole sectors); a 1024-bit Bloom
// filter per thread in shared memory screens the revisit test, which scans the column only
// on a filter hit. Chains longer than LT_CAP go to tier 2 (list1). Finished lanes wait until
// LT_BATCH of them (or the whole warp) are idle; then they store their sets and claim new
// ones together: in chains of some forty steps nearly every step of a warp ends one, and the
// claim, the store and the filter's clearing took several times the step's own work.
// (58.8M members of R-MAT 20, 1/indeg weights: handled as each chain ended, columns
// interleaved by lane, 4.4 ms with the reads that follow; here 1.9 ms; LT_BATCH 1, 4, 8, 12, 16:
// 2.4, 1.9, 1.9, 2.0, 2.1.)
constexpr int LT_THREADS = 128;
constexpr int LT_CAP = 1024;                 // members per chain in this pass
constexpr int LT_BLOOM_WORDS = 32;           // 1024 bits per thread
constexpr int LT_BATCH = 8;                  // idle lanes of a warp handled together
enum : int { LT_IDLE = 0, LT_WALK = 1, LT_DONE = 2, LT_NONE = 3 };  // a lane's chain
constexpr size_t LT_SMEM = (size_t)LT_BLOOM_WORDS * LT_THREADS * sizeof(uint32_t);

__device__ __forceinline__ void lt_bloom_bits(uint32_t u, uint32_t& w1, uint32_t& m1, uint32_t& w2,
                                              uint32_t& m2) {
    const uint32_t h = u * 0x9E3779B1u;
    const uint32_t b1 = h >> 22, b2 = (h >> 12) & 1023u;
    w1 = b1 >> 5;
    m1 = 1u << (b1 & 31);
    w2 = b2 >> 5;
    m2 = 1u << (b2 & 31);
}

__device__ __forceinline__ void lane_bloom_add(uint32_t* bloom, uint32_t u) {
    uint32_t w1, m1, w2, m2;
    lt_bloom_bits(u, w1, m1, w2, m2);
    bloom[w1 * LT_THREADS] |= m1;
    bloom[w2 * LT_THREADS] |= m2;
}

__device__ __forceinline__ bool lane_bloom_test(const uint32_t* bloom, uint32_t u) {
    uint32_t w1, m1, w2, m2;
    lt_bloom_bits(u, w1, m1, w2, m2);
    return (bloom[w1 * LT_THREADS] & m1) && (bloom[w2 * LT_THREADS] & m2);
}

// Revisit test of the lanes with hit set: does lane l's column (wcol + l LT_CAP) hold u among
// its first len members? All lanes scan each such column together. Warp-collective.
__device__ __forceinline__ bool lane_cols_contain(const uint32_t* wcol, int lane, bool hit,
                                                  uint32_t u, int len) {
    bool seen = false;
    const unsigned hits = __ballot_sync(0xffffffffu, hit);
    if (hits) __syncwarp();
    for (unsigned hm = hits; hm; hm &= hm - 1) {
        const int l = __ffs(hm) - 1;
        const uint32_t ul = __shfl_sync(0xffffffffu, u, l);
        const int ll = __shfl_sync(0xffffffffu, len, l);
        bool f = false;
        for (int k = lane; k < ll; k += 32) f |= wcol[l * LT_CAP + k] == ul;
        f = __any_sync(0xffffffffu, f);
        if (lane == l) seen = f;
    }
    return seen;
}

__global__ void __launch_bounds__(LT_THREADS) rr_lt_lane_kernel(SampleArgs a) {
    extern __shared__ uint32_t bloom_all[];
    const int tid = threadIdx.x, lane = tid & 31;
    uint32_t* bloom = bloom_all + tid;  // word w at bloom[w * LT_THREADS]
    for (int w = 0; w < LT_BLOOM_WORDS; w++) bloom[w * LT_THREADS] = 0u;
    // member k of lane l of this warp's columns: wcol[l * LT_CAP + k]
    uint32_t* wcol = a.lt_col + ((uint64_t)blockIdx.x * LT_THREADS + (tid & ~31)) * LT_CAP;
    uint32_t* col = wcol + lane * LT_CAP;
    const bool emit = a.flags & SAMPLE_EMIT, kap = a.flags & SAMPLE_KAPPA,
               cover = a.flags & SAMPLE_COVER;
    unsigned long long k_lo = 0, k_hi = 0, wsum = 0, cov = 0, live = 0, memb = 0;
    int state = LT_IDLE;
    uint64_t j = 0, sid = 0;
    uint32_t v = 0;
    int len = 0;
    bool covered = false, ovf = false;
    uint32_t width = 0;  // a chain's nodes are distinct: below m < 2^32
    // bounded: every step either advances a chain (at most LT_CAP steps each) or
    // finishes it, and the lanes take at most count sets between them
    const uint64_t steps = (a.count + 1) * (uint64_t)(LT_CAP + 2) + 64;
    for (uint64_t guard = 0; guard < steps; guard++) {
        const unsigned idle = __ballot_sync(0xffffffffu, state == LT_IDLE || state == LT_DONE);
        const unsigned walk = __ballot_sync(0xffffffffu, state == LT_WALK);
        if (__popc(idle) >= LT_BATCH || (idle && !walk)) {
            const bool fin = state == LT_DONE;
            if (fin && ovf) {
                const unsigned idx = atomicAdd(&a.ds->cnt1, 1u);
                if (idx < a.list_cap)
                    a.list1[idx] = (uint32_t)j;
                else
                    atomicOr(&a.ds->err, TIM_DEV_ERR_OVF_LIST);
            } else if (fin) {
                wsum += width;
                memb += len;
                if (covered) cov++;
                if (kap) {
                    const unsigned long long kf = kappa_fixed(kappa_fp64(width, a.m, a.k));
                    k_lo += kf;
                    if (k_lo < kf) k_hi++;
                }
            }
            // finished chains reserve their store space together and the warp copies each
            // one's column with all its lanes
            const bool put = emit && fin && !ovf;
            const unsigned pm = __ballot_sync(0xffffffffu, put);
            if (pm) {
                unsigned incl = put ? (unsigned)len : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(&a.ds->pool_used, (unsigned long long)total);
                base = __shfl_sync(0xffffffffu, base, 0);
                const unsigned first = incl - (put ? (unsigned)len : 0u);
                const bool fits = base + total <= a.pool_cap;
                if (put) {
                    if (fits) {
                        a.set_start[j] = base + first;
                        a.set_len[j] = (uint32_t)len;
                        a.set_width[j] = width;
                    } else {
                        atomicOr(&a.ds->err, TIM_DEV_ERR_POOL);
                    }
                }
                __syncwarp();
                for (unsigned m = fits ? pm : 0u; m; m &= m - 1) {
                    const int l = __ffs(m) - 1;
                    const unsigned long long sl = base + __shfl_sync(0xffffffffu, first, l);
                    const int ll = __shfl_sync(0xffffffffu, len, l);
                    const uint32_t jl = (uint32_t)__shfl_sync(0xffffffffu, j, l);
                    for (int k = lane; k < ll; k += 32) {
                        a.pool[sl + k] = wcol[l * LT_CAP + k];
                        a.pool_sid[sl + k] = jl;
                    }
                }
                __syncwarp();
            }
            if (fin)
                for (int w = 0; w < LT_BLOOM_WORDS; w++) bloom[w * LT_THREADS] = 0u;
            // the idle lanes claim the next sets, one atomic for the warp
            const int leader = __ffs(idle) - 1;
            unsigned long long base = 0;
            if (lane == leader) base = atomicAdd(&a.ds->next_set, (unsigned long long)__popc(idle));
            base = __shfl_sync(0xffffffffu, base, leader);
            if ((idle >> lane) & 1u) {
                const unsigned long long mine = base + __popc(idle & ((1u << lane) - 1u));
                state = LT_NONE;
                if (mine < a.count) {
                    j = mine;
                    sid = sid_of(a.ids, j);
                    v = rr_root(sid, a.n, a.K);
                    col[0] = v;
                    len = 1;
                    width = 0;
                    ovf = false;
                    lane_bloom_add(bloom, v);
                    covered = cover && marked(a.seed_mark, v);
                    state = LT_WALK;
                }
            }
        }
        if (!__any_sync(0xffffffffu, state == LT_WALK)) {
            if (__any_sync(0xffffffffu, state == LT_DONE)) continue;
            break;
        }
        // one step of every lane's chain: the next member u, if any
        bool cand = false;
        uint32_t u = 0;
        if (state == LT_WALK) {
            if (covered) {
                state = LT_DONE;
            } else {
                const uint4 rec = __ldg(a.node + v);
                const uint64_t beg = rec.x, end = rec.y;
                const unsigned long long nt = node_nt(rec);
                width += rec.y - rec.x;
                uint64_t jj = end;
                if (beg < end) {
                    const uint32_t x =
                        philox4x32_10((uint32_t)sid, (uint32_t)(sid >> 32), v, TIM_TAG_LT, a.K).x;
                    jj = (nt >> 32) ? lt_uniform_pick(nt, beg, end, x)
                                    : lane_lt_search(a.thr, beg, end, x);
                }
                if (jj >= end) {
                    state = LT_DONE;
                } else {
                    u = __ldg(a.src + jj);
                    live++;
                    cand = true;
                }
            }
        }
        // revisit test: the filter first; on a hit the whole warp scans that column
        const bool seen =
            lane_cols_contain(wcol, lane, cand && lane_bloom_test(bloom, u), u, len);
        if (cand) {
            if (seen) {
                state = LT_DONE;
            } else if (len == LT_CAP) {
                state = LT_DONE;
                ovf = true;
            } else {
                col[len] = u;
                len++;
                lane_bloom_add(bloom, u);
                covered = cover && marked(a.seed_mark, u);
                v = u;
            }
        }
    }
    live = warp_sum_u64(live);
    wsum = warp_sum_u64(wsum);
    memb = warp_sum_u64(memb);
    cov = warp_sum_u64(cov);
    if (lane == 0) {
        if (live) atomicAdd(&a.ds->live[0], live);
        if (wsum) {
            atomicAdd(&a.ds->wsum, wsum);
            atomicAdd(&a.ds->width[0], wsum);
        }
        if (memb) atomicAdd(&a.ds->memb[0], memb);
        if (cov) atomicAdd(&a.ds->covered, cov);
    }
    if (kap && (k_lo || k_hi)) atomic_add_u128(&a.ds->ksum_lo, &a.ds->ksum_hi, k_lo, k_hi);
}

// ---------------------------------------------------------- tier 3 (LT chains)

// One CTA per listed set; warp 0 walks the chain with a visited bitmap and a queue of
// up to n members in global memory.
__global__ void __launch_bounds__(BIG_THREADS) rr_lt_chain_kernel(SampleArgs a) {
    __shared__ unsigned long long s_j;
    __shared__ int s_tail, s_status;
    __shared__ unsigned long long s_width, s_base;
    const int tid = threadIdx.x, lane = tid & 31;
    uint32_t* bitmap = a.big_bitmap + (uint64_t)blockIdx.x * a.big_words;
    uint32_t* queue = a.big_queue + (uint64_t)blockIdx.x * a.n;
    const bool emit = a.flags & SAMPLE_EMIT, kap = a.flags & SAMPLE_KAPPA,
               cover = a.flags & SAMPLE_COVER;
    unsigned long long k_lo = 0, k_hi = 0, wsum = 0, cov = 0, live = 0, memb = 0;
    const unsigned nlist = min(((volatile unsigned*)&a.ds->cnt2)[0], a.list_cap);
    for (;;) {
        if (tid == 0) s_j = atomicAdd(&a.ds->next3, 1ull);
        __syncthreads();
        unsigned long long idx = s_j;
        if (idx >= nlist) break;
        uint64_t j = a.list2[idx];
        uint64_t sid = sid_of(a.ids, j);
        uint32_t root = rr_root(sid, a.n, a.K);
        if (tid == 0) {
            atomicOr(&bitmap[root >> 5], 1u << (root & 31));
            queue[0] = root;
            s_tail = 1;
            s_status = (cover && marked(a.seed_mark, root)) ? ST_COVERED : 0;
            s_width = 0;
        }
        __syncthreads();
        if (tid < 32) {
            uint32_t v = root;
            unsigned long long width = 0;
            int tail = 1;
            int status = s_status;
            for (uint64_t guard = 0; guard <= a.n && !status; guard++) {
                const uint4 rec = __ldg(a.node + v);
                const uint64_t beg = rec.x, end = rec.y;
                width += end - beg;
                if (beg == end) break;
                uint32_t x = draw(a, sid, v, TIM_TAG_LT).x;
                const unsigned long long nt = node_nt(rec);
                uint64_t jj = (nt >> 32) ? lt_uniform_pick(nt, beg, end, x)
                                         : warp_lt_search(a.thr, beg, end, x, lane);
                if (jj >= end) break;
                uint32_t u = __ldg(a.src + jj);
                int fresh = 0;
                if (lane == 0) {
                    live++;
                    uint32_t bit = 1u << (u & 31);
                    uint32_t old = atomicOr(&bitmap[u >> 5], bit);
                    fresh = !(old & bit);
                    if (fresh) queue[tail] = u;
                }
                fresh = __shfl_sync(0xffffffffu, fresh, 0);
                if (!fresh) break;
                tail++;
                if (cover && marked(a.seed_mark, u)) status |= ST_COVERED;
                v = u;
            }
            __syncwarp();
            if (lane == 0) {
                s_width = width;
                s_tail = tail;
                s_status = status;
            }
        }
        __syncthreads();
        const int tail = s_tail;
        const unsigned long long width = s_width;
        if (tid == 0) {
            wsum += width;
            memb += tail;
            if (s_status & ST_COVERED) cov++;
            if (kap) {
                unsigned long long kf = kappa_fixed(kappa_fp64(width, a.m, a.k));
                k_lo += kf;
                if (k_lo < kf) k_hi++;
            }
            if (emit) s_base = atomicAdd(&a.ds->pool_used, (unsigned long long)tail);
        }
        __syncthreads();
        if (emit) {
            unsigned long long base = s_base;
            if (base + tail <= a.pool_cap) {
                for (int i = tid; i < tail; i += BIG_THREADS) {
                    a.pool[base + i] = queue[i];
                    a.pool_sid[base + i] = (uint32_t)j;
                }
                if (tid == 0) {
                    a.set_start[j] = base;
                    a.set_len[j] = (uint32_t)tail;
                    a.set_width[j] = width;
                }
            } else if (tid == 0) {
                atomicOr(&a.ds->err, TIM_DEV_ERR_POOL);
            }
        }
        for (int i = tid; i < tail; i += BIG_THREADS) {
            uint32_t u = queue[i];
            atomicAnd(&bitmap[u >> 5], ~(1u << (u & 31)));
        }
        __syncthreads();
    }
    if (tid == 0) {
        if (kap && (k_lo || k_hi)) atomic_add_u128(&a.ds->ksum_lo, &a.ds->ksum_hi, k_lo, k_hi);
        if (wsum) {
            atomicAdd(&a.ds->wsum, wsum);
            atomicAdd(&a.ds->width[2], wsum);
        }
        if (cov) atomicAdd(&a.ds->covered, cov);
        if (memb) atomicAdd(&a.ds->memb[2], memb);
        if (live) atomicAdd(&a.ds->live[2], live);
    }
}

// ------------------------------------------------- tier 3 (triggering model)

// One CTA per listed set, level-synchronous: the warps claim 32 queued nodes of the
// current level at a time, each lane draws its node's option, and the options' in-edges
// are flattened over the lanes; a new member sets its bit in the slot's visited bitmap
// (n bits) and takes the next entry of the slot's queue (n entries). A level ends when
// every warp has drained it; the set ends at an empty level (or, COVER, at the first
// member in the seed set).
__global__ void __launch_bounds__(BIG_THREADS) rr_trig_big_kernel(SampleArgs a) {
    __shared__ unsigned long long s_j, s_base;
    __shared__ unsigned long long s_width[BIG_THREADS / 32];
    __shared__ unsigned s_head, s_tail;
    __shared__ int s_status;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t* bitmap = a.big_bitmap + (uint64_t)blockIdx.x * a.big_words;
    uint32_t* queue = a.big_queue + (uint64_t)blockIdx.x * a.n;
    const bool emit = a.flags & SAMPLE_EMIT, kap = a.flags & SAMPLE_KAPPA,
               cover = a.flags & SAMPLE_COVER;
    volatile int* vstatus = &s_status;
    unsigned long long k_lo = 0, k_hi = 0, wsum = 0, cov = 0, live = 0, memb = 0;
    const unsigned nlist = min(((volatile unsigned*)&a.ds->cnt2)[0], a.list_cap);
    for (;;) {
        if (tid == 0) s_j = atomicAdd(&a.ds->next3, 1ull);
        __syncthreads();
        const unsigned long long idx = s_j;
        if (idx >= nlist) break;
        const uint64_t j = a.list2[idx];
        const uint64_t sid = sid_of(a.ids, j);
        const uint32_t root = rr_root(sid, a.n, a.K);
        if (tid == 0) {
            atomicOr(&bitmap[root >> 5], 1u << (root & 31));
            queue[0] = root;
            s_tail = 1;
            s_head = 0;
            s_status = (cover && marked(a.seed_mark, root)) ? ST_COVERED : 0;
        }
        __syncthreads();
        unsigned long long width = 0;
        unsigned lvl_end = 1;
        // at most n levels: every level but the last adds a member
        for (uint64_t level = 0; level <= a.n; level++) {
            for (;;) {
                unsigned h0 = 0;
                if (lane == 0) h0 = atomicAdd(&s_head, 32u);
                h0 = __shfl_sync(0xffffffffu, h0, 0);
                if (h0 >= lvl_end || *vstatus) break;
                const unsigned nb = min(32u, lvl_end - h0);
                uint64_t beg = 0, end = 0, ob = 0, oe = 0;
                if (lane < nb) {
                    const uint32_t v = queue[h0 + lane];
                    const uint4 r = __ldg(a.node + v);
                    beg = r.x;
                    end = r.y;
                    const uint64_t o0 = __ldg(a.node_opt + v), o1 = __ldg(a.node_opt + v + 1);
                    if (o1 > o0) {
                        const uint32_t x = draw(a, sid, v, TIM_TAG_LT).x;
                        const uint64_t o = lane_lt_search(a.opt_cum, o0, o1, x);
                        if (o < o1) {
                            ob = __ldg(a.opt_off + o);
                            oe = __ldg(a.opt_off + o + 1);
                        }
                    }
                }
                width += __reduce_add_sync(0xffffffffu, (unsigned)(end - beg));
                const uint32_t ne = (uint32_t)(oe - ob);
                uint32_t incl = ne;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
                const uint32_t excl = incl - ne;
                for (uint32_t base = 0; base < total; base += 32) {
                    const uint32_t t = base + lane;
                    int own = 0;
#pragma unroll
                    for (int sft = 16; sft > 0; sft >>= 1) {
                        const uint32_t ic = __shfl_sync(0xffffffffu, incl, own + sft - 1);
                        if (ic <= t) own += sft;
                    }
                    const uint64_t o_b = __shfl_sync(0xffffffffu, ob, own);
                    const uint32_t o_x = __shfl_sync(0xffffffffu, excl, own);
                    if (t < total) {
                        live++;
                        const uint32_t u = __ldg(a.src + __ldg(a.opt_pos + o_b + (t - o_x)));
                        const uint32_t bit = 1u << (u & 31);
                        if (!(atomicOr(&bitmap[u >> 5], bit) & bit)) {
                            queue[atomicAdd(&s_tail, 1u)] = u;
                            if (cover && marked(a.seed_mark, u)) atomicOr(&s_status, ST_COVERED);
                        }
                    }
                }
            }
            __syncthreads();
            const unsigned next_end = s_tail;
            const bool done = s_status || next_end == lvl_end;
            __syncthreads();  // every thread has read s_tail and s_status
            if (done) break;
            if (tid == 0) s_head = lvl_end;
            lvl_end = next_end;
            __syncthreads();
        }
        if (lane == 0) s_width[wid] = width;
        __syncthreads();
        const unsigned tail = s_tail;
        if (tid == 0) {
            width = 0;
            for (int w = 0; w < BIG_THREADS / 32; w++) width += s_width[w];
            s_width[0] = width;
            wsum += width;
            memb += tail;
            if (s_status & ST_COVERED) cov++;
            if (kap) {
                const unsigned long long kf = kappa_fixed(kappa_fp64(width, a.m, a.k));
                k_lo += kf;
                if (k_lo < kf) k_hi++;
            }
            if (emit) s_base = atomicAdd(&a.ds->pool_used, (unsigned long long)tail);
        }
        __syncthreads();
        if (emit) {
            const unsigned long long base = s_base;
            if (base + tail <= a.pool_cap) {
                for (unsigned i = tid; i < tail; i += BIG_THREADS) {
                    a.pool[base + i] = queue[i];
                    a.pool_sid[base + i] = (uint32_t)j;
                }
                if (tid == 0) {
                    a.set_start[j] = base;
                    a.set_len[j] = tail;
                    a.set_width[j] = s_width[0];
                }
            } else if (tid == 0) {
                atomicOr(&a.ds->err, TIM_DEV_ERR_POOL);
            }
        }
        for (unsigned i = tid; i < tail; i += BIG_THREADS) {
            const uint32_t u = queue[i];
            atomicAnd(&bitmap[u >> 5], ~(1u << (u & 31)));
        }
        __syncthreads();
    }
    live = warp_sum_u64(live);
    if (lane == 0 && live) atomicAdd(&a.ds->live[2], live);
    if (tid == 0) {
        if (kap && (k_lo || k_hi)) atomic_add_u128(&a.ds->ksum_lo, &a.ds->ksum_hi, k_lo, k_hi);
        if (wsum) {
            atomicAdd(&a.ds->wsum, wsum);
            atomicAdd(&a.ds->width[2], wsum);
        }
        if (cov) atomicAdd(&a.ds->covered, cov);
        if (memb) atomicAdd(&a.ds->memb[2], memb);
    }
}

// Resident blocks per SM of a kernel of WARPS warps with smem bytes of dynamic shared memory.
template <class K>
int occupancy(K kernel, size_t smem) {
    int nb = 0;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, WARPS * 32, smem) != cudaSuccess ||
        nb < 1) {
        cudaGetLastError();
        nb = 1;
    }
    return nb;
}

// First pass of IC over `sets` sets: sets in flight per warp, members per set, kernel. With no more
// sets than warps a warp has one set, and hands it over at 16 members whatever the capacity: what
// counts then is the largest set, and the teams of pass 2 expand it faster than one warp (R-MAT 14
// query: 16, 32, 64 members 1.56, 1.61, 1.63 ms; a kernel for one set of 256 per warp 1.68).
template <class Args>
struct PackPlan {
    int inflight, members;
    size_t smem;
    unsigned grid;
    void (*kernel)(Args);
};

template <class C, class Args>
PackPlan<Args> pack_plan_of(const tim_ctx* ctx, void (*kernel)(Args)) {
    const size_t smem = (size_t)WARPS * sizeof(uint32_t) * Pack<C>::WORDS;
    return {PACK_SETS, C::Q, smem, (unsigned)(ctx->num_sms * occupancy(kernel, smem)), kernel};
}

// small, middle, large: the kernel for PackS, PackM and PackL.
template <class Args>
PackPlan<Args> pack_plan(const tim_ctx* ctx, uint64_t sets, void (*small)(Args),
                         void (*middle)(Args), void (*large)(Args)) {
    PackPlan<Args> p = pack_plan_of<PackS>(ctx, small);
    if (sets > (uint64_t)p.grid * WARPS && ctx->cap1 != 128)
        p = ctx->cap1 == 512 ? pack_plan_of<PackL>(ctx, large) : pack_plan_of<PackM>(ctx, middle);
    const uint64_t warps = (uint64_t)p.grid * WARPS;
    p.inflight = (int)std::min<uint64_t>(p.inflight, std::max<uint64_t>(1, (sets + warps - 1) / warps));
    return p;
}

int launch_tier1(tim_ctx* ctx, const SampleArgs& a, const PackPlan<SampleArgs>& plan, unsigned grid,
                 size_t smem) {
    if (ctx->model == TIM_IC) {
        plan.kernel<<<plan.grid, WARPS * 32, plan.smem, ctx->stream>>>(a);
        LAUNCH_CHECK(ctx, "rr_pack_kernel (tier 1)");
    } else if (ctx->model == TIM_TRIG) {
        rr_team_kernel<TIM_TRIG, Tier1, 1, 1><<<grid, WARPS * 32, smem, ctx->stream>>>(a);
        LAUNCH_CHECK(ctx, "rr_team_kernel (tier 1, triggering)");
    } else {
        int nb = 0;
        CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, rr_lt_lane_kernel,
                                                                    LT_THREADS, LT_SMEM));
        const unsigned g = (unsigned)(ctx->num_sms * std::max(nb, 1));
        SampleArgs b = a;
        TIM_TRY(tim_ensure(ctx, ctx->lt_col,
                           (size_t)g * LT_THREADS * LT_CAP * sizeof(uint32_t)));
        b.lt_col = (uint32_t*)ctx->lt_col.p;
        rr_lt_lane_kernel<<<g, LT_THREADS, LT_SMEM, ctx->stream>>>(b);
        LAUNCH_CHECK(ctx, "rr_lt_lane_kernel (tier 1)");
    }
    return TIM_OK;
}

// Bytes of shared memory for the bitmaps of tier 2's teams of T warps (`words` words each), or 0:
// they don't go there.
size_t bitmap_smem(uint64_t words, int T) {
    const size_t bytes = (size_t)(WARPS / T) * words * sizeof(uint32_t);
    return bytes <= (T == 8 ? BITMAP_SMEM_FEW : BITMAP_SMEM) ? bytes : 0;
}

// Blocks of a tier-2 launch with bitmaps in shared memory: at most `grid` (the arena's slots).
template <class K>
int bitmap_grid(tim_ctx* ctx, K kernel, size_t smem, unsigned grid, unsigned* out) {
    CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)BITMAP_SMEM_FEW));
    int nb = 0;
    CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, WARPS * 32, smem));
    *out = std::min(grid, (unsigned)(ctx->num_sms * std::max(nb, 1)));
    return TIM_OK;
}

template <class K>
int launch_bitmap(tim_ctx* ctx, K kernel, const SampleArgs& a, unsigned grid, size_t smem) {
    if (smem) TIM_TRY(bitmap_grid(ctx, kernel, smem, grid, &grid));
    kernel<<<grid, WARPS * 32, smem, ctx->stream>>>(a);
    return TIM_OK;
}

int launch_tier2(tim_ctx* ctx, SampleArgs& a, unsigned grid, int T) {
    const size_t smem = bitmap_smem(a.bm_words, T);
    a.bm_shared = smem > 0;
    if (ctx->model != TIM_LT && (smem || a.bm_words <= BITMAP_GLOBAL)) {
        if (ctx->model == TIM_TRIG)
            TIM_TRY(launch_bitmap(ctx, rr_team_kernel<TIM_TRIG, Tier2B, 2, 1>, a, grid, smem));
        else if (T == 1)
            TIM_TRY(launch_bitmap(ctx, rr_team_kernel<TIM_IC, Tier2B, 2, 1>, a, grid, smem));
        else if (T == 2)
            TIM_TRY(launch_bitmap(ctx, rr_team_kernel<TIM_IC, Tier2B, 2, 2>, a, grid, smem));
        else if (T == 4)
            TIM_TRY(launch_bitmap(ctx, rr_team_kernel<TIM_IC, Tier2B, 2, 4>, a, grid, smem));
        else
            TIM_TRY(launch_bitmap(ctx, rr_team_kernel<TIM_IC, Tier2B, 2, 8>, a, grid, smem));
    } else if (ctx->model != TIM_IC || T == 1) {
        if (ctx->model == TIM_IC)
            rr_team_kernel<TIM_IC, Tier2, 2, 1><<<grid, WARPS * 32, 0, ctx->stream>>>(a);
        else if (ctx->model == TIM_TRIG)
            rr_team_kernel<TIM_TRIG, Tier2, 2, 1><<<grid, WARPS * 32, 0, ctx->stream>>>(a);
        else
            rr_team_kernel<TIM_LT, Tier2, 2, 1><<<grid, WARPS * 32, 0, ctx->stream>>>(a);
    } else if (T == 2) {
        rr_team_kernel<TIM_IC, Tier2, 2, 2><<<grid, WARPS * 32, 0, ctx->stream>>>(a);
    } else if (T == 4) {
        rr_team_kernel<TIM_IC, Tier2, 2, 4><<<grid, WARPS * 32, 0, ctx->stream>>>(a);
    } else {
        rr_team_kernel<TIM_IC, Tier2, 2, 8><<<grid, WARPS * 32, 0, ctx->stream>>>(a);
    }
    LAUNCH_CHECK(ctx, "rr_team_kernel (tier 2)");
    return TIM_OK;
}


// ------------------------------------------------------- several queries at once

// One query of a multi-query launch (device memory).
struct QueryDesc {
    const uint4* node;
    const uint32_t* src;
    const uint32_t* thr;
    const unsigned long long* qtab;
    uint64_t n, m;
    uint64_t sid0, count;
    int model, flags, k, pad;
    const uint32_t* seed_mark;
    uint32_t* pool;
    uint32_t* pool_sid;
    uint64_t pool_cap;
    uint64_t* set_start;
    uint32_t* set_len;
    uint64_t* set_width;
    DevScalars* ds;
    unsigned long long width_budget, width_budget2;
};

struct MultiArgs {
    PhiloxKeys K;
    const QueryDesc* q;
    const unsigned long long* prefix;  // prefix[i] = sets of queries before i; [nq] = total
    int nq;
    int chunk;
    int inflight;                      // tier 1 IC: sets in flight per warp
    unsigned long long* next;  // [0] tier-1, [1] tier-2 work counters
    unsigned* cnt;             // [0] sets listed for tier 2, [1] for tier 3
    int* err;
    uint2* list1;  // (query, set index)
    uint2* list2;
    uint32_t list_cap;
    uint32_t* arena;
    uint32_t bm_words;   // tier 2 with bitmaps: words of each
    uint32_t bm_shared;  // they are in shared memory (otherwise in the hash regions)
    // IC: pass-1 state handed to pass 2 for list1 position i < hcap (as in SampleArgs)
    uint32_t* hand;
    uint32_t hcap, hw;
};

constexpr int MAXQ = 256;  // queries per multi-query launch

struct QAcc {
    unsigned long long k_lo, k_hi, wsum, cov, live, memb, exam;
};

template <int TIER>
__device__ __forceinline__ void flush_acc(const QueryDesc* qd, int qi, QAcc& acc, int lane) {
    const unsigned long long lv = warp_sum_u64(acc.live);
    if (qi >= 0 && lane == 0) {
        DevScalars* ds = qd[qi].ds;
        if (acc.k_lo || acc.k_hi) atomic_add_u128(&ds->ksum_lo, &ds->ksum_hi, acc.k_lo, acc.k_hi);
        if (acc.wsum) {
            atomicAdd(&ds->wsum, acc.wsum);
            atomicAdd(&ds->width[TIER - 1], acc.wsum);
        }
        if (acc.cov) atomicAdd(&ds->covered, acc.cov);
        if (lv) atomicAdd(&ds->live[TIER - 1], lv);
        if (acc.memb) atomicAdd(&ds->memb[TIER - 1], acc.memb);
        if (acc.exam) atomicAdd(&ds->exam[TIER - 1], acc.exam);
    }
    acc = QAcc{0, 0, 0, 0, 0, 0, 0};
}

// Tier 2: the listed (query, set) pairs with a global arena and teams of T warps.
template <class C, int T>
__global__ void __launch_bounds__(WARPS * 32, 4) rr_multi_kernel(MultiArgs ma) {
    extern __shared__ uint32_t smem[];
    __shared__ unsigned long long s_claim[WARPS];
    __shared__ int s_ctl[WARPS][4];  // tier 2: a team's tail and status (shared atomics)
    __shared__ WarpScratch s_scratch[WARPS];
    __shared__ uint32_t s_tot[WARPS][4];  // a team's batch sums
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int wt = wid % T, team = wid / T;
    const int tl = wt * 32 + lane;
    const uint64_t slot_id = (uint64_t)blockIdx.x * (WARPS / T) + team;
    uint32_t* hash = ma.arena + slot_id * C::WORDS;
    uint32_t* queue = hash + C::H;
    if (C::BITMAP && ma.bm_shared) {
        hash = smem + team * ma.bm_words;
        set_clear_all<C>(hash, ma.bm_words, tl, 32 * T);
    }
    team_sync<T>(team);
    uint16_t* slot = reinterpret_cast<uint16_t*>(queue + C::Q);
    int* ctl = s_ctl[team];
    unsigned long long* counter = &ma.next[1];
    const uint64_t items = min(((volatile unsigned*)ma.cnt)[0], ma.list_cap);
    const bool leader = wt == 0 && lane == 0;
    QAcc acc{0, 0, 0, 0, 0, 0, 0};
    int cur_q = -1;
    // kappa of the current query's completed sets, 32 at a time, one per lane (warp 0 of
    // the team): pending widths, the query's m and k, and each lane's 128-bit sum
    unsigned long long kw = 0, km = 0, klo = 0, khi = 0;
    unsigned kcnt = 0;
    int kk = 0;
    auto kflush = [&](int qi) {
        kappa_lanes(kw, kcnt, lane, km, kk, klo, khi);
        kcnt = 0;
        if (qi >= 0 && (klo || khi))
            atomic_add_u128(&ma.q[qi].ds->ksum_lo, &ma.q[qi].ds->ksum_hi, klo, khi);
        klo = khi = 0;
    };
    for (;;) {
        unsigned long long i0 = 0;
        if (leader) i0 = atomicAdd(counter, (unsigned long long)ma.chunk);
        if (T == 1) {
            i0 = __shfl_sync(0xffffffffu, i0, 0);
        } else {
            if (leader) s_claim[team] = i0;
            team_sync<T>(team);
            i0 = s_claim[team];
            team_sync<T>(team);
        }
        if (i0 >= items) break;
        const unsigned long long i1 = min(i0 + (unsigned long long)ma.chunk, (unsigned long long)items);
        for (unsigned long long it = i0; it < i1; it++) {
            const uint2 e = ma.list1[it];
            const int qi = (int)e.x;
            const uint64_t j = e.y;
            if (qi != cur_q) {
                if (wt == 0) kflush(cur_q);
                flush_acc<2>(ma.q, cur_q, acc, lane);
                cur_q = qi;
            }
            const QueryDesc& d = ma.q[qi];
            const QArgs qa{d.node, d.src, d.thr, d.qtab, d.n, d.m, d.flags, d.k, d.seed_mark};
            const int model = d.model;
            const unsigned long long budget =
                model != TIM_IC ? ~0ull : d.width_budget2;
            unsigned long long width;
            int st;
            // IC: pass 2 goes on from the state pass 1 handed over (see rr_team_kernel)
            Resume rin{0, 0ull};
            bool resumed = false;
            if (model == TIM_IC && ma.hand && it < ma.hcap) {
                const uint32_t* hs = ma.hand + it * (uint64_t)ma.hw;
                const uint32_t t0 = hs[0];
                if (t0 > 0 && t0 <= (uint32_t)C::Q) {
                    if (leader) {
                        ctl[0] = (int)t0;
                        ctl[1] = 0;
                    }
                    team_sync<T>(team);
                    for (uint32_t i = tl; i < t0; i += 32 * T) {
                        const uint32_t u = hs[4 + i];
                        queue[i] = u;
                        set_restore<C>(hash, slot, i, u);
                        if ((d.flags & SAMPLE_COVER) && marked(d.seed_mark, u))
                            atomicOr(&ctl[1], ST_COVERED);
                    }
                    rin.head = (int)min(hs[1], t0);
                    rin.width = (unsigned long long)hs[2] | ((unsigned long long)hs[3] << 32);
                    resumed = true;
                }
                team_sync<T>(team);
            }
            if (model == TIM_IC)
                st = team_rr<TIM_IC, C, T, QArgs>(qa, ma.K, d.sid0 + j, hash, queue, slot, ctl,
                                                  budget, ~0ull, wt, team, &width, &acc.live,
                                                  &acc.exam, &s_scratch[wid], s_tot[team],
                                                  resumed ? &rin : nullptr);
            else
                st = team_rr<TIM_LT, C, T, QArgs>(qa, ma.K, d.sid0 + j, hash, queue, slot, ctl,
                                                  budget, ~0ull, wt, team, &width, &acc.live,
                                                  &acc.exam, nullptr, nullptr);
            const int tail = min(T == 1 ? __shfl_sync(0xffffffffu, ((volatile int*)ctl)[0], 0)
                                        : ((volatile int*)ctl)[0],
                                 C::Q);
            team_sync<T>(team);
            if (st & ST_OVERFLOW) {
                if (leader) {
                    const unsigned idx = atomicAdd(&ma.cnt[1], 1u);
                    if (idx < ma.list_cap)
                        ma.list2[idx] = make_uint2((uint32_t)qi, (uint32_t)j);
                    else
                        atomicOr(ma.err, TIM_DEV_ERR_OVF_LIST);
                }
                set_clear_all<C>(hash, ma.bm_words, tl, 32 * T);
                team_sync<T>(team);
                continue;
            }
            if (leader) {
                acc.wsum += width;
                acc.memb += tail;
                if (st & ST_COVERED) acc.cov++;
            }
            if ((d.flags & SAMPLE_KAPPA) && wt == 0) {  // width is the same on every lane
                if ((unsigned)lane == kcnt) kw = width;
                km = d.m;
                kk = d.k;
                if (++kcnt == 32) {
                    kappa_lanes(kw, kcnt, lane, km, kk, klo, khi);
                    kcnt = 0;
                }
            }
            if (d.flags & SAMPLE_EMIT) {
                unsigned long long base = 0;
                if (leader) base = atomicAdd(&d.ds->pool_used, (unsigned long long)tail);
                if (T == 1) {
                    base = __shfl_sync(0xffffffffu, base, 0);
                } else {
                    if (leader) s_claim[team] = base;
                    team_sync<T>(team);
                    base = s_claim[team];
                }
                if (base + tail <= d.pool_cap) {
                    for (int i = tl; i < tail; i += 32 * T) {
                        d.pool[base + i] = queue[i];
                        d.pool_sid[base + i] = (uint32_t)j;
                    }
                    if (leader) {
                        d.set_start[j] = base;
                        d.set_len[j] = (uint32_t)tail;
                        d.set_width[j] = width;
                    }
                } else if (leader) {
                    atomicOr(&d.ds->err, TIM_DEV_ERR_POOL);
                }
            }
            set_clear<C>(hash, queue, slot, tail, tl, 32 * T);
            team_sync<T>(team);
        }
    }
    if (wt == 0) kflush(cur_q);
    flush_acc<2>(ma.q, cur_q, acc, lane);
}

// Tier 1 of the IC queries of a multi-query launch (several sets of one query per warp); a warp
// drains a query's sets before it goes on to the next query's.
template <class C>
__global__ void __launch_bounds__(WARPS * 32, 3) rr_pack_multi_kernel(MultiArgs ma) {
    extern __shared__ uint4 smem4[];
    __shared__ PackScratch s_scratch[WARPS];
    __shared__ unsigned long long s_prefix[MAXQ + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t* mem = reinterpret_cast<uint32_t*>(smem4) + wid * Pack<C>::WORDS;
    for (int i = lane; i < PACK_SETS * C::H; i += 32) mem[i] = EMPTY;
    for (int i = threadIdx.x; i <= ma.nq; i += blockDim.x) s_prefix[i] = ma.prefix[i];
    __syncthreads();
    const unsigned long long items = s_prefix[ma.nq];
    unsigned long long ci = 0, ce = 0;  // claimed
    bool more = true;
    auto claim = [&](int want) {
        if (ci != ce || !more) return;
        const int step = max(ma.chunk, want);
        if (lane == 0) ci = atomicAdd(&ma.next[0], (unsigned long long)step);
        ci = __shfl_sync(0xffffffffu, ci, 0);
        more = ci < items;
        if (!more) ci = items;
        ce = min(ci + step, items);
    };
    for (;;) {
        claim(ma.inflight);
        if (ci == ce) break;
        int lo = 0, hi = ma.nq;  // s_prefix[lo] <= ci < s_prefix[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_prefix[mid] <= ci)
                lo = mid;
            else
                hi = mid;
        }
        const unsigned long long q0 = s_prefix[lo], q1 = s_prefix[lo + 1];
        const QueryDesc& d = ma.q[lo];
        const QArgs qa{d.node, d.src, d.thr, d.qtab, d.n, d.m, d.flags, d.k, d.seed_mark};
        const uint64_t sid0 = d.sid0;
        pack_run<C>(
            qa, d, ma.K, d.width_budget, ma.inflight, mem, &s_scratch[wid], ma.hand, ma.hcap,
            ma.hw, [&](uint32_t j) { return sid0 + j; },
            [&](int want, unsigned long long* first) -> unsigned {
                claim(want);
                if (ci >= q1) return 0u;
                *first = ci - q0;
                const unsigned got = (unsigned)min((unsigned long long)want, min(ce, q1) - ci);
                ci += got;
                return got;
            },
            [&](uint32_t j) {
                const uint32_t at = atomicAdd(&ma.cnt[0], 1u);
                if (at < ma.list_cap)
                    ma.list1[at] = make_uint2((uint32_t)lo, j);
                else
                    atomicOr(ma.err, TIM_DEV_ERR_OVF_LIST);
                return at;
            });
    }
}

// Tier 1 of the LT queries of a multi-query launch: one chain per thread as in
// rr_lt_lane_kernel, over the set index space of the LT queries (lt_prefix; IC queries
// have no sets there). Each thread keeps its query's totals and flushes them when it
// moves to another query; store space is reserved per set; chains longer than LT_CAP
// join the tier-2 list of the launch.
__global__ void __launch_bounds__(LT_THREADS)
rr_lt_lane_multi_kernel(MultiArgs ma, const unsigned long long* lt_prefix,
                        unsigned long long* lt_next, uint32_t* lt_col) {
    extern __shared__ uint32_t bloom_all[];
    __shared__ unsigned long long s_prefix[MAXQ + 1];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i <= ma.nq; i += blockDim.x) s_prefix[i] = lt_prefix[i];
    uint32_t* bloom = bloom_all + tid;
    for (int w = 0; w < LT_BLOOM_WORDS; w++) bloom[w * LT_THREADS] = 0u;
    __syncthreads();
    const uint64_t total = s_prefix[ma.nq];
    uint32_t* wcol = lt_col + ((uint64_t)blockIdx.x * LT_THREADS + (tid & ~31)) * LT_CAP;
    uint32_t* col = wcol + lane * LT_CAP;
    QAcc acc{0, 0, 0, 0, 0, 0, 0};
    int cur_q = -1;
    auto flush = [&]() {
        if (cur_q < 0) return;
        DevScalars* ds = ma.q[cur_q].ds;
        if (acc.k_lo || acc.k_hi)
            atomic_add_u128(&ds->ksum_lo, &ds->ksum_hi, acc.k_lo, acc.k_hi);
        if (acc.wsum) {
            atomicAdd(&ds->wsum, acc.wsum);
            atomicAdd(&ds->width[0], acc.wsum);
        }
        if (acc.cov) atomicAdd(&ds->covered, acc.cov);
        if (acc.live) atomicAdd(&ds->live[0], acc.live);
        if (acc.memb) atomicAdd(&ds->memb[0], acc.memb);
        acc = QAcc{0, 0, 0, 0, 0, 0, 0};
    };
    int state = LT_IDLE;
    int flags = 0, kk = 0, len = 0;
    bool covered = false, ovf = false;
    uint64_t j = 0, sid = 0, n = 0, m = 0;
    const uint4* node = nullptr;
    const uint32_t* src = nullptr;
    const uint32_t* thr = nullptr;
    const uint32_t* seed_mark = nullptr;
    uint32_t v = 0, width = 0;
    const uint64_t steps = (total + 1) * (uint64_t)(LT_CAP + 2) + 64;
    for (uint64_t guard = 0; guard < steps; guard++) {
        const unsigned idle = __ballot_sync(0xffffffffu, state == LT_IDLE || state == LT_DONE);
        const unsigned walk = __ballot_sync(0xffffffffu, state == LT_WALK);
        if (__popc(idle) >= LT_BATCH || (idle && !walk)) {
            bool put = false;
            unsigned long long st = 0;
            uint32_t* pool = nullptr;
            uint32_t* pool_sid = nullptr;
            if (state == LT_DONE && ovf) {
                const unsigned idx = atomicAdd(&ma.cnt[0], 1u);
                if (idx < ma.list_cap)
                    ma.list1[idx] = make_uint2((uint32_t)cur_q, (uint32_t)j);
                else
                    atomicOr(ma.err, TIM_DEV_ERR_OVF_LIST);
            } else if (state == LT_DONE) {
                acc.wsum += width;
                acc.memb += len;
                if (covered) acc.cov++;
                if (flags & SAMPLE_KAPPA) {
                    const unsigned long long kf = kappa_fixed(kappa_fp64(width, m, kk));
                    acc.k_lo += kf;
                    if (acc.k_lo < kf) acc.k_hi++;
                }
                if (flags & SAMPLE_EMIT) {
                    const QueryDesc& d = ma.q[cur_q];
                    st = atomicAdd(&d.ds->pool_used, (unsigned long long)len);
                    if (st + (unsigned)len <= d.pool_cap) {
                        put = true;
                        pool = d.pool;
                        pool_sid = d.pool_sid;
                        d.set_start[j] = st;
                        d.set_len[j] = (uint32_t)len;
                        d.set_width[j] = width;
                    } else {
                        atomicOr(&d.ds->err, TIM_DEV_ERR_POOL);
                    }
                }
            }
            // the warp copies each stored chain's column with all its lanes
            __syncwarp();
            for (unsigned pm = __ballot_sync(0xffffffffu, put); pm; pm &= pm - 1) {
                const int l = __ffs(pm) - 1;
                const unsigned long long sl = __shfl_sync(0xffffffffu, st, l);
                const int ll = __shfl_sync(0xffffffffu, len, l);
                const uint32_t jl = (uint32_t)__shfl_sync(0xffffffffu, (unsigned long long)j, l);
                uint32_t* pl = (uint32_t*)__shfl_sync(0xffffffffu, (unsigned long long)pool, l);
                uint32_t* psl = (uint32_t*)__shfl_sync(0xffffffffu, (unsigned long long)pool_sid, l);
                for (int k = lane; k < ll; k += 32) {
                    pl[sl + k] = wcol[l * LT_CAP + k];
                    psl[sl + k] = jl;
                }
            }
            __syncwarp();
            if (state == LT_DONE)
                for (int w = 0; w < LT_BLOOM_WORDS; w++) bloom[w * LT_THREADS] = 0u;
            // the idle lanes claim the next sets, one atomic for the warp
            const int leader = __ffs(idle) - 1;
            unsigned long long base = 0;
            if (lane == leader) base = atomicAdd(lt_next, (unsigned long long)__popc(idle));
            base = __shfl_sync(0xffffffffu, base, leader);
            if ((idle >> lane) & 1u) {
                const unsigned long long mine = base + __popc(idle & ((1u << lane) - 1u));
                state = LT_NONE;
                if (mine < total) {
                    int lo = 0, hi = ma.nq;  // s_prefix[lo] <= mine < s_prefix[hi]
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (s_prefix[mid] <= mine)
                            lo = mid;
                        else
                            hi = mid;
                    }
                    if (lo != cur_q) {
                        flush();
                        cur_q = lo;
                        const QueryDesc& d = ma.q[lo];
                        node = d.node;
                        src = d.src;
                        thr = d.thr;
                        seed_mark = d.seed_mark;
                        n = d.n;
                        m = d.m;
                        flags = d.flags;
                        kk = d.k;
                    }
                    j = mine - s_prefix[lo];
                    sid = ma.q[lo].sid0 + j;
                    v = rr_root(sid, n, ma.K);
                    col[0] = v;
                    len = 1;
                    width = 0;
                    ovf = false;
                    lane_bloom_add(bloom, v);
                    covered = (flags & SAMPLE_COVER) && marked(seed_mark, v);
                    state = LT_WALK;
                }
            }
        }
        if (!__any_sync(0xffffffffu, state == LT_WALK)) {
            if (__any_sync(0xffffffffu, state == LT_DONE)) continue;
            break;
        }
        bool cand = false;
        uint32_t u = 0;
        if (state == LT_WALK) {
            if (covered) {
                state = LT_DONE;
            } else {
                const uint4 rec = __ldg(node + v);
                const uint64_t beg = rec.x, end = rec.y;
                const unsigned long long nt = node_nt(rec);
                width += rec.y - rec.x;
                uint64_t jj = end;
                if (beg < end) {
                    const uint32_t x =
                        philox4x32_10((uint32_t)sid, (uint32_t)(sid >> 32), v, TIM_TAG_LT, ma.K).x;
                    jj = (nt >> 32) ? lt_uniform_pick(nt, beg, end, x)
                                    : lane_lt_search(thr, beg, end, x);
                }
                if (jj >= end) {
                    state = LT_DONE;
                } else {
                    u = __ldg(src + jj);
                    acc.live++;
                    cand = true;
                }
            }
        }
        const bool seen =
            lane_cols_contain(wcol, lane, cand && lane_bloom_test(bloom, u), u, len);
        if (cand) {
            if (seen) {
                state = LT_DONE;
            } else if (len == LT_CAP) {
                state = LT_DONE;
                ovf = true;
            } else {
                col[len] = u;
                len++;
                lane_bloom_add(bloom, u);
                covered = (flags & SAMPLE_COVER) && marked(seed_mark, u);
                v = u;
            }
        }
    }
    flush();
}

// Tier 2 of a multi-query launch with teams of T warps.
int launch_multi(tim_ctx* owner, const MultiArgs& ma, int T, unsigned grid) {
    if (ma.bm_shared || ma.bm_words <= BITMAP_GLOBAL) {
        const size_t bytes = bitmap_smem(ma.bm_words, T);
        auto* kernel = T == 1   ? rr_multi_kernel<Tier2B, 1>
                       : T == 2 ? rr_multi_kernel<Tier2B, 2>
                       : T == 4 ? rr_multi_kernel<Tier2B, 4>
                                : rr_multi_kernel<Tier2B, 8>;
        if (bytes) TIM_TRY(bitmap_grid(owner, kernel, bytes, grid, &grid));
        kernel<<<grid, WARPS * 32, bytes, owner->stream>>>(ma);
    } else if (T == 1) {
        rr_multi_kernel<Tier2, 1><<<grid, WARPS * 32, 0, owner->stream>>>(ma);
    } else if (T == 2) {
        rr_multi_kernel<Tier2, 2><<<grid, WARPS * 32, 0, owner->stream>>>(ma);
    } else if (T == 4) {
        rr_multi_kernel<Tier2, 4><<<grid, WARPS * 32, 0, owner->stream>>>(ma);
    } else {
        rr_multi_kernel<Tier2, 8><<<grid, WARPS * 32, 0, owner->stream>>>(ma);
    }
    LAUNCH_CHECK(owner, "rr_multi_kernel (tier 2)");
    return TIM_OK;
}

}  // namespace

// Room for `entries` members in the store: both arrays, whatever an earlier call that ran out of
// memory left of them.
static int ensure_pool(tim_ctx* ctx, uint64_t entries) {
    TIM_TRY(tim_ensure(ctx, ctx->pool, entries * sizeof(uint32_t)));
    return tim_ensure(ctx, ctx->pool_sid, entries * sizeof(uint32_t));
}

static uint64_t pool_entries(const tim_ctx* ctx) {
    return std::min(ctx->pool.bytes, ctx->pool_sid.bytes) / sizeof(uint32_t);
}

static int regrow_pool(tim_ctx* ctx, uint64_t used) {
    tim_free(ctx->pool);
    tim_free(ctx->pool_sid);
    return ensure_pool(ctx, used + used / 16 + 4096);
}

// The store and what refers to it while a call writes into it: empty until the call succeeds, since
// a failed one may have given its arrays back.
static void open_store(tim_ctx* ctx) {
    ctx->n_sets = ctx->members = 0;
    ctx->select_open = false;
    ctx->have_kpt = false;
    ctx->rounds_kept = false;
}

int tim_sample(tim_ctx* ctx, const SampleRequest& req, SampleResult* res) {
    if (!ctx->have_graph) return tim_fail(ctx, TIM_ERR_STATE, "no graph loaded");
    const uint64_t count = req.count;
    const bool emit = req.flags & SAMPLE_EMIT;
    if (count > 0xFFFFFFF0ull) return tim_fail(ctx, TIM_ERR_ARG, "too many RR sets in one call");
    // per-set arrays grow to the next power of two so that the doubling rounds of
    // Algorithm 2 do not reallocate every round
    uint64_t cap_sets = 1024;
    while (cap_sets < count + 1) cap_sets <<= 1;
    const bool have_kpt = ctx->have_kpt;
    if (emit) {
        open_store(ctx);
        TIM_TRY(tim_ensure(ctx, ctx->set_start, cap_sets * sizeof(uint64_t)));
        TIM_TRY(tim_ensure(ctx, ctx->set_len, cap_sets * sizeof(uint32_t)));
        TIM_TRY(tim_ensure(ctx, ctx->set_width, cap_sets * sizeof(uint64_t)));
        TIM_TRY(ensure_pool(ctx, cap_sets * 8 + 4096));
    }
    const uint32_t list_cap = (uint32_t)(count + 1);
    TIM_TRY(tim_ensure(ctx, ctx->ovf_list, (size_t)cap_sets * sizeof(uint32_t)));
    TIM_TRY(tim_ensure(ctx, ctx->ovf_list2, (size_t)cap_sets * sizeof(uint32_t)));

    // tier 2 arena: one slot per resident warp, hash regions kept EMPTY between sets
    PackPlan<SampleArgs> plan{};
    size_t smem1 = 0;
    unsigned grid1 = 0;  // triggering
    if (ctx->model == TIM_IC) {
        plan = pack_plan(ctx, count, rr_pack_kernel<PackS>,
                         rr_pack_kernel<PackM>, rr_pack_kernel<PackL>);
    } else if (ctx->model == TIM_TRIG) {
        smem1 = (size_t)WARPS * sizeof(uint32_t) * Tier1::WORDS;
        grid1 = (unsigned)(ctx->num_sms * occupancy(rr_team_kernel<TIM_TRIG, Tier1, 1, 1>, smem1));
    }
    const int nb2 = ctx->model == TIM_IC     ? occupancy(rr_team_kernel<TIM_IC, Tier2, 2, 1>, 0)
                    : ctx->model == TIM_TRIG ? occupancy(rr_team_kernel<TIM_TRIG, Tier2, 2, 1>, 0)
                                             : occupancy(rr_team_kernel<TIM_LT, Tier2, 2, 1>, 0);
    const unsigned grid2 = (unsigned)(ctx->num_sms * nb2);
    const size_t arena_bytes = (size_t)grid2 * WARPS * Tier2::WORDS * sizeof(uint32_t);
    const uint64_t made_arena = ctx->arena.made;
    TIM_TRY(tim_ensure(ctx, ctx->arena, arena_bytes));
    if (ctx->arena.made != made_arena || !ctx->arena_clean) {
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->arena.p, 0xFF, ctx->arena.bytes, ctx->stream));
        ctx->arena_clean = true;
    }
    // tier 3 LT and triggering slots: a bitmap of n bits and a queue of n entries each,
    // at most ~2 GiB
    const uint64_t words = (uint64_t)(ctx->n + 31) / 32 + 1;
    int slots = 0;
    if (ctx->model != TIM_IC) {
        const uint64_t per_slot = (words + (uint64_t)ctx->n) * sizeof(uint32_t);
        slots = ctx->num_sms;
        const uint64_t budget = 2ull << 30;
        if ((uint64_t)slots * per_slot > budget)
            slots = (int)std::max<uint64_t>(1, budget / per_slot);
        const uint64_t made_bm = ctx->big_bitmap.made;
        TIM_TRY(tim_ensure(ctx, ctx->big_bitmap, (size_t)slots * words * sizeof(uint32_t)));
        TIM_TRY(tim_ensure(ctx, ctx->big_queue,
                           (size_t)slots * (uint64_t)ctx->n * sizeof(uint32_t)));
        if (ctx->big_bitmap.made != made_bm || !ctx->big_bitmap_clean) {
            CUDA_TRY(ctx, cudaMemsetAsync(ctx->big_bitmap.p, 0, ctx->big_bitmap.bytes, ctx->stream));
            ctx->big_bitmap_clean = true;
        }
    }
    SampleArgs a;
    a.node = (const uint4*)ctx->node.p;
    a.src = (const uint32_t*)ctx->src.p;
    a.thr = (const uint32_t*)ctx->thr.p;
    a.qtab = (const unsigned long long*)ctx->qtab.p;
    a.n = (uint64_t)ctx->n;
    a.m = (uint64_t)ctx->m;
    a.K = tim_philox_keys(req.seed);
    a.ids = tim_sid_map(req);
    a.count = count;
    a.flags = req.flags;
    a.k = req.k;
    a.seed_mark = req.seed_mark;
    a.ds = tim_dscal(ctx);
    a.list1 = (uint32_t*)ctx->ovf_list.p;
    a.list2 = (uint32_t*)ctx->ovf_list2.p;
    a.list_cap = list_cap;
    a.arena = (uint32_t*)ctx->arena.p;
    a.bm_words = (uint32_t)((uint64_t)ctx->n / 32 + 1);
    a.big_bitmap = (uint32_t*)ctx->big_bitmap.p;
    a.big_queue = (uint32_t*)ctx->big_queue.p;
    a.big_words = words;
    a.set_start = (uint64_t*)ctx->set_start.p;
    a.set_len = (uint32_t*)ctx->set_len.p;
    a.set_width = (uint64_t*)ctx->set_width.p;
    a.width_budget = ctx->width_budget;
    a.width_budget2 = ctx->width_budget2;
    a.long_budget2 = count <= LONG_FEW_SETS || (uint64_t)ctx->m <= LONG_FEW_EDGES
                         ? LONG_BUDGET2_FEW : LONG_BUDGET2;
    a.chunk = std::max(1, ctx->chunk);
    a.inflight = plan.inflight;
    // IC: room for the pass-1 state of up to count / 2 + 4096 handed-over sets (at most
    // 1 GiB); sets listed beyond it start over in pass 2
    a.hand = nullptr;
    a.hcap = 0;
    a.hw = 4u + (uint32_t)plan.members;
    if (ctx->model == TIM_IC && count > 0) {
        const uint64_t maxslots = (1ull << 30) / ((uint64_t)a.hw * sizeof(uint32_t));
        const uint64_t hcap = std::min<uint64_t>(std::min<uint64_t>(count / 2 + 4096, maxslots),
                                                 list_cap);
        TIM_TRY(tim_ensure(ctx, ctx->hand, (size_t)hcap * a.hw * sizeof(uint32_t)));
        a.hand = (uint32_t*)ctx->hand.p;
        a.hcap = (uint32_t)hcap;
    }
    a.hand2 = nullptr;
    a.h2cap = 0;
    a.h2w = 4u + (uint32_t)Tier2::Q;
    if (ctx->model == TIM_IC && count > 0) {  // at most 1 GiB; later sets start over
        const uint64_t h2cap = std::min<uint64_t>((1ull << 30) / ((uint64_t)a.h2w * 4), list_cap);
        TIM_TRY(tim_ensure(ctx, ctx->hand2, (size_t)h2cap * a.h2w * sizeof(uint32_t)));
        a.hand2 = (uint32_t*)ctx->hand2.p;
        a.h2cap = (uint32_t)h2cap;
    }
    a.node_opt = (const uint64_t*)ctx->node_opt.p;
    a.opt_cum = (const uint32_t*)ctx->opt_cum.p;
    a.opt_off = (const uint64_t*)ctx->opt_off.p;
    a.opt_pos = (const uint32_t*)ctx->opt_pos.p;
    for (int attempt = 0; attempt < 4; attempt++) {
        a.pool = (uint32_t*)ctx->pool.p;
        a.pool_sid = (uint32_t*)ctx->pool_sid.p;
        a.pool_cap = emit ? pool_entries(ctx) : 0;
        TIM_TRY(tim_zero_scalars(ctx));
        uint64_t live3 = 0;
        bool read = false;
        if (count > 0) {
            cudaEventRecord(ctx->kev[0], ctx->stream);
            TIM_TRY(launch_tier1(ctx, a, plan, grid1, smem1));
            cudaEventRecord(ctx->kev[1], ctx->stream);
            // team size of tier 2: intra-set parallelism when the listed sets are few
            int T = 1;
            if (ctx->model == TIM_IC) {
                TIM_TRY(tim_read_scalars(ctx));
                const uint64_t listed = ctx->h_scal->cnt1;
                const uint64_t slots1 = (uint64_t)grid2 * WARPS;
                T = ctx->team_size;
                if (T <= 0) {
                    T = 1;
                    while (T < 8 && listed * (uint64_t)ctx->team_factor < slots1 / T) T *= 2;
                }
                ctx->last_team = T;
            }
            TIM_TRY(launch_tier2(ctx, a, grid2, T));
            cudaEventRecord(ctx->kev[2], ctx->stream);
            if (ctx->model == TIM_IC) {
                TIM_TRY(tim_read_scalars(ctx));
                const unsigned n3 = std::min(ctx->h_scal->cnt2, list_cap);
                read = n3 == 0;  // nothing runs after this read
                TIM_TRY(tim_bulk_ic(ctx, req, a.list2, n3, a.pool, a.pool_sid, a.pool_cap, a.ds,
                                    &live3, a.hand2, a.h2cap, a.h2w));
            } else if (ctx->model == TIM_TRIG) {
                rr_trig_big_kernel<<<slots, BIG_THREADS, 0, ctx->stream>>>(a);
                LAUNCH_CHECK(ctx, "rr_trig_big_kernel");
            } else {
                rr_lt_chain_kernel<<<slots, BIG_THREADS, 0, ctx->stream>>>(a);
                LAUNCH_CHECK(ctx, "rr_lt_chain_kernel");
            }
            cudaEventRecord(ctx->kev[3], ctx->stream);
        }
        if (!read) TIM_TRY(tim_read_scalars(ctx));
        DevScalars& h = *ctx->h_scal;
        if (ctx->model == TIM_IC) h.live[2] = live3;
        if (h.err & TIM_DEV_ERR_POOL) {
            TIM_TRY(regrow_pool(ctx, h.pool_used));
            continue;
        }
        if (h.err) {
            ctx->arena_clean = ctx->big_bitmap_clean = false;
            return tim_fail(ctx, TIM_ERR_CUDA, "device error flags set by the RR sampler");
        }
        if (count > 0) {
            float t[3] = {0.f, 0.f, 0.f};
            for (int i = 0; i < (read ? 2 : 3); i++) cudaEventElapsedTime(&t[i], ctx->kev[i], ctx->kev[i + 1]);
            const uint64_t sets[3] = {count - h.cnt1, (uint64_t)h.cnt1 - h.cnt2, h.cnt2};
            tim_profile& P = ctx->prof;
            uint64_t* L[3] = {&P.pass1_launches, &P.pass2_launches, &P.pass3_launches};
            double* T[3] = {&P.pass1_ms, &P.pass2_ms, &P.pass3_ms};
            uint64_t* S[3] = {&P.pass1_sets, &P.pass2_sets, &P.pass3_sets};
            uint64_t* W[3] = {&P.pass1_width, &P.pass2_width, &P.pass3_width};
            uint64_t* V[3] = {&P.pass1_live, &P.pass2_live, &P.pass3_live};
            uint64_t* M[3] = {&P.pass1_members, &P.pass2_members, &P.pass3_members};
            uint64_t* X[3] = {&P.pass1_examined, &P.pass2_examined, &P.pass3_examined};
            for (int i = 0; i < 3; i++) {
                *L[i] += 1;
                *T[i] += t[i];
                *S[i] += sets[i];
                *W[i] += h.width[i];
                *V[i] += h.live[i];
                *M[i] += h.memb[i];
                *X[i] += h.exam[i];
            }
        }
        if (res) {
            res->ksum = ((unsigned __int128)h.ksum_hi << 64) | h.ksum_lo;
            res->wsum = h.wsum;
            res->live = h.live[0] + h.live[1] + h.live[2];
            res->covered = h.covered;
            res->members = emit ? h.pool_used : 0;
            res->big_sets = h.cnt1;
        }
        if (emit) {
            ctx->n_sets = count;
            ctx->members = h.pool_used;
            ctx->have_kpt = have_kpt;
        }
        return TIM_OK;
    }
    return tim_fail(ctx, TIM_ERR_OOM, "RR-set store kept overflowing");
}

// --------------------------------------------- several rounds of Algorithm 2 at once

namespace {

// Round blockIdx.y: sum of kappa over its sets' widths, of the widths and of the sizes.
__global__ void round_sums_kernel(SidMap ids, uint64_t count, const uint64_t* __restrict__ width,
                                  const uint32_t* __restrict__ len, uint64_t m, int k,
                                  RoundSums* __restrict__ out) {
    const uint32_t r = blockIdx.y;
    const uint64_t end = r + 1 < ids.n ? ids.start[r + 1] : count;
    unsigned long long lo = 0, hi = 0, w = 0, memb = 0;
    for (uint64_t j = ids.start[r] + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < end;
         j += (uint64_t)gridDim.x * blockDim.x) {
        const unsigned long long kf = kappa_fixed(kappa_fp64(width[j], m, k));
        lo += kf;
        if (lo < kf) hi++;
        w += width[j];
        memb += len[j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
        lo += l2;
        if (lo < l2) hi++;
    }
    w = warp_sum_u64(w);
    memb = warp_sum_u64(memb);
    if ((threadIdx.x & 31) == 0 && memb) {
        if (lo || hi) atomic_add_u128(&out[r].lo, &out[r].hi, lo, hi);
        atomicAdd(&out[r].width, w);
        atomicAdd(&out[r].members, memb);
    }
}

// Sets [start, start + count) of one store into another, one warp per set.
__global__ void keep_round_kernel(uint64_t start, uint64_t count,
                                  const uint32_t* __restrict__ pool,
                                  const uint64_t* __restrict__ set_start,
                                  const uint32_t* __restrict__ set_len,
                                  const uint64_t* __restrict__ set_width,
                                  uint32_t* __restrict__ pool_out, uint32_t* __restrict__ sid_out,
                                  uint64_t* __restrict__ start_out, uint32_t* __restrict__ len_out,
                                  uint64_t* __restrict__ width_out, DevScalars* ds) {
    const int lane = threadIdx.x & 31;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t j = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; j < count; j += nw) {
        const uint64_t from = set_start[start + j];
        const uint32_t len = set_len[start + j];
        unsigned long long to = 0;
        if (lane == 0) {
            to = atomicAdd(&ds->pool_used, (unsigned long long)len);
            start_out[j] = to;
            len_out[j] = len;
            width_out[j] = set_width[start + j];
        }
        to = __shfl_sync(0xffffffffu, to, 0);
        for (uint32_t i = lane; i < len; i += 32) {
            pool_out[to + i] = pool[from + i];
            sid_out[to + i] = (uint32_t)j;
        }
    }
}

void swap_stores(tim_ctx* ctx) {
    std::swap(ctx->pool, ctx->pool2);
    std::swap(ctx->pool_sid, ctx->pool_sid2);
    std::swap(ctx->set_start, ctx->set_start2);
    std::swap(ctx->set_len, ctx->set_len2);
    std::swap(ctx->set_width, ctx->set_width2);
}

}  // namespace

bool tim_drop_rounds(tim_ctx* ctx, bool all) {
    bool any = false;
    for (DevBuf* b : {&ctx->pool2, &ctx->pool_sid2, &ctx->set_start2, &ctx->set_len2,
                      &ctx->set_width2}) {
        any = any || b->p;
        tim_free(*b);
    }
    if (all)
        for (DevBuf* b : {&ctx->ovf_list, &ctx->ovf_list2, &ctx->hand, &ctx->hand2,
                          &ctx->bulk_bitmap, &ctx->bulk_slot})
            tim_free(*b);
    ctx->rounds_kept = false;
    return any;
}

int tim_sample_rounds(tim_ctx* ctx, SampleRequest req, const uint64_t* counts, int rounds,
                      RoundSums* sums) {
    req.rounds = rounds;
    req.count = 0;
    for (int r = 0; r < rounds; r++) {
        req.round_start[r] = (uint32_t)req.count;
        req.count += counts[r];
    }
    req.flags = SAMPLE_EMIT;
    swap_stores(ctx);
    SampleResult res;
    const int rc = tim_sample(ctx, req, &res);
    swap_stores(ctx);
    ctx->n_sets = ctx->members = 0;
    TIM_TRY(rc);
    ctx->rounds_kept = true;
    TIM_TRY(tim_ensure(ctx, ctx->round_sums, SID_ROUNDS * sizeof(RoundSums)));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->round_sums.p, 0, rounds * sizeof(RoundSums), ctx->stream));
    round_sums_kernel<<<dim3(ctx->num_sms, rounds), 128, 0, ctx->stream>>>(
        tim_sid_map(req), req.count, (const uint64_t*)ctx->set_width2.p,
        (const uint32_t*)ctx->set_len2.p, (uint64_t)ctx->m, req.k, (RoundSums*)ctx->round_sums.p);
    LAUNCH_CHECK(ctx, "round_sums_kernel");
    CUDA_TRY(ctx, cudaMemcpyAsync(sums, ctx->round_sums.p, rounds * sizeof(RoundSums),
                                  cudaMemcpyDeviceToHost, ctx->stream));
    return tim_sync(ctx);
}

int tim_keep_round(tim_ctx* ctx, uint64_t start, uint64_t count, uint64_t members) {
    TIM_TRY(tim_ensure(ctx, ctx->set_start, (count + 1) * sizeof(uint64_t)));
    TIM_TRY(tim_ensure(ctx, ctx->set_len, (count + 1) * sizeof(uint32_t)));
    TIM_TRY(tim_ensure(ctx, ctx->set_width, (count + 1) * sizeof(uint64_t)));
    TIM_TRY(ensure_pool(ctx, members));
    TIM_TRY(tim_zero_scalars(ctx));
    keep_round_kernel<<<(unsigned)(ctx->num_sms * 4), 256, 0, ctx->stream>>>(
        start, count, (const uint32_t*)ctx->pool2.p, (const uint64_t*)ctx->set_start2.p,
        (const uint32_t*)ctx->set_len2.p, (const uint64_t*)ctx->set_width2.p,
        (uint32_t*)ctx->pool.p, (uint32_t*)ctx->pool_sid.p, (uint64_t*)ctx->set_start.p,
        (uint32_t*)ctx->set_len.p, (uint64_t*)ctx->set_width.p, tim_dscal(ctx));
    LAUNCH_CHECK(ctx, "keep_round_kernel");
    ctx->n_sets = count;
    ctx->members = members;
    ctx->rounds_kept = false;
    return TIM_OK;
}

// ----------------------------------------------------- multi-query host driver

namespace {

// Tier-3 LT slots of one context: a visited bitmap of n bits and a queue of n entries
// each, at most ~2 GiB in total.
int ensure_lt_slots(tim_ctx* ctx, int* slots_out, uint64_t* words_out) {
    const uint64_t words = (uint64_t)(ctx->n + 31) / 32 + 1;
    const uint64_t per_slot = (words + (uint64_t)ctx->n) * sizeof(uint32_t);
    int slots = ctx->num_sms;
    const uint64_t budget = 2ull << 30;
    if ((uint64_t)slots * per_slot > budget) slots = (int)std::max<uint64_t>(1, budget / per_slot);
    const uint64_t made_bm = ctx->big_bitmap.made;
    TIM_TRY(tim_ensure(ctx, ctx->big_bitmap, (size_t)slots * words * sizeof(uint32_t)));
    TIM_TRY(tim_ensure(ctx, ctx->big_queue, (size_t)slots * (uint64_t)ctx->n * sizeof(uint32_t)));
    if (ctx->big_bitmap.made != made_bm || !ctx->big_bitmap_clean) {
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->big_bitmap.p, 0, ctx->big_bitmap.bytes, ctx->stream));
        ctx->big_bitmap_clean = true;
    }
    *slots_out = slots;
    *words_out = words;
    return TIM_OK;
}

// Tier 3 for one query of a multi-query launch: the sets list_dev[0 .. n3) of ctx's
// graph, accumulating into ds. Runs on `stream`.
int run_tier3(tim_ctx* ctx, cudaStream_t stream, const SampleRequest& req, DevScalars* ds,
              uint32_t* pool, uint32_t* pool_sid, uint64_t pool_cap, const uint32_t* list_dev,
              unsigned n3, uint64_t* live3) {
    cudaStream_t saved = ctx->stream;
    ctx->stream = stream;
    int rc = TIM_OK;
    if (ctx->model == TIM_IC) {
        rc = tim_bulk_ic(ctx, req, list_dev, n3, pool, pool_sid, pool_cap, ds, live3);
    } else {
        int slots = 0;
        uint64_t words = 0;
        rc = ensure_lt_slots(ctx, &slots, &words);
        if (rc == TIM_OK) {
            SampleArgs a{};
            a.node = (const uint4*)ctx->node.p;
            a.src = (const uint32_t*)ctx->src.p;
            a.thr = (const uint32_t*)ctx->thr.p;
            a.n = (uint64_t)ctx->n;
            a.m = (uint64_t)ctx->m;
            a.K = tim_philox_keys(req.seed);
            a.ids = tim_sid_map(req);
            a.count = req.count;
            a.flags = req.flags;
            a.k = req.k;
            a.seed_mark = req.seed_mark;
            a.pool = pool;
            a.pool_sid = pool_sid;
            a.pool_cap = pool_cap;
            a.set_start = (uint64_t*)ctx->set_start.p;
            a.set_len = (uint32_t*)ctx->set_len.p;
            a.set_width = (uint64_t*)ctx->set_width.p;
            a.ds = ds;
            a.list2 = const_cast<uint32_t*>(list_dev);
            a.list_cap = n3 + 1;
            a.big_bitmap = (uint32_t*)ctx->big_bitmap.p;
            a.big_queue = (uint32_t*)ctx->big_queue.p;
            a.big_words = words;
            a.chunk = 1;
            rc = tim_cuda_check(ctx, cudaMemcpyAsync(&ds->cnt2, &n3, sizeof(unsigned),
                                                     cudaMemcpyHostToDevice, stream),
                                "tier-3 count");
            if (rc == TIM_OK) rc = tim_cuda_check(ctx, cudaMemsetAsync(&ds->next3, 0, 8, stream), "memset");
            if (rc == TIM_OK) rc = tim_cuda_check(ctx, cudaStreamSynchronize(stream), "sync");
            if (rc == TIM_OK) {
                rr_lt_chain_kernel<<<slots, BIG_THREADS, 0, stream>>>(a);
                ctx->launches++;
                rc = tim_cuda_check(ctx, cudaGetLastError(), "rr_lt_chain_kernel");
            }
        }
        *live3 = 0;
    }
    ctx->stream = saved;
    return rc;
}

}  // namespace

int tim_sample_multi(tim_ctx* owner, MultiQuery* qs, int nq, uint64_t seed) {
    if (nq <= 0) return TIM_OK;
    if (nq > MAXQ) return tim_fail(owner, TIM_ERR_ARG, "too many queries in one launch");
    // IC queries are sampled by rr_multi_kernel over their own set index space, LT
    // queries by rr_lt_lane_multi_kernel over theirs
    std::vector<unsigned long long> prefix(nq + 1, 0), prefix_lt(nq + 1, 0);
    uint64_t total = 0, total_ic = 0, total_lt = 0;
    for (int i = 0; i < nq; i++) {
        tim_ctx* c = qs[i].ctx;
        if (!c || !c->have_graph) return tim_fail(owner, TIM_ERR_STATE, "query without a graph");
        if (c->device != owner->device) return tim_fail(owner, TIM_ERR_ARG, "queries on several devices");
        if (c->model == TIM_TRIG)
            return tim_fail(owner, TIM_ERR_ARG,
                            "the multi-query sampler takes IC and LT graphs; a triggering-model "
                            "graph runs one query at a time");
        const uint64_t count = qs[i].req.count;
        if (count > 0xFFFFFFF0ull) return tim_fail(owner, TIM_ERR_ARG, "too many RR sets in one call");
        prefix[i] = total_ic;
        prefix_lt[i] = total_lt;
        if (c->model == TIM_LT)
            total_lt += count;
        else
            total_ic += count;
        total += count;
        if (qs[i].req.flags & SAMPLE_EMIT) {
            open_store(c);
            uint64_t cap_sets = 1024;
            while (cap_sets < count + 1) cap_sets <<= 1;
            TIM_TRY(tim_ensure(c, c->set_start, cap_sets * sizeof(uint64_t)));
            TIM_TRY(tim_ensure(c, c->set_len, cap_sets * sizeof(uint32_t)));
            TIM_TRY(tim_ensure(c, c->set_width, cap_sets * sizeof(uint64_t)));
            TIM_TRY(ensure_pool(c, cap_sets * 8 + 4096));
        }
    }
    prefix[nq] = total_ic;
    prefix_lt[nq] = total_lt;
    if (total > 0xFFFFFFF0ull) return tim_fail(owner, TIM_ERR_ARG, "too many RR sets in one launch");
    // owner scratch: descriptors | IC prefix | per-query scalars | next[2] | cnt[2] | err |
    // LT work counter | LT prefix
    const size_t off_prefix = ((size_t)nq * sizeof(QueryDesc) + 255) & ~size_t(255);
    const size_t off_scal = (off_prefix + (size_t)(nq + 1) * 8 + 255) & ~size_t(255);
    const size_t off_ctr = (off_scal + (size_t)nq * sizeof(DevScalars) + 255) & ~size_t(255);
    const size_t off_prefix_lt = off_ctr + 64;
    const size_t batch_bytes = off_prefix_lt + (size_t)(nq + 1) * 8;
    TIM_TRY(tim_ensure(owner, owner->batch, batch_bytes));
    char* bb = (char*)owner->batch.p;
    QueryDesc* d_desc = (QueryDesc*)bb;
    unsigned long long* d_prefix = (unsigned long long*)(bb + off_prefix);
    DevScalars* d_scal = (DevScalars*)(bb + off_scal);
    unsigned long long* d_next = (unsigned long long*)(bb + off_ctr);
    unsigned* d_cnt = (unsigned*)(bb + off_ctr + 16);
    int* d_err = (int*)(bb + off_ctr + 24);
    unsigned long long* d_lt_next = (unsigned long long*)(bb + off_ctr + 32);
    unsigned long long* d_prefix_lt = (unsigned long long*)(bb + off_prefix_lt);
    unsigned grid_lt = 0;
    if (total_lt > 0) {
        int nb = 0;
        CUDA_TRY(owner, cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                            &nb, rr_lt_lane_multi_kernel, LT_THREADS, LT_SMEM));
        grid_lt = (unsigned)(owner->num_sms * std::max(nb, 1));
        TIM_TRY(tim_ensure(owner, owner->lt_col,
                           (size_t)grid_lt * LT_THREADS * LT_CAP * sizeof(uint32_t)));
    }
    TIM_TRY(tim_ensure(owner, owner->ovf_list, (size_t)(total + 1) * sizeof(uint2)));
    TIM_TRY(tim_ensure(owner, owner->ovf_list2, (size_t)(total + 1) * sizeof(uint2)));
    // arena and occupancy as in the single-query path
    const PackPlan<MultiArgs> plan =
        pack_plan(owner, total_ic, rr_pack_multi_kernel<PackS>,
                  rr_pack_multi_kernel<PackM>, rr_pack_multi_kernel<PackL>);
    const int nb2 = occupancy(rr_multi_kernel<Tier2, 1>, 0);
    const unsigned grid2 = (unsigned)(owner->num_sms * nb2);
    const size_t arena_bytes = (size_t)grid2 * WARPS * Tier2::WORDS * sizeof(uint32_t);
    const uint64_t made_arena = owner->arena.made;
    TIM_TRY(tim_ensure(owner, owner->arena, arena_bytes));
    if (owner->arena.made != made_arena || !owner->arena_clean) {
        CUDA_TRY(owner, cudaMemsetAsync(owner->arena.p, 0xFF, owner->arena.bytes, owner->stream));
        owner->arena_clean = true;
    }
    MultiArgs ma;
    ma.K = tim_philox_keys(seed);
    ma.q = d_desc;
    ma.prefix = d_prefix;
    ma.nq = nq;
    ma.chunk = std::max(1, owner->chunk);
    ma.inflight = plan.inflight;
    ma.next = d_next;
    ma.cnt = d_cnt;
    ma.err = d_err;
    ma.list1 = (uint2*)owner->ovf_list.p;
    ma.list2 = (uint2*)owner->ovf_list2.p;
    ma.list_cap = (uint32_t)(total + 1);
    ma.arena = (uint32_t*)owner->arena.p;
    ma.bm_words = 1;
    for (int i = 0; i < nq; i++)
        ma.bm_words = std::max(ma.bm_words, (uint32_t)((uint64_t)qs[i].ctx->n / 32 + 1));
    // pass-1 state handed to pass 2 (IC queries), in the owner's scratch
    ma.hw = 4u + (uint32_t)plan.members;
    {
        const uint64_t maxslots = (1ull << 30) / ((uint64_t)ma.hw * sizeof(uint32_t));
        const uint64_t hcap =
            std::min<uint64_t>(std::min<uint64_t>(total_ic / 2 + 4096, maxslots), total + 1);
        TIM_TRY(tim_ensure(owner, owner->hand, (size_t)hcap * ma.hw * sizeof(uint32_t)));
        ma.hand = (uint32_t*)owner->hand.p;
        ma.hcap = (uint32_t)hcap;
    }
    std::vector<QueryDesc> h_desc(nq);
    std::vector<DevScalars> h_scal(nq);
    for (int attempt = 0; attempt < 4; attempt++) {
        for (int i = 0; i < nq; i++) {
            tim_ctx* c = qs[i].ctx;
            const SampleRequest& r = qs[i].req;
            QueryDesc& d = h_desc[i];
            d.node = (const uint4*)c->node.p;
            d.src = (const uint32_t*)c->src.p;
            d.thr = (const uint32_t*)c->thr.p;
            d.qtab = (const unsigned long long*)c->qtab.p;
            d.n = (uint64_t)c->n;
            d.m = (uint64_t)c->m;
            d.sid0 = r.sid0;
            d.count = r.count;
            d.model = c->model;
            d.flags = r.flags;
            d.k = r.k;
            d.pad = 0;
            d.seed_mark = r.seed_mark;
            const bool emit = r.flags & SAMPLE_EMIT;
            d.pool = emit ? (uint32_t*)c->pool.p : nullptr;
            d.pool_sid = emit ? (uint32_t*)c->pool_sid.p : nullptr;
            d.pool_cap = emit ? pool_entries(c) : 0;
            d.set_start = (uint64_t*)c->set_start.p;
            d.set_len = (uint32_t*)c->set_len.p;
            d.set_width = (uint64_t*)c->set_width.p;
            d.ds = d_scal + i;
            d.width_budget = c->width_budget;
            d.width_budget2 = c->width_budget2;
        }
        CUDA_TRY(owner, cudaMemcpyAsync(d_desc, h_desc.data(), (size_t)nq * sizeof(QueryDesc),
                                        cudaMemcpyHostToDevice, owner->stream));
        CUDA_TRY(owner, cudaMemcpyAsync(d_prefix, prefix.data(), (size_t)(nq + 1) * 8,
                                        cudaMemcpyHostToDevice, owner->stream));
        CUDA_TRY(owner, cudaMemcpyAsync(d_prefix_lt, prefix_lt.data(), (size_t)(nq + 1) * 8,
                                        cudaMemcpyHostToDevice, owner->stream));
        CUDA_TRY(owner, cudaMemsetAsync(d_scal, 0, (size_t)nq * sizeof(DevScalars), owner->stream));
        CUDA_TRY(owner, cudaMemsetAsync(d_next, 0, 64, owner->stream));
        uint64_t live3_total = 0;
        std::vector<uint64_t> live3(nq, 0);
        if (total > 0) {
            if (total_ic > 0) {
                plan.kernel<<<plan.grid, WARPS * 32, plan.smem, owner->stream>>>(ma);
                LAUNCH_CHECK(owner, "rr_pack_multi_kernel (tier 1)");
            }
            if (total_lt > 0) {
                rr_lt_lane_multi_kernel<<<grid_lt, LT_THREADS, LT_SMEM, owner->stream>>>(
                    ma, d_prefix_lt, d_lt_next, (uint32_t*)owner->lt_col.p);
                LAUNCH_CHECK(owner, "rr_lt_lane_multi_kernel (tier 1)");
            }
            unsigned h_cnt[2] = {0, 0};
            CUDA_TRY(owner, cudaMemcpyAsync(h_cnt, d_cnt, sizeof h_cnt, cudaMemcpyDeviceToHost,
                                            owner->stream));
            TIM_TRY(tim_sync(owner));
            int T = owner->team_size;
            if (T <= 0) {
                T = 1;
                const uint64_t slots1 = (uint64_t)grid2 * WARPS;
                while (T < 8 && (uint64_t)h_cnt[0] * (uint64_t)owner->team_factor < slots1 / T)
                    T *= 2;
            }
            ma.bm_shared = bitmap_smem(ma.bm_words, T) > 0;
            TIM_TRY(launch_multi(owner, ma, T, grid2));
            CUDA_TRY(owner, cudaMemcpyAsync(h_cnt, d_cnt, sizeof h_cnt, cudaMemcpyDeviceToHost,
                                            owner->stream));
            TIM_TRY(tim_sync(owner));
            const unsigned n3 = std::min<unsigned>(h_cnt[1], ma.list_cap);
            if (n3 > 0) {
                // the rare sets beyond tier 2: per query, with that query's context
                std::vector<uint2> l2(n3);
                CUDA_TRY(owner, cudaMemcpyAsync(l2.data(), ma.list2, (size_t)n3 * sizeof(uint2),
                                                cudaMemcpyDeviceToHost, owner->stream));
                TIM_TRY(tim_sync(owner));
                std::vector<std::vector<uint32_t>> per(nq);
                for (const uint2& e : l2) per[e.x].push_back(e.y);
                for (int i = 0; i < nq; i++) {
                    if (per[i].empty()) continue;
                    tim_ctx* c = qs[i].ctx;
                    TIM_TRY(tim_ensure(c, c->ovf_list2, per[i].size() * sizeof(uint32_t)));
                    CUDA_TRY(owner, cudaMemcpyAsync(c->ovf_list2.p, per[i].data(),
                                                    per[i].size() * sizeof(uint32_t),
                                                    cudaMemcpyHostToDevice, owner->stream));
                    SampleRequest r = qs[i].req;
                    TIM_TRY(run_tier3(c, owner->stream, r, d_scal + i, h_desc[i].pool,
                                      h_desc[i].pool_sid, h_desc[i].pool_cap,
                                      (const uint32_t*)c->ovf_list2.p, (unsigned)per[i].size(),
                                      &live3[i]));
                    live3_total += live3[i];
                }
            }
        }
        CUDA_TRY(owner, cudaMemcpyAsync(h_scal.data(), d_scal, (size_t)nq * sizeof(DevScalars),
                                        cudaMemcpyDeviceToHost, owner->stream));
        int h_err = 0;
        CUDA_TRY(owner, cudaMemcpyAsync(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost,
                                        owner->stream));
        TIM_TRY(tim_sync(owner));
        bool regrow = false;
        for (int i = 0; i < nq; i++) {
            if (h_scal[i].err & TIM_DEV_ERR_POOL) {
                TIM_TRY(regrow_pool(qs[i].ctx, h_scal[i].pool_used));
                regrow = true;
            } else if (h_scal[i].err) {
                h_err |= h_scal[i].err;
            }
        }
        if (regrow) continue;
        if (h_err) {
            owner->arena_clean = false;
            return tim_fail(owner, TIM_ERR_CUDA, "device error flags set by the multi-query sampler");
        }
        for (int i = 0; i < nq; i++) {
            const DevScalars& h = h_scal[i];
            SampleResult& res = qs[i].res;
            res.ksum = ((unsigned __int128)h.ksum_hi << 64) | h.ksum_lo;
            res.wsum = h.wsum;
            res.live = h.live[0] + h.live[1] + live3[i];
            res.covered = h.covered;
            const bool emit = qs[i].req.flags & SAMPLE_EMIT;
            res.members = emit ? h.pool_used : 0;
            res.big_sets = 0;
            if (emit) {
                qs[i].ctx->n_sets = qs[i].req.count;
                qs[i].ctx->members = h.pool_used;
            }
        }
        (void)live3_total;
        return TIM_OK;
    }
    return tim_fail(owner, TIM_ERR_OOM, "RR-set stores kept overflowing");
}
