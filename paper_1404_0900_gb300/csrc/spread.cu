// spread.cu -- forward Monte-Carlo spread of a seed set (Section 2.1: E[I(S)] estimated
// as the average number of nodes reachable from S in random graphs g, every edge kept
// with its propagation probability; Section 4.2: under a triggering model every node
// keeps the in-edges of its sampled triggering set; Section 7 averages 10^5 cascades).
//
// Cascade c walks the world of set id sid = first_set_id + c with the keys of the RR
// sets: the IC in-edge at in-CSR position j is kept iff word (j & 3) of Philox(seed;
// sid, j >> 2, TAG_IC) is below its threshold (one coin per in-edge, also in lists that
// RR sampling treats by geometric skipping), under LT node v keeps the in-edge that
// word 0 of Philox(seed; sid, v, TAG_LT) picks, and under a general triggering model the
// in-edges of the option that the same word picks. Where no list is skipped, the RR set
// of sid is then exactly the set of nodes that reach its root in this cascade's world.
//
// The walk needs G itself: out-records {in-CSR position, destination} grouped by
// source, and the inverse (out-record index of every in-CSR position), built from G^T on
// first use. A block per cascade, after a pass of a warp per cascade over calls of many (the
// small ones end there, mc_light_kernel). The visited bitmap (n bits) sits in shared memory
// when it fits there, the queue (the activated nodes, n slots) and the live-edge bits
// (below) in global memory, one set per resident block. A round expands the nodes the
// round before added; a round that adds nothing ends the cascade.
//
// A round runs in one of two ways. Walking tests every out-edge of the round's nodes by
// its own draw (a Philox block per edge: the in-CSR positions of one node's out-edges are
// scattered). Drawing evaluates the cascade's whole world once: IC draws the coins of
// four consecutive in-CSR positions with one Philox block and 16 contiguous bytes of
// thresholds, LT and triggering models make one pick per unvisited node, and every live
// edge sets one bit at its out-record; from then on a node's live out-edges are read 32
// to a word. A cascade starts walking and draws its world when the out-edges it
// would have walked by the end of the next round pass a fixed share (MC_WALK) of the draws
// that the world takes (m / 4 blocks for IC, n picks otherwise) and it grows: small cascades
// never pay for a world, large ones walk little before they do. Against walking alone (one 256-thread
// block per cascade, one warp per node): 50 seeds on R-MAT 18, 2000 IC cascades 42.2 -> 10.9
// ms, 1000 LT cascades 70.4 -> 7.4 ms. Drawing is bound by issue (Philox) and by the one L1
// sector per clock of scattered out-record indexes and bit updates, the rounds by their
// chains of dependent loads.
#include <algorithm>

#include "common.cuh"

namespace {

// largest visited bitmaps kept in shared memory, one and two per SM (n up to 1.55 million
// and 0.65 million nodes), beside the blocks' stages
constexpr uint64_t MC_SMEM_MAX = 190 * 1024, MC_SMEM_TWO = 80 * 1024;

__global__ void out_count_kernel(const uint32_t* __restrict__ src, uint64_t m,
                                 uint32_t* __restrict__ cnt) {
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < m;
         j += (uint64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[__ldg(src + j)], 1u);
}

// Rows of the out-records as one 8-byte word per node (m < 2^32): one load per node.
__global__ void out_rows_kernel(const uint64_t* __restrict__ out_rowptr, uint64_t n,
                                uint2* __restrict__ out_row) {
    for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n;
         v += (uint64_t)gridDim.x * blockDim.x)
        out_row[v] = make_uint2((uint32_t)out_rowptr[v], (uint32_t)out_rowptr[v + 1]);
}

// One warp per destination v: each in-edge j = (u -> v) becomes out-record {j, v} of u.
__global__ void out_scatter_kernel(const uint64_t* __restrict__ rowptr,
                                   const uint32_t* __restrict__ src, uint64_t n,
                                   const uint64_t* __restrict__ out_rowptr,
                                   uint32_t* __restrict__ cursor, uint2* __restrict__ out_rec,
                                   uint32_t* __restrict__ out_pos) {
    const int lane = threadIdx.x & 31;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t v = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
        const uint64_t b = rowptr[v], e = rowptr[v + 1];
        for (uint64_t j = b + lane; j < e; j += 32) {
            const uint32_t u = __ldg(src + j);
            const uint32_t slot = atomicAdd(&cursor[u], 1u);
            const uint64_t at = out_rowptr[u] + slot;
            out_rec[at] = make_uint2((uint32_t)j, (uint32_t)v);
            if (out_pos) out_pos[j] = (uint32_t)at;
        }
    }
}

struct McArgs {
    const uint4* node;  // node records
    const uint32_t* thr;
    const uint2* out_row;
    const uint2* out_rec;
    const uint32_t* out_pos;
    int model;
    uint64_t n, m;
    PhiloxKeys K;
    uint64_t sid0, count;
    const int32_t* seeds;
    int k;
    uint32_t* bitmap;  // slots * words (unless the bitmaps sit in shared memory)
    uint32_t* queue;   // slots * n
    uint64_t words;
    uint32_t* live;    // slots * live_words: bit e = out-record e is live
    uint64_t live_words;          // a multiple of 4
    unsigned long long draw_at;   // out-edges a cascade walks at most; ~0: never draws
    uint32_t* counts;              // per cascade
    unsigned long long* scal;      // [0] next cascade, [1] total activated, [2] cascades listed
    uint32_t* list;                // cascades that the warps left to the blocks; null: all
    // triggering model: options per node, cumulative thresholds, sorted in-CSR positions
    const uint64_t* node_opt;
    const uint32_t* opt_cum;
    const uint64_t* opt_off;
    const uint32_t* opt_pos;
};

// The in-edge node v keeps in the world of sid (LT), or the end of its in-list for none.
__device__ __forceinline__ uint64_t lt_pick(const McArgs& a, uint32_t s0, uint32_t s1, uint32_t v,
                                            uint64_t* end_out) {
    const uint4 rec = __ldg(a.node + v);
    const uint64_t beg = rec.x, end = rec.y;
    const uint32_t x = philox4x32_10(s0, s1, v, TIM_TAG_LT, a.K).x;
    const unsigned long long nt = node_nt(rec);
    *end_out = end;
    return (nt >> 32) ? lt_uniform_pick(nt, beg, end, x) : lane_lt_search(a.thr, beg, end, x);
}

// The option node v picks in the world of sid (triggering model): its positions are
// opt_pos[*lo .. *hi), none when they are equal.
__device__ __forceinline__ void trig_pick(const McArgs& a, uint32_t s0, uint32_t s1, uint32_t v,
                                          uint64_t* lo, uint64_t* hi) {
    *lo = *hi = 0;
    const uint64_t o0 = __ldg(a.node_opt + v), o1 = __ldg(a.node_opt + v + 1);
    if (o1 == o0) return;
    const uint32_t x = philox4x32_10(s0, s1, v, TIM_TAG_LT, a.K).x;
    const uint64_t o = lane_lt_search(a.opt_cum, o0, o1, x);
    if (o >= o1) return;
    *lo = __ldg(a.opt_off + o);
    *hi = __ldg(a.opt_off + o + 1);
}

// Does v keep in-edge j in the world of sid?
__device__ __forceinline__ bool edge_kept(const McArgs& a, uint32_t s0, uint32_t s1, uint32_t v,
                                          uint32_t j) {
    if (a.model == TIM_IC) {
        const uint4 x = philox4x32_10(s0, s1, j >> 2, TIM_TAG_IC, a.K);
        const uint32_t w = (j & 3) == 0 ? x.x : (j & 3) == 1 ? x.y : (j & 3) == 2 ? x.z : x.w;
        const uint32_t t = __ldg(a.thr + j);
        return t == 0xFFFFFFFFu || w < t;
    }
    if (a.model == TIM_TRIG) {
        uint64_t lo, hi;
        trig_pick(a, s0, s1, v, &lo, &hi);
        const uint64_t stop = hi;
        for (int it = 0; it < 40 && lo < hi; it++) {  // first position >= j (ascending)
            const uint64_t mid = lo + ((hi - lo) >> 1);
            if (__ldg(a.opt_pos + mid) < j)
                lo = mid + 1;
            else
                hi = mid;
        }
        return lo < stop && __ldg(a.opt_pos + lo) == j;
    }
    uint64_t end;
    const uint64_t p = lt_pick(a, s0, s1, v, &end);
    return p < end && p == (uint64_t)j;
}

__device__ __forceinline__ void set_live(const McArgs& a, uint32_t* live, uint64_t j) {
    const uint32_t e = __ldg(a.out_pos + j);
    atomicOr(&live[e >> 5], 1u << (e & 31));
}

// A cascade walks at most 1 / MC_WALK as many out-edges as drawing its world takes draws: a
// walked edge costs about three of them, and a cascade that has walked this much mostly
// goes on (MC_WALK 2, 4, 12, 24: 50 seeds on R-MAT 18, IC, 16.0, 15.0, 11.1, 11.1 ms; one
// seed on a 200,001-node Chung-Lu graph, 1000 cascades, 6.2, 4.9, 3.7, 3.6 ms).
constexpr unsigned MC_WALK = 12;
// It goes on walking, up to MC_SURE times that share, while its rounds are small (a world costs
// 20 of them or more) and do not grow: a cascade that neither grows nor dies out walks a
// fraction of what its world takes. Growing: the next round has an eighth of the out-edges of all
// rounds before it and half as many again as their average. (Random graph of 600,001 nodes, 38M
// edges, p = 0.0155, 500 cascades of 200 seeds: drawing at the share alone 25.3 ms, walking alone
// 14.2, here 14.8; 60,001 nodes, 2000 of 10 seeds 2.74, 1.81, 1.24.)
constexpr float MC_SURE = 6.f;

// Live in-CSR positions a warp collects (in shared memory) before it sets their bits, four
// per lane in flight: setting each one as it is found would wait for its out-record index
// every time.
constexpr uint32_t MC_STAGE = 256;

__device__ __forceinline__ void flush_live(const McArgs& a, uint32_t* live, const uint32_t* st,
                                           uint32_t cnt, int lane) {
    __syncwarp();
    for (uint32_t i = lane; i < cnt; i += 128) {
        uint32_t e[4];
#pragma unroll
        for (int k = 0; k < 4; k++) e[k] = i + 32 * k < cnt ? __ldg(a.out_pos + st[i + 32 * k]) : 0u;
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (i + 32 * k < cnt) atomicOr(&live[e[k] >> 5], 1u << (e[k] & 31));
    }
    __syncwarp();
}

// The world of sid as live bits over the out-records (all of the block's threads). Bound by
// issue for IC (the Philox rounds of m / 4 blocks); nodes already visited need no pick.
__device__ __forceinline__ void draw_world(const McArgs& a, uint32_t s0, uint32_t s1,
                                           const uint32_t* bm, uint32_t* live,
                                           uint32_t* stage) {
    const int lane = threadIdx.x & 31;
    uint4* l4 = reinterpret_cast<uint4*>(live);
    for (uint64_t w = threadIdx.x; w < a.live_words >> 2; w += blockDim.x)
        l4[w] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (a.model == TIM_IC) {
        const uint4* thr4 = reinterpret_cast<const uint4*>(a.thr);
        const uint32_t groups = (uint32_t)((a.m + 3) >> 2);  // thr is zero past its end
        uint32_t* st = stage + (threadIdx.x >> 5) * MC_STAGE;
        uint32_t held = 0;
        // four groups per thread and step: their loads overlap, and the live in-edges of all
        // four (about one in sixteen coins under weighted cascade) share one loop
        for (uint32_t gw = threadIdx.x & ~31u; gw < groups; gw += 4 * blockDim.x) {
            const uint32_t g0 = gw + lane;
            uint32_t lm = 0;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint32_t g = g0 + i * blockDim.x;
                const uint4 t = g < groups ? __ldg(thr4 + g) : make_uint4(0u, 0u, 0u, 0u);
                const uint4 x = philox4x32_10(s0, s1, g, TIM_TAG_IC, a.K);
                lm |= ((x.x < t.x || t.x == 0xFFFFFFFFu ? 1u : 0u) |
                       (x.y < t.y || t.y == 0xFFFFFFFFu ? 2u : 0u) |
                       (x.z < t.z || t.z == 0xFFFFFFFFu ? 4u : 0u) |
                       (x.w < t.w || t.w == 0xFFFFFFFFu ? 8u : 0u)) << (4 * i);
            }
            const uint32_t cnt = __popc(lm);
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            if (held + total > MC_STAGE) {
                flush_live(a, live, st, held, lane);
                held = 0;
            }
            uint32_t at = held + incl - cnt;
            const bool fits = total <= MC_STAGE;
            for (; lm; lm &= lm - 1) {
                const uint32_t b = __ffs(lm) - 1;
                const uint32_t j = ((g0 + (b >> 2) * blockDim.x) << 2) + (b & 3);
                if (fits)
                    st[at++] = j;
                else
                    set_live(a, live, j);
            }
            if (fits) held += total;
        }
        flush_live(a, live, st, held, lane);
    } else if (a.model == TIM_TRIG) {
        // the picked options' positions, flattened over the warp's lanes
        for (uint64_t vw = threadIdx.x & ~31u; vw < a.n; vw += blockDim.x) {
            const uint64_t v = vw + lane;
            uint64_t lo = 0, hi = 0;
            if (v < a.n && !((bm[v >> 5] >> (v & 31)) & 1u))
                trig_pick(a, s0, s1, (uint32_t)v, &lo, &hi);
            const uint32_t cnt = (uint32_t)(hi - lo);
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            for (uint32_t base = 0; base < total; base += 32) {
                const uint32_t t = base + lane;
                int own = 0;  // number of lanes whose inclusive count is <= t
#pragma unroll
                for (int sft = 16; sft > 0; sft >>= 1) {
                    const uint32_t ic = __shfl_sync(0xffffffffu, incl, own + sft - 1);
                    if (ic <= t) own += sft;
                }
                const uint64_t ol = __shfl_sync(0xffffffffu, lo, own);
                const uint32_t ox = __shfl_sync(0xffffffffu, incl - cnt, own);
                if (t < total) set_live(a, live, __ldg(a.opt_pos + ol + (t - ox)));
            }
        }
    } else {
        // four picks per thread in flight
        for (uint64_t v0 = threadIdx.x; v0 < a.n; v0 += 4 * blockDim.x) {
            uint64_t p[4], end[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint64_t v = v0 + i * blockDim.x;
                p[i] = end[i] = 0;
                if (v < a.n && !((bm[v >> 5] >> (v & 31)) & 1u))
                    p[i] = lt_pick(a, s0, s1, (uint32_t)v, &end[i]);
            }
            uint32_t e[4];
#pragma unroll
            for (int i = 0; i < 4; i++) e[i] = p[i] < end[i] ? __ldg(a.out_pos + p[i]) : 0u;
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (p[i] < end[i]) atomicOr(&live[e[i] >> 5], 1u << (e[i] & 31));
        }
    }
    __syncthreads();
}

// Cascades that stay small, a warp each: members and their hash in shared memory, walked edge by
// edge. One that outgrows LIGHT_Q members or LIGHT_EDGES out-edges is listed and starts over in
// a block of mc_cascade_kernel. What such a cascade takes is its chain of dependent loads, so what
// counts is how many are in flight: 7,296 warps, against 152 or 304 blocks, each of which
// also has barriers to pass and a bitmap to clear. Used for calls of more than four times as many
// cascades as blocks (with fewer the blocks are faster) from at most LIGHT_Q / 2 seeds.
// (20,000 weighted-cascade cascades of one node of low out-degree, Chung-Lu 600,001 and 1,000,003
// nodes, R-MAT 16: a block of 256 threads each 0.19, 0.20, 1.47 ms; the large blocks alone 0.37,
// 0.68, 0.77; here 0.12, 0.14, 0.53. LIGHT_Q 256 with 2048 out-edges: within 10 % either way.)
constexpr int LIGHT_THREADS = 256, LIGHT_BLOCKS = 6;
constexpr int LIGHT_Q = 128;
constexpr int LIGHT_LOG2H = 8;  // 256 slots for at most LIGHT_Q + 31 nodes
constexpr uint32_t LIGHT_EDGES = 1024;

__global__ void __launch_bounds__(LIGHT_THREADS, LIGHT_BLOCKS) mc_light_kernel(McArgs a) {
    constexpr uint32_t H = 1u << LIGHT_LOG2H, NONE = 0xFFFFFFFFu;
    __shared__ uint32_t s_hash[LIGHT_THREADS / 32][H], s_queue[LIGHT_THREADS / 32][LIGHT_Q];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *hash = s_hash[wid], *q = s_queue[wid];
    for (uint32_t i = lane; i < H; i += 32) hash[i] = NONE;
    __syncwarp();
    const uint64_t nw = (uint64_t)gridDim.x * (LIGHT_THREADS / 32);
    unsigned long long all = 0;
    for (uint64_t c = blockIdx.x * (uint64_t)(LIGHT_THREADS / 32) + wid; c < a.count; c += nw) {
        const uint64_t sid = a.sid0 + c;
        const uint32_t s0 = (uint32_t)sid, s1 = (uint32_t)(sid >> 32);
        int tail = 0;
        bool heavy = false;
        auto add = [&](bool want, uint32_t v) {
            bool fresh = false;
            if (want) {
                uint32_t h = (v * 0x9E3779B1u) >> (32 - LIGHT_LOG2H);
                for (uint32_t p = 0; p < H; p++) {
                    const uint32_t old = atomicCAS(&hash[h], NONE, v);
                    fresh = old == NONE;
                    if (fresh || old == v) break;
                    h = (h + 1) & (H - 1);
                }
            }
            const uint32_t fm = __ballot_sync(0xffffffffu, fresh);
            const int at = tail + __popc(fm & ((1u << lane) - 1u));
            if (fresh && at < LIGHT_Q) q[at] = v;
            tail += __popc(fm);
            heavy = tail > LIGHT_Q;
            __syncwarp();
        };
        for (int i = 0; i < a.k && !heavy; i += 32)
            add(i + lane < a.k, i + lane < a.k ? (uint32_t)a.seeds[i + lane] : 0u);
        uint32_t edges = 0;
        for (int head = 0; head < tail && !heavy;) {
            const int nb = min(32, tail - head);
            uint2 row = make_uint2(0u, 0u);
            if (lane < nb) row = __ldg(a.out_row + q[head + lane]);
            head += nb;
            uint32_t incl = row.y - row.x;  // distinct rows: fewer than 2^32 edges together
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            heavy = total > LIGHT_EDGES - edges;
            if (heavy) break;
            edges += total;
            const uint32_t first = row.x - (incl - (row.y - row.x));
            for (uint32_t base = 0; base < total && !heavy; base += 32) {
                const uint32_t t = base + lane;
                int own = 0;  // number of lanes whose inclusive count is <= t
#pragma unroll
                for (int sft = 16; sft > 0; sft >>= 1) {
                    const uint32_t ic = __shfl_sync(0xffffffffu, incl, own + sft - 1);
                    if (ic <= t) own += sft;
                }
                const uint32_t at = __shfl_sync(0xffffffffu, first, own) + t;
                uint2 r = make_uint2(0u, 0u);
                if (t < total) r = __ldg(a.out_rec + at);
                add(t < total && edge_kept(a, s0, s1, r.y, r.x), r.y);
            }
        }
        for (uint32_t i = lane; i < H; i += 32) hash[i] = NONE;
        __syncwarp();
        if (lane == 0 && heavy) {
            a.list[atomicAdd(&a.scal[2], 1ull)] = (uint32_t)c;
        } else if (lane == 0) {
            a.counts[c] = (uint32_t)tail;
            all += tail;
        }
    }
    if (lane == 0 && all) atomicAdd(&a.scal[1], all);
}

// With the bitmap in shared memory: members up to which it is cleared through the queue (clearing
// all of its words takes about as long as this many stores).
constexpr uint32_t MC_LIST = 4096;

// SM: the visited bitmap in shared memory (n bits of dynamic shared memory).
template <bool SM, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS) mc_cascade_kernel(McArgs a) {
    extern __shared__ uint32_t s_bm[];
    __shared__ uint32_t s_stage[THREADS / 32 * MC_STAGE];
    __shared__ unsigned long long s_c, s_edges;
    // round r expands s_tail[r % 3] nodes, claimed through s_next[r % 2], and counts the next
    // round's in s_tail[(r + 1) % 3]; the third and the other are cleared meanwhile
    __shared__ uint32_t s_tail[3], s_next[2], s_draw;
    const uint32_t count = (uint32_t)(a.list ? __ldcg(&a.scal[2]) : a.count);
    if (blockIdx.x >= count) return;
    const int lane = threadIdx.x & 31;
    constexpr uint32_t W = THREADS / 32;
    uint32_t* bm = SM ? s_bm : a.bitmap + (uint64_t)blockIdx.x * a.words;
    uint32_t* q = a.queue + (uint64_t)blockIdx.x * a.n;
    uint32_t* live = a.live + (uint64_t)blockIdx.x * a.live_words;
    uint32_t* st = s_stage + (threadIdx.x >> 5) * MC_STAGE;
    if (SM)
        for (uint32_t w = threadIdx.x; w < (uint32_t)a.words; w += blockDim.x) bm[w] = 0u;
    // The round's nodes are q[cur .. ] and the next round's q[nxt .. ], step +1 or -1. The
    // rounds follow one another, so that the bitmap can be cleared through the queue. With the
    // bitmap in shared memory the rounds of a cascade of more than MC_LIST nodes fill the queue
    // from its two ends in turn (the nodes of two rounds are distinct, so they fit), which
    // keeps its lines in L2.
    int cur = 0, nxt = 0, dcur = 1, dnxt = 1;
    uint32_t to = 0;  // the next round's nodes are counted in s_tail[to]
    auto add = [&](uint32_t v) {
        const uint32_t b = 1u << (v & 31);
        if (!(atomicOr(&bm[v >> 5], b) & b))
            q[nxt + dnxt * (int)atomicAdd(&s_tail[to], 1u)] = v;
    };
    // a plain read first: a stale zero only costs a draw or an atomic
    auto seen = [&](uint32_t v) {
        return ((SM ? ((volatile uint32_t*)bm)[v >> 5] : __ldcg(bm + (v >> 5))) >> (v & 31)) & 1u;
    };
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned long long i = atomicAdd(&a.scal[0], 1ull);
            s_c = i >= count ? ~0ull : a.list ? __ldcg(a.list + i) : i;
            s_tail[0] = s_tail[1] = s_next[0] = s_draw = 0u;
        }
        __syncthreads();
        const unsigned long long c = s_c;
        if (c == ~0ull) break;
        const uint64_t sid = a.sid0 + c;
        const uint32_t s0 = (uint32_t)sid, s1 = (uint32_t)(sid >> 32);
        nxt = 0;
        dnxt = 1;
        to = 0;
        bool ends = false;
        for (int i = threadIdx.x; i < a.k; i += blockDim.x) add((uint32_t)a.seeds[i]);
        __syncthreads();
        uint32_t act = 0;  // nodes of the rounds before
        bool drawn = false;
        float walked = 0.f;  // out-edges of the rounds before
        // every round either adds a node or ends the cascade: at most n + 1 rounds
        for (uint32_t round = 0; round <= (uint32_t)a.n; round++) {
            const uint32_t f = s_tail[to];
            if (f == 0) break;
            cur = nxt;
            dcur = dnxt;
            if (SM && act + f > MC_LIST) {
                nxt = ends && dcur < 0 ? 0 : (int)a.n - 1;
                dnxt = ends ? -dcur : -1;
                ends = true;
            } else {
                nxt = cur + (int)f;
            }
            act += f;
            to = to == 2 ? 0 : to + 1;
            if (threadIdx.x == 0) {
                s_tail[to == 2 ? 0 : to + 1] = 0;
                s_next[(round + 1) & 1] = 0;
            }
            // a round of at most 32 nodes: every warp holds all their rows and takes its share of
            // their edges, without claims. One barrier ends such a round (three when its nodes
            // are more; with four a round and rows claimed one by one: 500 cascades of 600 nodes in
            // fifty rounds 0.44 ms, here 0.37; one hub on R-MAT 18, 1000 cascades, 3.93 -> 3.15)
            const bool few = f <= 32;
            auto load_rows = [&]() {
                return few && (uint32_t)lane < f
                           ? __ldg(a.out_row + __ldcg(q + (cur + dcur * lane)))
                           : make_uint2(0u, 0u);
            };
            uint2 rows = load_rows();
            if (!drawn && a.draw_at != ~0ull) {
                float out;  // of this round
                if (few) {
                    out = (float)__reduce_add_sync(0xffffffffu, rows.y - rows.x);
                } else {
                    if (threadIdx.x == 0) s_edges = 0;
                    __syncthreads();
                    unsigned long long d = 0;
                    for (uint32_t i = threadIdx.x; i < f; i += THREADS) {
                        const uint32_t u = __ldcg(q + (cur + dcur * (int)i));
                        const uint2 row = __ldg(a.out_row + u);
                        d += row.y - row.x;
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                    if (lane == 0 && d) atomicAdd(&s_edges, d);
                    __syncthreads();
                    out = (float)s_edges;
                }
                const float at = (float)a.draw_at;
                const bool grows = 5.f * out >= at ||
                                   (8.f * out >= walked && 2.f * (float)round * out >= 3.f * walked);
                walked += out;
                if (walked > at && (grows || walked > MC_SURE * at)) {
                    if (threadIdx.x == 0) s_draw = 1u;
                    __syncthreads();
                }
            }
            // (decided by shared memory alone, as the set id comes from it: so that the branch and
            // the id are known to be the same for the whole block. The drawing takes a quarter
            // to 40 % longer otherwise: 1000 cascades of 50 seeds on R-MAT 18 3.4 -> 4.3 to 4.8 ms)
            if (s_draw) {
                draw_world(a, s0, s1, bm, live, s_stage);
                drawn = true;
                if (threadIdx.x == 0) s_draw = 0u;
                rows = load_rows();  // again: the drawing is 1.4 % faster with their registers
            }
            // otherwise warps claim the round's nodes, up to 32 at a time (fewer when the round
            // has few nodes for its warps). Rows are flattened over the lanes: one out-edge
            // per lane, or one word of 32 live bits
            const uint32_t per = min(32u, max(1u, f / W));
            const uint32_t start = few ? threadIdx.x & ~31u : 0u, half = few ? W * 32u : 32u;
            uint32_t held = 0;  // live out-records staged by this warp
            // destinations of the staged records, four per lane in flight; the new ones join
            // the queue with one counter update per warp
            auto take = [&]() {
                __syncwarp();
                for (uint32_t i = 0; i < held; i += 128) {
                    uint32_t v[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const uint32_t x = i + 32 * k + lane;
                        v[k] = x < held ? __ldg(&a.out_rec[st[x]].y) : ~0u;
                    }
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const uint32_t b = 1u << (v[k] & 31);
                        const bool fresh = v[k] != ~0u && !seen(v[k]) &&
                                           !(atomicOr(&bm[v[k] >> 5], b) & b);
                        const uint32_t fm = __ballot_sync(0xffffffffu, fresh);
                        if (!fm) continue;
                        uint32_t base = 0;
                        if (lane == 0) base = atomicAdd(&s_tail[to], (uint32_t)__popc(fm));
                        base = __shfl_sync(0xffffffffu, base, 0) + __popc(fm & ((1u << lane) - 1u));
                        if (fresh) q[nxt + dnxt * (int)base] = v[k];
                    }
                }
                __syncwarp();
            };
            do {
                uint2 row = rows;
                if (!few) {
                    uint32_t i0 = 0;
                    if (lane == 0) i0 = atomicAdd(&s_next[round & 1], per);
                    i0 = __shfl_sync(0xffffffffu, i0, 0);
                    if (i0 >= f) break;
                    if ((uint32_t)lane < per && i0 + lane < f)
                        row = __ldg(a.out_row + __ldcg(q + (cur + dcur * (int)(i0 + lane))));
                }
                // m < 2^32: a warp's distinct rows have fewer than 2^32 edges together
                const uint32_t n32 = row.y - row.x;
                const uint32_t r0 = drawn ? row.x >> 5 : row.x;
                const uint32_t cnt = n32 == 0 || !drawn ? n32 : ((row.y - 1) >> 5) - r0 + 1;
                uint32_t incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
                const uint32_t excl = incl - cnt;
                // the lane whose row holds unit t of the flattened rows
                auto owner = [&](uint32_t t) {
                    int own = 0;  // number of lanes whose inclusive count is <= t
#pragma unroll
                    for (int sft = 16; sft > 0; sft >>= 1) {
                        const uint32_t ic = __shfl_sync(0xffffffffu, incl, own + sft - 1);
                        if (ic <= t) own += sft;
                    }
                    return own;
                };
                if (!drawn) {
                    for (uint32_t base = start; base < total; base += min(2 * half, total - base)) {
                        uint2 r[2];
#pragma unroll
                        for (int i = 0; i < 2; i++) {
                            const uint32_t t = base + half * i + lane;
                            const int own = owner(t);
                            const uint32_t at = __shfl_sync(0xffffffffu, r0, own) +
                                                (t - __shfl_sync(0xffffffffu, excl, own));
                            r[i] = t < total ? __ldg(a.out_rec + at) : make_uint2(0u, ~0u);
                        }
#pragma unroll
                        for (int i = 0; i < 2; i++)
                            if (r[i].y != ~0u && !seen(r[i].y) &&
                                edge_kept(a, s0, s1, r[i].y, r[i].x))
                                add(r[i].y);
                    }
                    continue;  // (few: the last turn)
                }
                for (uint32_t base = start; base < total; base += min(2 * half, total - base)) {
                    uint32_t at[2], w[2];
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const uint32_t t = base + half * i + lane;
                        const int own = owner(t);
                        at[i] = __shfl_sync(0xffffffffu, r0, own) +
                                (t - __shfl_sync(0xffffffffu, excl, own));
                        const uint32_t ob = __shfl_sync(0xffffffffu, row.x, own);
                        const uint32_t oe = __shfl_sync(0xffffffffu, row.y, own);
                        w[i] = 0;
                        if (t < total) {  // bits of word `at` of the out-records ob .. oe - 1
                            w[i] = __ldcg(live + at[i]);
                            if (at[i] == ob >> 5) w[i] &= 0xFFFFFFFFu << (ob & 31);
                            if (at[i] == (oe - 1) >> 5) w[i] &= 0xFFFFFFFFu >> (31 - ((oe - 1) & 31));
                        }
                    }
                    const uint32_t wc = __popc(w[0]) + __popc(w[1]);
                    uint32_t wi = wc;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
                        if (lane >= o) wi += y;
                    }
                    const uint32_t wt = __shfl_sync(0xffffffffu, wi, 31);
                    if (wt == 0) continue;
                    if (held + wt > MC_STAGE) {
                        take();
                        held = 0;
                    }
                    uint32_t p = held + wi - wc;
                    const bool fits = wt <= MC_STAGE;
#pragma unroll
                    for (int i = 0; i < 2; i++)
                        for (uint32_t x = w[i]; x; x &= x - 1) {
                            const uint32_t e = (at[i] << 5) + (__ffs(x) - 1);
                            if (fits) {
                                st[p++] = e;
                            } else {
                                const uint32_t v = __ldg(&a.out_rec[e].y);
                                if (!seen(v)) add(v);
                            }
                        }
                    if (fits) held += wt;
                }
            } while (!few);
            take();
            held = 0;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            a.counts[c] = act;
            atomicAdd(&a.scal[1], (unsigned long long)act);
        }
        // leave the bitmap all-zero
        if (SM && ends)
            for (uint32_t w = threadIdx.x; w < (uint32_t)a.words; w += blockDim.x) bm[w] = 0u;
        else  // every set bit belongs to a queued node
            for (uint32_t i = threadIdx.x; i < act; i += blockDim.x) bm[__ldcg(q + i) >> 5] = 0u;
    }
}

// out_pos (4 B per edge) only when worlds are drawn (a function of the graph's size).
int build_out_records(tim_ctx* ctx, bool draws) {
    if (ctx->have_out) return TIM_OK;
    const uint64_t n = (uint64_t)ctx->n, m = (uint64_t)ctx->m;
    // (the 64-bit offsets are needed here alone)
    TIM_TRY(tim_ensure(ctx, ctx->scratch_d, (n + 1) * sizeof(uint64_t)));
    auto* off = (uint64_t*)ctx->scratch_d.p;
    TIM_TRY(tim_ensure(ctx, ctx->out_rec, std::max<uint64_t>(m, 1) * sizeof(uint2)));
    if (draws)
        TIM_TRY(tim_ensure(ctx, ctx->out_pos, std::max<uint64_t>(m, 1) * sizeof(uint32_t)));
    TIM_TRY(tim_ensure(ctx, ctx->scratch_a, (n + 1) * sizeof(uint32_t)));
    auto* cnt = (uint32_t*)ctx->scratch_a.p;
    CUDA_TRY(ctx, cudaMemsetAsync(cnt, 0, (n + 1) * sizeof(uint32_t), ctx->stream));
    const unsigned G = (unsigned)(ctx->num_sms * 8);
    if (m) {
        out_count_kernel<<<G, 256, 0, ctx->stream>>>((const uint32_t*)ctx->src.p, m, cnt);
        LAUNCH_CHECK(ctx, "out_count_kernel");
    }
    TIM_TRY(tim_scan_u32_to_u64(ctx, cnt, off, n));
    TIM_TRY(tim_ensure(ctx, ctx->out_row, n * sizeof(uint2)));
    out_rows_kernel<<<G, 256, 0, ctx->stream>>>(off, n, (uint2*)ctx->out_row.p);
    LAUNCH_CHECK(ctx, "out_rows_kernel");
    CUDA_TRY(ctx, cudaMemsetAsync(cnt, 0, (n + 1) * sizeof(uint32_t), ctx->stream));
    if (m) {
        out_scatter_kernel<<<G, 256, 0, ctx->stream>>>(
            (const uint64_t*)ctx->rowptr.p, (const uint32_t*)ctx->src.p, n, off, cnt,
            (uint2*)ctx->out_rec.p,
            draws ? (uint32_t*)ctx->out_pos.p : nullptr);
        LAUNCH_CHECK(ctx, "out_scatter_kernel");
    }
    ctx->have_out = true;
    return TIM_OK;
}

}  // namespace

extern "C" int tim_spread_mc(tim_ctx* ctx, const int32_t* seeds, int k, uint64_t count,
                             uint64_t seed, uint64_t first_set_id, uint64_t* total, double* mean,
                             uint32_t* counts_out) {
    if (!ctx) return TIM_ERR_ARG;
    if (!ctx->have_graph) return tim_fail(ctx, TIM_ERR_STATE, "no graph loaded");
    if (k < 0 || (k > 0 && !seeds)) return tim_fail(ctx, TIM_ERR_ARG, "bad seed list");
    const uint64_t n = (uint64_t)ctx->n;
    for (int i = 0; i < k; i++)
        if (seeds[i] < 0 || (uint64_t)seeds[i] >= n)
            return tim_fail(ctx, TIM_ERR_ARG, "seed out of range");
    if (count > 0xFFFFFFFFull) return tim_fail(ctx, TIM_ERR_ARG, "count must be below 2^32");
    DeviceGuard g(ctx->device);
    if (total) *total = 0;
    if (mean) *mean = 0.0;
    if (count == 0) return TIM_OK;
    // visited bitmap in shared memory while one block of it fits on an SM; two blocks of 768
    // threads per SM while two bitmaps fit, one of 1024 beyond that (50 seeds on R-MAT 18, 2000
    // IC and 1000 LT cascades: 2 x 768 threads 10.9 and 7.4 ms, 1 x 1024 12.4 and 8.8, 3 x 512
    // 10.9 and 8.2)
    const uint64_t words = n / 32 + 1;
    const bool sm = words * 4 <= MC_SMEM_MAX, two = words * 4 <= MC_SMEM_TWO;
    const size_t smem = sm ? (size_t)words * 4 : 0;
    const int threads = sm && !two ? 1024 : 768;
    const void* kernel = !sm ? (const void*)mc_cascade_kernel<false, 768, 2>
                       : two ? (const void*)mc_cascade_kernel<true, 768, 2>
                             : (const void*)mc_cascade_kernel<true, 1024, 1>;
    if (sm)
        CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)(two ? MC_SMEM_TWO : MC_SMEM_MAX)));
    int nb = 0;
    CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem));
    nb = std::max(nb, 1);
    // queue, live bits and (outside shared memory) bitmap per resident block, within
    // ~4 GiB; worlds are drawn when that leaves at least a block per SM and the device has room
    // for them
    const uint64_t budget = 4ull << 30;
    const uint64_t live_words = ((uint64_t)ctx->m + 127) / 128 * 4;
    const uint64_t base = n * 4 + (sm ? 0 : words * 4);
    bool draws = !ctx->mc_walk_only && budget / (base + live_words * 4) >= (uint64_t)ctx->num_sms;
    uint64_t slots = 0;
    // the records, queues and live bits of as many blocks as the budget holds
    auto prepare = [&]() -> int {
        TIM_TRY(build_out_records(ctx, draws));
        const uint64_t per_slot = base + (draws ? live_words * 4 : 0);
        slots = std::max<uint64_t>(1, budget / per_slot);
        slots = std::min<uint64_t>(slots, (uint64_t)ctx->num_sms * nb);
        slots = std::min<uint64_t>(slots, count);
        TIM_TRY(tim_ensure(ctx, ctx->mc_queue, slots * n * 4));
        return tim_ensure(ctx, ctx->mc_live, draws ? slots * live_words * 4 : 16);
    };
    int rc = prepare();
    if (rc == TIM_ERR_OOM && draws) {
        tim_free(ctx->out_pos);
        tim_free(ctx->mc_live);
        ctx->have_out = draws = false;
        rc = prepare();
        ctx->mc_walk_only = rc == TIM_OK;
    }
    TIM_TRY(rc);
    if (!sm) {
        const uint64_t made = ctx->mc_bitmap.made;
        TIM_TRY(tim_ensure(ctx, ctx->mc_bitmap, slots * words * 4));
        if (ctx->mc_bitmap.made != made || !ctx->mc_clean) {
            CUDA_TRY(ctx, cudaMemsetAsync(ctx->mc_bitmap.p, 0, ctx->mc_bitmap.bytes, ctx->stream));
            ctx->mc_clean = true;
        }
    }
    TIM_TRY(tim_ensure(ctx, ctx->mc_counts, count * 4));
    TIM_TRY(tim_ensure(ctx, ctx->mc_seeds, std::max(k, 1) * sizeof(int32_t)));
    TIM_TRY(tim_ensure(ctx, ctx->mc_scal, 3 * sizeof(unsigned long long)));
    // by warps first where there are several times more cascades than blocks at once
    const bool light = k <= LIGHT_Q / 2 && count > 4 * (uint64_t)ctx->num_sms * nb &&
                       tim_ensure(ctx, ctx->mc_list, count * sizeof(uint32_t)) == TIM_OK;
    if (k > 0)
        CUDA_TRY(ctx, cudaMemcpyAsync(ctx->mc_seeds.p, seeds, (size_t)k * sizeof(int32_t),
                                      cudaMemcpyHostToDevice, ctx->stream));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->mc_scal.p, 0, 3 * sizeof(unsigned long long), ctx->stream));
    McArgs a;
    a.node = (const uint4*)ctx->node.p;
    a.thr = (const uint32_t*)ctx->thr.p;
    a.out_row = (const uint2*)ctx->out_row.p;
    a.out_rec = (const uint2*)ctx->out_rec.p;
    a.out_pos = (const uint32_t*)ctx->out_pos.p;
    a.model = ctx->model;
    a.n = n;
    a.m = (uint64_t)ctx->m;
    a.K = tim_philox_keys(seed);
    a.sid0 = first_set_id;
    a.count = count;
    a.seeds = (const int32_t*)ctx->mc_seeds.p;
    a.k = k;
    a.bitmap = (uint32_t*)ctx->mc_bitmap.p;
    a.queue = (uint32_t*)ctx->mc_queue.p;
    a.words = words;
    a.live = (uint32_t*)ctx->mc_live.p;
    a.live_words = draws ? live_words : 0;
    a.draw_at = !draws ? ~0ull
                       : (ctx->model == TIM_IC ? (unsigned long long)ctx->m / 4 : n) / MC_WALK;
    a.counts = (uint32_t*)ctx->mc_counts.p;
    a.scal = (unsigned long long*)ctx->mc_scal.p;
    a.node_opt = (const uint64_t*)ctx->node_opt.p;
    a.opt_cum = (const uint32_t*)ctx->opt_cum.p;
    a.opt_off = (const uint64_t*)ctx->opt_off.p;
    a.opt_pos = (const uint32_t*)ctx->opt_pos.p;
    a.list = light ? (uint32_t*)ctx->mc_list.p : nullptr;
    if (light) {
        const uint64_t blocks = (count + LIGHT_THREADS / 32 - 1) / (LIGHT_THREADS / 32);
        mc_light_kernel<<<(unsigned)std::min<uint64_t>(blocks, (uint64_t)ctx->num_sms * LIGHT_BLOCKS),
                          LIGHT_THREADS, 0, ctx->stream>>>(a);
        LAUNCH_CHECK(ctx, "mc_light_kernel");
    }
    if (!sm) ctx->mc_clean = false;
    void* args[] = {&a};
    CUDA_TRY(ctx, cudaLaunchKernel(kernel, dim3((unsigned)slots), dim3(threads), args, smem, ctx->stream));
    LAUNCH_CHECK(ctx, "mc_cascade_kernel");
    unsigned long long h[2] = {0, 0};
    CUDA_TRY(ctx, cudaMemcpyAsync(h, ctx->mc_scal.p, sizeof h, cudaMemcpyDeviceToHost,
                                  ctx->stream));
    if (counts_out)
        CUDA_TRY(ctx, cudaMemcpyAsync(counts_out, ctx->mc_counts.p, count * 4,
                                      cudaMemcpyDeviceToHost, ctx->stream));
    TIM_TRY(tim_sync(ctx));
    if (!sm) ctx->mc_clean = true;
    if (total) *total = h[1];
    if (mean) *mean = (double)h[1] / (double)count;
    return TIM_OK;
}
