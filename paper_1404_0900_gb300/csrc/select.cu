// select.cu -- greedy maximum coverage over the RR-set store (the selection of
// Algorithm 1; also the greedy on R' of Algorithm 3).
//
// Only nodes with large counts are ever chosen: the counts (a histogram over the store) pick at
// most CAND candidate nodes, only their lists are built, and the rounds run over them in one
// cooperative launch, in epochs (see CandState).
// Where that does not pay, the full index: an exclusive scan of the counts into node offsets,
// and a scatter of set ids into per-node lists (node -> sets).
// Its greedy round r: an argmax over the counts with a warp-shuffle reduction of the key
// (count << 32 | ~node) so ties go to the smallest id and chosen nodes are skipped
// (counts read four at a time, several loads in flight per thread: the scan runs at
// DRAM speed when the counts outgrow L2); then every not-yet-covered set in the chosen
// node's list is marked covered and each of its members loses one from its count (in
// the cooperative launch, sets of more than COVER_CHUNK members are cut into chunks
// that all warps share). The chosen node is read on the device, so the k rounds run
// without host round trips.
#include <stddef.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "common.cuh"

namespace {

constexpr uint32_t NONE = 0xFFFFFFFFu;

// Coverage counts. The members of RR sets are skewed (a few hub nodes sit in a large part of
// all sets), and atomics on one address take turns: each block therefore keeps a direct-mapped
// table of counts in shared memory, whose slot goes to the first node that hashes to it --
// hubs, met within the first few thousand members, take theirs almost always -- and sends
// only the other nodes' members to the global counts. LIVE: only the members of sets that are
// not covered. (38.4M members of R-MAT 20 weighted cascade 667 -> 277 us, 28.4M of a Chung-Lu
// graph 2660 -> 230 us.)
constexpr uint32_t CNT_SLOTS = 8192;
constexpr int CNT_THREADS = 512;

template <bool LIVE>
__global__ void __launch_bounds__(CNT_THREADS)
count_members_kernel(const uint32_t* __restrict__ pool, const uint32_t* __restrict__ pool_sid,
                     const uint8_t* __restrict__ covered, uint64_t members,
                     uint32_t* __restrict__ cnt) {
    extern __shared__ uint32_t cs[];
    uint32_t *tag = cs, *num = cs + CNT_SLOTS;
    for (uint32_t i = threadIdx.x; i < CNT_SLOTS; i += CNT_THREADS) {
        tag[i] = NONE;
        num[i] = 0u;
    }
    __syncthreads();
    auto add = [&](uint32_t u) {
        const uint32_t h = (u * 0x9E3779B1u) >> 19;  // 13 bits
        uint32_t t = ((volatile uint32_t*)tag)[h];
        if (t == NONE) {
            t = atomicCAS(&tag[h], NONE, u);
            if (t == NONE) t = u;
        }
        if (t == u)
            atomicAdd(&num[h], 1u);
        else
            atomicAdd(&cnt[u], 1u);
    };
    const uint64_t stride = (uint64_t)gridDim.x * CNT_THREADS;
    const uint64_t tid = blockIdx.x * (uint64_t)CNT_THREADS + threadIdx.x;
    const uint64_t quads = members >> 2;
    const uint4* pool4 = reinterpret_cast<const uint4*>(pool);
    const uint4* sid4 = reinterpret_cast<const uint4*>(pool_sid);
    for (uint64_t q = tid; q < quads; q += stride) {
        const uint4 u = __ldg(pool4 + q);
        uint4 c = make_uint4(0u, 0u, 0u, 0u);
        if (LIVE) {
            const uint4 j = __ldg(sid4 + q);
            c = make_uint4(covered[j.x], covered[j.y], covered[j.z], covered[j.w]);
        }
        if (!c.x) add(u.x);
        if (!c.y) add(u.y);
        if (!c.z) add(u.z);
        if (!c.w) add(u.w);
    }
    for (uint64_t p = (quads << 2) + tid; p < members; p += stride)
        if (!LIVE || !covered[pool_sid[p]]) add(pool[p]);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < CNT_SLOTS; i += CNT_THREADS)
        if (num[i]) atomicAdd(&cnt[tag[i]], num[i]);
}

// Four members per thread and step (16-byte loads of the pool, which is 16-byte aligned):
// four independent atomics per thread are in flight at once.
// Node v's sets: node_sets[start(v) .. start(v + 1)). next[v] holds start(v) on entry
// (next = node_off + 1, the exclusive scan written one place to the right); each member
// takes its position with one atomic on it, so that afterwards next[v] = start(v + 1):
// node_off[0 .. n] are the node offsets with no cursor array and no offset load.
__global__ void scatter_sets_kernel(const uint32_t* __restrict__ pool,
                                    const uint32_t* __restrict__ pool_sid, uint64_t members,
                                    unsigned long long* __restrict__ next,
                                    uint32_t* __restrict__ node_sets) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const uint64_t quads = members >> 2;
    const uint4* pool4 = reinterpret_cast<const uint4*>(pool);
    const uint4* sid4 = reinterpret_cast<const uint4*>(pool_sid);
    for (uint64_t q = tid; q < quads; q += stride) {
        const uint4 u = __ldg(pool4 + q);
        const uint4 j = __ldg(sid4 + q);
        const unsigned long long p0 = atomicAdd(&next[u.x], 1ull), p1 = atomicAdd(&next[u.y], 1ull);
        const unsigned long long p2 = atomicAdd(&next[u.z], 1ull), p3 = atomicAdd(&next[u.w], 1ull);
        node_sets[p0] = j.x;
        node_sets[p1] = j.y;
        node_sets[p2] = j.z;
        node_sets[p3] = j.w;
    }
    for (uint64_t p = (quads << 2) + tid; p < members; p += stride)
        node_sets[atomicAdd(&next[pool[p]], 1ull)] = pool_sid[p];
}

__global__ void argmax_kernel(const int* __restrict__ counts, const uint8_t* __restrict__ chosen,
                              uint64_t n, unsigned long long* __restrict__ best) {
    unsigned long long b = slice_argmax(counts, chosen, n,
                                        blockIdx.x * (uint64_t)blockDim.x + threadIdx.x,
                                        (uint64_t)gridDim.x * blockDim.x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
        b = y > b ? y : b;
    }
    __shared__ unsigned long long wb[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) wb[wid] = b;
    __syncthreads();
    if (wid == 0) {
        b = lane < (int)(blockDim.x >> 5) ? wb[lane] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
            b = y > b ? y : b;
        }
        if (lane == 0 && b) atomicMax(best, b);
    }
}

__global__ void set_key_kernel(unsigned long long* key, unsigned long long value) { *key = value; }

__global__ void cover_kernel(const unsigned long long* __restrict__ best,
                             const uint64_t* __restrict__ node_off,
                             const uint32_t* __restrict__ node_sets,
                             const uint64_t* __restrict__ set_start,
                             const uint32_t* __restrict__ set_len,
                             const uint32_t* __restrict__ pool, uint8_t* __restrict__ covered,
                             int* __restrict__ counts, uint8_t* __restrict__ chosen,
                             int32_t* __restrict__ seed_out, unsigned long long* __restrict__ ncov) {
    const unsigned long long key = *best;
    if (key == 0) return;  // no candidate (cannot happen for k <= n)
    const uint32_t v = ~(uint32_t)(key & 0xFFFFFFFFull);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        chosen[v] = 1;
        *seed_out = (int32_t)v;
    }
    const int lane = threadIdx.x & 31;
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t a = node_off[v], b = node_off[v + 1];
    unsigned long long fresh = 0;
    for (uint64_t i = a + warp; i < b; i += nwarps) {
        uint32_t s = node_sets[i];
        if (covered[s]) continue;  // uniform across the warp
        __syncwarp();
        if (lane == 0) {
            covered[s] = 1;
            fresh++;
        }
        const uint64_t st = set_start[s];
        const uint32_t len = set_len[s];
        for (uint32_t t = lane; t < len; t += 32) atomicSub(&counts[pool[st + t]], 1);
    }
    if (lane == 0 && fresh) atomicAdd(ncov, fresh);
}

// Members per chunk of a large set in the cooperative greedy: a newly covered set with
// more members is split into chunks that all warps share after the cover step (one warp
// walking a set of 10^4 - 10^6 members would hold up the round).
constexpr uint32_t COVER_CHUNK = 4096;

// Greedy rounds r0 .. k - 1 in one cooperative launch: per round an argmax over the counts
// (every block reduces a slice, atomicMax into best[r]), a grid barrier, the cover step
// of the chosen node (warps over its set list; a set of more than COVER_CHUNK members is
// only marked, and its member chunks listed), a second barrier, and when chunks were
// listed, the chunks over all warps and a third barrier. chunks holds at most
// chunk_cap entries (set id | chunk << 32); nchunk[r] counts round r's.
__global__ void __launch_bounds__(256)
greedy_rounds_kernel(int* __restrict__ counts, uint8_t* __restrict__ chosen, uint64_t n,
                     const uint64_t* __restrict__ node_off, const uint32_t* __restrict__ node_sets,
                     const uint64_t* __restrict__ set_start, const uint32_t* __restrict__ set_len,
                     const uint32_t* __restrict__ pool, uint8_t* __restrict__ covered, int r0,
                     int k, unsigned long long* __restrict__ best, int32_t* __restrict__ seeds,
                     unsigned long long* __restrict__ ncov, GridBarrier* bar, int* err,
                     unsigned limit, unsigned long long* __restrict__ chunks,
                     unsigned long long* __restrict__ nchunk, unsigned long long chunk_cap) {
    __shared__ unsigned long long wb[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long fresh = 0;
    for (int r = r0; r < k; r++) {
        unsigned long long b = slice_argmax(counts, chosen, n,
                                            blockIdx.x * (uint64_t)blockDim.x + threadIdx.x,
                                            (uint64_t)gridDim.x * blockDim.x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
            b = y > b ? y : b;
        }
        if (lane == 0) wb[wid] = b;
        __syncthreads();
        if (wid == 0) {
            b = lane < (int)(blockDim.x >> 5) ? wb[lane] : 0ull;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
                b = y > b ? y : b;
            }
            if (lane == 0 && b) atomicMax(best + r, b);
        }
        if (!grid_barrier(bar, err, limit)) return;
        const unsigned long long key = ((volatile unsigned long long*)best)[r];
        if (key != 0) {
            const uint32_t v = ~(uint32_t)(key & 0xFFFFFFFFull);
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                chosen[v] = 1;
                seeds[r] = (int32_t)v;
            }
            const uint64_t a = node_off[v], e = node_off[v + 1];
            for (uint64_t i = a + warp; i < e; i += nwarps) {
                const uint32_t s = node_sets[i];
                if (((volatile uint8_t*)covered)[s]) continue;  // uniform across the warp
                __syncwarp();
                if (lane == 0) {
                    covered[s] = 1;
                    fresh++;
                }
                const uint64_t st = set_start[s];
                const uint32_t len = set_len[s];
                if (len <= COVER_CHUNK) {
                    for (uint32_t t = lane; t < len; t += 32) atomicSub(&counts[pool[st + t]], 1);
                } else {
                    const uint32_t nc = (len + COVER_CHUNK - 1) / COVER_CHUNK;
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(nchunk + r, (unsigned long long)nc);
                    base = __shfl_sync(0xffffffffu, base, 0);
                    for (uint32_t c = lane; c < nc; c += 32) {
                        if (base + c < chunk_cap)
                            chunks[base + c] = (unsigned long long)s | ((unsigned long long)c << 32);
                        else
                            atomicOr(err, TIM_DEV_ERR_BOUNDS);
                    }
                }
            }
        }
        if (!grid_barrier(bar, err, limit)) return;
        // the large sets' member chunks, over all warps, eight loads in flight per lane
        const unsigned long long nc = min(((volatile unsigned long long*)nchunk)[r], chunk_cap);
        if (nc) {
            for (uint64_t w = warp; w < nc; w += nwarps) {
                const unsigned long long e = chunks[w];
                const uint32_t s = (uint32_t)e, c = (uint32_t)(e >> 32);
                const uint64_t st = set_start[s] + (uint64_t)c * COVER_CHUNK;
                const uint32_t len = min(COVER_CHUNK, set_len[s] - c * COVER_CHUNK);
                for (uint32_t t = lane; t < len; t += 256) {
                    uint32_t u[8];
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        u[q] = t + 32u * q < len ? __ldg(pool + st + t + 32u * q) : 0u;
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        if (t + 32u * q < len) atomicSub(&counts[u[q]], 1);
                }
            }
            if (!grid_barrier(bar, err, limit)) return;
        }
    }
    if (lane == 0 && fresh) atomicAdd(ncov, fresh);
}


// ------------------------------------------------------- greedy over candidate nodes
//
// The greedy picks nodes of large counts, and counts only fall: while the largest current
// count among the C nodes whose counts were at least tau is itself at least tau, it is the
// largest of all nodes (ties too: no other node reaches tau). So only these candidates get a
// list of their sets, only their counts are lowered, and a round needs no pass over the n
// counts. When the best candidate falls below tau (or the candidates cannot be told apart
// within CAND), the host starts again on the sets still uncovered, or goes on with the full
// index. The candidates' table (node -> candidate) sits in the shared memory of every block,
// as do the running counts, so that a round costs one grid barrier.
constexpr uint32_t CAND = 8192;         // candidates at most
constexpr uint32_t CAND_SLOTS = 16384;  // hash slots of their table
constexpr int CAND_BINS = 1024;         // bins of counts (CAND_BINS >= 64 + 26 * 32)
constexpr int CG_THREADS = 1024;
constexpr uint32_t TILE_ITEMS = 16;     // members per thread of an index tile
constexpr uint32_t CAND_BITS = 1u << 17;  // bits of the filter in front of the table
// candidates in play at the start (128, 512, 2048: 50 seeds of 1.8M members 0.645, 0.642, 0.682 ms,
// of 0.2 to 38M others within 2 %)
constexpr uint32_t CAND_PREFIX = 512;
// stores up to this many members are selected from by one block, without grid barriers (50 seeds,
// all blocks / one: 21K members 0.518 / 0.345 ms, 97K 0.524 / 0.407, 211K 0.535 / 0.512, 331K 0.585 /
// 0.621)
constexpr uint64_t CAND_SOLO = 100'000;
// members of a set that one block lowers, and per chunk of a larger one (8192 to 131072, 512 and
// 2048: 50 seeds of 4.6M members in sets of up to 10^5 within 3 %)
constexpr uint32_t CG_BLOCK = 32768;
constexpr uint32_t CG_CHUNK = 512;
// shared memory of a table and its filter; then the rounds' counts, decrements, list offsets
// and the sets of a tile, or the index's counts of a tile
constexpr size_t TABLE_SMEM = (size_t)CAND_SLOTS * 6 + CAND_BITS / 8;
constexpr size_t CG_SMEM = TABLE_SMEM + (size_t)CAND * 12 + 16 + (size_t)(CG_THREADS + 4) * 12;
constexpr size_t CI_SMEM = TABLE_SMEM + (size_t)CAND * 4;

// State of one greedy over candidates (device memory; cleared before each epoch).
struct CandState {
    uint32_t bins[CAND_BINS];
    uint32_t taken[CAND_BINS];
    uint32_t ncand;
    uint32_t tau;
    uint32_t pad[2];
    uint32_t off[CAND + 4];  // CAND + 1 used
    uint32_t cursor[CAND];
    uint32_t cnt[CAND];
    uint32_t node[CAND];
    uint32_t delta[3][CAND];  // decrements of round r in delta[r % 3]
    uint32_t late[CAND];      // decrements of candidates from before they came into play
    uint32_t key[CAND_SLOTS];
    uint16_t val[CAND_SLOTS];
};
static_assert(offsetof(CandState, key) % 16 == 0 && offsetof(CandState, val) % 16 == 0,
              "the table is read 16 bytes at a time");

// Bin of a count >= 1: exact below 64, then 32 per factor of two; bins ascend with counts.
__device__ __forceinline__ uint32_t count_bin(uint32_t c) {
    if (c < 64u) return c;
    const int e = 31 - __clz((int)c);
    return 64u + (uint32_t)(e - 6) * 32u + ((c >> (e - 5)) & 31u);
}

// Smallest count of a bin.
__device__ __forceinline__ uint32_t bin_floor(uint32_t b) {
    if (b < 64u) return b;
    const uint32_t e = 6u + (b - 64u) / 32u, m = (b - 64u) % 32u;
    return (32u + m) << (e - 5u);
}

__global__ void __launch_bounds__(256) count_bins_kernel(const uint32_t* __restrict__ counts,
                                                         uint64_t n, CandState* st) {
    __shared__ uint32_t h[CAND_BINS];
    for (int i = threadIdx.x; i < CAND_BINS; i += 256) h[i] = 0u;
    __syncthreads();
    for (uint64_t v = blockIdx.x * 256ull + threadIdx.x; v < n; v += (uint64_t)gridDim.x * 256ull) {
        const uint32_t c = __ldg(counts + v);
        if (c) atomicAdd(&h[count_bin(c)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < CAND_BINS; i += 256)
        if (h[i]) atomicAdd(&st->bins[i], h[i]);
}

// tau = the smallest bin floor that leaves at most CAND nodes at or above it (every block
// finds it from the bins), and the nodes there, in the order of descending bins. tau = 0, no
// candidates: there are more than CAND in the highest bin, or fewer than `need` among more nodes
// that have sets.
__global__ void __launch_bounds__(256) candidates_kernel(const uint32_t* __restrict__ counts,
                                                         uint64_t n, uint32_t need,
                                                         CandState* st) {
    __shared__ uint32_t sfx[256];
    __shared__ uint32_t s_bin, s_cand;
    // thread t owns bins 4 t .. 4 t + 3; sfx[t] = nodes in its bins and above
    uint32_t b[4], sum = 0;
    for (int i = 0; i < 4; i++) sum += b[i] = st->bins[threadIdx.x * 4 + i];
    sfx[threadIdx.x] = sum;
    if (threadIdx.x == 0) s_bin = CAND_BINS, s_cand = 0u;
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {
        const uint32_t y = threadIdx.x + o < 256 ? sfx[threadIdx.x + o] : 0u;
        __syncthreads();
        sfx[threadIdx.x] += y;
        __syncthreads();
    }
    uint32_t above = sfx[threadIdx.x] - sum;  // fewer than n < 2^31
    for (int i = 3; i >= 0; i--) {
        above += b[i];
        const int bin = threadIdx.x * 4 + i;
        if (bin >= 1 && above <= CAND) atomicMin(&s_bin, (uint32_t)bin);
    }
    __syncthreads();
    above = sfx[threadIdx.x] - sum;
    for (int i = 3; i >= 0; i--) {
        above += b[i];
        if (threadIdx.x * 4 + i == (int)s_bin) s_cand = above;
    }
    __syncthreads();
    const uint32_t tau =
        s_bin == 1u || (s_bin < CAND_BINS && s_cand >= need) ? bin_floor(s_bin) : 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->tau = tau;
    if (tau == 0u) return;
    // a bin's candidates follow those of the bins above it
    __shared__ uint32_t first[CAND_BINS];
    above = sfx[threadIdx.x] - sum;
    for (int i = 3; i >= 0; i--) {
        first[threadIdx.x * 4 + i] = above;
        above += b[i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->ncand = s_cand;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (uint64_t v0 = blockIdx.x * 256ull + (threadIdx.x & ~31u); v0 < n;
         v0 += (uint64_t)gridDim.x * 256ull) {
        const uint32_t c = v0 + lane < n ? __ldg(counts + v0 + lane) : 0u;
        if (c < tau) continue;
        const uint32_t bin = count_bin(c);
        const uint32_t at = first[bin] + atomicAdd(&st->taken[bin], 1u);
        if (at < CAND) {
            st->node[at] = (uint32_t)(v0 + lane);
            st->cnt[at] = c;
        }
    }
}

__device__ __forceinline__ uint32_t cand_hash(uint32_t u) { return u * 0x9E3779B1u; }

// One block: list offsets of the candidates and the node -> candidate table (keys NONE on
// entry).
__global__ void __launch_bounds__(1024) cand_table_kernel(CandState* st) {
    __shared__ uint32_t wsum[32];
    if (st->tau == 0u) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t nc = min(st->ncand, CAND);
    constexpr uint32_t PER = CAND / 1024;
    uint32_t c[PER], sum = 0;
    for (uint32_t i = 0; i < PER; i++) {
        const uint32_t x = threadIdx.x * PER + i;
        sum += c[i] = x < nc ? st->cnt[x] : 0u;
    }
    uint32_t inc = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    uint32_t at = inc - sum;
    for (int i = 0; i < w; i++) at += wsum[i];
    for (uint32_t i = 0; i < PER; i++) {
        const uint32_t x = threadIdx.x * PER + i;
        st->off[x] = st->cursor[x] = at;
        at += c[i];
        if (x == CAND - 1) st->off[CAND] = at;
        if (x >= nc) continue;
        const uint32_t v = st->node[x];
        uint32_t h = cand_hash(v) >> 18;  // 14 bits
        for (uint32_t p = 0; p < CAND_SLOTS; p++, h = (h + 1) & (CAND_SLOTS - 1))
            if (atomicCAS(&st->key[h], NONE, v) == NONE) break;
        st->val[h] = (uint16_t)x;
    }
}

// The table in a block's shared memory, with a bit filter in front (about 6 % of the other
// nodes pass it): most members are no candidates, and one look at the filter says so.
struct CandTable {
    uint32_t* key;
    uint16_t* val;
    uint32_t* bits;
};

// Followed by __syncthreads in the caller.
__device__ __forceinline__ CandTable load_table(const CandState* st, uint32_t* smem) {
    CandTable t{smem, reinterpret_cast<uint16_t*>(smem + CAND_SLOTS),
                smem + CAND_SLOTS + CAND_SLOTS / 2};
    for (uint32_t i = threadIdx.x; i < CAND_BITS / 32; i += blockDim.x) t.bits[i] = 0u;
    __syncthreads();
    const uint4* v4 = reinterpret_cast<const uint4*>(st->val);
    for (uint32_t i = threadIdx.x; i < CAND_SLOTS; i += blockDim.x) {
        const uint32_t k = st->key[i];
        t.key[i] = k;
        if (k != NONE) {
            const uint32_t b = cand_hash(k) >> 15;  // 17 bits
            atomicOr(&t.bits[b >> 5], 1u << (b & 31));
        }
    }
    for (uint32_t i = threadIdx.x; i < CAND_SLOTS / 8; i += blockDim.x)
        reinterpret_cast<uint4*>(t.val)[i] = v4[i];
    return t;
}

__device__ __forceinline__ bool maybe_cand(const CandTable& t, uint32_t u) {
    const uint32_t b = cand_hash(u) >> 15;
    return (t.bits[b >> 5] >> (b & 31)) & 1u;
}

// Candidate of node u, or NONE (at most half of the slots are taken, so a probe ends).
__device__ __forceinline__ uint32_t find_cand(const CandTable& t, uint32_t u) {
    uint32_t h = cand_hash(u) >> 18;
    for (uint32_t p = 0; p < CAND_SLOTS; p++) {
        const uint32_t k = t.key[h];
        if (k == u) return t.val[h];
        if (k == NONE) break;
        h = (h + 1) & (CAND_SLOTS - 1);
    }
    return NONE;
}

// Sets of every candidate: sets[off[c] .. off[c + 1]). A block takes tiles of members, counts
// each candidate's members of the tile in shared memory (which also ranks them) and reserves
// their places with one global atomic per candidate and tile.
template <bool LIVE>
__global__ void __launch_bounds__(CG_THREADS)
cand_index_kernel(const uint32_t* __restrict__ pool, const uint32_t* __restrict__ pool_sid,
                  const uint8_t* __restrict__ covered, uint64_t members, CandState* st,
                  uint32_t* __restrict__ sets) {
    extern __shared__ __align__(16) uint32_t sm[];
    if (st->tau == 0u) return;
    const CandTable tab = load_table(st, sm);
    uint32_t* num = sm + TABLE_SMEM / 4;  // [CAND]
    constexpr uint64_t TILE = (uint64_t)CG_THREADS * TILE_ITEMS;
    const uint4* pool4 = reinterpret_cast<const uint4*>(pool);
    const uint4* sid4 = reinterpret_cast<const uint4*>(pool_sid);
    const uint32_t nc = min(st->ncand, CAND);
    for (uint64_t t0 = blockIdx.x * TILE; t0 < members; t0 += gridDim.x * TILE) {
        for (uint32_t i = threadIdx.x; i < nc; i += CG_THREADS) num[i] = 0u;
        __syncthreads();
        // the members (NONE: past the end), all loads first, then the filter for all
        uint32_t hit[TILE_ITEMS];
#pragma unroll
        for (uint32_t q = 0; q < TILE_ITEMS / 4; q++) {
            const uint64_t p = t0 + (uint64_t)q * CG_THREADS * 4 + threadIdx.x * 4ull;
            if (p + 4 <= members) {
                const uint4 x = __ldg(pool4 + (p >> 2));
                hit[q * 4] = x.x, hit[q * 4 + 1] = x.y, hit[q * 4 + 2] = x.z, hit[q * 4 + 3] = x.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; k++) hit[q * 4 + k] = p + k < members ? pool[p + k] : NONE;
            }
        }
#pragma unroll
        for (uint32_t i = 0; i < TILE_ITEMS; i++)
            if (!maybe_cand(tab, hit[i])) hit[i] = NONE;
        // candidate | rank in the tile << 13 (13 and 14 bits)
#pragma unroll
        for (uint32_t i = 0; i < TILE_ITEMS; i++) {
            if (hit[i] == NONE) continue;
            const uint32_t c = find_cand(tab, hit[i]);
            const uint64_t p = t0 + (uint64_t)(i / 4) * CG_THREADS * 4 + threadIdx.x * 4ull + i % 4;
            const bool live = c != NONE && (!LIVE || !covered[pool_sid[p]]);
            hit[i] = live ? c | (atomicAdd(&num[c], 1u) << 13) : NONE;
        }
        __syncthreads();
        {
            uint32_t x[CAND / CG_THREADS];  // independent atomics in flight
#pragma unroll
            for (uint32_t i = 0; i < CAND / CG_THREADS; i++) {
                const uint32_t c = threadIdx.x + i * CG_THREADS;
                x[i] = c < nc ? num[c] : 0u;
                if (x[i]) x[i] = atomicAdd(&st->cursor[c], x[i]);
            }
#pragma unroll
            for (uint32_t i = 0; i < CAND / CG_THREADS; i++) {
                const uint32_t c = threadIdx.x + i * CG_THREADS;
                if (c < nc) num[c] = x[i];
            }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t q = 0; q < TILE_ITEMS / 4; q++) {
            const uint64_t p = t0 + (uint64_t)q * CG_THREADS * 4 + threadIdx.x * 4ull;
            const bool any = (hit[q * 4] & hit[q * 4 + 1] & hit[q * 4 + 2] & hit[q * 4 + 3]) != NONE;
            if (!any) continue;
            uint32_t j[4];
            if (p + 4 <= members) {
                const uint4 x = __ldg(sid4 + (p >> 2));
                j[0] = x.x, j[1] = x.y, j[2] = x.z, j[3] = x.w;
            } else {
                for (int k = 0; k < 4; k++) j[k] = p + k < members ? pool_sid[p + k] : 0u;
            }
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t h = hit[q * 4 + k];
                if (h != NONE) sets[num[h & (CAND - 1)] + (h >> 13)] = j[k];
            }
        }
        __syncthreads();
    }
}

// One 16-byte record per set for the rounds: {start (2 words), length, covered}.
__global__ void set_rec_kernel(const uint64_t* __restrict__ set_start,
                               const uint32_t* __restrict__ set_len, uint64_t n_sets,
                               uint4* __restrict__ rec) {
    for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < n_sets;
         s += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t a = set_start[s];
        rec[s] = make_uint4((uint32_t)a, (uint32_t)(a >> 32), set_len[s], 0u);
    }
}

// Rounds r0 .. k - 1 over the candidates (cooperative launch). Every block keeps its own copy
// of the candidates' counts and finds the same best one. The blocks share out its sets; a
// block lists the members of those not yet covered one after another, and its warps take
// equal ranges of them (whole sets per warp left most warps waiting for the one with the
// longest sets) and lower the candidates' counts in shared memory. The block then adds its
// decrements to the round's global ones, and after the barrier every block takes them off
// its counts. Sets of more than CG_BLOCK members are listed in chunks that all blocks share
// after the barrier.
//   The candidates come in descending order of their initial counts (by bins), and only a
// prefix of them is in play: counts only fall, so the rest cannot win while the best exceeds
// their bins. Their decrements stay in the blocks until the prefix doubles. Rounds are bound
// by their chain of loads, atomics and the barrier.
__global__ void __launch_bounds__(CG_THREADS)
cand_rounds_kernel(CandState* st, const uint32_t* __restrict__ sets,
                   uint4* __restrict__ rec, const uint32_t* __restrict__ pool,
                   uint8_t* __restrict__ covered, int r0, int k,
                   uint8_t* __restrict__ chosen, int32_t* __restrict__ seeds,
                   unsigned long long* __restrict__ ncov, unsigned* __restrict__ done,
                   GridBarrier* bar, int* err,
                   unsigned limit, unsigned long long* __restrict__ chunks,
                   unsigned long long* __restrict__ nchunk, unsigned long long chunk_cap) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ unsigned long long wbest[CG_THREADS / 32];
    __shared__ uint32_t wcand[CG_THREADS / 32];
    __shared__ unsigned long long wsum[CG_THREADS / 32];
    if (st->tau == 0u) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *done = (uint32_t)r0;
        return;
    }
    const CandTable tab = load_table(st, sm);
    int* cnt = reinterpret_cast<int*>(sm + TABLE_SMEM / 4);               // [CAND]
    uint32_t* dec = reinterpret_cast<uint32_t*>(cnt + CAND);              // [CAND]
    uint32_t* off = dec + CAND;                                           // [CAND + 1]
    uint32_t* pre = off + CAND + 4;                                       // [CG_THREADS + 1]
    uint64_t* frm = reinterpret_cast<uint64_t*>(pre + CG_THREADS + 4);    // [CG_THREADS + 1]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t nc = min(st->ncand, CAND), tau = st->tau;
    const uint64_t warp = blockIdx.x * (uint64_t)(CG_THREADS / 32) + wid;
    const uint64_t nwarps = (uint64_t)gridDim.x * (CG_THREADS / 32);
    for (uint32_t i = threadIdx.x; i < nc; i += CG_THREADS) {
        cnt[i] = (int)st->cnt[i];
        dec[i] = 0u;
        off[i] = st->off[i];
        if (i == nc - 1) off[nc] = st->off[nc];
    }
    __syncthreads();
    unsigned long long fresh = 0;
    const bool solo = gridDim.x == 1;  // no other block: counts are lowered in place
    auto lower = [&](uint32_t u) {
        if (u == NONE || !maybe_cand(tab, u)) return;
        const uint32_t c = find_cand(tab, u);
        if (c == NONE) return;
        if (solo)
            atomicSub(&cnt[c], 1);
        else
            atomicAdd(&dec[c], 1u);
    };
    // add the block's decrements of candidates lo .. hi - 1 to the global ones
    auto flush = [&](uint32_t* delta, uint32_t lo, uint32_t hi) {
        __syncthreads();
        for (uint32_t i = lo + threadIdx.x; i < hi; i += CG_THREADS)
            if (dec[i]) {
                atomicAdd(&delta[i], dec[i]);
                dec[i] = 0u;
            }
    };
    uint32_t np = min(nc, CAND_PREFIX);  // candidates in play
    int r = r0;
    for (; r < k;) {
        uint32_t* delta = st->delta[r % 3];
        // the best candidate in play: (count, smallest node), by every block for itself
        unsigned long long b = 0;
        uint32_t bc = 0;
        for (uint32_t i = threadIdx.x; i < np; i += CG_THREADS) {
            if (cnt[i] < 0) continue;  // chosen
            const unsigned long long key = greedy_key(cnt[i], __ldg(&st->node[i]));
            if (key > b) {
                b = key;
                bc = i;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
            const uint32_t yc = __shfl_xor_sync(0xffffffffu, bc, o);
            if (y > b) b = y, bc = yc;
        }
        if (lane == 0) wbest[wid] = b, wcand[wid] = bc;
        __syncthreads();
        b = wbest[lane];
        bc = wcand[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
            const uint32_t yc = __shfl_xor_sync(0xffffffffu, bc, o);
            if (y > b) b = y, bc = yc;
        }
        // the same in every block. No candidate out of play exceeds the largest count of the
        // next one's bin; when the best does not, bring more into play
        if (np < nc && (uint32_t)(b >> 32) < bin_floor(count_bin(__ldg(&st->cnt[np])) + 1u)) {
            const uint32_t more = min(nc, 2 * np);
            uint32_t* late = st->late;
            if (!solo) {
                flush(late, np, more);
                if (!grid_barrier(bar, err, limit)) return;
                for (uint32_t i = np + threadIdx.x; i < more; i += CG_THREADS)
                    cnt[i] -= (int)__ldcg(late + i);
            }
            np = more;
            __syncthreads();
            continue;
        }
        if (b == 0 || (uint32_t)(b >> 32) < tau) break;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            const uint32_t v = st->node[bc];
            chosen[v] = 1;
            seeds[r] = (int32_t)v;
        }
        const uint32_t a = off[bc], e = off[bc + 1];
        for (uint64_t p0 = a + blockIdx.x; p0 < e; p0 += (uint64_t)gridDim.x * CG_THREADS) {
            // one set per thread: the new ones' starts and lengths, compacted, with the prefix
            // of the lengths
            const uint64_t i = p0 + (uint64_t)threadIdx.x * gridDim.x;
            uint32_t len = 0;
            uint64_t from = 0;
            if (i < e) {
                const uint32_t s = sets[i];
                const uint4 x = __ldcg(rec + s);
                if (x.w == 0u) {
                    len = x.z;
                    from = (uint64_t)x.x | ((uint64_t)x.y << 32);
                    reinterpret_cast<uint32_t*>(rec + s)[3] = 1u;
                    covered[s] = 1;
                    fresh++;
                    if (len > CG_BLOCK && !solo) {
                        const uint32_t n = (len + CG_CHUNK - 1) / CG_CHUNK;
                        const unsigned long long base =
                            atomicAdd(nchunk + r, (unsigned long long)n);
                        for (uint32_t c = 0; c < n; c++) {
                            if (base + c < chunk_cap)
                                chunks[base + c] =
                                    (unsigned long long)s | ((unsigned long long)c << 32);
                            else
                                atomicOr(err, TIM_DEV_ERR_BOUNDS);
                        }
                        len = 0;
                    }
                }
            }
            // at most CG_THREADS x CG_BLOCK = 2^25 members (solo: CAND_SOLO)
            const unsigned long long v = len ? (1ull << 32) | len : 0ull;
            unsigned long long inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) wsum[wid] = inc;
            __syncthreads();
            unsigned long long ws = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, ws, o);
                if (lane >= o) ws += y;
            }
            const unsigned long long all = __shfl_sync(0xffffffffu, ws, 31);
            const unsigned long long before = __shfl_sync(0xffffffffu, ws, wid ? wid - 1 : 0);
            const uint32_t ns = (uint32_t)(all >> 32), total = (uint32_t)all;
            if (len) {
                const unsigned long long ex = (wid ? before : 0ull) + inc - v;
                pre[ex >> 32] = (uint32_t)ex;
                frm[ex >> 32] = from;
            }
            if (threadIdx.x == 0) pre[ns] = total;
            __syncthreads();
            // the members in steps of 32, a contiguous range of steps per warp
            const uint32_t steps = (total + 31) / 32;
            const uint32_t s0 = steps * (uint64_t)wid / (CG_THREADS / 32);
            const uint32_t s1 = steps * (uint64_t)(wid + 1) / (CG_THREADS / 32);
            uint32_t c = 0;  // the set that holds member 32 s0: pre[c] <= 32 s0 < pre[c + 1]
            if (s0 < s1) {
                uint32_t hi = ns;
                while (hi - c > 1) {
                    const uint32_t mid = (c + hi) >> 1;
                    if (pre[mid] <= s0 * 32)
                        c = mid;
                    else
                        hi = mid;
                }
            }
            for (uint32_t st0 = s0; st0 < s1; st0 += 4) {
                uint32_t u[4];
#pragma unroll
                for (uint32_t q = 0; q < 4; q++) {
                    u[q] = NONE;
                    if (st0 + q >= s1) continue;
                    const uint32_t base = (st0 + q) * 32;
                    // every set has a member, so at most 32 sets end within the step
                    const uint32_t end = c + 1 + lane <= ns ? pre[c + 1 + lane] : NONE;
                    const uint32_t marks = __reduce_or_sync(
                        0xffffffffu, end - base < 32u ? 1u << (end - base) : 0u);
                    const uint32_t own = c + __popc(marks & (0xFFFFFFFFu >> (31 - lane)));
                    if (base + lane < total) u[q] = __ldg(pool + frm[own] + (base + lane - pre[own]));
                    c += __popc(__ballot_sync(0xffffffffu, end - base <= 32u));
                }
#pragma unroll
                for (uint32_t q = 0; q < 4; q++) lower(u[q]);
            }
            __syncthreads();
        }
        if (solo) {  // the tiles end with a barrier of the block
            __syncthreads();
            if (threadIdx.x == 0) cnt[bc] = -1;
            __syncthreads();
            r++;
            continue;
        }
        flush(delta, 0, np);
        if (!grid_barrier(bar, err, limit)) return;
        const unsigned long long nch = min(((volatile unsigned long long*)nchunk)[r], chunk_cap);
        if (nch) {
            for (uint64_t w = warp; w < nch; w += nwarps) {
                const unsigned long long x = __ldcg(chunks + w);
                const uint32_t s = (uint32_t)x, c = (uint32_t)(x >> 32);
                const uint4 y = __ldcg(rec + s);
                const uint64_t from =
                    ((uint64_t)y.x | ((uint64_t)y.y << 32)) + (uint64_t)c * CG_CHUNK;
                const uint32_t len = min(CG_CHUNK, y.z - c * CG_CHUNK);
                for (uint32_t t = lane; t < len; t += 256) {
                    uint32_t u[8];
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        u[q] = t + 32u * q < len ? __ldg(pool + from + t + 32u * q) : NONE;
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        lower(u[q]);
                }
            }
            flush(delta, 0, np);
            if (!grid_barrier(bar, err, limit)) return;
        }
        // the round's decrements; and round r + 2's buffer, last read before this barrier
        uint32_t* next = st->delta[(r + 2) % 3];
        for (uint32_t i = threadIdx.x; i < np; i += CG_THREADS) cnt[i] -= (int)__ldcg(delta + i);
        for (uint32_t i = blockIdx.x * CG_THREADS + threadIdx.x; i < np; i += gridDim.x * CG_THREADS)
            next[i] = 0u;
        __syncthreads();
        if (threadIdx.x == 0) cnt[bc] = -1;
        __syncthreads();
        r++;
    }
    // rounds done; bit 31: the candidates are all nodes that have a set
    if (blockIdx.x == 0 && threadIdx.x == 0) *done = (uint32_t)r | (tau == 1u ? 0x80000000u : 0u);
    fresh += __shfl_xor_sync(0xffffffffu, fresh, 16);
    fresh += __shfl_xor_sync(0xffffffffu, fresh, 8);
    fresh += __shfl_xor_sync(0xffffffffu, fresh, 4);
    fresh += __shfl_xor_sync(0xffffffffu, fresh, 2);
    fresh += __shfl_xor_sync(0xffffffffu, fresh, 1);
    if (lane == 0 && fresh) atomicAdd(ncov, fresh);
}

}  // namespace

// The coverage count of every node over the store (LIVE: over its uncovered sets).
static int count_members(tim_ctx* ctx, bool live) {
    const uint64_t n = (uint64_t)ctx->n, members = ctx->members;
    TIM_TRY(tim_ensure(ctx, ctx->counts, (n + 1) * sizeof(int)));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->counts.p, 0, (n + 1) * sizeof(int), ctx->stream));
    if (!members) return TIM_OK;
    constexpr size_t smem = 2 * CNT_SLOTS * sizeof(uint32_t);
    auto* kernel = live ? count_members_kernel<true> : count_members_kernel<false>;
    CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
    const uint64_t blocks = members / (CNT_THREADS * 16) + 1;
    kernel<<<(unsigned)std::min<uint64_t>(blocks, (uint64_t)ctx->num_sms * 3), CNT_THREADS, smem,
             ctx->stream>>>((const uint32_t*)ctx->pool.p, (const uint32_t*)ctx->pool_sid.p,
                            (const uint8_t*)ctx->covered.p, members, (uint32_t*)ctx->counts.p);
    LAUNCH_CHECK(ctx, "count_members_kernel");
    return TIM_OK;
}

int tim_count_members(tim_ctx* ctx) { return count_members(ctx, false); }

// counted: the counts are already those of the store.
static int build_index(tim_ctx* ctx, bool counted) {
    const uint64_t n = (uint64_t)ctx->n, members = ctx->members;
    TIM_TRY(tim_ensure(ctx, ctx->node_off, (n + 2) * sizeof(uint64_t)));
    TIM_TRY(tim_ensure(ctx, ctx->node_sets, (members + 1) * sizeof(uint32_t)));
    if (!counted) TIM_TRY(count_members(ctx, false));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->node_off.p, 0, sizeof(uint64_t), ctx->stream));
    const unsigned G = (unsigned)(ctx->num_sms * 8);
    // node_off[v + 1] = start of node v's sets (node_off[0] = 0); the scatter turns it
    // into start(v + 1)
    TIM_TRY(tim_scan_u32_to_u64(ctx, (const uint32_t*)ctx->counts.p,
                                (uint64_t*)ctx->node_off.p + 1, n));
    if (members) {
        scatter_sets_kernel<<<G, 256, 0, ctx->stream>>>(
            (const uint32_t*)ctx->pool.p, (const uint32_t*)ctx->pool_sid.p, members,
            (unsigned long long*)ctx->node_off.p + 1, (uint32_t*)ctx->node_sets.p);
        LAUNCH_CHECK(ctx, "scatter_sets_kernel");
    }
    return TIM_OK;
}

int tim_build_index(tim_ctx* ctx) { return build_index(ctx, false); }

// Rounds r0 .. k - 1 over the full index; with r0 > 0 the flags of the sets and nodes and the
// covered counter are those of the rounds before, and counts holds the uncovered sets'.
static int greedy_full(tim_ctx* ctx, int k, int r0, int32_t* host_seeds, uint64_t* covered) {
    const uint64_t n = (uint64_t)ctx->n;
    if (k < 1 || (uint64_t)k > n) return tim_fail(ctx, TIM_ERR_ARG, "k must be in [1, n]");
    TIM_TRY(tim_ensure(ctx, ctx->covered, ctx->n_sets + 1));
    TIM_TRY(tim_ensure(ctx, ctx->chosen, n + 1));
    TIM_TRY(tim_ensure(ctx, ctx->best, (size_t)k * sizeof(unsigned long long)));
    TIM_TRY(tim_ensure(ctx, ctx->seeds_dev, (size_t)k * sizeof(int32_t)));
    if (r0 == 0) {
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->covered.p, 0, ctx->n_sets + 1, ctx->stream));
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->chosen.p, 0, n + 1, ctx->stream));
        TIM_TRY(tim_zero_scalars(ctx));
    }
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->best.p, 0, (size_t)k * sizeof(unsigned long long),
                                  ctx->stream));
    DevScalars* ds = tim_dscal(ctx);
    auto* best = (unsigned long long*)ctx->best.p;
    // all rounds in one cooperative launch when the device supports it
    int coop = 0, nb = 0;
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device);
    if (coop &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, greedy_rounds_kernel, 256, 0) ==
            cudaSuccess &&
        nb > 0) {
        TIM_TRY(tim_ensure(ctx, ctx->greedy_bar, sizeof(GridBarrier)));
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->greedy_bar.p, 0, sizeof(GridBarrier), ctx->stream));
        // every covered set is listed at most once, in ceil(len / COVER_CHUNK) chunks
        unsigned long long chunk_cap = ctx->n_sets + ctx->members / COVER_CHUNK + 1;
        TIM_TRY(tim_ensure(ctx, ctx->greedy_chunks, chunk_cap * sizeof(unsigned long long)));
        TIM_TRY(tim_ensure(ctx, ctx->greedy_nchunk, (size_t)k * sizeof(unsigned long long)));
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->greedy_nchunk.p, 0, (size_t)k * sizeof(unsigned long long),
                                      ctx->stream));
        auto* d_chunks = (unsigned long long*)ctx->greedy_chunks.p;
        auto* d_nchunk = (unsigned long long*)ctx->greedy_nchunk.p;
        const unsigned grid = (unsigned)(ctx->num_sms * std::min(nb, 4));
        int* d_counts = (int*)ctx->counts.p;
        uint8_t* d_chosen = (uint8_t*)ctx->chosen.p;
        uint64_t nn = n;
        const uint64_t* d_off = (const uint64_t*)ctx->node_off.p;
        const uint32_t* d_ns = (const uint32_t*)ctx->node_sets.p;
        const uint64_t* d_ss = (const uint64_t*)ctx->set_start.p;
        const uint32_t* d_sl = (const uint32_t*)ctx->set_len.p;
        const uint32_t* d_pool = (const uint32_t*)ctx->pool.p;
        uint8_t* d_cov = (uint8_t*)ctx->covered.p;
        int kk = k;
        int32_t* d_seeds = (int32_t*)ctx->seeds_dev.p;
        unsigned long long* d_ncov = &ds->covered;
        GridBarrier* d_bar = (GridBarrier*)ctx->greedy_bar.p;
        int* d_err = &ds->err;
        unsigned limit = ctx->wait_limit;
        void* args[] = {&d_counts, &d_chosen, &nn, &d_off, &d_ns, &d_ss, &d_sl, &d_pool,
                        &d_cov, &r0, &kk, &best, &d_seeds, &d_ncov, &d_bar, &d_err, &limit,
                        &d_chunks, &d_nchunk, &chunk_cap};
        CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void*)greedy_rounds_kernel, dim3(grid),
                                                  dim3(256), args, 0, ctx->stream));
        LAUNCH_CHECK(ctx, "greedy_rounds_kernel");
        if (host_seeds)
            CUDA_TRY(ctx, cudaMemcpyAsync(host_seeds, ctx->seeds_dev.p, (size_t)k * sizeof(int32_t),
                                          cudaMemcpyDeviceToHost, ctx->stream));
        TIM_TRY(tim_read_scalars(ctx));
        if (ctx->h_scal->err & TIM_DEV_ERR_TIMEOUT)
            return tim_fail(ctx, TIM_ERR_TIMEOUT, "greedy grid barrier timed out");
        if (ctx->h_scal->err)
            return tim_fail(ctx, TIM_ERR_CUDA, "device error flags set by the greedy");
        if (covered) *covered = ctx->h_scal->covered;
        return TIM_OK;
    }
    const unsigned GA = (unsigned)(ctx->num_sms * 4);
    const unsigned GC = (unsigned)(ctx->num_sms * 2);
    for (int r = r0; r < k; r++) {
        argmax_kernel<<<GA, 512, 0, ctx->stream>>>((const int*)ctx->counts.p,
                                                   (const uint8_t*)ctx->chosen.p, n, best + r);
        LAUNCH_CHECK(ctx, "argmax_kernel");
        cover_kernel<<<GC, 256, 0, ctx->stream>>>(
            best + r, (const uint64_t*)ctx->node_off.p, (const uint32_t*)ctx->node_sets.p,
            (const uint64_t*)ctx->set_start.p, (const uint32_t*)ctx->set_len.p,
            (const uint32_t*)ctx->pool.p, (uint8_t*)ctx->covered.p, (int*)ctx->counts.p,
            (uint8_t*)ctx->chosen.p, (int32_t*)ctx->seeds_dev.p + r, &ds->covered);
        LAUNCH_CHECK(ctx, "cover_kernel");
    }
    if (host_seeds)
        CUDA_TRY(ctx, cudaMemcpyAsync(host_seeds, ctx->seeds_dev.p, (size_t)k * sizeof(int32_t),
                                      cudaMemcpyDeviceToHost, ctx->stream));
    TIM_TRY(tim_read_scalars(ctx));
    if (covered) *covered = ctx->h_scal->covered;
    return TIM_OK;
}

// Seeds r0 .. k - 1 when every set is covered: the smallest ids not chosen yet (one thread).
__global__ void fill_seeds_kernel(int r0, int k, uint64_t n, uint8_t* __restrict__ chosen,
                                  int32_t* __restrict__ seeds) {
    uint64_t v = 0;
    for (int r = r0; r < k; r++, v++) {
        while (v < n && chosen[v]) v++;  // k <= n: there is one
        chosen[v] = 1;
        seeds[r] = (int32_t)v;
    }
}

// Greedy over candidates in epochs (see above), the full index for what they leave. An epoch
// is a pass over the members that counts, one that indexes the candidates, and the rounds: an
// epoch that did not do CAND_MIN_ROUNDS hands the rest to the full index.
constexpr int CAND_MIN_ROUNDS = 8;
// The candidates cost some 50 us before the first round and save some 4 us a round, and more the
// more members there are: selections of at most CAND_MIN_K seeds from stores of at most
// CAND_MIN_MEMBERS take the full index. (One, three and six seeds, candidates / full index, Chung-Lu
// 20,001 nodes: 113,528 members 0.140 / 0.110, 0.160 / 0.134, 0.185 / 0.166 ms; 226,602 0.152 / 0.135,
// 0.163 / 0.162, 0.187 / 0.195; 458,240 0.153 / 0.188, 0.166 / 0.220, 0.191 / 0.257. 5,001 nodes cross
// at 200,000 members, R-MAT 19 at a million for one seed and, at any size, between three and six.)
constexpr int CAND_MIN_K = 5;
constexpr uint64_t CAND_MIN_MEMBERS = 150'000;
// an epoch needs a candidate for every round left, or this many
constexpr int CAND_NEED = 128;

int tim_greedy(tim_ctx* ctx, int k, int32_t* host_seeds, uint64_t* covered) {
    const uint64_t n = (uint64_t)ctx->n, members = ctx->members;
    if (k < 1 || (uint64_t)k > n) return tim_fail(ctx, TIM_ERR_ARG, "k must be in [1, n]");
    int coop = 0, nb = 0;
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device);
    // 32-bit offsets and counts; an open stepwise selection keeps the full index's counts
    bool cand = coop && !ctx->select_open && members < 0xFFFFFFFFull &&
                ctx->n_sets < 0x7FFFFFFFull && (k > CAND_MIN_K || members > CAND_MIN_MEMBERS);
    if (cand) {
        CUDA_TRY(ctx, cudaFuncSetAttribute(cand_rounds_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)CG_SMEM));
        CUDA_TRY(ctx, cudaFuncSetAttribute(cand_index_kernel<false>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)CI_SMEM));
        CUDA_TRY(ctx, cudaFuncSetAttribute(cand_index_kernel<true>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)CI_SMEM));
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, cand_rounds_kernel, CG_THREADS,
                                                          CG_SMEM) != cudaSuccess) {
            cudaGetLastError();
            nb = 0;
        }
        cand = nb > 0;
    }
    unsigned long long chunk_cap = 2 * (members / CG_CHUNK) + 1;
    if (cand) {  // what the full index does without; it also does where this has no room
        const std::pair<DevBuf*, size_t> need[] = {
            {&ctx->set_rec, (ctx->n_sets + 1) * sizeof(uint4)},
            {&ctx->cand, sizeof(CandState)},
            {&ctx->greedy_chunks, chunk_cap * sizeof(unsigned long long)},
            {&ctx->node_sets, (members + 1) * sizeof(uint32_t)}};
        for (const auto& b : need) {
            const int rc = cand ? tim_ensure(ctx, *b.first, b.second) : TIM_OK;
            if (rc != TIM_OK && rc != TIM_ERR_OOM) return rc;
            cand = cand && rc == TIM_OK;
        }
        if (!cand)
            for (DevBuf* b : {&ctx->set_rec, &ctx->cand, &ctx->greedy_chunks}) tim_free(*b);
    }
    if (!cand) {
        TIM_TRY(tim_build_index(ctx));
        return greedy_full(ctx, k, 0, host_seeds, covered);
    }
    TIM_TRY(tim_ensure(ctx, ctx->covered, ctx->n_sets + 1));
    TIM_TRY(tim_ensure(ctx, ctx->chosen, n + 1));
    TIM_TRY(tim_ensure(ctx, ctx->seeds_dev, (size_t)k * sizeof(int32_t)));
    TIM_TRY(tim_ensure(ctx, ctx->greedy_bar, sizeof(GridBarrier)));
    TIM_TRY(tim_ensure(ctx, ctx->greedy_nchunk, (size_t)k * sizeof(unsigned long long)));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->covered.p, 0, ctx->n_sets + 1, ctx->stream));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->chosen.p, 0, n + 1, ctx->stream));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->greedy_nchunk.p, 0, (size_t)k * sizeof(unsigned long long),
                                  ctx->stream));
    TIM_TRY(tim_zero_scalars(ctx));
    DevScalars* ds = tim_dscal(ctx);
    auto* st = (CandState*)ctx->cand.p;
    // (chunks of sets above CG_CHUNK members: ceil(len / CG_CHUNK) < 2 len / CG_CHUNK each)
    // blocks: one per SM, fewer for few members (a barrier of few blocks is shorter)
    const uint64_t tiles = members / ((uint64_t)CG_THREADS * TILE_ITEMS) + 1;
    const unsigned GN = (unsigned)std::min<uint64_t>(n / 1024 + 1, (uint64_t)ctx->num_sms * 4);
    const unsigned GT = (unsigned)std::min<uint64_t>(tiles, (uint64_t)ctx->num_sms);
    const unsigned GR =
        members <= CAND_SOLO
            ? 1u
            : (unsigned)std::min<uint64_t>(members / 8192 + 1, (uint64_t)ctx->num_sms);
    if (ctx->n_sets) {
        set_rec_kernel<<<(unsigned)std::min<uint64_t>(ctx->n_sets / 256 + 1,
                                                      (uint64_t)ctx->num_sms * 8),
                         256, 0, ctx->stream>>>((const uint64_t*)ctx->set_start.p,
                                                (const uint32_t*)ctx->set_len.p, ctx->n_sets,
                                                (uint4*)ctx->set_rec.p);
        LAUNCH_CHECK(ctx, "set_rec_kernel");
    }
    int r = 0;
    for (bool live = false;; live = true) {
        TIM_TRY(count_members(ctx, live));
        CUDA_TRY(ctx, cudaMemsetAsync(st, 0, sizeof(CandState), ctx->stream));
        CUDA_TRY(ctx, cudaMemsetAsync(st->key, 0xFF, sizeof st->key, ctx->stream));
        CUDA_TRY(ctx, cudaMemsetAsync(ctx->greedy_bar.p, 0, sizeof(GridBarrier), ctx->stream));
        count_bins_kernel<<<GN, 256, 0, ctx->stream>>>((const uint32_t*)ctx->counts.p, n, st);
        LAUNCH_CHECK(ctx, "count_bins_kernel");
        candidates_kernel<<<GN, 256, 0, ctx->stream>>>((const uint32_t*)ctx->counts.p, n,
                                                    (uint32_t)std::min(k - r, CAND_NEED), st);
        LAUNCH_CHECK(ctx, "candidates_kernel");
        cand_table_kernel<<<1, 1024, 0, ctx->stream>>>(st);
        LAUNCH_CHECK(ctx, "cand_table_kernel");
        auto* index = live ? cand_index_kernel<true> : cand_index_kernel<false>;
        index<<<GT, CG_THREADS, CI_SMEM, ctx->stream>>>(
            (const uint32_t*)ctx->pool.p, (const uint32_t*)ctx->pool_sid.p,
            (const uint8_t*)ctx->covered.p, members, st, (uint32_t*)ctx->node_sets.p);
        LAUNCH_CHECK(ctx, "cand_index_kernel");
        const uint32_t* d_sets = (const uint32_t*)ctx->node_sets.p;
        uint4* d_rec = (uint4*)ctx->set_rec.p;
        const uint32_t* d_pool = (const uint32_t*)ctx->pool.p;
        uint8_t* d_cov = (uint8_t*)ctx->covered.p;
        uint8_t* d_chosen = (uint8_t*)ctx->chosen.p;
        int32_t* d_seeds = (int32_t*)ctx->seeds_dev.p;
        unsigned long long* d_ncov = &ds->covered;
        unsigned* d_done = &ds->done;
        GridBarrier* d_bar = (GridBarrier*)ctx->greedy_bar.p;
        int* d_err = &ds->err;
        unsigned limit = ctx->wait_limit;
        auto* d_chunks = (unsigned long long*)ctx->greedy_chunks.p;
        auto* d_nchunk = (unsigned long long*)ctx->greedy_nchunk.p;
        int r0 = r, kk = k;
        void* args[] = {&st,     &d_sets, &d_rec, &d_pool, &d_cov, &r0,       &kk,       &d_chosen,
                        &d_seeds, &d_ncov, &d_done, &d_bar, &d_err, &limit, &d_chunks, &d_nchunk,
                        &chunk_cap};
        CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void*)cand_rounds_kernel, dim3(GR),
                                                  dim3(CG_THREADS), args, CG_SMEM, ctx->stream));
        LAUNCH_CHECK(ctx, "cand_rounds_kernel");
        if (host_seeds)
            CUDA_TRY(ctx, cudaMemcpyAsync(host_seeds, d_seeds, (size_t)k * sizeof(int32_t),
                                          cudaMemcpyDeviceToHost, ctx->stream));
        TIM_TRY(tim_read_scalars(ctx));
        if (ctx->h_scal->err & TIM_DEV_ERR_TIMEOUT)
            return tim_fail(ctx, TIM_ERR_TIMEOUT, "greedy grid barrier timed out");
        if (ctx->h_scal->err)
            return tim_fail(ctx, TIM_ERR_CUDA, "device error flags set by the greedy");
        const int done = (int)(ctx->h_scal->done & 0x7FFFFFFFu);
        const bool all = ctx->h_scal->done >> 31;  // every node with a set was a candidate
        if (done < k && all && k - done <= 1024) {
            fill_seeds_kernel<<<1, 1, 0, ctx->stream>>>(done, k, n, d_chosen, d_seeds);
            LAUNCH_CHECK(ctx, "fill_seeds_kernel");
            if (host_seeds)
                CUDA_TRY(ctx, cudaMemcpyAsync(host_seeds, d_seeds, (size_t)k * sizeof(int32_t),
                                              cudaMemcpyDeviceToHost, ctx->stream));
            TIM_TRY(tim_sync(ctx));
        } else if (done < k && done - r < CAND_MIN_ROUNDS) {
            TIM_TRY(build_index(ctx, !live));
            if (done > 0) TIM_TRY(count_members(ctx, true));
            return greedy_full(ctx, k, done, host_seeds, covered);
        } else if (done < k) {
            r = done;
            continue;
        }
        if (covered) *covered = ctx->h_scal->covered;
        return TIM_OK;
    }
}

// Bitmap of a seed set held in device memory (for Algorithm 3's coverage test).
__global__ void mark_seeds_kernel(const int32_t* __restrict__ seeds, int k,
                                  uint32_t* __restrict__ mark) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) {
        uint32_t u = (uint32_t)seeds[i];
        atomicOr(&mark[u >> 5], 1u << (u & 31));
    }
}

// Stepwise greedy: the caller chooses each node (for example from coverage counts summed
// over several contexts), the context covers that node's sets of its own store.
int tim_greedy_begin(tim_ctx* ctx) {
    TIM_TRY(tim_build_index(ctx));
    TIM_TRY(tim_ensure(ctx, ctx->covered, ctx->n_sets + 1));
    TIM_TRY(tim_ensure(ctx, ctx->chosen, (uint64_t)ctx->n + 1));
    TIM_TRY(tim_ensure(ctx, ctx->best, sizeof(unsigned long long)));
    TIM_TRY(tim_ensure(ctx, ctx->seeds_dev, sizeof(int32_t)));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->covered.p, 0, ctx->n_sets + 1, ctx->stream));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->chosen.p, 0, (uint64_t)ctx->n + 1, ctx->stream));
    return TIM_OK;
}

int tim_greedy_take(tim_ctx* ctx, int32_t v, uint64_t* newly_covered) {
    // the key cover_kernel decodes: any count, node v
    const unsigned long long key = (1ull << 32) | (unsigned long long)(~(uint32_t)v);
    // (a selection between the steps that ran out of memory may have given these back)
    TIM_TRY(tim_ensure(ctx, ctx->best, sizeof(unsigned long long)));
    TIM_TRY(tim_ensure(ctx, ctx->seeds_dev, sizeof(int32_t)));
    TIM_TRY(tim_zero_scalars(ctx));
    DevScalars* ds = tim_dscal(ctx);
    set_key_kernel<<<1, 1, 0, ctx->stream>>>((unsigned long long*)ctx->best.p, key);
    LAUNCH_CHECK(ctx, "set_key_kernel");
    cover_kernel<<<(unsigned)(ctx->num_sms * 2), 256, 0, ctx->stream>>>(
        (const unsigned long long*)ctx->best.p, (const uint64_t*)ctx->node_off.p,
        (const uint32_t*)ctx->node_sets.p, (const uint64_t*)ctx->set_start.p,
        (const uint32_t*)ctx->set_len.p, (const uint32_t*)ctx->pool.p, (uint8_t*)ctx->covered.p,
        (int*)ctx->counts.p, (uint8_t*)ctx->chosen.p, (int32_t*)ctx->seeds_dev.p, &ds->covered);
    LAUNCH_CHECK(ctx, "cover_kernel");
    TIM_TRY(tim_read_scalars(ctx));
    if (newly_covered) *newly_covered = ctx->h_scal->covered;
    return TIM_OK;
}

int tim_mark_seeds(tim_ctx* ctx, const int32_t* d_seeds, int k) {
    const uint64_t words = (uint64_t)(ctx->n + 31) / 32 + 1;
    TIM_TRY(tim_ensure(ctx, ctx->seed_mark, words * sizeof(uint32_t)));
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->seed_mark.p, 0, words * sizeof(uint32_t), ctx->stream));
    if (k > 0) {
        mark_seeds_kernel<<<(k + 255) / 256, 256, 0, ctx->stream>>>(d_seeds, k,
                                                                    (uint32_t*)ctx->seed_mark.p);
        LAUNCH_CHECK(ctx, "mark_seeds_kernel");
    }
    return TIM_OK;
}

// ------------------------------------------------------ several queries at once
//
// The greedy of Algorithm 1 for a batch of queries, each over its own context's
// RR-set store: every kernel covers all queries (each query owns a range of blocks in
// proportion to its work), so one round of the batch is two launches whatever the
// number of queries, and the whole sequence
// (index build and the k rounds) is captured once into a CUDA graph and launched as
// one unit.

namespace {

struct GreedyDesc {
    const uint32_t* pool;
    const uint32_t* pool_sid;
    uint64_t members;
    const uint64_t* set_start;
    const uint32_t* set_len;
    int* counts;
    uint64_t* node_off;
    uint32_t* cursor;
    uint32_t* node_sets;
    uint8_t* covered;
    uint8_t* chosen;
    unsigned long long* best;
    int32_t* seeds;
    unsigned long long* ncov;
    uint64_t n;
    int k;
    int pad;
};

// Blocks are shared out among the queries in proportion to their work; block b belongs
// to the query q with bstart[q] <= b < bstart[q + 1] and is its (b - bstart[q])-th.
__device__ __forceinline__ int block_query(const unsigned* __restrict__ bstart, int nq,
                                           unsigned* local, unsigned* count) {
    int lo = 0, hi = nq;  // bstart[lo] <= b < bstart[hi]
    const unsigned b = blockIdx.x;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (bstart[mid] <= b)
            lo = mid;
        else
            hi = mid;
    }
    *local = b - bstart[lo];
    *count = bstart[lo + 1] - bstart[lo];
    return lo;
}

__global__ void mcount_kernel(const GreedyDesc* __restrict__ gd, const unsigned* __restrict__ bstart,
                              int nq) {
    unsigned lb, nb;
    const GreedyDesc& d = gd[block_query(bstart, nq, &lb, &nb)];
    for (uint64_t p = lb * (uint64_t)blockDim.x + threadIdx.x; p < d.members;
         p += (uint64_t)nb * blockDim.x)
        atomicAdd((unsigned*)&d.counts[d.pool[p]], 1u);
}

__global__ void mscatter_kernel(const GreedyDesc* __restrict__ gd,
                                const unsigned* __restrict__ bstart, int nq) {
    unsigned lb, nb;
    const GreedyDesc& d = gd[block_query(bstart, nq, &lb, &nb)];
    for (uint64_t p = lb * (uint64_t)blockDim.x + threadIdx.x; p < d.members;
         p += (uint64_t)nb * blockDim.x) {
        const uint32_t u = d.pool[p];
        const uint32_t slot = atomicAdd(&d.cursor[u], 1u);
        d.node_sets[d.node_off[u] + slot] = d.pool_sid[p];
    }
}

__global__ void margmax_kernel(const GreedyDesc* __restrict__ gd, const unsigned* __restrict__ bstart,
                               int nq, int r) {
    unsigned lb, nb;
    const GreedyDesc& d = gd[block_query(bstart, nq, &lb, &nb)];
    if (r >= d.k) return;
    unsigned long long b = slice_argmax(d.counts, d.chosen, d.n,
                                        lb * (uint64_t)blockDim.x + threadIdx.x,
                                        (uint64_t)nb * blockDim.x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
        b = y > b ? y : b;
    }
    if ((threadIdx.x & 31) == 0 && b) atomicMax(&d.best[r], b);
}

__global__ void mcover_kernel(const GreedyDesc* __restrict__ gd, const unsigned* __restrict__ bstart,
                              int nq, int r) {
    unsigned lb, nb;
    const GreedyDesc& d = gd[block_query(bstart, nq, &lb, &nb)];
    if (r >= d.k) return;
    const unsigned long long key = d.best[r];
    if (key == 0) return;
    const uint32_t v = ~(uint32_t)(key & 0xFFFFFFFFull);
    if (lb == 0 && threadIdx.x == 0) {
        d.chosen[v] = 1;
        d.seeds[r] = (int32_t)v;
    }
    const int lane = threadIdx.x & 31;
    const uint64_t warp = (lb * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)nb * blockDim.x) >> 5;
    const uint64_t a = d.node_off[v], b = d.node_off[v + 1];
    unsigned long long fresh = 0;
    for (uint64_t i = a + warp; i < b; i += nwarps) {
        const uint32_t s = d.node_sets[i];
        if (d.covered[s]) continue;
        __syncwarp();
        if (lane == 0) {
            d.covered[s] = 1;
            fresh++;
        }
        const uint64_t st = d.set_start[s];
        const uint32_t len = d.set_len[s];
        for (uint32_t t = lane; t < len; t += 32) atomicSub(&d.counts[d.pool[st + t]], 1);
    }
    if (lane == 0 && fresh) atomicAdd(d.ncov, fresh);
}

}  // namespace

int tim_greedy_batch(tim_ctx* owner, tim_ctx* const* ctxs, const int* ks, int nq,
                     int32_t* const* host_seeds, uint64_t* covered, bool use_graph) {
    if (nq <= 0) return TIM_OK;
    int kmax = 0;
    std::vector<GreedyDesc> gd(nq);
    for (int i = 0; i < nq; i++) {
        tim_ctx* c = ctxs[i];
        const uint64_t n = (uint64_t)c->n;
        const int k = ks[i];
        if (k < 1 || (uint64_t)k > n) return tim_fail(owner, TIM_ERR_ARG, "k must be in [1, n]");
        kmax = std::max(kmax, k);
        TIM_TRY(tim_ensure(c, c->counts, (n + 1) * sizeof(int)));
        TIM_TRY(tim_ensure(c, c->node_off, (n + 1) * sizeof(uint64_t)));
        TIM_TRY(tim_ensure(c, c->cursor, (n + 1) * sizeof(uint32_t)));
        TIM_TRY(tim_ensure(c, c->node_sets, (c->members + 1) * sizeof(uint32_t)));
        TIM_TRY(tim_ensure(c, c->covered, c->n_sets + 1));
        TIM_TRY(tim_ensure(c, c->chosen, n + 1));
        TIM_TRY(tim_ensure(c, c->best, (size_t)k * sizeof(unsigned long long) + 8));
        TIM_TRY(tim_ensure(c, c->seeds_dev, (size_t)k * sizeof(int32_t)));
        // the scan's block sums, so that nothing is allocated inside the capture
        TIM_TRY(tim_ensure(c, c->scratch_e, ((n + 4095) / 4096 + 1) * sizeof(unsigned long long)));
        if (!c->pool.p) TIM_TRY(tim_ensure(c, c->pool, 16));
        if (!c->pool_sid.p) TIM_TRY(tim_ensure(c, c->pool_sid, 16));
        if (!c->set_start.p) TIM_TRY(tim_ensure(c, c->set_start, 16));
        if (!c->set_len.p) TIM_TRY(tim_ensure(c, c->set_len, 16));
        GreedyDesc& d = gd[i];
        d.pool = (const uint32_t*)c->pool.p;
        d.pool_sid = (const uint32_t*)c->pool_sid.p;
        d.members = c->members;
        d.set_start = (const uint64_t*)c->set_start.p;
        d.set_len = (const uint32_t*)c->set_len.p;
        d.counts = (int*)c->counts.p;
        d.node_off = (uint64_t*)c->node_off.p;
        d.cursor = (uint32_t*)c->cursor.p;
        d.node_sets = (uint32_t*)c->node_sets.p;
        d.covered = (uint8_t*)c->covered.p;
        d.chosen = (uint8_t*)c->chosen.p;
        d.best = (unsigned long long*)c->best.p;
        d.seeds = (int32_t*)c->seeds_dev.p;
        d.n = n;
        d.k = k;
        d.pad = 0;
    }
    // blocks per query in proportion to its work: nodes (argmax) and members (index,
    // cover); every query gets at least one block
    const unsigned total_blocks = (unsigned)std::max(nq, owner->num_sms * 8);
    std::vector<unsigned> bs_nodes(nq + 1, 0), bs_memb(nq + 1, 0);
    {
        double wn = 0, wm = 0;
        for (int i = 0; i < nq; i++) {
            wn += (double)gd[i].n;
            wm += (double)gd[i].members + 1.0;
        }
        for (int i = 0; i < nq; i++) {
            bs_nodes[i + 1] = bs_nodes[i] +
                              std::max(1u, (unsigned)(total_blocks * ((double)gd[i].n / wn)));
            bs_memb[i + 1] = bs_memb[i] + std::max(1u, (unsigned)(total_blocks *
                                                                  (((double)gd[i].members + 1.0) / wm)));
        }
    }
    // descriptors | covered counters | block starts (nodes) | block starts (members)
    const size_t off_cov = ((size_t)nq * sizeof(GreedyDesc) + 255) & ~size_t(255);
    const size_t off_bn = (off_cov + (size_t)nq * 8 + 255) & ~size_t(255);
    const size_t off_bm = (off_bn + (size_t)(nq + 1) * 4 + 255) & ~size_t(255);
    TIM_TRY(tim_ensure(owner, owner->greedy_batch, off_bm + (size_t)(nq + 1) * 4));
    GreedyDesc* d_gd = (GreedyDesc*)owner->greedy_batch.p;
    unsigned long long* d_cov = (unsigned long long*)((char*)owner->greedy_batch.p + off_cov);
    unsigned* d_bn = (unsigned*)((char*)owner->greedy_batch.p + off_bn);
    unsigned* d_bm = (unsigned*)((char*)owner->greedy_batch.p + off_bm);
    for (int i = 0; i < nq; i++) gd[i].ncov = d_cov + i;
    cudaStream_t st = owner->stream;
    CUDA_TRY(owner, cudaMemcpyAsync(d_gd, gd.data(), (size_t)nq * sizeof(GreedyDesc),
                                    cudaMemcpyHostToDevice, st));
    CUDA_TRY(owner, cudaMemcpyAsync(d_bn, bs_nodes.data(), (size_t)(nq + 1) * 4,
                                    cudaMemcpyHostToDevice, st));
    CUDA_TRY(owner, cudaMemcpyAsync(d_bm, bs_memb.data(), (size_t)(nq + 1) * 4,
                                    cudaMemcpyHostToDevice, st));
    CUDA_TRY(owner, cudaStreamSynchronize(st));
    std::vector<cudaStream_t> saved(nq);
    for (int i = 0; i < nq; i++) {
        saved[i] = ctxs[i]->stream;
        ctxs[i]->stream = st;
    }
    cudaGraph_t graph = nullptr;
    int rc = TIM_OK;
    if (use_graph &&
        cudaStreamBeginCapture(st, cudaStreamCaptureModeRelaxed) != cudaSuccess) {
        cudaGetLastError();
        use_graph = false;
    }
    do {
        if ((rc = tim_cuda_check(owner, cudaMemsetAsync(d_cov, 0, (size_t)nq * 8, st), "memset")))
            break;
        for (int i = 0; i < nq && rc == TIM_OK; i++) {
            const GreedyDesc& d = gd[i];
            if ((rc = tim_cuda_check(owner, cudaMemsetAsync(d.counts, 0, (d.n + 1) * 4, st), "memset")))
                break;
            if ((rc = tim_cuda_check(owner, cudaMemsetAsync(d.cursor, 0, (d.n + 1) * 4, st), "memset")))
                break;
            if ((rc = tim_cuda_check(owner, cudaMemsetAsync(d.covered, 0, ctxs[i]->n_sets + 1, st),
                                     "memset")))
                break;
            if ((rc = tim_cuda_check(owner, cudaMemsetAsync(d.chosen, 0, d.n + 1, st), "memset")))
                break;
            if ((rc = tim_cuda_check(owner, cudaMemsetAsync(d.best, 0, (size_t)d.k * 8, st), "memset")))
                break;
        }
        if (rc) break;
        mcount_kernel<<<bs_memb[nq], 256, 0, st>>>(d_gd, d_bm, nq);
        owner->launches++;
        for (int i = 0; i < nq && rc == TIM_OK; i++)
            rc = tim_scan_u32_to_u64(ctxs[i], (const uint32_t*)gd[i].counts, gd[i].node_off, gd[i].n);
        if (rc) break;
        mscatter_kernel<<<bs_memb[nq], 256, 0, st>>>(d_gd, d_bm, nq);
        owner->launches++;
        for (int r = 0; r < kmax; r++) {
            margmax_kernel<<<bs_nodes[nq], 512, 0, st>>>(d_gd, d_bn, nq, r);
            mcover_kernel<<<bs_memb[nq], 256, 0, st>>>(d_gd, d_bm, nq, r);
            owner->launches += 2;
        }
        rc = tim_cuda_check(owner, cudaGetLastError(), "batched greedy kernels");
    } while (0);
    if (use_graph) {
        cudaError_t e = cudaStreamEndCapture(st, &graph);
        if (rc == TIM_OK && e != cudaSuccess) rc = tim_cuda_check(owner, e, "cudaStreamEndCapture");
        if (rc == TIM_OK) {
            cudaGraphExec_t exec = nullptr;
            e = cudaGraphInstantiate(&exec, graph, 0);
            if (e == cudaSuccess) {
                e = cudaGraphLaunch(exec, st);
                if (e == cudaSuccess) e = cudaStreamSynchronize(st);
                cudaGraphExecDestroy(exec);
            }
            rc = tim_cuda_check(owner, e, "batched greedy graph");
        }
        if (graph) cudaGraphDestroy(graph);
    }
    for (int i = 0; i < nq; i++) ctxs[i]->stream = saved[i];
    if (rc) return rc;
    std::vector<unsigned long long> hc(nq);
    CUDA_TRY(owner, cudaMemcpyAsync(hc.data(), d_cov, (size_t)nq * 8, cudaMemcpyDeviceToHost, st));
    for (int i = 0; i < nq; i++)
        if (host_seeds && host_seeds[i])
            CUDA_TRY(owner, cudaMemcpyAsync(host_seeds[i], gd[i].seeds, (size_t)gd[i].k * 4,
                                            cudaMemcpyDeviceToHost, st));
    CUDA_TRY(owner, cudaStreamSynchronize(st));
    for (int i = 0; i < nq; i++)
        if (covered) covered[i] = hc[i];
    return TIM_OK;
}
