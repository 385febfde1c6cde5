// noalloc.cu -- tim_node_select_noalloc: the greedy node selection of tim_node_select
// (node -> set index, exclusive scan, k rounds of argmax and cover) over a CSR of RR
// sets that the caller owns, for callers that cannot let the library allocate device
// memory: code whose device memory is owned by another allocator or a fixed budget,
// and code that must not trigger the device-wide synchronisation that cudaMalloc and
// cudaFree imply. Nothing here calls cudaMalloc, cudaFree or an allocating library.
//
// All scratch lives in one file-scope __device__ array of NA_SCRATCH_BYTES (about
// 13.3 MiB), which every GPU that loads the library holds until the process exits. Host code
// cannot use the array's name as a device address, so the first call on each device
// looks the address up with cudaGetSymbolAddress (with that device current) and keeps
// it; make that first call before any stream capture. Every call also reads two
// offsets back to the host and waits for its stream. Every call shares the array and
// leaves its contents behind: each call clears what must start at zero, and calls
// whose work overlaps on the GPU (other streams, other host threads) race. Members
// must be distinct within a set; a repeated member is not detected.
#include <mutex>

#include "common.cuh"

namespace {

// Limits of the caller's problem, fixed by the size of the scratch array.
constexpr int64_t NA_MAX_NODES = 1 << 18;        // n
constexpr uint64_t NA_MAX_SETS = 1 << 20;        // number of RR sets
constexpr uint64_t NA_MAX_MEMBERS = 1 << 21;     // sum of |R|
constexpr int NA_MAX_K = 1024;                   // seeds
constexpr uint64_t NA_MAX_BLOCKS = 1024;         // blocks of the launch (one per SM)

// Layout of the scratch array (byte offsets, each a multiple of 256).
constexpr uint64_t al(uint64_t x) { return (x + 255) & ~uint64_t(255); }
constexpr uint64_t OFF_COUNTS = 0;                                           // int32[n]
constexpr uint64_t OFF_NODE_OFF = al(OFF_COUNTS + 4 * NA_MAX_NODES);         // u64[n+1]
constexpr uint64_t OFF_CURSOR = al(OFF_NODE_OFF + 8 * (NA_MAX_NODES + 1));   // u32[n]
constexpr uint64_t OFF_NODE_SETS = al(OFF_CURSOR + 4 * NA_MAX_NODES);        // u32[members]
constexpr uint64_t OFF_COVERED = al(OFF_NODE_SETS + 4 * NA_MAX_MEMBERS);     // u8[sets]
constexpr uint64_t OFF_CHOSEN = al(OFF_COVERED + NA_MAX_SETS);               // u8[n]
constexpr uint64_t OFF_BEST = al(OFF_CHOSEN + NA_MAX_NODES);                 // u64[k]
constexpr uint64_t OFF_SUMS = al(OFF_BEST + 8 * NA_MAX_K);                   // u64[blocks]
constexpr uint64_t OFF_FLAGS = al(OFF_SUMS + 8 * NA_MAX_BLOCKS);             // u64[8]
constexpr uint64_t NA_SCRATCH_BYTES = al(OFF_FLAGS + 64);

static __device__ __align__(256) unsigned char na_scratch[NA_SCRATCH_BYTES];

struct NaView {
    int* counts;
    uint64_t* node_off;
    uint32_t* cursor;
    uint32_t* node_sets;
    uint8_t* covered;
    uint8_t* chosen;
    unsigned long long* best;
    unsigned long long* sums;
    unsigned long long* flags;  // [0] covered count, [1] error bits, [2] barrier, [3] its error,
                                // [4] the rounds' barrier
};

NaView view_of(unsigned char* base) {
    NaView v;
    v.counts = (int*)(base + OFF_COUNTS);
    v.node_off = (uint64_t*)(base + OFF_NODE_OFF);
    v.cursor = (uint32_t*)(base + OFF_CURSOR);
    v.node_sets = (uint32_t*)(base + OFF_NODE_SETS);
    v.covered = base + OFF_COVERED;
    v.chosen = base + OFF_CHOSEN;
    v.best = (unsigned long long*)(base + OFF_BEST);
    v.sums = (unsigned long long*)(base + OFF_SUMS);
    v.flags = (unsigned long long*)(base + OFF_FLAGS);
    return v;
}

constexpr int NA_THREADS = 512;
// blocks that run the greedy rounds (8, 16, 32, 64, 152 blocks: 951, 762, 700, 672, 673 us at
// the size below)
constexpr unsigned NA_ROUNDS_GRID = 64;
constexpr uint32_t NA_SLOTS = 4096;  // hot-node table of the histogram
constexpr uint32_t NA_EMPTY = 0xFFFFFFFFu;

// Exclusive scan of one value per thread over the block.
__device__ unsigned long long na_block_scan(unsigned long long x, unsigned long long* wsum,
                                            unsigned long long* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    unsigned long long before = 0, all = 0;
    for (int i = 0; i < NA_THREADS / 32; i++) {
        if (i < w) before += wsum[i];
        all += wsum[i];
    }
    *total = all;
    return before + inc - x;
}

struct NaArgs {
    const int64_t* off;
    const int32_t* mem;
    uint64_t n_sets;
    int64_t n;
    uint64_t members;
    int k;
    int32_t* seeds;
    uint64_t* covered_out;
    unsigned rounds_grid;
    NaView v;
    unsigned limit;
};

// The whole selection in one cooperative launch; a grid barrier separates its phases:
// clearing, the histogram of members (hub nodes counted in a shared-memory table first, since
// atomics on one address take turns), the scan into node offsets, node -> sets, and per round
// an argmax over the counts and the cover of the chosen node's sets (eight lanes per set).
// One launch per phase and two per round: 150,001 nodes, 250,007 sets of six members, k = 50,
// 870 us, this 672 us; bound by a round's chain of about fourteen dependent L2 accesses, two
// barriers among them.
__global__ void __launch_bounds__(NA_THREADS) na_select_kernel(NaArgs a) {
    __shared__ uint32_t tag[NA_SLOTS], num[NA_SLOTS];
    __shared__ unsigned long long wsum[NA_THREADS / 32];
    const NaView v = a.v;
    GridBarrier* bar = reinterpret_cast<GridBarrier*>(v.flags + 2);
    int* err = reinterpret_cast<int*>(v.flags + 3);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t tid = blockIdx.x * (uint64_t)NA_THREADS + threadIdx.x;
    const uint64_t nt = (uint64_t)gridDim.x * NA_THREADS;
    const uint64_t n = (uint64_t)a.n;
    for (uint64_t i = tid; i < n; i += nt) {
        v.counts[i] = 0;
        v.chosen[i] = 0;
    }
    for (uint64_t i = tid; i < a.n_sets; i += nt) v.covered[i] = 0;
    for (uint64_t i = tid; i < (uint64_t)a.k; i += nt) v.best[i] = 0;
    for (uint32_t i = threadIdx.x; i < NA_SLOTS; i += NA_THREADS) {
        tag[i] = NA_EMPTY;
        num[i] = 0u;
    }
    if (!grid_barrier(bar, err, a.limit)) return;
    // histogram; members outside [0, n) are skipped and flagged
    for (uint64_t p = tid; p < a.members; p += nt) {
        const int32_t u = a.mem[p];
        if (u < 0 || u >= a.n) {
            atomicOr(&v.flags[1], 1ull);
            continue;
        }
        const uint32_t h = ((uint32_t)u * 0x9E3779B1u) >> 20;  // 12 bits
        uint32_t t = ((volatile uint32_t*)tag)[h];
        if (t == NA_EMPTY) {
            t = atomicCAS(&tag[h], NA_EMPTY, (uint32_t)u);
            if (t == NA_EMPTY) t = (uint32_t)u;
        }
        if (t == (uint32_t)u)
            atomicAdd(&num[h], 1u);
        else
            atomicAdd(&v.counts[u], 1);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < NA_SLOTS; i += NA_THREADS)
        if (num[i]) atomicAdd(&v.counts[tag[i]], (int)num[i]);
    if (!grid_barrier(bar, err, a.limit)) return;
    // node offsets: every block scans a contiguous range of nodes
    const uint64_t per = (n + gridDim.x - 1) / gridDim.x;
    const uint64_t ib = min(blockIdx.x * per, n), ie = min(ib + per, n);
    unsigned long long sum = 0, tot = 0;
    for (uint64_t i = ib + threadIdx.x; i < ie; i += NA_THREADS) sum += (uint32_t)__ldcg(v.counts + i);
    na_block_scan(sum, wsum, &tot);
    if (threadIdx.x == 0) v.sums[blockIdx.x] = tot;
    if (!grid_barrier(bar, err, a.limit)) return;
    unsigned long long before = 0;
    for (uint32_t b = threadIdx.x; b < blockIdx.x; b += NA_THREADS) before += __ldcg(v.sums + b);
    na_block_scan(before, wsum, &before);  // the blocks' totals below this one
    for (uint64_t c = ib; c < ie; c += NA_THREADS) {
        const uint64_t i = c + threadIdx.x;
        const unsigned long long x = i < ie ? (uint32_t)__ldcg(v.counts + i) : 0ull;
        const unsigned long long ex = na_block_scan(x, wsum, &tot);
        if (i < ie) {
            v.node_off[i] = before + ex;
            v.cursor[i] = (uint32_t)(before + ex);  // at most NA_MAX_MEMBERS
        }
        before += tot;
    }
    if (ie == n && ib < n && threadIdx.x == 0) v.node_off[n] = before;
    if (!grid_barrier(bar, err, a.limit)) return;
    // node -> sets, eight lanes per set
    const int sub = lane & 7;
    for (uint64_t s = tid >> 3; s < a.n_sets; s += nt >> 3) {
        const int64_t pa = a.off[s], pb = a.off[s + 1];
        if (pa < 0 || pb < pa || (uint64_t)pb > a.members) {  // malformed offsets: skip the set
            if (sub == 0) atomicOr(&v.flags[1], 2ull);
            continue;
        }
        for (int64_t p = pa + sub; p < pb; p += 8) {
            const int32_t u = a.mem[p];
            if (u < 0 || u >= a.n) continue;
            const uint32_t at = atomicAdd(&v.cursor[u], 1u);
            if (at < __ldcg(v.node_off + u + 1))
                v.node_sets[at] = (uint32_t)s;
            else
                atomicOr(&v.flags[1], 2ull);
        }
    }
    if (!grid_barrier(bar, err, a.limit)) return;
    // the rounds are short: the first few blocks run them, with barriers of their own
    if (blockIdx.x >= a.rounds_grid) return;
    bar = reinterpret_cast<GridBarrier*>(v.flags + 4);
    const uint64_t nr = (uint64_t)a.rounds_grid * NA_THREADS;
    unsigned long long fresh = 0;
    for (int r = 0; r < a.k; r++) {
        unsigned long long b = slice_argmax(v.counts, v.chosen, n, tid, nr);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
            b = y > b ? y : b;
        }
        __syncthreads();
        if (lane == 0) wsum[wid] = b;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < NA_THREADS / 32; i++) b = wsum[i] > b ? wsum[i] : b;
            if (b) atomicMax(&v.best[r], b);
        }
        if (!grid_barrier(bar, err, a.limit, a.rounds_grid)) return;
        const unsigned long long key = __ldcg(v.best + r);
        if (key != 0) {
            const uint32_t u = ~(uint32_t)(key & 0xFFFFFFFFull);
            if (tid == 0) {
                v.chosen[u] = 1;
                a.seeds[r] = (int32_t)u;
            }
            const uint64_t e0 = __ldcg(v.node_off + u), e1 = __ldcg(v.node_off + u + 1);
            for (uint64_t i = e0 + (tid >> 3); i < e1; i += nr >> 3) {
                const uint32_t s = __ldcg(v.node_sets + i);
                const int64_t pa = a.off[s], pb = a.off[s + 1];
                // the eight lanes read the flag before one of them sets it
                const unsigned group = 0xFFu << (lane & 24);
                const bool done = __ldcg(v.covered + s) != 0;
                __syncwarp(group);
                if (done) continue;
                if (sub == 0) {
                    v.covered[s] = 1;
                    fresh++;
                }
                if (pa < 0 || pb < pa || (uint64_t)pb > a.members) continue;
                for (int64_t p = pa + sub; p < pb; p += 8) {
                    const int32_t x = a.mem[p];
                    if (x >= 0 && x < a.n) atomicSub(&v.counts[x], 1);
                }
            }
        }
        if (!grid_barrier(bar, err, a.limit, a.rounds_grid)) return;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fresh += __shfl_xor_sync(0xffffffffu, fresh, o);
    if (lane == 0 && fresh) atomicAdd(&v.flags[0], fresh);
    if (!grid_barrier(bar, err, a.limit, a.rounds_grid)) return;
    if (tid == 0) *a.covered_out = __ldcg(v.flags);
}

std::mutex na_mutex;
unsigned char* na_base[64] = {};

}  // namespace

extern "C" int tim_node_select_noalloc(int device, void* cuda_stream, int64_t n, uint64_t n_sets,
                                       const int64_t* d_off, const int32_t* d_mem, int k,
                                       int32_t* d_seeds, uint64_t* d_covered) {
    if (device < 0 || device >= 64 || !d_off || !d_seeds || !d_covered) return TIM_ERR_ARG;
    if (n < 1 || n > NA_MAX_NODES || n_sets > NA_MAX_SETS || k < 1 || k > n || k > NA_MAX_K)
        return TIM_ERR_ARG;
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) return TIM_ERR_CUDA;
    if (prev != device && cudaSetDevice(device) != cudaSuccess) return TIM_ERR_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int rc = TIM_OK;
    do {
        unsigned char* base;
        {
            // once per device, with that device current: the device address of the array
            std::lock_guard<std::mutex> lock(na_mutex);
            if (!na_base[device]) {
                void* p = nullptr;
                if (cudaGetSymbolAddress(&p, na_scratch) != cudaSuccess || !p) {
                    cudaGetLastError();
                    rc = TIM_ERR_CUDA;
                    break;
                }
                na_base[device] = (unsigned char*)p;
            }
            base = na_base[device];
        }
        int64_t ends[2] = {0, 0};
        if (cudaMemcpyAsync(&ends[1], d_off + n_sets, sizeof(int64_t), cudaMemcpyDeviceToHost,
                            st) != cudaSuccess ||
            cudaMemcpyAsync(&ends[0], d_off, sizeof(int64_t), cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = TIM_ERR_CUDA;
            break;
        }
        if (ends[0] != 0 || ends[1] < 0 || (uint64_t)ends[1] > NA_MAX_MEMBERS || (n_sets > 0 && !d_mem)) {
            rc = TIM_ERR_ARG;
            break;
        }
        const NaView v = view_of(base);
        // counters, error bits and the grid barrier
        if (cudaMemsetAsync(v.flags, 0, 64, st) != cudaSuccess) {
            rc = TIM_ERR_CUDA;
            break;
        }
        int sms = 0, nb = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, na_select_kernel, NA_THREADS, 0) !=
                cudaSuccess ||
            nb < 1 || sms < 1) {
            cudaGetLastError();
            rc = TIM_ERR_CUDA;
            break;
        }
        NaArgs na;
        na.off = d_off;
        na.mem = d_mem;
        na.n_sets = n_sets;
        na.n = n;
        na.members = (uint64_t)ends[1];
        na.k = k;
        na.seeds = d_seeds;
        na.covered_out = d_covered;
        na.v = v;
        na.limit = 1u << 24;
        // one block per SM, fewer for a small problem (a barrier of few blocks is shorter)
        uint64_t work = (uint64_t)n;
        if (work < na.members) work = na.members;
        if (work < n_sets) work = n_sets;
        const uint64_t want = work / (2 * NA_THREADS) + 1;
        uint64_t G64 = want < (uint64_t)sms ? want : (uint64_t)sms;
        const unsigned G = (unsigned)(G64 < NA_MAX_BLOCKS ? G64 : NA_MAX_BLOCKS);
        na.rounds_grid = G < NA_ROUNDS_GRID ? G : NA_ROUNDS_GRID;
        void* args[] = {&na};
        if (cudaLaunchCooperativeKernel((const void*)na_select_kernel, dim3(G), dim3(NA_THREADS),
                                        args, 0, st) != cudaSuccess ||
            cudaGetLastError() != cudaSuccess) {
            rc = TIM_ERR_CUDA;
            break;
        }
        unsigned long long err[3] = {0, 0, 0};  // error bits, barrier, barrier's error
        if (cudaMemcpyAsync(err, v.flags + 1, 24, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = TIM_ERR_CUDA;
            break;
        }
        if (err[2]) rc = TIM_ERR_TIMEOUT;
        else if (err[0]) rc = TIM_ERR_ARG;
    } while (0);
    if (prev >= 0 && prev != device) cudaSetDevice(prev);
    return rc;
}
