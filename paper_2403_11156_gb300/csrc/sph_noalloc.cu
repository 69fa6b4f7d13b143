// sph_noalloc.cu -- grid order of a point set without any memory allocation.
//
// Some callers cannot let a library allocate device memory: code that enqueues work while
// another component is capturing a CUDA graph (cudaMalloc is not permitted inside such a
// capture), host applications such as rendering or game engines and plugins that own the
// GPU's memory budget and forbid libraries from allocating, and real-time loops in which
// an allocation's latency or a possible out-of-memory failure is not acceptable.  For them
// sph_grid_order_noalloc runs the same counting sort as the per-step neighbour search
// (cell keys, histogram, prefix sum, scatter, rank by index, with the crowded cells in order by a
// bitmap each) with its scratch in one file-scope static device array of fixed size, which
// every GPU that loads the library holds until the process exits.
#include "sph.h"
#include "sph_blocksort.cuh"
#include "sph_internal.cuh"
#include "sph_sweep.cuh"

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <mutex>

using namespace sph;

namespace {

constexpr int64_t kMaxPoints = SPH_NOALLOC_MAX_POINTS;
constexpr int64_t kMaxCells = SPH_NOALLOC_MAX_CELLS;
constexpr int kOrderBlocks = 152;   // at most one block per SM

// Byte offsets of the scratch regions (each a multiple of 256).
constexpr size_t kOffCount = 0;                                          // u32 [kMaxCells]
constexpr size_t kOffStart = kOffCount + 4 * kMaxCells;                  // u32 [kMaxCells + 1]
constexpr size_t kOffKey = kOffStart + ((4 * (kMaxCells + 1) + 255) / 256) * 256;  // u32 [kMaxPoints]
constexpr size_t kOffSlot = kOffKey + 4 * kMaxPoints;                    // u32 [kMaxPoints]
constexpr size_t kOffSid = kOffSlot + 4 * kMaxPoints;                    // u32 [kMaxPoints]
constexpr size_t kOffCell = kOffSid + 4 * kMaxPoints;                    // u32 [kMaxPoints]
constexpr size_t kOffSums = kOffCell + 4 * kMaxPoints;                    // u32 [kOrderBlocks]
constexpr size_t kOffBar = kOffSums + ((4 * kOrderBlocks + 255) / 256) * 256;  // u64, see OrderBarrier
constexpr size_t kOffCtl = kOffBar + 256;                                // Control
constexpr int64_t kMaxLarge = kMaxPoints / (kRankSmall + 1) + 1;
constexpr size_t kOffLarge = kOffCtl + ((sizeof(Control) + 255) / 256) * 256;  // u32 [kMaxLarge]
constexpr size_t kScratchBytes = kOffLarge + ((4 * kMaxLarge + 255) / 256) * 256;

static __device__ __align__(256) unsigned char g_grid_scratch[kScratchBytes];

struct View {
    uint32_t *count, *start, *key, *slot, *sid, *cell;
    uint32_t *sums;
    uint64_t *bar;
    Control *ctl;
    uint32_t *large;
};

View carve(unsigned char *base)
{
    View v;
    v.count = reinterpret_cast<uint32_t *>(base + kOffCount);
    v.start = reinterpret_cast<uint32_t *>(base + kOffStart);
    v.key = reinterpret_cast<uint32_t *>(base + kOffKey);
    v.slot = reinterpret_cast<uint32_t *>(base + kOffSlot);
    v.sid = reinterpret_cast<uint32_t *>(base + kOffSid);
    v.cell = reinterpret_cast<uint32_t *>(base + kOffCell);
    v.sums = reinterpret_cast<uint32_t *>(base + kOffSums);
    v.bar = reinterpret_cast<uint64_t *>(base + kOffBar);
    v.ctl = reinterpret_cast<Control *>(base + kOffCtl);
    v.large = reinterpret_cast<uint32_t *>(base + kOffLarge);
    return v;
}

struct Grid {
    float origin[3], cell;
    int32_t dims[3];
};

// Exclusive sum over the block's threads of one value each, and the total.
__device__ uint32_t block_scan(uint32_t v, uint32_t &total)
{
    __shared__ uint32_t s_warp[kLargeThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();   // the previous call's reads are done
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    const uint32_t w = s_warp[lane];
    uint32_t before = lane < warp ? w : 0u, all = w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    total = all;
    return before + x - v;
}

__device__ __forceinline__ uint32_t key_of(const Grid &g, const float *__restrict__ x, int64_t i)
{
    const int32_t ix = cell_coord(x[3 * i + 0], g.origin[0], g.cell, g.dims[0]);
    const int32_t iy = cell_coord(x[3 * i + 1], g.origin[1], g.cell, g.dims[1]);
    const int32_t iz = cell_coord(x[3 * i + 2], g.origin[2], g.cell, g.dims[2]);
    return (uint32_t)ix + (uint32_t)g.dims[0] * ((uint32_t)iy + (uint32_t)g.dims[1] * (uint32_t)iz);
}

// A crowded cell's indices sid[b..e), each below n and there once, in ascending order to order[b..e):
// an index's place is the number of bits below its own in a bitmap of the members.  Linear in the
// members and n / 32 words whatever their number; the radix sort of the step's crowded cells takes
// four passes of several barriers, 5 us for a cell of 65 and 2,110 for one of 262,000.
// By the whole block (every thread calls it).
__device__ void order_crowd(const uint32_t *sid, uint32_t b, uint32_t e, uint32_t n, int32_t *order)
{
    __shared__ __align__(16) uint32_t s_map[kMaxPoints / 32];
    __shared__ uint32_t s_before[kLargeThreads];   // bits before each 256
    static_assert(kMaxPoints == 256 * kLargeThreads, "eight words a thread");
    uint4 *mine = reinterpret_cast<uint4 *>(s_map) + 2 * threadIdx.x;
    mine[0] = mine[1] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    for (uint32_t t = b + threadIdx.x; t < e; t += kLargeThreads) {
        const uint32_t i = sid[t];
        if (i < n) atomicOr(&s_map[i >> 5], 1u << (i & 31u));
    }
    __syncthreads();
    const uint4 p = mine[0], q = mine[1];
    uint32_t total;
    s_before[threadIdx.x] = block_scan(__popc(p.x) + __popc(p.y) + __popc(p.z) + __popc(p.w) + __popc(q.x) + __popc(q.y) +
                                           __popc(q.z) + __popc(q.w), total);
    __syncthreads();
    for (uint32_t t = b + threadIdx.x; t < e; t += kLargeThreads) {
        const uint32_t i = sid[t];
        if (i >= n) continue;
        uint32_t at = b + s_before[i >> 8] + __popc(s_map[i >> 5] & ((1u << (i & 31u)) - 1u));
        for (uint32_t w = (i >> 8) * 8u; w < i >> 5; ++w) at += __popc(s_map[w]);
        if (at < e) order[at] = (int32_t)i;
    }
    __syncthreads();
}

// The same by one warp, for indices below 8,192, with 256 words of its own and as many counts.
constexpr int kWarpMap = 256;
__device__ void order_crowd_warp(const uint32_t *sid, uint32_t b, uint32_t e, uint32_t *map, uint16_t *before, int32_t *order)
{
    const int lane = threadIdx.x & 31;
    uint4 *mine = reinterpret_cast<uint4 *>(map) + 2 * lane;
    mine[0] = mine[1] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    for (uint32_t t = b + lane; t < e; t += 32u) atomicOr(&map[sid[t] >> 5], 1u << (sid[t] & 31u));
    __syncwarp();
    const uint4 p = mine[0], q = mine[1];
    const uint32_t w[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
    uint32_t sum = 0u, x;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += __popc(w[k]);
    x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    x -= sum;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        before[8 * lane + k] = (uint16_t)x;
        x += __popc(w[k]);
    }
    __syncwarp();
    for (uint32_t t = b + lane; t < e; t += 32u) {
        const uint32_t i = sid[t];
        order[b + before[i >> 5] + __popc(map[i >> 5] & ((1u << (i & 31u)) - 1u))] = (int32_t)i;
    }
    __syncwarp();
}

// The barrier over the blocks of a call, on a word that no call resets: a captured call is replayed
// with the arguments of its capture and cannot be given a fresh one, and a memset before the
// launch takes 4 us.  High half: arrivals.  A barrier's sum to kArrivals whatever
// the grid (block 0 makes up the difference), so that every block knows from the value it met
// which barrier it is in.  Low half: blocks that gave up a bounded wait; a change since a block's
// start ends its waits (the blocks of a cooperative launch start together).
// A block of any call leaves exactly kBarriers barriers' arrivals behind (those that it did not
// come to are added as it leaves), so the word is whole again after calls that gave up or overlapped.
struct OrderBarrier {
    static constexpr uint32_t kArrivals = 1u << 16;
    static constexpr int kBarriers = 7;   // the most that a call meets
    uint64_t *word;
    int32_t *error;
    uint32_t fails;
    int left = kBarriers;
    __device__ OrderBarrier(uint64_t *w, int32_t *e) : word(w), error(e), fails((uint32_t)*reinterpret_cast<volatile uint64_t *>(w)) {}
    __device__ static uint64_t share() { return blockIdx.x == 0 ? kArrivals - (gridDim.x - 1u) : 1u; }
    __device__ void leave(bool gave_up)
    {
        if (threadIdx.x == 0 && left > 0) atomicAdd(reinterpret_cast<unsigned long long *>(word), (unsigned long long)((share() * left << 32) + (gave_up ? 1u : 0u)));
        left = 0;
    }
    // Whether all blocks came; if not, the block has left.
    __device__ bool wait()
    {
        bool ok = true;
        __syncthreads();
        --left;
        if (threadIdx.x == 0) {
            const uint64_t add = share() << 32;
            uint64_t met;
            asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], %2;" : "=l"(met) : "l"(word), "l"(add) : "memory");
            const uint32_t base = (uint32_t)(met >> 32) & ~(kArrivals - 1u);
            auto open = [&](uint64_t w) { return (uint32_t)(w >> 32) - base >= kArrivals; };
            auto whole = [&](uint64_t w) { return (uint32_t)w == fails; };
            uint64_t now = met + add;
            for (uint32_t spins = 0; !open(now) && whole(now) && spins < kBarrierSpins; ++spins)
                asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(now) : "l"(word) : "memory");
            ok = open(now) && whole(now);
            if (!ok) atomicExch(error, 5);
        }
        ok = __syncthreads_and(ok);
        if (!ok) leave(true);
        return ok;
    }
};

// The whole order in one cooperative launch: keys and histogram, prefix sum (each block sums its
// share of the cells, then adds the shares before it), scatter, rank inside the cell by index or,
// for the crowded cells, which the prefix sum queues, by bitmap; four barriers.  The histogram
// is zero between calls: the prefix sum clears what it has read.  Its total has to be n; where an
// earlier call left something in it, it is cleared and filled once more.  Calls that overlap race
// on the scratch: what is read from it is checked (places below n, the queue's length) before it
// is used as an index.
// As six launches it was bound by them: 262,143 points 39.0 -> 22.5 us (24.6 with the barrier's
// count and generation in two words, 28.7 with a memset that cleared both and the histogram before
// every call); 100,000 points in 1,000 crowded cells 77 -> 40.
__global__ void __launch_bounds__(kLargeThreads) k_na_order(View v, Grid g, const float *__restrict__ x, int64_t n,
                                                            int64_t ncell, uint32_t *keys_out, int32_t *order)
{
    Control *ctl = v.ctl;
    OrderBarrier bar(v.bar, &ctl->error);
    const int64_t first = (int64_t)blockIdx.x * kLargeThreads + threadIdx.x, stride = (int64_t)gridDim.x * kLargeThreads;
    if (first == 0) {
        ctl->error = 0;   // (no block can have given up yet)
        ctl->nlarge[0] = 0;
    }
    // cells [c0, c1) are this block's share, a multiple of the block's width
    const int64_t share = ((ncell + gridDim.x - 1) / gridDim.x + kLargeThreads - 1) / kLargeThreads * kLargeThreads;
    const int64_t c0 = (int64_t)blockIdx.x * share, c1 = min(c0 + share, ncell);
    __shared__ uint32_t s_run;
    uint32_t total;
    for (int attempt = 0;; ++attempt) {
        for (int64_t i = first; i < n; i += stride) {
            const uint32_t key = key_of(g, x, i);
            v.key[i] = key;
            v.slot[i] = atomicAdd(&v.count[key], 1u);
            if (keys_out) keys_out[i] = key;
        }
        if (!bar.wait()) return;
        uint32_t sum = 0u;
        for (int64_t c = c0 + threadIdx.x; c < c1; c += kLargeThreads) sum += v.count[c];
        block_scan(sum, total);
        if (threadIdx.x == 0) v.sums[blockIdx.x] = total;
        if (!bar.wait()) return;
        const uint32_t before_me = block_scan(threadIdx.x < gridDim.x ? v.sums[threadIdx.x] : 0u, total);
        if (threadIdx.x == blockIdx.x) s_run = before_me;   // shares before this one
        if (total == (uint32_t)n) break;
        // the histogram was not this call's alone (every block alike)
        for (int64_t c = c0 + threadIdx.x; c < c1; c += kLargeThreads) v.count[c] = 0u;
        if (attempt > 0) {   // not a leftover: another call writes it now
            if (threadIdx.x == 0) atomicExch(&ctl->error, 7);
            bar.leave(false);
            return;
        }
        if (!bar.wait()) return;
    }
    {
        __syncthreads();
        uint32_t run = s_run;
        for (int64_t c = c0; c < c1; c += kLargeThreads) {
            const int64_t at = c + threadIdx.x;
            const uint32_t k = at < c1 ? v.count[at] : 0u;
            const uint32_t before = block_scan(k, total);
            if (at < c1) {
                v.start[at] = run + before;
                v.count[at] = 0u;
                if (k > kRankSmall) {
                    const int q = atomicAdd(&ctl->nlarge[0], 1);
                    if (q < kMaxLarge) v.large[q] = (uint32_t)at;
                }
            }
            run += total;
        }
        if (c1 == ncell && c0 < c1 && threadIdx.x == 0) v.start[ncell] = run;
    }
    if (!bar.wait()) return;
    for (int64_t i = first; i < n; i += stride) {
        const uint32_t key = v.key[i], s = v.start[key] + v.slot[i];
        if (s >= (uint32_t)n) continue;
        v.sid[s] = (uint32_t)i;
        v.cell[s] = key;
    }
    if (!bar.wait()) return;
    for (int64_t s = first; s < n; s += stride) {
        const uint32_t c = v.cell[s], b = v.start[c], e = min(v.start[c + 1], (uint32_t)n);
        if (e - b > kRankSmall) continue;   // queued
        const uint32_t my = v.sid[s];
        uint32_t rank = 0;
        for (uint32_t t = b; t < e; ++t) rank += (v.sid[t] < my) ? 1u : 0u;
        if (b + rank < e) order[b + rank] = (int32_t)my;
    }
    // the queued cells, one block per cell at a time
    __shared__ uint32_t s_seg[2];
    const int nq = min(*reinterpret_cast<volatile int32_t *>(&ctl->nlarge[0]), (int)kMaxLarge);
    for (int q = blockIdx.x; q < nq; q += gridDim.x) {
        if (threadIdx.x == 0) {
            const uint32_t c = v.large[q];
            s_seg[0] = v.start[c];
            s_seg[1] = min(v.start[c + 1], (uint32_t)n);
        }
        __syncthreads();
        order_crowd(v.sid, s_seg[0], s_seg[1], (uint32_t)n, order);
    }
    bar.leave(false);
}

// Few points in few cells: the same in one block, histogram, starts and order in shared memory, a
// warp for each crowded cell.  3,001 points in 10,648 cells: 28.7 us as six launches, 8.2 us here
// (a barrier over blocks costs more than this range's work); 8,192 in 21,952 cells 15.5 us, as the
// cooperative kernel's 15.6, in 64 crowded cells 13.0 against 19.5, with 126 cells of 65 17.2 (35.8
// as six launches, 610 with the block's radix sort for one cell after the other).
constexpr int64_t kOneBlockPoints = 8 * kLargeThreads, kOneBlockCells = 24 * kLargeThreads;
static_assert(kOneBlockPoints == 32 * kWarpMap, "a bit for each point");
constexpr int kOneBlockMaps = kLargeThreads / 32 * (kWarpMap + kWarpMap / 2);   // words
__global__ void __launch_bounds__(kLargeThreads) k_na_order_one(Control *ctl, Grid g, const float *__restrict__ x, int n, int ncell,
                                                                uint32_t *keys_out, int32_t *order)
{
    extern __shared__ __align__(16) uint32_t sm[];
    // a bitmap and its counts for each warp, the cells' starts, the order inside them not yet fixed
    uint32_t *map = sm + (threadIdx.x >> 5) * kWarpMap;
    uint16_t *before = reinterpret_cast<uint16_t *>(sm + kLargeThreads / 32 * kWarpMap) + (threadIdx.x >> 5) * kWarpMap;
    uint32_t *start = sm + kOneBlockMaps, *sid = start + ncell + 1;
    __shared__ int s_large;
    __shared__ uint32_t s_cells[kOneBlockPoints / (kRankSmall + 1)];   // the crowded ones
    constexpr int kOwn = (int)(kOneBlockPoints / kLargeThreads);
    const int t = threadIdx.x;
    for (int c = t; c < ncell; c += kLargeThreads) start[c] = 0u;
    if (t == 0) {
        s_large = 0;
        ctl->error = 0;
    }
    __syncthreads();
    uint32_t key[kOwn], at[kOwn];
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
        const int i = k * kLargeThreads + t;
        if (i < n) {
            key[k] = key_of(g, x, i);
            at[k] = atomicAdd(&start[key[k]], 1u);
            if (keys_out) keys_out[i] = key[k];
        }
    }
    __syncthreads();
    // a thread's consecutive cells, an odd number of them (no bank conflicts)
    const int per = ((ncell + kLargeThreads - 1) / kLargeThreads) | 1;
    const int c0 = min(t * per, ncell), c1 = min(c0 + per, ncell);
    uint32_t sum = 0u, total;
    for (int c = c0; c < c1; ++c) sum += start[c];
    uint32_t run = block_scan(sum, total);
    for (int c = c0; c < c1; ++c) {
        const uint32_t k = start[c];
        start[c] = run;
        run += k;
    }
    if (t == 0) start[ncell] = (uint32_t)n;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
        const int i = k * kLargeThreads + t;
        if (i < n) sid[start[key[k]] + at[k]] = (uint32_t)i;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
        const int i = k * kLargeThreads + t;
        if (i >= n) continue;
        const uint32_t b = start[key[k]], e = start[key[k] + 1];
        if (e - b > kRankSmall) {
            if (at[k] == 0u) s_cells[atomicAdd(&s_large, 1)] = key[k];
            continue;
        }
        uint32_t rank = 0;
        for (uint32_t q = b; q < e; ++q) rank += (sid[q] < (uint32_t)i) ? 1u : 0u;
        order[b + rank] = i;
    }
    __syncthreads();
    for (int q = t >> 5; q < s_large; q += kLargeThreads / 32) {
        const uint32_t c = s_cells[q];
        order_crowd_warp(sid, start[c], start[c + 1], map, before, order);
    }
}

std::mutex g_mu;
unsigned char *g_base[256] = {};

}  // namespace

extern "C" sph_status sph_grid_order_noalloc(const float *x, int64_t n, const float *domain_min,
                                             const float *domain_max, float cell_size, int32_t *order,
                                             uint32_t *keys, void *stream)
{
    if (n < 0 || n > kMaxPoints) return SPH_EINVAL;
    if (n > 0 && (!x || !order)) return SPH_EINVAL;
    if (!domain_min || !domain_max || !(cell_size > 0.0f) || !std::isfinite(cell_size)) return SPH_EINVAL;
    Grid g;
    g.cell = cell_size;
    int64_t ncell = 1;
    for (int a = 0; a < 3; ++a) {
        if (!std::isfinite(domain_min[a]) || !std::isfinite(domain_max[a]) || !(domain_max[a] > domain_min[a]))
            return SPH_EINVAL;
        g.origin[a] = domain_min[a] - cell_size;
        float ext = (domain_max[a] - domain_min[a]) / cell_size;
        if (!(ext < 1e7f)) return SPH_EINVAL;
        g.dims[a] = (int32_t)std::ceil(ext) + 2;
        ncell *= g.dims[a];
        if (ncell > kMaxCells) return SPH_EINVAL;
    }
    if (n == 0) return SPH_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return SPH_ECUDA;
    unsigned char *base;
    {
        // once per device, with that device current: the device address of the array
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_base[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_grid_scratch) != cudaSuccess || !p) return SPH_ECUDA;
            g_base[dev] = static_cast<unsigned char *>(p);
        }
        base = g_base[dev];
    }
    View v = carve(base);
    cudaStream_t s = (cudaStream_t)stream;
    if (n <= kOneBlockPoints && ncell <= kOneBlockCells) {
        const size_t bytes = sizeof(uint32_t) * (size_t)(kOneBlockMaps + ncell + 1 + n);
        if (cudaFuncSetAttribute(k_na_order_one, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(uint32_t) * (kOneBlockMaps + kOneBlockCells + 1 + kOneBlockPoints))) != cudaSuccess)
            return SPH_ECUDA;
        k_na_order_one<<<1, kLargeThreads, bytes, s>>>(v.ctl, g, x, (int)n, (int)ncell, keys, order);
        return cudaGetLastError() == cudaSuccess ? SPH_OK : SPH_ECUDA;
    }
    // a block of 1024 threads per 1024 points or cells, at most one per SM
    int nsm = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1) return SPH_ECUDA;
    const int64_t want = (std::max(n, ncell) + kLargeThreads - 1) / kLargeThreads;
    const int blocks = (int)std::min<int64_t>(want, std::min(nsm, kOrderBlocks));
    void *args[] = {&v, &g, (void *)&x, &n, &ncell, &keys, &order};
    const cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(&k_na_order), dim3((unsigned)blocks),
                                                      dim3(kLargeThreads), args, 0, s);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? SPH_OK : SPH_ECUDA;
}

extern "C" sph_status sph_grid_order_noalloc_status(void *stream)
{
    // a call that found its histogram disturbed or gave up a bounded wait records it in the
    // scratch's error word, which each call clears: read it back once the stream's work is done
    // (a copy from the symbol into a host integer, nothing allocated)
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return SPH_ECUDA;
    int32_t err = 0;
    const size_t off = kOffCtl + offsetof(Control, error);
    if (cudaMemcpyFromSymbol(&err, g_grid_scratch, sizeof(err), off, cudaMemcpyDeviceToHost) != cudaSuccess)
        return SPH_ECUDA;
    return err != 0 ? SPH_ETIMEOUT : SPH_OK;
}
