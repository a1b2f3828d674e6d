// Ragged batches: many segments, each with its own kmax (e.g. the shell
// quartets of an ERI batch, kmax_s = la+lb+lc+ld).  Two ways to cut the work: flat
// tiles that a persistent kernel takes from a counter (a 256-byte workspace, the
// no-alloc entry point, some plans, and where a tile table does not fit), or a table
// of one-segment tiles sorted by kmax (larger workspaces, most plans; further below).
//
// Flat tiles: the concatenated argument array x[0, total) is cut into
// flat tiles of blockDim*XPT arguments; resident CTAs take tiles from a
// global atomic counter (the only scratch memory) until none are left, which
// balances the very uneven per-argument cost of different kmax.  A thread
// finds the segment of each of its arguments by binary search over seg_off
// restricted to the tile's segment range, and evaluates it with exactly the
// code boys_eval uses for that segment's kmax (bitwise-identical results).
// A warp whose lanes straddle segments with different kmax loops over the
// distinct values (rare: only warps that cross a segment boundary).
//
// Output of segment s (length len_s = seg_off[s+1] - seg_off[s]) is its own
// order-major block: F_k(x[seg_off[s] + j]) at out[out_off[s] + k*len_s + j].
#include <algorithm>
#include <array>
#include <chrono>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <unordered_map>
#include <utility>
#include <vector>

#include "boys_internal.h"
#include "boys_region.cuh"

namespace boys {
namespace ragged {
constexpr int kMaxBlock = 256;
// Resident blocks of kMaxBlock threads per SM: 8 caps the kernels at 32 registers.
// The tile kernel spills one register there; the persistent one 8 (two arguments a
// thread: 15), its out-of-line evaluations one or two from order 6 on, and it is
// the fastest all the same (4096 segments at mean kmax 4.07, 3.5e7 arguments:
// 560 us with 8, 612 with 6, 742 with 4).
#ifndef BOYS_RAGGED_MIN_BLOCKS
#define BOYS_RAGGED_MIN_BLOCKS 8
#endif

struct Workspace {
    unsigned long long next_tile;  // work counter, zeroed before every launch
    unsigned long long error;      // nonzero: a segment had kmax outside [0, 32]
};
static_assert(sizeof(Workspace) <= 256, "workspace fits its published size");

// One argument's orders 0..K to dst[k * row]: the stored mode's evaluation (same bits).
template <int K>
__device__ __noinline__ void eval_store(double xv, double* __restrict__ dst, int64_t row) {
    region::eval_store<K, true>(xv, dst, row);
}

__device__ __forceinline__ void dispatch(int k, double xv, double* dst, int64_t row) {
#define BOYS_RAGGED_CASE(K) \
    case K: eval_store<K>(xv, dst, row); break;
    switch (k) {
        BOYS_RAGGED_CASE(0) BOYS_RAGGED_CASE(1) BOYS_RAGGED_CASE(2) BOYS_RAGGED_CASE(3)
        BOYS_RAGGED_CASE(4) BOYS_RAGGED_CASE(5) BOYS_RAGGED_CASE(6) BOYS_RAGGED_CASE(7)
        BOYS_RAGGED_CASE(8) BOYS_RAGGED_CASE(9) BOYS_RAGGED_CASE(10) BOYS_RAGGED_CASE(11)
        BOYS_RAGGED_CASE(12) BOYS_RAGGED_CASE(13) BOYS_RAGGED_CASE(14) BOYS_RAGGED_CASE(15)
        BOYS_RAGGED_CASE(16) BOYS_RAGGED_CASE(17) BOYS_RAGGED_CASE(18) BOYS_RAGGED_CASE(19)
        BOYS_RAGGED_CASE(20) BOYS_RAGGED_CASE(21) BOYS_RAGGED_CASE(22) BOYS_RAGGED_CASE(23)
        BOYS_RAGGED_CASE(24) BOYS_RAGGED_CASE(25) BOYS_RAGGED_CASE(26) BOYS_RAGGED_CASE(27)
        BOYS_RAGGED_CASE(28) BOYS_RAGGED_CASE(29) BOYS_RAGGED_CASE(30) BOYS_RAGGED_CASE(31)
        BOYS_RAGGED_CASE(32)
        default: break;
    }
#undef BOYS_RAGGED_CASE
}

// Largest s in [lo, hi] with seg_off[s] <= i (seg_off non-decreasing; lo if
// there is none): a 32-way search by a whole warp.  Each round the lanes
// probe 32 evenly spaced offsets and a ballot keeps the interval between the
// last probe at or below i and the next one, so 4096 segments take three
// dependent loads instead of twelve.  All 32 lanes must call it together;
// every lane returns the result.
__device__ __forceinline__ int find_segment_warp(const int64_t* __restrict__ seg_off, int lo, int hi, int64_t i) {
    const int lane = threadIdx.x & 31;
    while (hi > lo) {
        const int span = hi - lo + 1;
        const int step = (span + 31) / 32;
        const int probe = lo + lane * step;
        const bool le = probe <= hi && __ldg(seg_off + probe) <= i;
        const unsigned m = __ballot_sync(0xffffffffu, le);
        const int last = m ? 31 - __clz((int)m) : 0;  // none at or below i: stay at lo, as the binary search does
        lo = lo + last * step;
        hi = min(hi, lo + step - 1);
        if (step == 1) break;
    }
    return lo;
}

// Largest s in [lo, hi] with seg_off[s] <= i (seg_off non-decreasing).
__device__ __forceinline__ int find_segment(const int64_t* __restrict__ seg_off, int lo, int hi, int64_t i) {
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(seg_off + mid) <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <int XPT>
__global__ void __launch_bounds__(kMaxBlock, BOYS_RAGGED_MIN_BLOCKS) k_ragged(const double* __restrict__ x,
                                                      const int64_t* __restrict__ seg_off,
                                                      const int32_t* __restrict__ seg_kmax, int nseg,
                                                      double* __restrict__ out,
                                                      const int64_t* __restrict__ out_off,
                                                      Workspace* __restrict__ ws,
                                                      const unsigned* __restrict__ gate) {
    if (gate && *gate == 0) return;  // a fallback launch that is not needed
    __shared__ long long s_tile;
    __shared__ int s_seg_lo, s_seg_hi;
    const int64_t total = __ldg(seg_off + nseg);
    const int64_t per_tile = (int64_t)blockDim.x * XPT;
    const int64_t ntiles = (total + per_tile - 1) / per_tile;
    const unsigned lane = threadIdx.x & 31;
    for (;;) {
        if (threadIdx.x < 32) {  // warp 0 takes the next tile and finds its segments
            long long t = 0;
            if (threadIdx.x == 0) t = (long long)atomicAdd(&ws->next_tile, 1ULL);
            t = __shfl_sync(0xffffffffu, t, 0);
            if (threadIdx.x == 0) s_tile = t;
            if (t < ntiles) {
                const int64_t first = t * per_tile;
                const int64_t last = min(first + per_tile, total) - 1;
                const int lo = find_segment_warp(seg_off, 0, nseg - 1, first);
                const int hi = find_segment_warp(seg_off, lo, nseg - 1, last);
                if (threadIdx.x == 0) {
                    s_seg_lo = lo;
                    s_seg_hi = hi;
                }
            }
        }
        __syncthreads();
        const long long t = s_tile;
        const int seg_lo = s_seg_lo, seg_hi = s_seg_hi;
        __syncthreads();
        if (t >= ntiles) break;
        const int64_t base = t * per_tile;
#pragma unroll 1
        for (int j = 0; j < XPT; ++j) {
            const int64_t i = base + (int64_t)j * blockDim.x + threadIdx.x;
            bool valid = i < total;
            int km = 0;
            double xv = 0.0;
            double* dst = nullptr;
            int64_t row = 0;
            if (valid) {
                const int s = find_segment(seg_off, seg_lo, seg_hi, i);
                const int64_t s0 = __ldg(seg_off + s);
                row = __ldg(seg_off + s + 1) - s0;
                km = __ldg(seg_kmax + s);
                if (km < 0 || km > 32) {
                    atomicOr(&ws->error, 1ULL);
                    valid = false;
                } else {
                    xv = __ldcs(x + i);
                    dst = out + __ldg(out_off + s) + (i - s0);
                }
            }
            unsigned pending = __ballot_sync(0xffffffffu, valid);
            while (pending) {
                const int leader = __ffs(pending) - 1;
                const int k = __shfl_sync(0xffffffffu, km, leader);
                const bool mine = valid && km == k && ((pending >> lane) & 1u);
                if (mine) dispatch(k, xv, dst, row);
                pending &= ~__ballot_sync(0xffffffffu, mine);
            }
        }
    }
}

// ---------------------------------------------- kmax-grouped tiles
//
// The batch may instead be cut into tiles, each of up to blockDim consecutive
// arguments of one segment, in a table sorted by the segments' kmax: built on the
// host when a plan is created, or on the device at every plan-less call.  One
// launch walks the table, largest kmax first.  A tile's kmax is the same for the
// whole block, so the block takes one order's evaluation -- the stored mode's, same
// bits -- with no segment search and no loop over the kmax of a warp.  All orders
// fit in 32 registers but for one spill, so one kernel holds them all at full occupancy.  One kernel
// per kmax, as parallel graph branches of a plan or a chain of programmatic
// dependents without one, ran large batches as fast (plan: 4096 segments, 3.5e7
// arguments, 408 us either way) but paid for up to 33 launches (plan-less: 480 us
// against 422; 512 segments, 4.3e5 arguments: plan 20 us against 11, plan-less 78
// against 16, as fast as the persistent kernel).  The loop for irregular arguments is
// shared by the orders: a copy in each made the kernel's code larger (plan 432 us).

struct Tile {
    int32_t seg;    // segment index
    int32_t len;    // arguments in this tile (<= blockDim)
    int64_t start;  // first argument, relative to the segment
};
static_assert(sizeof(Tile) == 16, "tile table entries are 16 bytes");

// One tile: its arguments, one per thread.
template <int K>
__device__ __forceinline__ void group_tile(const double* __restrict__ x, const int64_t* __restrict__ seg_off,
                                           double* __restrict__ out, const int64_t* __restrict__ out_off,
                                           const Tile& tl) {
    if ((int)threadIdx.x < tl.len) {
        const int64_t s0 = __ldg(seg_off + tl.seg);
        const int64_t row = __ldg(seg_off + tl.seg + 1) - s0;
        const int64_t j = tl.start + threadIdx.x;
        region::eval_store<K, true>(__ldcs(x + s0 + j), out + __ldg(out_off + tl.seg) + j, row);
    }
}

constexpr int kGroupTile = 128;  // arguments per tile of a table built on the device

struct GroupHeader {
    Workspace ws;             // error word (the persistent kernel also uses next_tile)
    unsigned count[33];       // tiles per kmax
    unsigned cursor[33];      // of which are filled
    unsigned overflow;        // 1: the table does not fit, the persistent fallback runs
};
constexpr size_t kGroupHeaderBytes = 512;
static_assert(sizeof(GroupHeader) <= kGroupHeaderBytes, "group header fits its reserved bytes");

// The 33 counts summed up by a warp: lane k gets the first tile of order k + 1.
__device__ __forceinline__ unsigned group_ends(const GroupHeader* __restrict__ h, unsigned lane) {
    unsigned run = h->count[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, run, d);
        if (lane >= d) run += u;
    }
    return run;
}

__global__ void __launch_bounds__(kMaxBlock, BOYS_RAGGED_MIN_BLOCKS) k_group(
        const double* __restrict__ x, const int64_t* __restrict__ seg_off, double* __restrict__ out,
        const int64_t* __restrict__ out_off, const Tile* __restrict__ tiles, const GroupHeader* __restrict__ h) {
    if (h->overflow) return;
    const unsigned base = group_ends(h, threadIdx.x & 31);  // first tile of kmax lane + 1
    const unsigned total = __shfl_sync(0xffffffffu, base, 31) + h->count[32];
    for (unsigned i = blockIdx.x; i < total; i += gridDim.x) {
        const unsigned t = total - 1 - i;
        const int k = __popc(__ballot_sync(0xffffffffu, base <= t));
        const Tile tl = tiles[t];
#define BOYS_GROUP_CASE(K) \
    case K: group_tile<K>(x, seg_off, out, out_off, tl); break;
        switch (k) {
            BOYS_GROUP_CASE(0) BOYS_GROUP_CASE(1) BOYS_GROUP_CASE(2) BOYS_GROUP_CASE(3)
            BOYS_GROUP_CASE(4) BOYS_GROUP_CASE(5) BOYS_GROUP_CASE(6) BOYS_GROUP_CASE(7)
            BOYS_GROUP_CASE(8) BOYS_GROUP_CASE(9) BOYS_GROUP_CASE(10) BOYS_GROUP_CASE(11)
            BOYS_GROUP_CASE(12) BOYS_GROUP_CASE(13) BOYS_GROUP_CASE(14) BOYS_GROUP_CASE(15)
            BOYS_GROUP_CASE(16) BOYS_GROUP_CASE(17) BOYS_GROUP_CASE(18) BOYS_GROUP_CASE(19)
            BOYS_GROUP_CASE(20) BOYS_GROUP_CASE(21) BOYS_GROUP_CASE(22) BOYS_GROUP_CASE(23)
            BOYS_GROUP_CASE(24) BOYS_GROUP_CASE(25) BOYS_GROUP_CASE(26) BOYS_GROUP_CASE(27)
            BOYS_GROUP_CASE(28) BOYS_GROUP_CASE(29) BOYS_GROUP_CASE(30) BOYS_GROUP_CASE(31)
            BOYS_GROUP_CASE(32)
        }
#undef BOYS_GROUP_CASE
    }
}

// ------------------------------------ kmax-grouped tiles without a plan
//
// With a large enough workspace, boys_eval_ragged builds the table itself, on the
// device: a count of tiles per kmax, and a fill in which each segment takes a
// contiguous range of its group with one atomic and a warp writes it (the order of
// tiles inside a group varies, the values do not).  Every warp sums up the 33 counts
// for itself.  If the table
// would exceed the workspace's capacity, the tile kernel returns at once and a
// persistent launch, gated on that condition, evaluates the batch instead.

__device__ __forceinline__ bool bad_kmax(int k) { return k < 0 || k > 32; }

__global__ void k_group_count(const int64_t* __restrict__ seg_off, const int32_t* __restrict__ seg_kmax, int nseg,
                              GroupHeader* __restrict__ h) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nseg; s += gridDim.x * blockDim.x) {
        const int64_t len = __ldg(seg_off + s + 1) - __ldg(seg_off + s);
        const int k = __ldg(seg_kmax + s);
        if (len <= 0) continue;
        if (bad_kmax(k)) {
            atomicOr(&h->ws.error, 1ULL);
            continue;
        }
        atomicAdd(&h->count[k], (unsigned)((len + kGroupTile - 1) / kGroupTile));
    }
}

// A warp per segment: its tiles are written side by side.
__global__ void k_group_fill(const int64_t* __restrict__ seg_off, const int32_t* __restrict__ seg_kmax, int nseg,
                             GroupHeader* __restrict__ h, Tile* __restrict__ tiles, unsigned long long capacity) {
    const unsigned lane = threadIdx.x & 31, ends = group_ends(h, lane);
    if ((unsigned long long)__shfl_sync(0xffffffffu, ends, 31) + h->count[32] > capacity) {
        if (blockIdx.x == 0 && threadIdx.x == 0) h->overflow = 1;
        return;
    }
    const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; s < nseg; s += warps) {
        const int64_t len = __ldg(seg_off + s + 1) - __ldg(seg_off + s);
        const int k = __ldg(seg_kmax + s);
        if (len <= 0 || bad_kmax(k)) continue;
        const unsigned n = (unsigned)((len + kGroupTile - 1) / kGroupTile);
        unsigned p = 0;
        if (lane == 0) p = atomicAdd(&h->cursor[k], n);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (k > 0) p += __shfl_sync(0xffffffffu, ends, k - 1);
        for (unsigned t = lane; t < n; t += 32) {
            const int64_t a = (int64_t)t * kGroupTile;
            tiles[p + t] = Tile{(int32_t)s, (int32_t)min((int64_t)kGroupTile, len - a), a};
        }
    }
}

using KernelFn = void (*)(const double*, const int64_t*, const int32_t*, int, double*, const int64_t*, Workspace*,
                          const unsigned*);

inline KernelFn kernel_for(int xpt) { return xpt == 2 ? &k_ragged<2> : &k_ragged<1>; }

struct Config {
    int block = 128;
    int xpt = 1;
    int waves = 1;  // resident CTAs per SM multiplier for the persistent grid;
                    // 0: kmax-grouped tiles (plans only; tile = block)
};

inline int grid_size(const Config& c) {
    const int per_sm = blocks_per_sm((const void*)kernel_for(c.xpt), c.block);
    return std::max(1, sm_count() * per_sm * c.waves);
}

boys_status check_args(const double* x, const int64_t* seg_off, const int32_t* seg_kmax, int32_t nseg,
                       double* out, const int64_t* out_off, const char* fn) {
    if (nseg < 0) return fail(BOYS_ERR_INVALID_ARG, "%s: nseg=%d < 0", fn, nseg);
    if (nseg == 0) return BOYS_OK;
    if (!x || !seg_off || !seg_kmax || !out || !out_off) return fail(BOYS_ERR_INVALID_ARG, "%s: NULL pointer", fn);
    if (!aligned(x, 8) || !aligned(out, 8) || !aligned(seg_off, 8) || !aligned(out_off, 8) || !aligned(seg_kmax, 4))
        return fail(BOYS_ERR_ALIGNMENT, "%s: pointer not aligned to its element size", fn);
    return BOYS_OK;
}

boys_status launch(const Config& c, const double* x, const int64_t* seg_off, const int32_t* seg_kmax, int32_t nseg,
                   double* out, const int64_t* out_off, Workspace* ws, cudaStream_t stream) {
    boys_status st = check_cuda(cudaMemsetAsync(ws, 0, sizeof(Workspace), stream), "ragged workspace reset");
    if (st != BOYS_OK) return st;
    kernel_for(c.xpt)<<<grid_size(c), c.block, 0, stream>>>(x, seg_off, seg_kmax, nseg, out, out_off, ws, nullptr);
    return check_cuda(cudaGetLastError(), "ragged launch");
}

// Blocks of the tile kernel for `tiles` tiles of `block` arguments: at most 16
// waves of resident ones, so that the block scheduler evens out tiles of different
// cost (4096 segments, 3.5e7 arguments: 408 us with 16 waves, 440 with 4, 467 with
// 1, 416 with 64).
inline unsigned group_grid(int64_t tiles, int block) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sm_count() * (2048 / block) * 16));
}

// The plan-less kmax-grouped batch on a workspace of `bytes` >= kGroupHeaderBytes
// + 16: reset the header, build the table on the device, walk it, then the
// persistent kernel gated on the table's overflow flag.
boys_status launch_grouped(const double* x, const int64_t* seg_off, const int32_t* seg_kmax, int32_t nseg, double* out,
                           const int64_t* out_off, void* workspace, size_t bytes, cudaStream_t stream) {
    GroupHeader* h = (GroupHeader*)workspace;
    Tile* tiles = (Tile*)((char*)workspace + kGroupHeaderBytes);
    const unsigned long long capacity = std::min<unsigned long long>((bytes - kGroupHeaderBytes) / sizeof(Tile),
                                                                     0xFFFFFFFFull);  // tile indices are 32-bit
    boys_status st = check_cuda(cudaMemsetAsync(h, 0, sizeof(GroupHeader), stream), "ragged group header reset");
    if (st != BOYS_OK) return st;
    const int sgrid = (int)std::min<int64_t>((nseg + 255) / 256, (int64_t)sm_count() * 4);
    k_group_count<<<sgrid, 256, 0, stream>>>(seg_off, seg_kmax, nseg, h);
    const int fgrid = (int)std::min<int64_t>(((int64_t)nseg * 32 + 255) / 256, (int64_t)sm_count() * 8);
    k_group_fill<<<fgrid, 256, 0, stream>>>(seg_off, seg_kmax, nseg, h, tiles, capacity);
    st = check_cuda(cudaGetLastError(), "ragged group table");
    if (st != BOYS_OK) return st;
    k_group<<<group_grid((int64_t)capacity, kGroupTile), kGroupTile, 0, stream>>>(x, seg_off, out, out_off, tiles, h);
    const Config c;
    kernel_for(c.xpt)<<<grid_size(c), c.block, 0, stream>>>(x, seg_off, seg_kmax, nseg, out, out_off, &h->ws, &h->overflow);
    return check_cuda(cudaGetLastError(), "ragged group launch");
}

// ------------------------------------------------------------- autotuning

const std::vector<Config>& candidates() {
    static const std::vector<Config> c = [] {
        std::vector<Config> v;
        for (int block : {64, 128, 256})
            for (int xpt : {1, 2})
                for (int waves : {1, 2}) v.push_back(Config{block, xpt, waves});
        for (int block : {128, 256}) v.push_back(Config{block, 1, 0});
        return v;
    }();
    return c;
}

// Part of the cache's keys: raised whenever a shape stands for other kernels than
// before, so that a stored choice among the former ones is made anew (2: waves = 0 is one
// launch over a table of tiles, 512 segments 27 to 11 us; it was a launch per kmax).
constexpr int kShapes = 2;

std::string device_key() {
    int dev = 0, drv = 0;
    cudaGetDevice(&dev);
    cudaDriverGetVersion(&drv);
    cudaDeviceProp p;
    if (cudaGetDeviceProperties(&p, dev) != cudaSuccess) return "unknown";
    char buf[512];
    snprintf(buf, sizeof(buf), "%.200s|sm%d%d|%dSM|drv%d|lib%d|shapes%d", p.name, p.major, p.minor, p.multiProcessorCount, drv,
             boys_version(), kShapes);
    for (char* q = buf; *q; ++q)
        if (*q == ' ') *q = '_';
    return buf;
}

struct TuneCache {
    std::mutex mu;
    std::unordered_map<std::string, Config> mem;
    bool loaded = false;

    static const char* path() { return getenv("BOYS_AUTOTUNE_CACHE"); }

    void load() {
        if (loaded) return;
        loaded = true;
        const char* p = path();
        if (!p) return;
        FILE* f = fopen(p, "r");
        if (!f) return;
        char key[512];
        Config c;
        while (fscanf(f, "%511s %d %d %d", key, &c.block, &c.xpt, &c.waves) == 4) mem[key] = c;
        fclose(f);
    }

    bool get(const std::string& k, Config* c) {
        std::lock_guard<std::mutex> lk(mu);
        load();
        auto it = mem.find(k);
        if (it == mem.end()) return false;
        *c = it->second;
        return true;
    }

    void put(const std::string& k, const Config& c) {
        std::lock_guard<std::mutex> lk(mu);
        load();
        mem[k] = c;
        const char* p = path();
        if (!p) return;
        FILE* f = fopen(p, "a");
        if (!f) return;
        fprintf(f, "%s %d %d %d\n", k.c_str(), c.block, c.xpt, c.waves);
        fclose(f);
    }
};

TuneCache& cache() {
    static TuneCache c;
    return c;
}

}  // namespace ragged
}  // namespace boys

using namespace boys;

struct boys_ragged_plan {
    const double* x;
    const int64_t* seg_off;
    const int32_t* seg_kmax;
    int32_t nseg;
    double* out;
    const int64_t* out_off;
    ragged::Workspace* ws;
    ragged::Config cfg;
    int64_t total;
    cudaGraph_t graph;
    cudaGraphExec_t exec;
    float tuned_ms;
    // kmax-grouped tiles: host copies of the descriptors, the tile table and its header
    std::vector<int64_t> off_host;
    std::vector<int32_t> km_host;
    ragged::Tile* tiles;
    int tiles_block;
    ragged::GroupHeader* header;
    int64_t ntiles;
};

BOYS_API size_t boys_ragged_workspace_size(void) { return 256; }

BOYS_API size_t boys_ragged_workspace_size_grouped(int32_t nseg, int64_t total) {
    if (nseg < 0 || total < 0) return 0;
    // every segment of len arguments takes ceil(len / 128) <= len / 128 + 1 tiles
    return ragged::kGroupHeaderBytes + sizeof(ragged::Tile) * ((size_t)total / ragged::kGroupTile + (size_t)nseg + 1);
}

BOYS_API boys_status boys_eval_ragged(const double* x, const int64_t* seg_off, const int32_t* seg_kmax,
                                      int32_t nseg, double* out, const int64_t* out_off, void* workspace,
                                      size_t workspace_bytes, void* stream) {
    boys_status st = ragged::check_args(x, seg_off, seg_kmax, nseg, out, out_off, "boys_eval_ragged");
    if (st != BOYS_OK || nseg == 0) return st;
    if (!workspace) return fail(BOYS_ERR_INVALID_ARG, "boys_eval_ragged: NULL workspace");
    if (workspace_bytes < boys_ragged_workspace_size())
        return fail(BOYS_ERR_INVALID_ARG, "boys_eval_ragged: workspace_bytes=%zu < %zu", workspace_bytes,
                    boys_ragged_workspace_size());
    if (!aligned(workspace, 16)) return fail(BOYS_ERR_ALIGNMENT, "boys_eval_ragged: workspace not 16-byte aligned");
    if (workspace_bytes >= ragged::kGroupHeaderBytes + sizeof(ragged::Tile))
        return ragged::launch_grouped(x, seg_off, seg_kmax, nseg, out, out_off, workspace, workspace_bytes,
                                      (cudaStream_t)stream);
    ragged::Config c;
    return ragged::launch(c, x, seg_off, seg_kmax, nseg, out, out_off, (ragged::Workspace*)workspace,
                          (cudaStream_t)stream);
}

BOYS_API boys_status boys_ragged_status(const void* workspace, int* bad_kmax, void* stream) {
    if (!workspace || !bad_kmax) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_status: NULL pointer");
    unsigned long long err = 0;
    const ragged::Workspace* ws = (const ragged::Workspace*)workspace;
    boys_status st = check_cuda(cudaMemcpyAsync(&err, &ws->error, sizeof(err), cudaMemcpyDeviceToHost,
                                                (cudaStream_t)stream), "boys_ragged_status copy");
    if (st != BOYS_OK) return st;
    st = check_cuda(cudaStreamSynchronize((cudaStream_t)stream), "boys_ragged_status sync");
    *bad_kmax = err ? 1 : 0;
    return st;
}

// Tile table for tiles of `block` arguments, sorted by the segments' kmax, and
// its header.
static boys_status build_tiles(boys_ragged_plan* p, int block) {
    if (p->tiles_block == block) return BOYS_OK;
    std::vector<ragged::Tile> tab;
    ragged::GroupHeader h = {};
    for (int k = 0; k <= 32; ++k) {
        const size_t first = tab.size();
        for (int32_t sg = 0; sg < p->nseg; ++sg) {
            if (p->km_host[sg] != k) continue;
            const int64_t len = p->off_host[sg + 1] - p->off_host[sg];
            for (int64_t a = 0; a < len; a += block)
                tab.push_back(ragged::Tile{sg, (int32_t)std::min<int64_t>(block, len - a), a});
        }
        h.count[k] = (unsigned)(tab.size() - first);
    }
    if (tab.size() > 0xFFFFFFFFull) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_create: too many tiles");
    if (p->header) cudaFree(p->header);
    p->header = nullptr;
    p->tiles = nullptr;
    p->tiles_block = 0;
    p->ntiles = (int64_t)tab.size();
    const size_t bytes = ragged::kGroupHeaderBytes + std::max<size_t>(1, tab.size()) * sizeof(ragged::Tile);
    boys_status st = check_cuda(cudaMalloc((void**)&p->header, bytes), "plan tile table");
    if (st != BOYS_OK) return st;
    p->tiles = (ragged::Tile*)((char*)p->header + ragged::kGroupHeaderBytes);
    st = check_cuda(cudaMemcpy(p->header, &h, sizeof(h), cudaMemcpyHostToDevice), "plan tile table header");
    if (st == BOYS_OK && !tab.empty())
        st = check_cuda(cudaMemcpy(p->tiles, tab.data(), tab.size() * sizeof(ragged::Tile), cudaMemcpyHostToDevice),
                        "plan tile table upload");
    // A copy from pageable memory may return before its DMA has ended, and the plan's
    // graph is replayed on streams that do not wait for the default one.
    if (st == BOYS_OK) st = check_cuda(cudaStreamSynchronize(nullptr), "plan tile table upload");
    if (st == BOYS_OK) p->tiles_block = block;
    return st;
}

// Records the batch for configuration c on the capturing stream s: the workspace
// reset and the persistent kernel, or, for waves == 0, the tile kernel alone (the
// plan's kmax were checked when it was made).
static boys_status record_launch(boys_ragged_plan* p, const ragged::Config& c, cudaStream_t s) {
    if (c.waves != 0)
        return ragged::launch(c, p->x, p->seg_off, p->seg_kmax, p->nseg, p->out, p->out_off, p->ws, s);
    ragged::k_group<<<ragged::group_grid(p->ntiles, c.block), c.block, 0, s>>>(p->x, p->seg_off, p->out, p->out_off,
                                                                              p->tiles, p->header);
    return check_cuda(cudaGetLastError(), "ragged group launch");
}

static boys_status capture(boys_ragged_plan* p, const ragged::Config& c, cudaGraph_t* graph, cudaGraphExec_t* exec) {
    *graph = nullptr;
    *exec = nullptr;
    boys_status st = c.waves == 0 ? build_tiles(p, c.block) : BOYS_OK;  // allocates and copies: before any capture
    if (st != BOYS_OK) return st;
    cudaStream_t s;
    st = check_cuda(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking), "plan stream");
    if (st != BOYS_OK) return st;
    st = check_cuda(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "begin capture");
    if (st == BOYS_OK) {
        boys_status lst = record_launch(p, c, s);
        cudaGraph_t g = nullptr;
        boys_status est = check_cuda(cudaStreamEndCapture(s, &g), "end capture");
        st = lst != BOYS_OK ? lst : est;
        if (st == BOYS_OK) {
            *graph = g;
            st = check_cuda(cudaGraphInstantiate(exec, g, 0), "graph instantiate");
            if (st != BOYS_OK) {
                cudaGraphDestroy(g);
                *graph = nullptr;
            }
        } else if (g) {
            cudaGraphDestroy(g);
        }
    }
    cudaStreamDestroy(s);
    return st;
}

static boys_status capture_graph(boys_ragged_plan* p) { return capture(p, p->cfg, &p->graph, &p->exec); }

// Mean time of one replay of configuration c's captured graph (-1 on failure).
static float time_config(boys_ragged_plan* p, const ragged::Config& c, cudaStream_t s, int reps) {
    cudaGraph_t g;
    cudaGraphExec_t e;
    if (capture(p, c, &g, &e) != BOYS_OK) return -1.0f;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaGraphLaunch(e, s);  // warm
    cudaEventRecord(a, s);
    for (int r = 0; r < reps; ++r) cudaGraphLaunch(e, s);
    cudaEventRecord(b, s);
    float ms = -1.0f;
    if (cudaEventSynchronize(b) == cudaSuccess) cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaGraphExecDestroy(e);
    cudaGraphDestroy(g);
    return ms > 0 ? ms / reps : -1.0f;
}

BOYS_API boys_status boys_ragged_plan_create(const double* x, const int64_t* seg_off, const int32_t* seg_kmax,
                                             int32_t nseg, double* out, const int64_t* out_off, int flags,
                                             boys_ragged_plan** plan) {
    if (!plan) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_create: NULL plan");
    *plan = nullptr;
    boys_status st = ragged::check_args(x, seg_off, seg_kmax, nseg, out, out_off, "boys_ragged_plan_create");
    if (st != BOYS_OK) return st;
    if (nseg == 0) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_create: nseg must be > 0");
    // Read the descriptors once (plan creation is a set-up step and may synchronise).
    std::vector<int64_t> off(nseg + 1);
    std::vector<int32_t> km(nseg);
    st = check_cuda(cudaMemcpy(off.data(), seg_off, sizeof(int64_t) * (nseg + 1), cudaMemcpyDeviceToHost), "read seg_off");
    if (st != BOYS_OK) return st;
    st = check_cuda(cudaMemcpy(km.data(), seg_kmax, sizeof(int32_t) * nseg, cudaMemcpyDeviceToHost), "read seg_kmax");
    if (st != BOYS_OK) return st;
    int64_t hist[33] = {0};
    for (int32_t s = 0; s < nseg; ++s) {
        if (off[s + 1] < off[s]) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_create: seg_off decreases at %d", s);
        if (km[s] < 0 || km[s] > 32) return fail(BOYS_ERR_KMAX, "boys_ragged_plan_create: seg_kmax[%d]=%d", s, km[s]);
        hist[km[s]] += off[s + 1] - off[s];
    }
    if (off[0] != 0) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_create: seg_off[0] must be 0");

    boys_ragged_plan* p = new boys_ragged_plan{};
    p->x = x; p->seg_off = seg_off; p->seg_kmax = seg_kmax; p->nseg = nseg; p->out = out; p->out_off = out_off;
    p->total = off[nseg];
    p->off_host = off;
    p->km_host = km;
    st = check_cuda(cudaMalloc((void**)&p->ws, 256), "plan workspace");
    if (st != BOYS_OK) { delete p; return st; }

    if (flags & BOYS_PLAN_AUTOTUNE) {
        // workload key: device + size bucket + argument-weighted kmax histogram (coarse)
        char wk[256];
        int64_t wsum = 0;
        for (int k = 0; k <= 32; ++k) wsum += hist[k] * (k + 1);
        snprintf(wk, sizeof(wk), "|n2^%d|seg%d|w%.2f", 64 - __builtin_clzll((unsigned long long)std::max<int64_t>(1, p->total)),
                 nseg, p->total ? (double)wsum / p->total : 0.0);
        const std::string key = ragged::device_key() + wk;
        ragged::Config best;
        if (!ragged::cache().get(key, &best)) {
            cudaStream_t s;
            cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
            float best_ms = 1e30f;
            for (const auto& c : ragged::candidates()) {
                const float ms = time_config(p, c, s, 3);
                if (ms > 0 && ms < best_ms) { best_ms = ms; best = c; }
            }
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
            p->tuned_ms = best_ms;
            st = check_cuda(cudaGetLastError(), "autotune");
            if (st != BOYS_OK) { boys_ragged_plan_destroy(p); return st; }
            ragged::cache().put(key, best);
        }
        p->cfg = best;
    }
    if (flags & BOYS_PLAN_FORCE_CONFIG) {
        // BOYS_FORCE_CONFIG="block,xpt,waves" overrides tuning (tests use it)
        const char* f = getenv("BOYS_FORCE_CONFIG");
        ragged::Config c;
        if (f && sscanf(f, "%d,%d,%d", &c.block, &c.xpt, &c.waves) == 3 && (c.block == 64 || c.block == 128 || c.block == 256) &&
            (c.xpt == 1 || c.xpt == 2) && c.waves >= 0 && c.waves <= 8)
            p->cfg = c;
    }
    st = capture_graph(p);
    if (st != BOYS_OK) { boys_ragged_plan_destroy(p); return st; }
    *plan = p;
    return BOYS_OK;
}

BOYS_API boys_status boys_ragged_plan_launch(boys_ragged_plan* plan, void* stream) {
    if (!plan) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_launch: NULL plan");
    return check_cuda(cudaGraphLaunch(plan->exec, (cudaStream_t)stream), "graph launch");
}

BOYS_API boys_status boys_ragged_plan_config(const boys_ragged_plan* plan, int* block, int* xpt, int* waves) {
    if (!plan || !block || !xpt || !waves) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_plan_config: NULL pointer");
    *block = plan->cfg.block;
    *xpt = plan->cfg.xpt;
    *waves = plan->cfg.waves;
    return BOYS_OK;
}

BOYS_API void boys_ragged_plan_destroy(boys_ragged_plan* plan) {
    if (!plan) return;
    if (plan->exec) cudaGraphExecDestroy(plan->exec);
    if (plan->graph) cudaGraphDestroy(plan->graph);
    if (plan->ws) cudaFree(plan->ws);
    if (plan->header) cudaFree(plan->header);
    delete plan;
}

// ------------------------------------------------ ragged batch without allocation
//
// boys_eval_ragged_noalloc serves callers that cannot hand the library any
// device memory of their own: the ragged kernel's scratch (tile counter and
// error word, 16 bytes) lives instead in the array below, which is part of
// this library's device image.  Every GPU that loads the library holds the
// array (kNoAllocScratchBytes) until the process exits.

namespace boys {
namespace ragged {

constexpr size_t kNoAllocScratchBytes = 256;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
static_assert(sizeof(Workspace) <= kNoAllocScratchBytes, "ragged scratch must fit the static array");

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[kNoAllocMaxDevices];   // device address of the array, per device
static int g_noalloc_grid[kNoAllocMaxDevices];    // persistent grid of k_ragged<1> at 128 threads

// Per-device set-up on the first call with that device current: the array's
// name is only a host-side stand-in, so its device address comes from
// cudaGetSymbolAddress.  Nothing is allocated.
static boys_status noalloc_setup(int dev, void** ptr, int* grid) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return check_cuda(e, "boys_eval_ragged_noalloc: cudaGetSymbolAddress");
        int sms = 0, per_sm = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return check_cuda(e, "boys_eval_ragged_noalloc: SM count");
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ragged<1>, 128, 0);
        if (e != cudaSuccess) return check_cuda(e, "boys_eval_ragged_noalloc: occupancy");
        g_noalloc_grid[dev] = std::max(1, sms * std::max(1, per_sm));
        g_noalloc_ptr[dev] = p;
    }
    *ptr = g_noalloc_ptr[dev];
    *grid = g_noalloc_grid[dev];
    return BOYS_OK;
}

}  // namespace ragged
}  // namespace boys

BOYS_API boys_status boys_eval_ragged_noalloc(const double* x, const int64_t* seg_off, const int32_t* seg_kmax,
                                              int32_t nseg, double* out, const int64_t* out_off, void* stream) {
    boys_status st = ragged::check_args(x, seg_off, seg_kmax, nseg, out, out_off, "boys_eval_ragged_noalloc");
    if (st != BOYS_OK || nseg == 0) return st;
    // A call's scratch need does not grow with its sizes (one tile counter and
    // one error word); it is checked against the array all the same.
    if (sizeof(ragged::Workspace) > ragged::kNoAllocScratchBytes)
        return fail(BOYS_ERR_INVALID_ARG, "boys_eval_ragged_noalloc: needs %zu bytes of scratch, the static array holds %zu",
                    sizeof(ragged::Workspace), ragged::kNoAllocScratchBytes);
    int dev = 0;
    st = check_cuda(cudaGetDevice(&dev), "boys_eval_ragged_noalloc: cudaGetDevice");
    if (st != BOYS_OK) return st;
    if (dev < 0 || dev >= ragged::kNoAllocMaxDevices)
        return fail(BOYS_ERR_INVALID_ARG, "boys_eval_ragged_noalloc: device %d beyond the %d supported", dev,
                    ragged::kNoAllocMaxDevices);
    void* scratch = nullptr;
    int grid = 1;
    st = ragged::noalloc_setup(dev, &scratch, &grid);
    if (st != BOYS_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    // the array keeps the previous call's contents: the counter must restart at zero
    st = check_cuda(cudaMemsetAsync(scratch, 0, sizeof(ragged::Workspace), s), "boys_eval_ragged_noalloc: scratch reset");
    if (st != BOYS_OK) return st;
    ragged::k_ragged<1><<<grid, 128, 0, s>>>(x, seg_off, seg_kmax, nseg, out, out_off, (ragged::Workspace*)scratch,
                                             nullptr);
    return check_cuda(cudaGetLastError(), "boys_eval_ragged_noalloc launch");
}

// The error word of the static array on the current device, read after the
// stream's work so far; copying from the symbol needs no device address and
// no allocation.
BOYS_API boys_status boys_ragged_noalloc_status(int* bad_kmax, void* stream) {
    if (!bad_kmax) return fail(BOYS_ERR_INVALID_ARG, "boys_ragged_noalloc_status: NULL pointer");
    unsigned long long err = 0;
    cudaStream_t s = (cudaStream_t)stream;
    boys_status st = check_cuda(cudaMemcpyFromSymbolAsync(&err, ragged::g_noalloc_scratch, sizeof(err),
                                                          offsetof(ragged::Workspace, error), cudaMemcpyDeviceToHost, s),
                                "boys_ragged_noalloc_status copy");
    if (st != BOYS_OK) return st;
    st = check_cuda(cudaStreamSynchronize(s), "boys_ragged_noalloc_status sync");
    *bad_kmax = err ? 1 : 0;
    return st;
}
