// Binning by cell (counting sort into cell regions, each cell in pid order),
// the per-step commit of appended secondaries, and FP64 totals.
#include <algorithm>
#include <string>

#include "pcc_commit.cuh"
#include "pcc_internal.h"
#include "pcc_totals.cuh"

namespace pcc {

// Binning moves each particle record twice: into a temporary array of 32-byte
// records grouped by cell (one full sector per scattered write), and from
// there, in pid order, into the cell's region.  Both are bound by memory: 28 B
// read and 32 B written, then 32 B read and 28 B written, against the 56 B that
// one move would need; the 60 B more buy whole sectors where the input order is
// random (six scattered 4-8 byte writes per particle before).
constexpr int kMaxCellSort = 16384;
constexpr int kScanBlock = 1024;    // cells per block of the region scan
constexpr int kLocalCells = 8192;   // cells counted in a block's shared memory (32 KB)
constexpr int kLocalThreads = 512;
constexpr int kLocalBlocks = 3;      // of these on an SM

// What the host reads back, and what the later kernels check themselves, so
// that they can be enqueued before the host knows.
struct BinTotals {
    long long slots;        // sum of the regions
    long long largest;      // particles in the fullest cell
};
struct BinLimits {
    const BinTotals* t;
    long long capacity;
    __device__ __forceinline__ bool exceeded() const { return t->slots > capacity || t->largest > kMaxCellSort; }
};

// Lists of the cells each of the larger sort kernels takes.
constexpr int kSortClasses = 3;
struct SortLists {
    int* list[kSortClasses];   // [n_cells] each
    int* count;                // [kSortClasses]
};

struct Rec {
    const float *ux, *uy, *uz, *w, *x;
    const uint64_t* pid;
};
struct MRec {
    float *ux, *uy, *uz, *w, *x;
    uint64_t* pid;
};

// ---- histogram ----------------------------------------------------------------
__device__ __forceinline__ int valid_cell(const int* cell, int i, int n, int n_cells, DevStats* st)
{
    int c = i < n ? cell[i] : -1;
    if (i < n && (c < 0 || c >= n_cells)) {
        if (st) raise_status(st, PCC_ST_NONFINITE);
        c = -1;
    }
    return c;
}

// Lanes of the warp with this lane's cell, for the cells met in the first lanes:
// after a push a warp of nearly ordered particles holds about three cells, and
// three votes gather them; lanes of further cells count for themselves.  (The
// match instruction, which gathers all, takes about 70 clocks of the SM per
// warp, as much as the rest of the kernel; the votes take a few.)
__device__ __forceinline__ unsigned near_peers(int c)
{
    constexpr unsigned kFull = 0xffffffffu;
    unsigned peers = 1u << (threadIdx.x & 31), left = __ballot_sync(kFull, c >= 0);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        if (!left) break;   // warp-uniform
        const int cl = __shfl_sync(kFull, c, __ffs(left) - 1);
        const unsigned m = __ballot_sync(kFull, c == cl);
        if (c == cl) peers = m;
        left &= ~m;
    }
    return peers;
}

// One global atomic per group of lanes.
__global__ void bin_count_kernel(const int* cell, int n, int n_cells, int* counts, DevStats* st)
{
    pdl_begin();
    const int c = valid_cell(cell, blockIdx.x * blockDim.x + threadIdx.x, n, n_cells, st);
    const unsigned peers = near_peers(c);
    const int leader = __ffs(peers) - 1;
    if (c >= 0 && (threadIdx.x & 31) == leader) atomicAdd(&counts[c], __popc(peers));
}

// Few cells: a block counts a contiguous chunk of the input in shared memory
// and adds a cell's count once: 2048 cells of 8192 shuffled particles 0.70 -> 0.06
// ms (a global atomic per particle before).
__global__ void __launch_bounds__(kLocalThreads, kLocalBlocks) bin_count_local_kernel(const int* cell, int n, int n_cells,
                                                                                      int* counts, DevStats* st)
{
    pdl_begin();
    extern __shared__ int h[];
    const int lo = (int)((long long)n * blockIdx.x / gridDim.x), hi = (int)((long long)n * (blockIdx.x + 1) / gridDim.x);
    for (int c = threadIdx.x; c < n_cells; c += blockDim.x) h[c] = 0;
    __syncthreads();
    for (int i0 = lo; i0 < hi; i0 += blockDim.x) {
        const int c = valid_cell(cell, i0 + (int)threadIdx.x, hi, n_cells, st);
        const unsigned peers = near_peers(c);
        if (c >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&h[c], __popc(peers));
    }
    __syncthreads();
    for (int c = threadIdx.x; c < n_cells; c += blockDim.x)
        if (h[c]) atomicAdd(&counts[c], h[c]);
}

// ---- regions: sums per block of cells, then offsets ---------------------------------
__device__ __forceinline__ long long region_of(int count, int slack_abs, double slack_rel)
{
    const long long extra = (long long)ceil(slack_rel * (double)count);
    return (long long)count + (extra > slack_abs ? extra : slack_abs);
}

struct BlockSums {
    long long slots;
    int particles, largest;
};

__global__ void __launch_bounds__(kScanBlock) region_sums_kernel(const int* counts, int n, int slack_abs,
                                                                 double slack_rel, BlockSums* sums)
{
    pdl_begin();
    __shared__ long long s[32];
    __shared__ int sp[32], sm[32];
    const int i = blockIdx.x * kScanBlock + threadIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int c = i < n ? counts[i] : 0;
    const long long r = warp_sum(i < n ? region_of(c, slack_abs, slack_rel) : 0ll);
    const int p = warp_sum(c), m = __reduce_max_sync(0xffffffffu, c);
    if (lane == 0) { s[wid] = r; sp[wid] = p; sm[wid] = m; }
    __syncthreads();
    if (wid == 0) {
        const long long R = warp_sum(s[lane]);
        const int P = warp_sum(sp[lane]), M = __reduce_max_sync(0xffffffffu, sm[lane]);
        if (lane == 0) sums[blockIdx.x] = BlockSums{R, P, M};
    }
}

template <typename T>
__device__ __forceinline__ T warp_incl(T v)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) >= o) v += t;
    }
    return v;
}

// Sort class of a cell: -1 for the kernel that takes a warp per cell.
constexpr int kSortWarpCap = 256, kSortCap0 = 2048, kSortCap1 = 8192;
__device__ __forceinline__ int sort_class(int count)
{
    return count <= kSortWarpCap ? -1 : count <= kSortCap0 ? 0 : count <= kSortCap1 ? 1 : 2;
}

// Each block adds up the sums of the blocks before it and scans its own cells:
// the atomic maximum of every cell alone took 64 us of a 1e5-cell binning, and
// one thread walked the block sums.
__global__ void __launch_bounds__(kScanBlock) region_offsets_kernel(const BlockSums* sums, int nb, const int* counts, int n,
                                                                    int slack_abs, double slack_rel, int* cell_start,
                                                                    int* cell_count, int* cell_added, int* first,
                                                                    int* cursor, BinTotals* totals, SortLists L)
{
    pdl_begin();
    __shared__ long long sl[32];
    __shared__ int sp[32], sm[32], n_class[kSortClasses], at[kSortClasses];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the blocks before this one (and, for the totals, all of them)
    long long before = 0, all = 0;
    int pbefore = 0, largest = 0;
    for (int b = threadIdx.x; b < nb; b += kScanBlock) {
        const BlockSums v = sums[b];
        if (b < (int)blockIdx.x) { before += v.slots; pbefore += v.particles; }
        all += v.slots;
        largest = max(largest, v.largest);
    }
    before = warp_sum(before);
    pbefore = warp_sum(pbefore);
    if (lane == 0) { sl[wid] = before; sp[wid] = pbefore; }
    if (threadIdx.x < kSortClasses) n_class[threadIdx.x] = 0;
    __syncthreads();
    before = warp_sum(sl[lane]);
    pbefore = warp_sum(sp[lane]);
    __syncthreads();
    if (blockIdx.x == 0) {
        all = warp_sum(all);
        largest = __reduce_max_sync(0xffffffffu, largest);
        if (lane == 0) { sl[wid] = all; sm[wid] = largest; }
        __syncthreads();
        if (wid == 0) {
            all = warp_sum(sl[lane]);
            largest = __reduce_max_sync(0xffffffffu, sm[lane]);
            if (lane == 0) *totals = BinTotals{all, largest};
        }
        __syncthreads();
    }
    // this block's cells
    const int i = blockIdx.x * kScanBlock + threadIdx.x;
    const int c = i < n ? counts[i] : 0;
    const long long r = i < n ? region_of(c, slack_abs, slack_rel) : 0;
    const long long ri = warp_incl(r);
    const int ci = warp_incl(c);
    if (lane == 31) { sl[wid] = ri; sp[wid] = ci; }
    const int cls = i < n ? sort_class(c) : -1;
    int rank = 0;
    if (cls >= 0) rank = atomicAdd(&n_class[cls], 1);
    __syncthreads();
    const long long wl = warp_incl(sl[lane]);
    const int wp = warp_incl(sp[lane]);
    const long long end = before + ri + (wid ? __shfl_sync(0xffffffffu, wl, wid - 1) : 0);
    const int pstart = pbefore + ci - c + (wid ? __shfl_sync(0xffffffffu, wp, wid - 1) : 0);
    if (threadIdx.x < kSortClasses && n_class[threadIdx.x])
        at[threadIdx.x] = atomicAdd(&L.count[threadIdx.x], n_class[threadIdx.x]);
    __syncthreads();
    if (i >= n) return;
    if (end <= 0x7fffffffLL) cell_start[i + 1] = (int)end;
    if (i == 0) cell_start[0] = 0;
    cell_count[i] = c;
    cell_added[i] = 0;
    first[i] = pstart;
    cursor[i] = pstart;
    if (cls >= 0) L.list[cls][at[cls] + rank] = i;
}

// ---- scatter into the temporary records ---------------------------------------------
// A temporary record: one 32-byte sector, moved by one 256-bit access.
struct __align__(32) TmpRec {
    float ux, uy, uz, w, x, pad;
    uint32_t pid_lo, pid_hi;
};

__device__ __forceinline__ void put_record(const Rec& in, int i, TmpRec* tmp, int p)
{
    const uint64_t pid = in.pid[i];
    const float x = in.x ? in.x[i] : 0.f;
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(tmp + p), "f"(in.ux[i]), "f"(in.uy[i]),
                 "f"(in.uz[i]), "f"(in.w[i]), "f"(x), "f"(0.f), "f"(__uint_as_float((uint32_t)pid)),
                 "f"(__uint_as_float((uint32_t)(pid >> 32)))
                 : "memory");
}

__device__ __forceinline__ TmpRec get_record(const TmpRec* tmp, int p)
{
    TmpRec r;
    float lo, hi;
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r.ux), "=f"(r.uy), "=f"(r.uz), "=f"(r.w), "=f"(r.x), "=f"(r.pad), "=f"(lo), "=f"(hi)
                 : "l"(tmp + p));
    r.pid_lo = __float_as_uint(lo);
    r.pid_hi = __float_as_uint(hi);
    return r;
}

__device__ __forceinline__ uint64_t get_pid(const TmpRec* tmp, int p)
{
    return *reinterpret_cast<const uint64_t*>(&tmp[p].pid_lo);
}

__device__ __forceinline__ void store_record(const MRec& out, int dst, const TmpRec& r)
{
    out.ux[dst] = r.ux;
    out.uy[dst] = r.uy;
    out.uz[dst] = r.uz;
    out.w[dst] = r.w;
    if (out.x) out.x[dst] = r.x;
    out.pid[dst] = (uint64_t)r.pid_hi << 32 | r.pid_lo;
}

__global__ void bin_scatter_kernel(Rec in, const int* cell, int n, int n_cells, int* cursor, TmpRec* tmp, BinLimits lim)
{
    pdl_begin();
    if (lim.exceeded()) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = valid_cell(cell, i, n, n_cells, nullptr);
    const unsigned peers = near_peers(c);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (c >= 0 && lane == leader) base = atomicAdd(&cursor[c], __popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (c >= 0) put_record(in, i, tmp, base + __popc(peers & ((1u << lane) - 1u)));
}

// Few cells: a block takes places for the particles of a tile with one global
// atomic per cell of the tile and hands them out from shared memory.  Tiles of
// 4096 particles keep the records that are being filled in (32 B each, all
// blocks) within L2, so that its lines reach memory whole.
constexpr int kTileItems = 8;
__global__ void __launch_bounds__(kLocalThreads, kLocalBlocks) bin_scatter_local_kernel(Rec in, const int* cell, int n,
                                                                                        int n_cells, int* cursor,
                                                                                        TmpRec* tmp, BinLimits lim)
{
    pdl_begin();
    extern __shared__ int h[];
    if (lim.exceeded()) return;
    constexpr int kTile = kTileItems * kLocalThreads;
    const int lane = threadIdx.x & 31;
    for (long long t0 = (long long)blockIdx.x * kTile; t0 < n; t0 += (long long)gridDim.x * kTile) {
        for (int c = threadIdx.x; c < n_cells; c += blockDim.x) h[c] = 0;
        __syncthreads();
        int c[kTileItems], r[kTileItems];
#pragma unroll
        for (int k = 0; k < kTileItems; ++k) {
            const long long i = t0 + k * kLocalThreads + (int)threadIdx.x;
            c[k] = i < n ? valid_cell(cell, (int)i, n, n_cells, nullptr) : -1;
        }
#pragma unroll
        for (int k = 0; k < kTileItems; ++k) {
            const unsigned peers = near_peers(c[k]);
            const int leader = __ffs(peers) - 1;
            int base = 0;
            if (c[k] >= 0 && lane == leader) base = atomicAdd(&h[c[k]], __popc(peers));
            r[k] = __shfl_sync(0xffffffffu, base, leader) + __popc(peers & ((1u << lane) - 1u));
        }
        __syncthreads();
        for (int k = threadIdx.x; k < n_cells; k += blockDim.x)
            if (h[k]) h[k] = atomicAdd(&cursor[k], h[k]);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kTileItems; ++k)
            if (c[k] >= 0) put_record(in, (int)(t0 + k * kLocalThreads) + (int)threadIdx.x, tmp, h[c[k]] + r[k]);
        __syncthreads();
    }
}

// ---- per-cell sort by pid ---------------------------------------------------------------
// W warps order up to W 32 ITEMS records of a cell by pid and move them to its
// region; records already in order are only moved.
// Radix passes order 16-bit indices, eight bits a pass over the bits in which
// the pids differ only (two or three passes where pids are storage numbers, more
// for the wide ids of secondaries); ranks by eight votes per row of 32 against
// each warp's own digit counts, which keeps a pass stable.  A block (more than
// 256 records) first tries a counting sort: the pids' range cut into equal
// buckets, at least as many as records, and within a bucket each record compares
// itself with the few others; a bucket with more than kBucketMax sends the cell
// to the radix passes.  2048 cells of 8192 shuffled records: 0.56 ms, with radix
// passes only 0.70 ms (a bitonic network of 91 compare-exchange steps in shared
// memory took 2.7 ms); the cells of 257 to 2048 records of an uneven step 0.30
// against 0.34 ms.  Smaller cells hold ids of neighbours of any size, which
// crowd the buckets (one warp per cell of up to 512: 0.62 against 0.45 ms).
// Bound by shared memory and the latency of the phases, not by the two moves.
constexpr int kBucketMax = 12;
template <int W, int ITEMS>
struct SortSmem {
    static constexpr int kCap = W * 32 * ITEMS;
    uint64_t key[kCap];
    union {
        uint32_t count[kCap];                                       // buckets
        struct { uint16_t ord2[kCap], hist[W * 256]; } radix;
    };
    uint16_t ord[kCap];
    uint64_t lo, hi, diff;               // smallest and largest pid; bits in which they differ
    int unsorted, crowded;
    int wsum[32];
};

template <int W>
__device__ __forceinline__ void sort_sync()
{
    if (W == 1) __syncwarp();
    else __syncthreads();
}

// Exclusive scan of one value per thread over the group; the total is not needed.
template <int W>
__device__ __forceinline__ int group_excl(int v, int* wsum, int w, int lane)
{
    const int incl = warp_incl(v);
    if (W == 1) return incl - v;
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    int base = 0;
    for (int k = 0; k < w; ++k) base += wsum[k];
    return base + incl - v;
}

// Radix passes over the bits diff; the order ends in S.ord.
template <int W, int ITEMS>
__device__ __noinline__ void radix_order(SortSmem<W, ITEMS>& S, uint64_t diff, int n)
{
    constexpr unsigned kFull = 0xffffffffu;
    constexpr int T = 32 * W;
    const int lane = threadIdx.x & 31, w = W == 1 ? 0 : threadIdx.x >> 5, tid = w * 32 + lane;
    const int part = ((n + W - 1) / W + 31) & ~31;   // records per warp, whole rows of 32
    uint16_t* hw = S.radix.hist + 256 * w;
    uint16_t *from = S.radix.ord2, *to = S.ord;
    // an odd number of passes ends in S.ord; an even one starts the other way round
    int passes = 0;
    for (uint64_t d = diff; d; ++passes) d &= ~(0xFFull << (__ffsll((long long)d) - 1));
    if (!(passes & 1)) { uint16_t* t = from; from = to; to = t; }
    for (bool identity = true; diff; identity = false) {
        const int sh = __ffsll((long long)diff) - 1;
        diff &= ~(0xFFull << sh);
        for (int i = tid; i < W * 256; i += T) S.radix.hist[i] = 0;
        sort_sync<W>();
        uint32_t pk[ITEMS];   // index | rank among the warp's records of its digit << 16
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int i = w * part + it * 32 + lane;
            pk[it] = 0xFFFFu;
            if (it * 32 < part) {   // warp-uniform
                const bool in = i < n;
                const uint32_t idx = in ? (identity ? (uint32_t)i : from[i]) : 0u;
                const uint32_t d = (uint32_t)(S.key[idx] >> sh) & 255u;
                unsigned peers = __ballot_sync(kFull, in);   // lanes with this digit
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const unsigned m = __ballot_sync(kFull, d >> q & 1u);
                    peers &= d >> q & 1u ? m : ~m;
                }
                const uint32_t base = in ? hw[d] : 0u;
                __syncwarp();
                if (in && lane == __ffs(peers) - 1) hw[d] = (uint16_t)(base + __popc(peers));
                __syncwarp();
                if (in) pk[it] = idx | (base + __popc(peers & ((1u << lane) - 1u))) << 16;
            }
        }
        sort_sync<W>();
        // counts -> offsets, digits first, then warps
        if (W == 1) {
            uint32_t v[8], sum = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) { v[q] = S.radix.hist[8 * lane + q]; sum += v[q]; }
            uint32_t run = warp_incl(sum) - sum;
#pragma unroll
            for (int q = 0; q < 8; ++q) { S.radix.hist[8 * lane + q] = (uint16_t)run; run += v[q]; }
        } else {
            constexpr int D = T >= 256 ? 1 : 256 / T;   // digits per thread
            int sum = 0;
            if (tid < 256 / D)
                for (int q = 0; q < D; ++q)
                    for (int k = 0; k < W; ++k) sum += S.radix.hist[256 * k + D * tid + q];
            int run = group_excl<W>(sum, S.wsum, w, lane);
            if (tid < 256 / D)
                for (int q = 0; q < D; ++q)
                    for (int k = 0; k < W; ++k) {
                        uint16_t& x = S.radix.hist[256 * k + D * tid + q];
                        const int c = x;
                        x = (uint16_t)run;
                        run += c;
                    }
        }
        sort_sync<W>();
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            if (it * 32 + lane < part && w * part + it * 32 + lane < n) {
                const uint32_t idx = pk[it] & 0xFFFFu, d = (uint32_t)(S.key[idx] >> sh) & 255u;
                to[hw[d] + (pk[it] >> 16)] = (uint16_t)idx;
            }
        }
        sort_sync<W>();
        uint16_t* t = from; from = to; to = t;
    }
}

// One block per cell: the counting sort, or radix passes where it does not apply.
template <int W, int ITEMS>
__device__ __forceinline__ void sort_cell_block(SortSmem<W, ITEMS>& S, const TmpRec* tmp, int n, const MRec& out, int s0)
{
    constexpr int T = 32 * W;
    constexpr unsigned kFull = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) { S.lo = ~0ull; S.hi = S.diff = 0; S.unsorted = S.crowded = 0; }
    // buckets: a power of two, at least the records and a row per warp
    const int bits = max(W == 4 ? 7 : 9, 32 - __clz(n - 1)), nb = 1 << bits;
    for (int i = tid; i < nb; i += T) S.count[i] = 0;
    __syncthreads();
    const uint64_t k0 = get_pid(tmp, 0);
    uint64_t lo = ~0ull, hi = 0, diff = 0;
#pragma unroll 8
    for (int i = tid; i < n; i += T) {
        const uint64_t k = get_pid(tmp, i);
        S.key[i] = k;
        diff |= k ^ k0;
        lo = lo < k ? lo : k;
        hi = hi > k ? hi : k;
    }
    const uint32_t dl = __reduce_or_sync(kFull, (uint32_t)diff), dh = __reduce_or_sync(kFull, (uint32_t)(diff >> 32));
    if (lane == 0) atomicOr((unsigned long long*)&S.diff, (unsigned long long)dh << 32 | dl);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t a = __shfl_xor_sync(kFull, lo, o), b = __shfl_xor_sync(kFull, hi, o);
        lo = lo < a ? lo : a;
        hi = hi > b ? hi : b;
    }
    if (lane == 0) {
        atomicMin((unsigned long long*)&S.lo, (unsigned long long)lo);
        atomicMax((unsigned long long*)&S.hi, (unsigned long long)hi);
    }
    __syncthreads();
    lo = S.lo;
    const int shift = max(0, 64 - bits - __clzll((long long)(S.hi - lo)));   // bucket (pid - lo) >> shift < nb
    int r[ITEMS];
    bool bad = false, crowded = false;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = tid + k * T;
        r[k] = 0;
        if (k * T >= n) break;   // uniform, as below
        if (i < n) {
            const uint64_t key = S.key[i];
            bad |= i + 1 < n && key > S.key[i + 1];
            r[k] = (int)atomicAdd(&S.count[(uint32_t)((key - lo) >> shift)], 1u);
            crowded |= r[k] >= kBucketMax;
        }
    }
    if (__any_sync(kFull, bad) && lane == 0) S.unsorted = 1;
    if (__any_sync(kFull, crowded) && lane == 0) S.crowded = 1;
    __syncthreads();
    if (!S.unsorted) {
#pragma unroll 4
        for (int i = tid; i < n; i += T) store_record(out, s0 + i, get_record(tmp, i));
        return;
    }
    if (S.crowded) {
        radix_order<W, ITEMS>(S, S.diff, n);
    } else {
        // bucket counts -> first positions: a warp scans its part row by row
        const int rows = nb / T;
        uint32_t* part = S.count + w * 32 * rows;
        int run = 0;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            if (k >= rows) break;
            const int v = (int)part[32 * k + lane], incl = warp_incl(v);
            part[32 * k + lane] = (uint32_t)(run + incl - v);
            run += __shfl_sync(kFull, incl, 31);
        }
        if (lane == 0) S.wsum[w] = run;
        __syncthreads();
        int base = 0;
        for (int k = 0; k < w; ++k) base += S.wsum[k];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k)
            if (k < rows) part[32 * k + lane] += (uint32_t)base;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = tid + k * T;
            if (k * T >= n) break;
            if (i < n) S.ord[S.count[(uint32_t)((S.key[i] - lo) >> shift)] + r[k]] = (uint16_t)i;
        }
        __syncthreads();
        // a record's place in its bucket: the smaller pids there
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = tid + k * T;
            if (k * T >= n) break;
            if (i < n) {
                const uint64_t key = S.key[i];
                const uint32_t b = (uint32_t)((key - lo) >> shift);
                const int q0 = (int)S.count[b], q1 = (int)b + 1 < nb ? (int)S.count[b + 1] : n;
                int at = q0;
                for (int q = q0; q < q1; ++q) {
                    const int j = S.ord[q];
                    const uint64_t kj = S.key[j];
                    at += kj < key || (kj == key && j < i) ? 1 : 0;
                }
                r[k] = at;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = tid + k * T;
            if (k * T >= n) break;
            if (i < n) S.ord[r[k]] = (uint16_t)i;
        }
        __syncthreads();
    }
#pragma unroll 4
    for (int i = tid; i < n; i += T) store_record(out, s0 + i, get_record(tmp, S.ord[i]));
}

// One warp, up to 32 ITEMS records: the radix passes alone (the buckets would
// seldom do for so few records, whose ids come from cells of any size).
template <int ITEMS>
__device__ __forceinline__ void sort_cell_warp(SortSmem<1, ITEMS>& S, const TmpRec* tmp, int n, const MRec& out, int s0)
{
    constexpr unsigned kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint64_t k0 = get_pid(tmp, 0);
    uint64_t diff = 0, last = 0;
    bool bad = false;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int i = it * 32 + lane;
        if (it * 32 < n) {   // uniform
            const uint64_t k = i < n ? get_pid(tmp, i) : ~0ull;
            if (i < n) { S.key[i] = k; diff |= k ^ k0; }
            const uint64_t up = __shfl_up_sync(kFull, k, 1), carry = __shfl_sync(kFull, last, 31);
            bad |= (lane ? up : carry) > k;   // carry: the row before; 0 at first
            last = k;
        }
    }
    if (!__any_sync(kFull, bad)) {
        for (int i = lane; i < n; i += 32) store_record(out, s0 + i, get_record(tmp, i));
        return;
    }
    diff = (uint64_t)__reduce_or_sync(kFull, (uint32_t)(diff >> 32)) << 32 | __reduce_or_sync(kFull, (uint32_t)diff);
    __syncwarp();
    radix_order<1, ITEMS>(S, diff, n);
#pragma unroll 4
    for (int i = lane; i < n; i += 32) store_record(out, s0 + i, get_record(tmp, S.ord[i]));
}

// A warp per cell of up to kSortWarpCap records; up to 64 by counting the smaller pids.
constexpr int kSortWarps = 4;
__global__ void __launch_bounds__(32 * kSortWarps, 12) sort_warp_kernel(const int* cell_start, const int* cell_count,
                                                                        const int* first, int n_cells, const TmpRec* tmp,
                                                                        MRec out, BinLimits lim)
{
    pdl_begin();
    constexpr unsigned kFull = 0xffffffffu;
    __shared__ SortSmem<1, kSortWarpCap / 32> S[kSortWarps];
    const int c = blockIdx.x * kSortWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= n_cells) return;
    const int n = cell_count[c], s0 = cell_start[c];
    const TmpRec* t = tmp + first[c];
    if (n == 0 || n > kSortWarpCap || lim.exceeded()) return;
    if (n > 64) {
        sort_cell_warp<kSortWarpCap / 32>(S[threadIdx.x >> 5], t, n, out, s0);
        return;
    }
    // places by the number of smaller pids (or equal ones stored before)
    const int n1 = n - 32;
    const uint64_t k0 = lane < n ? get_pid(t, lane) : ~0ull, k1 = lane < n1 ? get_pid(t, 32 + lane) : ~0ull;
    int r0 = 0, r1 = 0;
    for (int i = 0; i < min(n, 32); ++i) {
        const uint64_t k = __shfl_sync(kFull, k0, i);
        r0 += k < k0 || (k == k0 && i < lane) ? 1 : 0;
        r1 += k <= k1 ? 1 : 0;
    }
    for (int i = 0; i < n1; ++i) {
        const uint64_t k = __shfl_sync(kFull, k1, i);
        r0 += k < k0 ? 1 : 0;
        r1 += k < k1 || (k == k1 && i < lane) ? 1 : 0;
    }
    if (lane < n) store_record(out, s0 + r0, get_record(t, lane));
    if (lane < n1) store_record(out, s0 + r1, get_record(t, 32 + lane));
}

// A block per cell of one class's list.
template <int W, int ITEMS>
__global__ void __launch_bounds__(32 * W, W == 4 ? 8 : 32 / ITEMS) sort_block_kernel(const int* cell_start, const int* cell_count,
                                                            const int* first, const int* list, const int* count,
                                                            const TmpRec* tmp, MRec out, BinLimits lim)
{
    pdl_begin();
    extern __shared__ __align__(16) unsigned char sort_smem[];
    auto& S = *reinterpret_cast<SortSmem<W, ITEMS>*>(sort_smem);
    if (lim.exceeded()) return;
    const int m = *count;
    for (int k = blockIdx.x; k < m; k += gridDim.x) {
        const int c = list[k];
        sort_cell_block<W, ITEMS>(S, tmp + first[c], cell_count[c], out, cell_start[c]);
        __syncthreads();
    }
}

// ---- commit of appended secondaries: order by pid, then make live
__global__ void commit_kernel(SpeciesView sp, int n_cells)
{
    pdl_begin();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n_cells) commit_cell(sp, c);
}

// For many blocks on an SM: the overlap's two instructions take a block of this kernel
// as long as its one load, which in the end is more than the overlap gains (4e6 cells,
// 103 blocks an SM: 17 us with them, 11 without; 2^20 cells, 27 blocks: 5.1 and 5.6).
__global__ void commit_many_kernel(SpeciesView sp, int n_cells)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n_cells) commit_cell(sp, c);
}

// ---- FP64 totals: slots shared out to the warps, fixed-order partials per block (see pcc_totals.cuh)
template <bool PHOTON>
__global__ void __launch_bounds__(256, 4) totals_kernel(const pcc_species sp, int n_cells, double* partial)
{
    pdl_begin();
    __shared__ double sh[3][32];
    const int nw = blockDim.x >> 5;
    TotalsAcc acc;
    totals_share<PHOTON>(sp, n_cells, blockIdx.x * nw + (threadIdx.x >> 5), gridDim.x * nw, threadIdx.x & 31, acc);
    totals_block_out(acc, sh, partial);
}

__global__ void totals_final_kernel(const double* partial, int nb, double* out) {
    pdl_begin(); totals_reduce(partial, nb, out); }

}  // namespace pcc

using namespace pcc;

// The pinned host copy of the totals and the event that says it is there.
static int ensure_bin_host(pcc_ctx* ctx)
{
    if (ctx->bin_host && ctx->bin_event) return PCC_OK;
    cudaError_t e = cudaSuccess;
    if (!ctx->bin_host) e = cudaMallocHost(&ctx->bin_host, sizeof(BinTotals));
    if (e == cudaSuccess && !ctx->bin_event) e = cudaEventCreateWithFlags(&ctx->bin_event, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(e, "pcc_bin: host buffer");
    // the larger sort classes need more shared memory than the default
    e = cudaFuncSetAttribute(sort_block_kernel<16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SortSmem<16, 16>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(sort_block_kernel<16, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SortSmem<16, 32>));
    return e == cudaSuccess ? PCC_OK : cuda_fail(e, "pcc_bin: shared memory");
}

// Resident blocks by shared memory and threads; every list is walked by a grid of them.
template <int W, int ITEMS>
static void launch_sort(pcc_ctx* ctx, int cls, const pcc_species* out, const int* first, const SortLists& L,
                        const TmpRec* tmp, const MRec& ro, const BinLimits& lim, cudaStream_t st)
{
    constexpr int smem = (int)sizeof(SortSmem<W, ITEMS>);
    constexpr int per_sm = std::min(2048 / (32 * W), 227 * 1024 / (smem + 1024));
    launch_pdl(sort_block_kernel<W, ITEMS>, per_sm * std::max(ctx->num_sms, 1), 32 * W, smem, st, 
        out->cell_start, out->cell_count, first, L.list[cls], L.count + cls, tmp, ro, lim);
    note_launches(1);
}

extern "C" int pcc_bin(pcc_ctx* ctx, const pcc_particles* in, int n_cells, pcc_species* out, int slack_abs,
                       double slack_rel, void* stream)
{
    if (!ctx || !in || !out) { set_error("pcc_bin: null argument"); return PCC_E_INVALID; }
    if (n_cells < 1 || in->n < 0 || slack_abs < 0 || !(slack_rel >= 0.0) || out->capacity < 0) {
        set_error("pcc_bin: invalid sizes");
        return PCC_E_INVALID;
    }
    if (in->n > 0 && (!in->ux || !in->uy || !in->uz || !in->w || !in->pid || !in->cell)) {
        set_error("pcc_bin: null input array");
        return PCC_E_INVALID;
    }
    if (!out->ux || !out->uy || !out->uz || !out->w || !out->pid || !out->cell_start || !out->cell_count ||
        !out->cell_added || ((in->x == nullptr) != (out->x == nullptr) && in->x != nullptr)) {
        set_error("pcc_bin: null output array (x must be given on both sides or only on the output)");
        return PCC_E_INVALID;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int n = in->n, nb = (n_cells + kScanBlock - 1) / kScanBlock;
    // scratch: counts with the class counters, offsets, cursors, block sums, totals,
    // class lists, records.  Its size goes by the capacity, not by the particles, so
    // that a run whose species grow allocates once and what a captured graph holds
    // of it stays; only where memory is too short for that, by the particles.
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
    const size_t o_counts = take(((size_t)n_cells + kSortClasses) * sizeof(int));
    const size_t o_first = take(n_cells * sizeof(int));
    const size_t o_cursor = take(n_cells * sizeof(int));
    const size_t o_sums = take(nb * sizeof(BlockSums));
    const size_t o_tot = take(sizeof(BinTotals));
    size_t o_list[kSortClasses];
    for (int k = 0; k < kSortClasses; ++k) o_list[k] = take((size_t)n_cells * sizeof(int));
    const size_t o_tmp = off, cap = (size_t)out->capacity;
    int rc = ensure_scratch(ctx, o_tmp + cap * sizeof(TmpRec));
    if (rc && (size_t)n < cap) {
        cudaGetLastError();
        rc = ensure_scratch(ctx, o_tmp + (size_t)n * sizeof(TmpRec));
    }
    if (rc) return rc;
    rc = ensure_bin_host(ctx);
    if (rc) return rc;
    char* base = (char*)ctx->scratch;
    int* counts = (int*)(base + o_counts);
    int* first = (int*)(base + o_first);
    int* cursor = (int*)(base + o_cursor);
    BlockSums* sums = (BlockSums*)(base + o_sums);
    BinTotals* tot = (BinTotals*)(base + o_tot);
    SortLists L;
    for (int k = 0; k < kSortClasses; ++k) L.list[k] = (int*)(base + o_list[k]);
    L.count = counts + n_cells;
    TmpRec* tmp = (TmpRec*)(base + o_tmp);

    // Counting and handing out places in shared memory pays where a block's
    // chunk holds several particles for each counter: 2048 cells x 8192
    // shuffled particles, count 0.70 -> 0.06 ms, scatter 1.18 -> 0.37 ms.
    const int blocks = kLocalBlocks * std::max(ctx->num_sms, 1);
    const bool local = n_cells <= kLocalCells && n >= 4ll * n_cells * blocks;
    const size_t local_smem = (size_t)n_cells * sizeof(int);

    cudaError_t e = cudaMemsetAsync(counts, 0, ((size_t)n_cells + kSortClasses) * sizeof(int), st);
    if (e != cudaSuccess) return cuda_fail(e, "pcc_bin: memset");
    if (n > 0) {
        if (local) launch_pdl(bin_count_local_kernel, blocks, kLocalThreads, local_smem, st, in->cell, n, n_cells, counts, ctx->stats);
        else launch_pdl(bin_count_kernel, (n + 255) / 256, 256, 0, st, in->cell, n, n_cells, counts, ctx->stats);
        note_launches(1);
    }
    launch_pdl(region_sums_kernel, nb, kScanBlock, 0, st, counts, n_cells, slack_abs, slack_rel, sums);
    launch_pdl(region_offsets_kernel, nb, kScanBlock, 0, st, sums, nb, counts, n_cells, slack_abs, slack_rel, out->cell_start,
                                                     out->cell_count, out->cell_added, first, cursor, tot, L);
    note_launches(2);
    // the host learns the totals while the records move: the kernels below
    // check the same limits themselves
    BinTotals* h_tot = static_cast<BinTotals*>(ctx->bin_host);
    e = cudaMemcpyAsync(h_tot, tot, sizeof(BinTotals), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaEventRecord(ctx->bin_event, st);
    if (e != cudaSuccess) return cuda_fail(e, "pcc_bin: totals");
    if (n > 0) {
        const BinLimits lim{tot, (long long)out->capacity};
        const Rec rin{in->ux, in->uy, in->uz, in->w, out->x ? in->x : nullptr, in->pid};
        const MRec ro{out->ux, out->uy, out->uz, out->w, out->x, out->pid};
        if (local) launch_pdl(bin_scatter_local_kernel, blocks, kLocalThreads, local_smem, st, rin, in->cell, n, n_cells, cursor, tmp, lim);
        else launch_pdl(bin_scatter_kernel, (n + 255) / 256, 256, 0, st, rin, in->cell, n, n_cells, cursor, tmp, lim);
        // the fullest cells first: their blocks run longest
        if (n > kSortCap1) launch_sort<16, 32>(ctx, 2, out, first, L, tmp, ro, lim, st);
        if (n > kSortCap0) launch_sort<16, 16>(ctx, 1, out, first, L, tmp, ro, lim, st);
        if (n > kSortWarpCap) launch_sort<4, 16>(ctx, 0, out, first, L, tmp, ro, lim, st);
        launch_pdl(sort_warp_kernel, (n_cells + kSortWarps - 1) / kSortWarps, 32 * kSortWarps, 0, st, 
            out->cell_start, out->cell_count, first, n_cells, tmp, ro, lim);
        note_launches(2);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaEventSynchronize(ctx->bin_event);
    if (e != cudaSuccess) return cuda_fail(e, "pcc_bin: kernels");
    if (h_tot->slots > (long long)out->capacity) {
        set_error("pcc_bin: regions need " + std::to_string(h_tot->slots) + " slots, capacity " +
                  std::to_string(out->capacity));
        return PCC_E_CAPACITY;
    }
    if (h_tot->largest > kMaxCellSort) {
        set_error("pcc_bin: a cell holds " + std::to_string(h_tot->largest) + " particles (max 16384)");
        return PCC_E_CAPACITY;
    }
    return PCC_OK;
}

extern "C" int pcc_append_secondaries(pcc_ctx* ctx, int n_cells, pcc_species* sp, void* stream)
{
    if (!ctx || !sp || n_cells < 1 || !sp->cell_start || !sp->cell_count || !sp->cell_added || !sp->pid) {
        set_error("pcc_append_secondaries: invalid argument");
        return PCC_E_INVALID;
    }
    const int blocks = (n_cells + 255) / 256;
    if (blocks <= 40 * ctx->num_sms) launch_pdl(commit_kernel, blocks, 256, 0, (cudaStream_t)stream, view_of(*sp), n_cells);
    else commit_many_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(view_of(*sp), n_cells);
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PCC_OK : cuda_fail(e, "pcc_append_secondaries");
}

extern "C" int pcc_totals(pcc_ctx* ctx, int n_cells, const pcc_species* sp, int is_photon, double* out,
                          void* stream)
{
    if (!ctx || !sp || !out || n_cells < 1) { set_error("pcc_totals: invalid argument"); return PCC_E_INVALID; }
    // four resident blocks per SM, fewer where the cells do not fill them
    const int most = 4 * std::max(ctx->num_sms, 1), blocks = std::min(most, (n_cells + 7) / 8);
    int rc = ensure_scratch(ctx, (size_t)most * 3 * sizeof(double));   // the same for every call, also in a later capture
    if (rc) return rc;
    double* partial = (double*)ctx->scratch;
    cudaStream_t st = (cudaStream_t)stream;
    if (is_photon) launch_pdl(totals_kernel<true>, blocks, 256, 0, st, *sp, n_cells, partial);
    else launch_pdl(totals_kernel<false>, blocks, 256, 0, st, *sp, n_cells, partial);
    launch_pdl(totals_final_kernel, 1, 96, 0, st, partial, blocks, out);
    note_launches(2);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PCC_OK : cuda_fail(e, "pcc_totals");
}
