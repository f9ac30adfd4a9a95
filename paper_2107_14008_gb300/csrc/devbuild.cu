// Device-side leaf and leaf-pair builder: the GPU counterpart of builder.cpp
// (paper, Section 2: contiguous leaves of at most MAXLEAF particles; Section
// 3.2: the task list grouped by target leaf, with start and length per leaf).
// It produces the arrays the host builder produces, bit for bit and in the
// same order:
//   1. keys      wrap positions into [0, L), 21-bit quantisation, 63-bit Morton key
//   2. sort      stable LSD radix sort of (key, index), 8 passes of 8 bits, one
//                launch each with decoupled look-back
//   3. leaves    a particle's leaf is its first ancestor cell, from the root, that
//                holds at most max_leaf particles; level-21 cells beyond max_leaf
//                are cut into chunks of max_leaf.  Since that cell contains the
//                particle and at most max_leaf particles, its extent is found by
//                binary searches inside a window of +-(max_leaf + 1) sorted keys.
//   4. groups    boxes of 32 consecutive leaves, of 32 such groups, and so on
//   5. pairs     per target leaf and periodic image, a walk of the groups that
//                keeps every leaf whose box comes closer than r_c.  A group's box
//                contains its leaves' boxes, so the kept set is exactly the set of
//                leaves that pass the leaf test, which the host's octree keeps too,
//                in leaf order like the host's Morton-ordered octree walk.
//                Counted in one pass, which also stores each row in a pair cache
//                of 16 words per particle; after a prefix sum of the counts the
//                cached rows are copied into place and only the rows the cache
//                could not hold are walked a second time.  The walk prunes with
//                FP32 bounds (boxes rounded outward, thresholds widened by
//                the rounding of the sums) and falls back to the host's FP64
//                leaf test only where the bounds cannot decide (gap^2 within about
//                1e-5 of the cutoff): FP64 throughput on this part is 1/64 of FP32.
//   6. schedule  target leaves sorted by evaluated work, largest first (stable)
// The FP64 steps use the same operations as the host (no contraction).
//
// Two calls: psr_device_build runs 1-5 (counting) on the caller's scratch and
// reads back the sizes; psr_device_build_finish writes the workspace.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstring>
#include <string>
#include <thread>

#include "kcommon.cuh"

namespace psr {

void set_last_error(const std::string& msg);

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;  // 4096 values per block
constexpr int kMaxLevels = 7;                         // of the groups: 32^6 > 2^28 leaves
constexpr int kDefaultTimeoutMs = 60000;
constexpr int64_t kMaxN = (int64_t)1 << 28;           // digit counts fit the look-back words' 30 bits

// counters in the scratch (int64 words)
enum : int {
    kCntMaxLeaf = 0,
    kCntPairs = 1,
    kCntEvaluated = 2,
    kCntMaxCost = 3,
    kCntMaxRow = 4,
    kCntError = 5,  // bit 0 non-finite input; kErrLookback
    kCntFar = 6,    // well-separated (M2L) entries of the multipole split
    kCntUncached = 7,  // rows the pair cache could not hold (re-walked by the write pass)
    kCntMassDiff = 8,  // nonzero if some particle's mass differs from particle 0's
    kCntMass0 = 9,     // particle 0's mass (the bits of a double)
    kCntLeaves = 10,   // plain octree leaves
    kCntPacked = 11,   // leaves after packing (kCntLeaves without it)
    kCntRedo = 12,     // split: rows whose near and far runs together did not fit
    kCntWords = 13,
};

// The pair cache: the count walk also records each row as runs of
// consecutive leaves of one image (the first leaf with its image code, and the
// run length: 8 bytes, one run for about ten entries on clustered sets), in a
// slot of equal size per row, so that the write step expands the runs instead
// of walking the tree again.  A row with more runs than its slot holds is
// walked again instead; with slots below kMinRuns runs the cache is not used.
constexpr int kCacheWordsPerParticle = 16;
constexpr int kMinRuns = 16;

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct BoxK {
    double L, scale, unit, inv2rs, rc2m;  // rc2m = r_c^2 (1 + 1e-5), the host's margin
    float thi, tlo;  // FP32 thresholds of the walk, above and below rc2m (box_k)
    float theta2;    // multipole split: theta^2 (0: no split)
    float gt2;       //   and theta^2 (2 r_s^2)^2 (the Gaussian length of the kernel)
    float rc2far;    // FP32 at most r_c^2 (1 - 1e-6): a far pair lies wholly inside the cutoff
};

// ------------------------------------------------------------ utilities --

__device__ __forceinline__ uint64_t spread3_d(uint64_t v)
{
    v &= 0x1fffffULL;
    v = (v | (v << 32)) & 0x1f00000000ffffULL;
    v = (v | (v << 16)) & 0x1f0000ff0000ffULL;
    v = (v | (v << 8)) & 0x100f00f00f00f00fULL;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ULL;
    v = (v | (v << 2)) & 0x1249249249249249ULL;
    return v;
}

__device__ __forceinline__ uint32_t compact3_d(uint64_t v)
{
    v &= 0x1249249249249249ULL;
    v = (v | (v >> 2)) & 0x10c30c30c30c30c3ULL;
    v = (v | (v >> 4)) & 0x100f00f00f00f00fULL;
    v = (v | (v >> 8)) & 0x1f0000ff0000ffULL;
    v = (v | (v >> 16)) & 0x1f00000000ffffULL;
    v = (v | (v >> 32)) & 0x1fffffULL;
    return (uint32_t)v;
}

// first index in [lo, hi) with a[index] >= x (hi if none)
__device__ __forceinline__ int64_t lower_bound_u64(const uint64_t* __restrict__ a, int64_t lo,
                                                   int64_t hi, uint64_t x)
{
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// FP64 gap^2 between box A and box B shifted by sh, in the host builder's
// order of operations (explicit roundings: no contraction).
__device__ __forceinline__ double gap2_d(const double* A, const double* B, const double sh[3])
{
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double l = __dadd_rn(B[a], sh[a]), h = __dadd_rn(B[3 + a], sh[a]);
        const double g = fmax(0.0, fmax(__dsub_rn(l, A[3 + a]), __dsub_rn(A[a], h)));
        s = __dadd_rn(s, __dmul_rn(g, g));
    }
    return s;
}

// ------------------------------------------------- single-pass scan and sort --
// Tiles of one launch pass their prefixes on: a block takes the next tile by a
// ticket, so every earlier tile has started; it publishes its own total, then
// adds up the published totals behind it until it meets a published prefix
// (decoupled look-back, Merrill and Garland 2016).  The waits are bounded: one
// that runs out sets kErrLookback (in the build's counters, and the build
// fails, or in the workspace's error word) and its prefix is too small.  What
// follows stays within its arrays: a scan's positions are at most the true
// ones; a sort pass, whose next pass then ranks stale keys against counts of
// the true ones, drops what would lie beyond the end; and the kernels that
// would follow the positions (k_leaf_box, k_rows) do nothing.
// The control words are zeroed by one memset per build call.
#ifndef PSR_SPIN_LIMIT  // a test lets every wait run out
#define PSR_SPIN_LIMIT (1 << 22)
#endif
constexpr int kSpinLimit = PSR_SPIN_LIMIT;
constexpr unsigned kSumReady = 1u << 30, kPrefixReady = 2u << 30, kValueMask = kSumReady - 1;

// Waits for a published word of the current look-back step; 0 when the wait
// runs out: the look-back then stops.
__device__ __forceinline__ unsigned wait_word(const volatile unsigned* p, unsigned* err)
{
    for (int k = 0; k < kSpinLimit; ++k) {
        const unsigned v = *p;
        if (v & (kSumReady | kPrefixReady)) return v;
    }
    atomicOr(err, kErrLookback);
    return 0u;
}

// Block-wide exclusive scan of one value per thread (blockDim.x a multiple of
// 32, at most 1024); sh has 33 words.  Returns the block total.
template <class T>
__device__ T block_exclusive(T v, T* ex, T* sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) sh[w] = inc;
    __syncthreads();
    if (w == 0) {
        const T s = lane < nw ? sh[lane] : T(0);
        T si = s;
        for (int o = 1; o < 32; o <<= 1) {
            const T t = __shfl_up_sync(kFull, si, o);
            if (lane >= o) si += t;
        }
        sh[lane] = si - s;
        if (lane == 31) sh[32] = si;
    }
    __syncthreads();
    *ex = inc - v + sh[w];
    const T total = sh[32];
    __syncthreads();
    return total;
}

// Control of one scan: ticket, then per tile a state word and two sums.
struct ScanCtl {
    unsigned* ticket;   // zeroed, followed by the tile states (zeroed)
    int64_t* sums;      // 2 per tile: own total, prefix through the tile
};

// Exclusive prefix sum of m int64 values (in == out is safe), or of the first
// *m_dev <= m; the total at *total.
__global__ void __launch_bounds__(kScanThreads) k_scan(const int64_t* in, int64_t m, const int64_t* m_dev, int64_t* out,
                                                       int64_t* total, ScanCtl ctl, unsigned* err)
{
    __shared__ int64_t sh[33];
    __shared__ int64_t s_prefix;
    __shared__ unsigned s_tile;
    if (m_dev) m = min(m, *m_dev);
    if (threadIdx.x == 0) s_tile = atomicAdd(ctl.ticket, 1u);
    __syncthreads();
    if ((int64_t)s_tile * kScanTile >= m) return;  // past the end: no tile waits for this one
    const int64_t tile = s_tile, base = tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int64_t loc[kScanItems], v = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        loc[k] = base + k < m ? in[base + k] : 0;
        v += loc[k];
    }
    int64_t ex;
    const int64_t sum = block_exclusive(v, &ex, sh);
    unsigned* const state = ctl.ticket + 1;
    if (threadIdx.x < 32) {  // 32 earlier tiles at a time
        const int lane = threadIdx.x;
        volatile int64_t* sums = ctl.sums;
        if (lane == 0 && tile > 0) {
            sums[2 * tile] = sum;
            __threadfence();
            *(volatile unsigned*)(state + tile) = kSumReady;
        }
        int64_t prefix = 0;
        for (int64_t t0 = tile - 1; t0 >= 0; t0 -= 32) {
            const int64_t t = t0 - lane;
            const unsigned s = t >= 0 ? wait_word(state + t, err) : kPrefixReady;
            __threadfence();
            const unsigned done = __ballot_sync(kFull, !s || (s & kPrefixReady));
            const int stop = done ? __ffs(done) - 1 : 32;  // the nearest tile whose prefix is known
            int64_t v = 0;
            if (t >= 0 && lane < stop) v = sums[2 * t];
            if (t >= 0 && lane == stop && s) v = sums[2 * t + 1];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
            prefix += v;
            if (done) break;
        }
        if (lane == 0) {
            sums[2 * tile + 1] = prefix + sum;
            __threadfence();
            *(volatile unsigned*)(state + tile) = kPrefixReady;
            s_prefix = prefix;
            if (tile == (m + kScanTile - 1) / kScanTile - 1) *total = prefix + sum;
        }
    }
    __syncthreads();
    ex += s_prefix;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < m) out[base + k] = ex;
        ex += loc[k];
    }
}

int64_t scan_tiles(int64_t m) { return (m + kScanTile - 1) / kScanTile; }

int scan_exclusive(const int64_t* in, int64_t* out, int64_t m, const int64_t* m_dev, int64_t* total, ScanCtl ctl,
                   unsigned* err, cudaStream_t st)
{
    k_scan<<<(unsigned)scan_tiles(m), kScanThreads, 0, st>>>(in, m, m_dev, out, total, ctl, err);
    return (int)cudaGetLastError();
}

// Stable LSD radix sort of (64-bit key, int32 value), 8 bits per pass.  One
// launch counts the digits of all passes; each pass is one launch whose tiles
// (4096 items: 256 threads, item t = 512 warp + 32 it + lane) rank their items
// by digit in item order (32 at a time, by votes), put them in digit order in
// shared memory, learn their digits' offsets by look-back (thread d: digit d)
// and write runs of a digit.  2.1 M keys, 8 passes: 40 launches and 0.52 ms
// with counts per tile and their scan before each pass.
// Up to 8192 items sort in one launch of one block, all passes in shared memory.
constexpr int kSortItems = 16, kSortThreads = 256, kSortTile = kSortItems * kSortThreads;
constexpr int kSmallItems = 8, kSmallThreads = 1024, kSmallTile = kSmallItems * kSmallThreads;

struct SortCtl {
    unsigned* hist;    // zeroed: 8 x 256 digit counts, then 8 tickets, then per pass 256 words per tile
    int64_t tiles;     // tiles the status words were sized for
};
__host__ __device__ inline int64_t sort_ctl_words(int passes, int64_t tiles) { return 2048 + 8 + 256 * tiles * passes; }
int64_t sort_tiles(int64_t n) { return (n + kSortTile - 1) / kSortTile; }

__global__ void __launch_bounds__(256) k_sort_hist(const uint64_t* __restrict__ keys, int64_t n, int passes,
                                                   unsigned* __restrict__ hist)
{
    __shared__ unsigned cnt[8][256];
    for (int d = threadIdx.x; d < 2048; d += blockDim.x) cnt[d >> 8][d & 255] = 0;
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[i];
        for (int p = 0; p < passes; ++p) atomicAdd(&cnt[p][(k >> (8 * p)) & 255], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256 * passes; d += blockDim.x)
        if (cnt[d >> 8][d & 255]) atomicAdd(hist + d, cnt[d >> 8][d & 255]);
}

// Ranks of a thread's items among the warp's items of the same digit before
// them, and the warp's digit counts in whist.
template <int ITEMS>
__device__ __forceinline__ void rank_items(const uint64_t* key, int shift, unsigned* whist, unsigned* rank)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const unsigned d = (unsigned)(key[it] >> shift) & 255u;
        unsigned peers = kFull;  // lanes with the same digit, by eight votes
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool on = (d >> b) & 1u;
            const unsigned v = __ballot_sync(kFull, on);
            peers &= on ? v : ~v;
        }
        const unsigned before = whist[d];
        rank[it] = before + __popc(peers & lt);
        __syncwarp();
        if (!(peers & lt)) whist[d] = before + __popc(peers);
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kSortThreads, 3) k_sort_pass(const uint64_t* __restrict__ kin,
                                                            const int32_t* __restrict__ vin,
                                                            uint64_t* __restrict__ kout, int32_t* __restrict__ vout,
                                                            int64_t n, int pass, SortCtl ctl, unsigned* err)
{
    extern __shared__ __align__(16) unsigned char smem_sort[];
    uint64_t* skey = reinterpret_cast<uint64_t*>(smem_sort);
    int32_t* sval = reinterpret_cast<int32_t*>(skey + kSortTile);
    unsigned (*whist)[256] = reinterpret_cast<unsigned (*)[256]>(sval + kSortTile);  // 8 warps
    __shared__ unsigned s_scan[33], s_start[256], s_tile;
    __shared__ int64_t s_base[256];  // global position of the tile's first item of each digit, minus s_start
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, shift = 8 * pass;
    unsigned* tickets = ctl.hist + 2048;
    if (tid == 0) s_tile = atomicAdd(tickets + pass, 1u);
    for (int d = tid; d < 2048; d += kSortThreads) whist[d >> 8][d & 255] = 0;
    __syncthreads();
    const int64_t tile = s_tile, t0 = tile * kSortTile;
    const int count = (int)(n - t0 < kSortTile ? n - t0 : kSortTile);
    uint64_t key[kSortItems];
    int32_t val[kSortItems];
    unsigned rank[kSortItems];
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const int t = w * (kSortItems * 32) + it * 32 + lane;
        // items beyond the end: the last digit's last
        key[it] = t < count ? kin[t0 + t] : ~0ULL;
        val[it] = t < count ? vin[t0 + t] : 0;
    }
    rank_items<kSortItems>(key, shift, whist[w], rank);
    __syncthreads();
    unsigned total = 0;  // of digit tid in the tile; whist: before each warp
#pragma unroll
    for (int k = 0; k < kSortThreads / 32; ++k) {
        const unsigned c = whist[k][tid];
        whist[k][tid] = total;
        total += c;
    }
    const unsigned real = tid == 255 ? total - (unsigned)(kSortTile - count) : total;
    volatile unsigned* status = ctl.hist + 2048 + 8 + 256 * (ctl.tiles * pass + tile);
    status[tid] = (tile == 0 ? kPrefixReady : kSumReady) | real;
    unsigned start;
    block_exclusive(total, &start, s_scan);
    unsigned gstart;  // items of smaller digits in the whole input
    block_exclusive(ctl.hist[256 * pass + tid], &gstart, s_scan);
    s_start[tid] = start;
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const unsigned d = (unsigned)(key[it] >> shift) & 255u;
        const unsigned pos = s_start[d] + whist[w][d] + rank[it];
        skey[pos] = key[it];
        sval[pos] = val[it];
    }
    // items of digit tid in earlier tiles, 16 of them read at a time: with all
    // tiles of a mid-sized sort resident at once, few prefixes are known early
    // and a tile adds up most of the totals before it
    unsigned prefix = 0;
    const unsigned* words = ctl.hist + 2048 + 8 + 256 * ctl.tiles * pass + tid;
    for (int64_t t = tile - 1; t >= 0; t -= 16) {
        unsigned s[16];
#pragma unroll
        for (int k = 0; k < 16; ++k)
            s[k] = t >= k ? *(const volatile unsigned*)(words + 256 * (t - k)) : kPrefixReady;
        bool done = false;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (!done) {
                if (!(s[k] & (kSumReady | kPrefixReady))) s[k] = wait_word(words + 256 * (t - k), err);
                prefix += s[k] & kValueMask;
                done = !s[k] || (s[k] & kPrefixReady);
            }
        if (done) break;
    }
    if (tile > 0) status[tid] = kPrefixReady | (prefix + real);
    s_base[tid] = (int64_t)gstart + prefix - start;
    __syncthreads();
    for (int i = tid; i < count; i += kSortThreads) {
        const uint64_t k = skey[i];
        const int64_t pos = s_base[(unsigned)(k >> shift) & 255u] + i;
        if (pos >= n) continue;  // only after a look-back that ran out
        kout[pos] = k;
        vout[pos] = sval[i];
    }
}
constexpr size_t kSortSmem = (size_t)kSortTile * 12 + 8 * 256 * 4;

__global__ void __launch_bounds__(kSmallThreads) k_sort_small(uint64_t* __restrict__ keys, int32_t* __restrict__ vals,
                                                              int n, int passes)
{
    extern __shared__ __align__(16) unsigned char smem_sort[];
    uint64_t* skey = reinterpret_cast<uint64_t*>(smem_sort);
    int32_t* sval = reinterpret_cast<int32_t*>(skey + kSmallTile);
    unsigned (*whist)[256] = reinterpret_cast<unsigned (*)[256]>(sval + kSmallTile);  // 32 warps
    __shared__ unsigned s_scan[33], s_start[256];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
    uint64_t key[kSmallItems];
    int32_t val[kSmallItems];
    unsigned rank[kSmallItems];
#pragma unroll
    for (int it = 0; it < kSmallItems; ++it) {
        const int t = w * (kSmallItems * 32) + it * 32 + lane;
        key[it] = t < n ? keys[t] : ~0ULL;  // beyond the end: stay last in every pass
        val[it] = t < n ? vals[t] : 0;
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        for (int d = tid; d < nw * 256; d += blockDim.x) whist[d >> 8][d & 255] = 0;
        __syncthreads();
        rank_items<kSmallItems>(key, shift, whist[w], rank);
        __syncthreads();
        unsigned total = 0, start;
        if (tid < 256)
            for (int k = 0; k < nw; ++k) {
                const unsigned c = whist[k][tid];
                whist[k][tid] = total;
                total += c;
            }
        block_exclusive(total, &start, s_scan);
        if (tid < 256) s_start[tid] = start;
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kSmallItems; ++it) {
            const unsigned d = (unsigned)(key[it] >> shift) & 255u;
            const unsigned pos = s_start[d] + whist[w][d] + rank[it];
            skey[pos] = key[it];
            sval[pos] = val[it];
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kSmallItems; ++it) {
            const int t = w * (kSmallItems * 32) + it * 32 + lane;
            key[it] = skey[t];
            val[it] = sval[t];
        }
        __syncthreads();
    }
#pragma unroll
    for (int it = 0; it < kSmallItems; ++it) {
        const int t = w * (kSmallItems * 32) + it * 32 + lane;
        if (t < n) {
            keys[t] = key[it];
            vals[t] = val[it];
        }
    }
}
constexpr size_t kSmallSmem = (size_t)kSmallTile * 12 + 32 * 256 * 4;

// Sorts on bits [0, bits) of the keys (bits <= 64) from (k0, v0), with (k1, v1)
// as the other buffers; the result is in (*kr, *vr).
int radix_sort(uint64_t* k0, int32_t* v0, uint64_t* k1, int32_t* v1, int64_t n, int bits, SortCtl ctl,
               unsigned* err, uint64_t** kr, int32_t** vr, cudaStream_t st)
{
    *kr = k0;
    *vr = v0;
    if (n <= 1) return 0;
    const int passes = (bits + 7) / 8;
    cudaError_t e;
    if (n <= kSmallTile) {
        e = cudaFuncSetAttribute(k_sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
        if (e != cudaSuccess) return (int)e;
        // as many warps as the items fill, at least one thread per digit
        const int warps = (int)((n + 32 * kSmallItems - 1) / (32 * kSmallItems));
        k_sort_small<<<1, 32 * (warps > 8 ? warps : 8), kSmallSmem, st>>>(k0, v0, (int)n, passes);
        return (int)cudaGetLastError();
    }
    e = cudaFuncSetAttribute(k_sort_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortSmem);
    if (e != cudaSuccess) return (int)e;
    const unsigned nb = (unsigned)sort_tiles(n);
    k_sort_hist<<<nb < 1216 ? nb : 1216, 256, 0, st>>>(k0, n, passes, ctl.hist);
    for (int p = 0; p < passes; ++p) {
        k_sort_pass<<<nb, kSortThreads, kSortSmem, st>>>(*kr, *vr, *kr == k0 ? k1 : k0, *vr == v0 ? v1 : v0, n, p,
                                                         ctl, err);
        *kr = *kr == k0 ? k1 : k0;
        *vr = *vr == v0 ? v1 : v0;
    }
    return (int)cudaGetLastError();
}

// The groups of the leaves (see k_groups).
struct Levels {
    int top;                        // the level of one group
    int64_t n[kMaxLevels];          // groups of each level
    const float4* box[kMaxLevels];  // and their boxes (two float4 each; level 0: lout)
};

// Scratch regions (byte offsets); leaf arrays are sized for n leaves (max_leaf 1).
struct Scratch {
    size_t wpos, key0, key1, val0, val1, flag, lid, lfirst, llevel, lkey, lbox, lcnt,
        lfar, lout, lcost, lkey2, lfirst2, llevel2, psize, groups, sums, levels, cnt, sort, scan0, scan1, zero_end,
        lruns, lfruns, cache, bytes;
    int64_t ncache;  // pair cache capacity in runs
};

Scratch scratch_layout(int64_t n)
{
    Scratch s{};
    size_t o = 0;
    const size_t N = (size_t)(n > 0 ? n : 1);
    const size_t nt = (N + kScanTile - 1) / kScanTile;
    s.wpos = o;   o = a256(o + 32 * N);  // x, y, z, m (wrapped, FP64)
    s.key0 = o;   o = a256(o + 8 * N);
    s.key1 = o;   o = a256(o + 8 * N);
    s.val0 = o;   o = a256(o + 4 * N);
    s.val1 = o;   o = a256(o + 4 * N);
    s.flag = o;   o = a256(o + 8 * N);
    s.lid = o;    o = a256(o + 8 * N);
    s.lfirst = o; o = a256(o + 4 * (N + 1));
    s.llevel = o; o = a256(o + 4 * N);
    s.lkey = o;   o = a256(o + 8 * N);
    s.lbox = o;   o = a256(o + 48 * N);
    s.lcnt = o;   o = a256(o + 8 * N);
    s.lfar = o;   o = a256(o + 8 * N);   // far entries per leaf (multipole split)
    s.lout = o;   o = a256(o + 32 * N);  // FP32 leaf box rounded outward, count, rho
    s.lcost = o;  o = a256(o + 8 * N);
    s.lkey2 = o;  o = a256(o + 8 * N);   // packed leaves, before they take the places of the plain ones
    s.lfirst2 = o; o = a256(o + 4 * (N + 1));
    s.llevel2 = o; o = a256(o + 4 * N);
    s.psize = o;  o = a256(o + 4 * N);
    s.groups = o; o = a256(o + 32 * (N / 31 + 2 * kMaxLevels));  // boxes of the groups of all levels
    s.sums = o;   o = a256(o + 2 * 16 * nt);  // two scans' tile sums
    s.levels = o; o = a256(o + sizeof(Levels));
    // zeroed at the start of each build call: counters, then the control words
    // of a sort and of two scans
    s.cnt = o;    o = a256(o + 8 * kCntWords);
    s.sort = o;   o = a256(o + 4 * (size_t)sort_ctl_words(8, (int64_t)((N + kSortTile - 1) / kSortTile)));
    s.scan0 = o;  o = a256(o + 4 * (1 + nt));
    s.scan1 = o;  o = a256(o + 4 * (1 + nt));
    s.zero_end = o;
    s.lruns = o;  o = a256(o + 4 * N);   // runs cached per row (-1: not cached)
    s.lfruns = o; o = a256(o + 4 * N);   // and far ones (multipole split)
    s.ncache = (int64_t)(kCacheWordsPerParticle / 2 * N);
    s.cache = o;  o = a256(o + 8 * (size_t)s.ncache);  // uint2 (first leaf << 5 | code, length)
    // The size callers are told has been about 430 bytes per particle, and is
    // kept (the regions take about 290): scratch of that size serves as before.
    s.bytes = a256(std::max(o, (size_t)430 * N));
    return s;
}

// -------------------------------------------------------- keys and leaves --

// Bound: the FP64 pipe (a warp instruction in 16 SM cycles), so a coordinate
// takes two FP64 instructions: its product with the scale, and floor by adding
// 2^52 rounded down.  Range checks compare the bits of the doubles; only a
// coordinate outside [0, L) takes the FP64 wrap.
__global__ void k_keys(const double* __restrict__ pos, const double* __restrict__ mass, int64_t n,
                       BoxK bx, double m_default, double* __restrict__ wpos, uint64_t* __restrict__ key,
                       int32_t* __restrict__ idx, long long* __restrict__ cnt)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned long long kInfBits = 0x7ff0000000000000ULL, kAbs = 0x7fffffffffffffffULL;
    auto bits = [](double x) { return (unsigned long long)__double_as_longlong(x); };
    uint32_t q[3];
    double v[4];
    bool bad = false;
    for (int a = 0; a < 3; ++a) {
        v[a] = pos[3 * i + a];
        if ((bits(v[a]) & kAbs) >= kInfBits) {
            bad = true;
            v[a] = 0.0;
        }
        if (bits(v[a]) >= bits(bx.L)) {  // outside [0, L), or -0.0
            v[a] = fmod(v[a], bx.L);  // fmod is exact, so values inside keep their bits
            if (v[a] < 0) v[a] += bx.L;
            if (!(v[a] < bx.L)) v[a] = 0.0;
        }
        // floor: the low word of x + 2^52 rounded down (0 <= x <= 2^21)
        const uint32_t f = (uint32_t)__double2loint(__dadd_rd(__dmul_rn(v[a], bx.scale), 4503599627370496.0));
        q[a] = min(f, (1u << kMortonBits) - 1u);
    }
    const double m0 = mass ? mass[0] : m_default;
    v[3] = mass ? mass[i] : m_default;
    if ((bits(v[3]) & kAbs) >= kInfBits) {
        bad = true;
        v[3] = 0.0;
    }
    double2* const w = reinterpret_cast<double2*>(wpos + 4 * i);
    w[0] = make_double2(v[0], v[1]);
    w[1] = make_double2(v[2], v[3]);
    if (bad) atomicOr((unsigned long long*)(cnt + kCntError), 1ULL);
    // one mass for every particle lets the FP32 kernels apply it once per target
    if (bits(v[3]) != bits(m0) && v[3] != m0) atomicOr((unsigned long long*)(cnt + kCntMassDiff), 1ULL);
    if (i == 0) cnt[kCntMass0] = __double_as_longlong(v[3]);
    key[i] = (spread3_d(q[0]) << 2) | (spread3_d(q[1]) << 1) | spread3_d(q[2]);
    idx[i] = (int32_t)i;
}

__device__ __forceinline__ uint64_t cell_prefix(uint64_t k, int level)
{
    const int sh = 3 * (kMortonBits - level);
    return sh >= 64 ? 0ULL : (k >> sh) << sh;
}

// levels (0..21) on which two keys share their cell
__device__ __forceinline__ int shared_levels(uint64_t a, uint64_t b)
{
    const uint64_t x = a ^ b;
    return x ? (__clzll((long long)x) - 1) / 3 : kMortonBits;
}

// Leaf level and leaf-start flag of each sorted particle.  A cell of level l
// around particle i holds more than max_leaf particles exactly when some window
// of max_leaf + 1 consecutive keys that contains i shares its first l levels,
// so the leaf level is one more than the largest number of levels shared by the
// ends of such a window: a sliding maximum over the windows that start at
// i - max_leaf .. i, taken in shared memory by doubling (8 searches of a key
// window per particle before: 124 us for 2.1 M particles).
constexpr int kLevelTile = 512;
__global__ void __launch_bounds__(kLevelTile) k_leaf_level(const uint64_t* __restrict__ key, int64_t n,
                                                           int max_leaf, int64_t* __restrict__ flag,
                                                           int32_t* __restrict__ level)
{
    __shared__ signed char s_max[2][kLevelTile + kMaxLeaf];
    const int64_t i0 = blockIdx.x * (int64_t)kLevelTile, i = i0 + threadIdx.x;
    // window starts i0 - max_leaf .. i0 + kLevelTile - 1
    const int m = kLevelTile + max_leaf;
    for (int k = threadIdx.x; k < m; k += kLevelTile) {
        const int64_t j = i0 - max_leaf + k;
        s_max[0][k] = j >= 0 && j + max_leaf < n ? (signed char)shared_levels(key[j], key[j + max_leaf]) : -1;
    }
    __syncthreads();
    // s_max[cur][k] = max over window starts k .. k + w - 1
    int cur = 0, w = 1;
    for (; 2 * w <= max_leaf + 1; w *= 2, cur ^= 1) {
        for (int k = threadIdx.x; k < m; k += kLevelTile)
            s_max[cur ^ 1][k] = k + w < m ? max(s_max[cur][k], s_max[cur][k + w]) : s_max[cur][k];
        __syncthreads();
    }
    if (i >= n) return;
    // starts i - max_leaf .. i are k = threadIdx.x .. threadIdx.x + max_leaf
    const int d = max(s_max[cur][threadIdx.x], s_max[cur][threadIdx.x + max_leaf + 1 - w]);
    bool start;
    int L = d + 1;
    if (d >= kMortonBits) {  // over-full finest cell: chunks of max_leaf from its start
        L = kMortonBits;
        const int64_t a0 = lower_bound_u64(key, 0, i, key[i]);
        start = ((i - a0) % max_leaf) == 0;
    } else {
        start = i == 0 || shared_levels(key[i - 1], key[i]) < L;
    }
    flag[i] = start ? 1 : 0;
    level[i] = L;
}

__global__ void k_leaf_fill(const int64_t* __restrict__ flag, const int64_t* __restrict__ lid,
                            const int32_t* __restrict__ level, const uint64_t* __restrict__ key,
                            int64_t n, int32_t* __restrict__ lfirst, int32_t* __restrict__ llevel,
                            uint64_t* __restrict__ lkey)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i == n - 1) lfirst[lid[i] + flag[i]] = (int32_t)n;  // lfirst[nl] = n
    if (i >= n || !flag[i]) return;
    const int64_t g = lid[i];
    lfirst[g] = (int32_t)i;
    llevel[g] = level[i];
    lkey[g] = cell_prefix(key[i], level[i]);
}

// Leaf packing (the host builder's rule): consecutive sibling leaves (the
// same level L >= 1 and the same parent cell; chunks of an over-full finest
// cell excluded) share one leaf while their total stays within max_leaf,
// taken greedily in Morton order.  A pack of several leaves takes the
// parent's cell (its level; its key stays that of its first member, whose
// top bits name the parent), a pack of one keeps its own.  The first leaf of each run of
// siblings (at most 8) packs the run: pstart[g] = 1 where a pack begins,
// psize[g] = the leaves of the pack that begins at g.
__device__ __forceinline__ bool packable(const int32_t* __restrict__ llevel,
                                         const uint64_t* __restrict__ lkey, int64_t nl, int64_t g)
{
    const int L = llevel[g];
    if (L < 1) return false;
    if (L == kMortonBits)  // a chunk of an over-full finest cell shares its key with a neighbour
        return !((g > 0 && llevel[g - 1] == L && lkey[g - 1] == lkey[g]) ||
                 (g + 1 < nl && llevel[g + 1] == L && lkey[g + 1] == lkey[g]));
    return true;
}

__device__ __forceinline__ bool siblings(const int32_t* __restrict__ llevel,
                                         const uint64_t* __restrict__ lkey, int64_t nl, int64_t g)
{
    const int L = llevel[g];
    return g > 0 && llevel[g - 1] == L && packable(llevel, lkey, nl, g - 1) &&
           packable(llevel, lkey, nl, g) &&
           cell_prefix(lkey[g - 1], L - 1) == cell_prefix(lkey[g], L - 1);
}

__global__ void k_pack_mark(const int32_t* __restrict__ lfirst, const int32_t* __restrict__ llevel,
                            const uint64_t* __restrict__ lkey, const int64_t* __restrict__ n_plain, int max_leaf,
                            int64_t* __restrict__ pstart, int32_t* __restrict__ psize)
{
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nl = *n_plain;
    if (g >= nl || siblings(llevel, lkey, nl, g)) return;  // not the first of its run
    int64_t start = g;
    int cnt = 0, k = 0;
    for (int64_t j = g; j < nl && (j == g || siblings(llevel, lkey, nl, j)); ++j) {
        const int c = lfirst[j + 1] - lfirst[j];
        if (j == g || cnt + c > max_leaf) {
            if (j > g) psize[start] = k;
            pstart[j] = 1;
            start = j;
            cnt = c;
            k = 1;
        } else {
            pstart[j] = 0;
            cnt += c;
            ++k;
        }
    }
    psize[start] = k;
}

__global__ void k_pack_fill(const int64_t* __restrict__ pstart, const int64_t* __restrict__ pid,
                            const int32_t* __restrict__ psize, const int32_t* __restrict__ lfirst,
                            const int32_t* __restrict__ llevel, const uint64_t* __restrict__ lkey,
                            const int64_t* __restrict__ n_plain, int32_t* __restrict__ lfirst2,
                            int32_t* __restrict__ llevel2, uint64_t* __restrict__ lkey2)
{
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nl = *n_plain;
    if (g == nl - 1) lfirst2[pid[g] + pstart[g]] = lfirst[nl];  // lfirst[packs] = n
    if (g >= nl || !pstart[g]) return;
    const int64_t p = pid[g];
    const bool multi = psize[g] > 1;
    lfirst2[p] = lfirst[g];
    llevel2[p] = multi ? llevel[g] - 1 : llevel[g];
    lkey2[p] = lkey[g];  // the first member's key keeps the keys sorted (an earlier,
                         // deeper sibling subtree can hold keys above the parent's prefix)
}

// Boxes of the leaves, 8 lanes per leaf (leaves average 20 to 40 particles).  Wrapped coordinates are not
// negative, so doubles compare as the integers of their bits (integer minima
// and maxima, off the FP64 pipe; -0.0 counts as the smallest, which equals 0).
// lbox: the FP64 box.  lout, for the walk and the multipole split: the box
// rounded outward in FP32 (lo down, hi up), the particle count and half the
// rounded box's diagonal.
__global__ void k_leaf_box(const int32_t* __restrict__ lfirst, int64_t n,
                           const double* __restrict__ wpos, const int32_t* __restrict__ idx,
                           double* __restrict__ lbox, float4* __restrict__ lout,
                           long long* __restrict__ cnt)
{
    if (cnt[kCntError] & kErrLookback) return;  // lfirst and idx may hold anything
    const int64_t nl = cnt[kCntPacked], step = (int64_t)gridDim.x * blockDim.x >> 3;
    const int sub = threadIdx.x & 7;
    int largest = 0;
    for (int64_t g0 = (blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31)) >> 3; g0 < nl; g0 += step) {
        const int64_t g = g0 + ((threadIdx.x & 31) >> 3);
        const bool live = g < nl;
        const int64_t f = live ? lfirst[g] : 0, e = !live ? 0 : g + 1 < nl ? lfirst[g + 1] : n;
        long long lo[3] = {LLONG_MAX, LLONG_MAX, LLONG_MAX}, hi[3] = {LLONG_MIN, LLONG_MIN, LLONG_MIN};
        for (int64_t k = f + sub; k < e; k += 8) {
            const double2* w = reinterpret_cast<const double2*>(wpos + 4 * (int64_t)idx[k]);
            const double2 xy = w[0], zm = w[1];
            const long long v[3] = {__double_as_longlong(xy.x), __double_as_longlong(xy.y),
                                    __double_as_longlong(zm.x)};
            for (int a = 0; a < 3; ++a) {
                lo[a] = min(lo[a], v[a]);
                hi[a] = max(hi[a], v[a]);
            }
        }
        for (int o = 4; o > 0; o >>= 1)
            for (int a = 0; a < 3; ++a) {
                lo[a] = min(lo[a], __shfl_xor_sync(kFull, lo[a], o));
                hi[a] = max(hi[a], __shfl_xor_sync(kFull, hi[a], o));
            }
        largest = max(largest, (int)(e - f));
        if (!live || sub) continue;
        float ol[3], oh[3], r2 = 0.f;
        for (int a = 0; a < 3; ++a) {
            const double l = __longlong_as_double(lo[a]), h = __longlong_as_double(hi[a]);
            lbox[6 * g + a] = l;
            lbox[6 * g + 3 + a] = h;
            ol[a] = __double2float_rd(l);
            oh[a] = __double2float_ru(h);
            const float ea = __fmul_rn(0.5f, __fsub_rn(oh[a], ol[a]));
            r2 = __fmaf_rn(ea, ea, r2);
        }
        lout[2 * g] = make_float4(ol[0], ol[1], ol[2], __int_as_float((int)(e - f)));
        lout[2 * g + 1] = make_float4(oh[0], oh[1], oh[2], __fsqrt_rn(r2));
    }
    for (int o = 16; o > 0; o >>= 1) largest = max(largest, __shfl_xor_sync(kFull, largest, o));
    if ((threadIdx.x & 31) == 0 && largest) atomicMax(cnt + kCntMaxLeaf, (long long)largest);
}

// ---------------------------------------------------------------- groups --
// A 32-ary tree over the leaves in their (Morton) order: a group of a level is
// 32 consecutive groups of the level below, level 0 the leaves, its box the
// union of theirs (FP32, rounded outward like them), up to one group.
__host__ __device__ inline Levels make_levels(int64_t nl, const float4* lout, const float4* groups)
{
    Levels w{};
    w.box[0] = lout;
    w.n[0] = nl;
    while (w.n[w.top] > 1 && w.top + 1 < kMaxLevels) {
        w.box[w.top + 1] = groups;
        w.n[w.top + 1] = (w.n[w.top] + 31) / 32;
        groups += 2 * w.n[++w.top];
    }
    return w;
}

__device__ __forceinline__ void group_box(const float4* __restrict__ below, int64_t n_below, int64_t g,
                                          float4* __restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t c = 32 * g + lane;
    float lo[3] = {kInf, kInf, kInf}, hi[3] = {-kInf, -kInf, -kInf};
    if (c < n_below) {
        const float4 l = below[2 * c], h = below[2 * c + 1];
        lo[0] = l.x; lo[1] = l.y; lo[2] = l.z;
        hi[0] = h.x; hi[1] = h.y; hi[2] = h.z;
    }
    for (int o = 16; o > 0; o >>= 1)
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(kFull, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(kFull, hi[a], o));
        }
    if (lane == 0) {
        out[2 * g] = make_float4(lo[0], lo[1], lo[2], 0.f);
        out[2 * g + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    }
}

// Boxes of levels 1 (level = 1, a warp per group over the grid) or 2 and up
// (level = 2, one block: at most a 1024th of the leaves); the latter writes the
// levels for the walks.
__global__ void __launch_bounds__(1024) k_groups(int level, const long long* __restrict__ cnt, const float4* lout,
                                                 float4* groups, Levels* out)
{
    const Levels v = make_levels(cnt[kCntPacked], lout, groups);
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 5);
    float4* dst = groups;
    for (int t = 1; t <= v.top; dst += 2 * v.n[t], ++t) {
        if (level == 1 ? t > 1 : t == 1) continue;
        for (int64_t g = w0; g < v.n[t]; g += step) group_box(t == 1 ? lout : dst - 2 * v.n[t - 1], v.n[t - 1], g, dst);
        __syncthreads();
    }
    if (level == 2 && threadIdx.x == 0) *out = v;
}

// ----------------------------------------------------------------- pairs --
// gap^2 between the target box [alo, ahi] (moved by minus the image's shift) and
// the box [blo, bhi], and the largest gap^2 of any point of that box, in FP32.
// Boxes are rounded outward, coordinates and shifts are at most 2 L: each
// component is off by less than 4 places of L (2^-21 L), the root by less than
// 2^-20 L, which the thresholds allow for (box_k).
__device__ __forceinline__ float gap2_f(const float* alo, const float* ahi, float4 blo, float4 bhi)
{
    const float x = fmaxf(fmaxf(blo.x - ahi[0], alo[0] - bhi.x), 0.f);
    const float y = fmaxf(fmaxf(blo.y - ahi[1], alo[1] - bhi.y), 0.f);
    const float z = fmaxf(fmaxf(blo.z - ahi[2], alo[2] - bhi.z), 0.f);
    return fmaf(x, x, fmaf(y, y, z * z));
}
__device__ __forceinline__ float maxgap2_f(const float* alo, const float* ahi, float4 blo, float4 bhi)
{
    const float x = fmaxf(fmaxf(bhi.x - ahi[0], alo[0] - blo.x), 0.f);
    const float y = fmaxf(fmaxf(bhi.y - ahi[1], alo[1] - blo.y), 0.f);
    const float z = fmaxf(fmaxf(bhi.z - ahi[2], alo[2] - blo.z), 0.f);
    return fmaf(x, x, fmaf(y, y, z * z));
}

// The multipole split: leaf J + shift is well separated from leaf I when
// every point of one box lies within r_c of every point of the other (a
// rigorous FP32 upper bound of the largest point-pair distance, from boxes
// rounded outward, against r_c^2 (1 - 1e-6) rounded down: the cutoff then
// removes no pair the expansion includes) and the box centres are R apart
// with theta |R| >= rho_I + rho_J (rho: half the diagonal of the outward
// box), and, with PSR_BUILD_SPLIT_GAUSSIAN, also theta 2 r_s^2 / |R| >=
// rho_I + rho_J: 2 r_s^2 / |R| is the length on which the kernel's Gaussian
// truncation varies (d/dR of -R^2 / 4 r_s^2), shorter than |R| beyond
// r = sqrt(2) r_s (gt2 = theta^2 (2 r_s^2)^2, or infinity without the flag).
// The opening test is taken in FP32 with explicit roundings so that the
// count and the write pass decide alike.
// alo/ahi, ra: box I and its rho; b0 = (lo of box J), b1 = (hi of box J,
// rho_J); sd/su: the shift rounded down and up.
__device__ __forceinline__ bool far_pair(const float* alo, const float* ahi, float ra, float4 b0,
                                         float4 b1, const float* sd, const float* su,
                                         float theta2, float gt2, float rc2far)
{
    const float blo[3] = {b0.x, b0.y, b0.z}, bhi[3] = {b1.x, b1.y, b1.z};
    float m2 = 0.f, d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float bl = __fadd_rd(blo[a], sd[a]), bh = __fadd_ru(bhi[a], su[a]);
        const float mx = fmaxf(__fsub_ru(bh, alo[a]), __fsub_ru(ahi[a], bl));
        m2 = __fmaf_ru(mx, mx, m2);
        const float d = __fsub_rn(__fmul_rn(0.5f, __fadd_rn(bl, bh)),
                                  __fmul_rn(0.5f, __fadd_rn(alo[a], ahi[a])));
        d2 = __fmaf_rn(d, d, d2);
    }
    const float r = __fadd_rn(ra, b1.w);
    const float r2 = __fmul_rn(r, r);
    return d2 > 0.f && m2 < rc2far && __fmul_rn(theta2, d2) >= r2 && __fmul_rn(r2, d2) <= gt2;
}

// The rows.  One WARP per target leaf (consecutive leaves on consecutive warps
// of a persistent grid, whose walks share their loads in L1), which walks the
// groups in order for each periodic image whose root comes close enough: a step
// tests the 32 members of a group, one per lane; of the members of a group of
// groups that survive, those wholly inside are kept as a range and the others
// are walked in turn; of a group of leaves, the kept ones are a bit mask.  So
// the row comes out in order, with every lane at work and no stack but one mask
// per level, which lane t holds for level t.
//   Bound: issue, about 60 steps of 40 instructions a row.  Against the walks
// it replaces (one thread per leaf over a binary radix tree): 17^3 uniform 820
// us, 64^3 NFW 930 us, 128^3 NFW 1.2 ms, split 3.26 + 0.65 ms.
//
// A member is pruned when its gap^2 reaches thi (then the host's FP64 test
// fails for every leaf below) and kept when its (largest) gap^2 is below tlo
// (then the host's FP64 test passes); only the leaves in between take the
// host's FP64 test itself.  One FP32 evaluation within known bounds instead of
// two with directed roundings: 5500 -> 3300 instructions a row.
//
// MODE: count (and, given a pair cache of kslot runs per row, record the row's
// runs: lruns[I] their number, or -1 when the slot is too small), or write the
// rows that were not recorded at rowptr (k_pairs_expand writes the others);
// SPLIT: each kept leaf goes to the near or the far list (far_pair), whose runs
// are recorded apart (lfruns the far ones).
constexpr int kWalkWarps = 4;
constexpr int kWalkBlocks = 8;  // per SM

struct WalkArgs {
    BoxK bx;
    const Levels* levels;
    const int32_t* lfirst;
    const double* lbox;
    int64_t *lcnt, *lcost, *lfar;         // count
    const int64_t *rowptr, *frowptr;      // write
    uint32_t *pairs, *fpairs;
    long long* cnt;
    unsigned* err;
    int32_t *lruns, *lfruns;
    uint2* cache;
    int64_t ncache;  // runs the cache holds, shared out over the rows
};

// runs per row in the pair cache (none below kMinRuns: rows walked twice)
__host__ __device__ inline int cache_slot(int64_t ncache, int64_t nl)
{
    const int64_t ks = ncache / nl;
    return ks < kMinRuns ? 0 : (int)(ks < (1 << 20) ? ks : (1 << 20));
}

// component a of an image code's periodic step, -1, 0 or 1
__device__ __forceinline__ int image_step(uint32_t code, int a)
{
    return (int)(a == 0 ? code / 9u : a == 1 ? (code / 3u) % 3u : code % 3u) - 1;
}

template <bool WRITE, bool SPLIT>
__global__ void __launch_bounds__(32 * kWalkWarps, kWalkBlocks) k_rows(const WalkArgs w)
{
    __shared__ long long s_pairs, s_far, s_eval, s_cost, s_row, s_uncached, s_redo;
    __shared__ Levels s_lv;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const float thi = w.bx.thi, tlo = w.bx.tlo;
    if (threadIdx.x == 0) s_lv = *w.levels;
    if (threadIdx.x == 0) s_pairs = s_far = s_eval = s_cost = s_row = s_uncached = s_redo = 0;
    __syncthreads();
    const float Lf = (float)w.bx.L, Lrd = __double2float_rd(w.bx.L), Lru = __double2float_ru(w.bx.L);
    const float4* const lout = s_lv.box[0];
    const int top = s_lv.top;
    // no rows after a look-back that ran out, and for more leaves than the host accepts
    const bool walk = s_lv.n[0] < (1 << 27) && (WRITE || !(*w.err & kErrLookback));
    const int nl = walk ? (int)s_lv.n[0] : 0;
    const int kslot = nl ? cache_slot(w.ncache, nl) : 0;
    const int W = (int)gridDim.x * kWalkWarps;
    for (int I = (int)blockIdx.x * kWalkWarps + wp; I < nl; I += W) {
        if (WRITE && kslot && w.lruns[I] >= 0) continue;  // recorded: k_pairs_expand writes it
        const float4 t0 = lout[2 * (int64_t)I], t1 = lout[2 * (int64_t)I + 1];
        const float ra = t1.w;  // rho of the outward box
        long long c = 0, cf = 0;  // entries so far (uniform)
        long long src = 0;        // this lane's part of their particles
        long long at = WRITE ? w.rowptr[I] : 0, fat = WRITE && SPLIT ? w.frowptr[I] : 0;
        const long long end = WRITE ? w.rowptr[I + 1] : 0, fend = WRITE && SPLIT ? w.frowptr[I + 1] : 0;
        // pair cache, [0] near and [1] far: runs so far, the open (last) run's
        // first entry and the entry after its end; near runs fill the row's
        // slot from its start, far ones from its end
        const bool caching = !WRITE && kslot;
        uint2* const slot = w.cache + I * (int64_t)kslot;
        int nrun[2] = {0, 0};
        uint32_t run0[2] = {0, 0}, runend[2] = {0xffffffffu, 0xffffffffu};
        int nall = 0;
        uint32_t allend = 0xffffffffu;
        uint32_t code = 0;
        float alo[3], ahi[3];  // the target box moved by minus the image's shift

        // records the leaves of mask M of the 32 from `base` on as runs
        auto record = [&](unsigned M, int base, const bool fr) {
            if (!M) return;
            const bool cont = (M & 1u) && (((uint32_t)base << 5) | code) == runend[fr];
            unsigned B = M & ~(M << 1);  // first leaves of runs
            if (cont) B &= ~1u;
            if (((B >> lane) & 1u) || (cont && lane == 0)) {
                const unsigned rest = ~(M >> lane);
                const int len = rest ? __ffs(rest) - 1 : 32;
                const bool old = cont && lane == 0;
                const int k = old ? nrun[fr] - 1 : nrun[fr] + __popc(B & lt);
                const uint32_t first = old ? run0[fr] : ((uint32_t)(base + lane) << 5) | code;
                if (k < kslot)
                    slot[fr ? kslot - 1 - k : k] = make_uint2(first, (uint32_t)(base + lane + len) - (first >> 5));
            }
            if (B) run0[fr] = ((uint32_t)(base + 31 - __clz(B)) << 5) | code;
            nrun[fr] += __popc(B);
            runend[fr] = ((uint32_t)(base + 32 - __clz(M)) << 5) | code;
        };
        // the leaves of mask M of the 32 from `base` on; b0, b1: this lane's leaf
        auto leaves = [&](unsigned M, int base, float4 b0, float4 b1) {
            if (!M) return;
            const bool mine = (M >> lane) & 1u;
            bool far = false;
            if (SPLIT && mine) {
                const float tlo3[3] = {t0.x, t0.y, t0.z}, thi3[3] = {t1.x, t1.y, t1.z};
                float sd[3], su[3];  // the image's shift rounded down and up
                for (int a = 0; a < 3; ++a) {
                    const int n = image_step(code, a);
                    sd[a] = n < 0 ? -Lru : n > 0 ? Lrd : 0.f;
                    su[a] = n < 0 ? -Lrd : n > 0 ? Lru : 0.f;
                }
                far = far_pair(tlo3, thi3, ra, b0, b1, sd, su, w.bx.theta2, w.bx.gt2, w.bx.rc2far);
            }
            const unsigned F = SPLIT ? __ballot_sync(kFull, far) : 0u, N = M & ~F;
            if (WRITE) {
                const long long p = far ? fat + __popc(F & lt) : at + __popc(N & lt);
                if (mine) {
                    if (p < (far ? fend : end))
                        (far ? w.fpairs : w.pairs)[p] = ((uint32_t)(base + lane) << 5) | code;
                    else
                        atomicOr(w.err, 4u);
                }
                at += __popc(N);
                fat += __popc(F);
                return;
            }
            c += __popc(N);
            cf += __popc(F);
            if (mine && !far) src += __float_as_int(b0.w);
            if (!caching) return;
            record(N, base, false);
            if (SPLIT) {
                record(F, base, true);
                // and the runs of the undivided row, which psr_info.rows_walked_twice
                // counts by
                nall += __popc(M & ~(M << 1)) - ((M & 1u) && (((uint32_t)base << 5) | code) == allend ? 1 : 0);
                allend = ((uint32_t)(base + 32 - __clz(M)) << 5) | code;
            }
        };
        // every leaf of [f, l]
        auto range = [&](int f, int l) {
            if (WRITE || SPLIT) {
                for (int base = f & ~31; base <= l; base += 32) {
                    const int J = base + lane;
                    const bool in = J >= f && J <= l;
                    float4 b0 = make_float4(0.f, 0.f, 0.f, 0.f), b1 = b0;
                    if (SPLIT && in) {
                        b0 = lout[2 * (int64_t)J];
                        b1 = lout[2 * (int64_t)J + 1];
                    }
                    leaves(__ballot_sync(kFull, in), base, b0, b1);
                }
                return;
            }
            c += l - f + 1;
            if (lane == 0) src += w.lfirst[l + 1] - w.lfirst[f];
            if (!caching) return;
            const uint32_t e0 = ((uint32_t)f << 5) | code;
            if (e0 != runend[0]) {
                run0[0] = e0;
                ++nrun[0];
            }
            runend[0] = ((uint32_t)(l + 1) << 5) | code;
            if (lane == 0 && nrun[0] <= kslot) slot[nrun[0] - 1] = make_uint2(run0[0], (runend[0] - run0[0]) >> 5);
        };
        auto set_image = [&](uint32_t cd) {
            code = cd;
            const float sx = (float)image_step(cd, 0) * Lf, sy = (float)image_step(cd, 1) * Lf,
                        sz = (float)image_step(cd, 2) * Lf;
            alo[0] = t0.x - sx; ahi[0] = t1.x - sx;
            alo[1] = t0.y - sy; ahi[1] = t1.y - sy;
            alo[2] = t0.z - sz; ahi[2] = t1.z - sz;
        };
        // the 32 leaves from `base` on
        auto test_leaves = [&](int base) {
            const int J = base + lane;
            float4 b0 = make_float4(0.f, 0.f, 0.f, 0.f), b1 = b0;
            bool keep = false;
            if (J < nl) {
                b0 = lout[2 * (int64_t)J];
                b1 = lout[2 * (int64_t)J + 1];
                const float g2 = gap2_f(alo, ahi, b0, b1);
                keep = g2 < tlo;
                if (!keep && g2 < thi) {
                    const double sh[3] = {image_step(code, 0) * w.bx.L, image_step(code, 1) * w.bx.L,
                                          image_step(code, 2) * w.bx.L};
                    keep = gap2_d(w.lbox + 6 * (int64_t)I, w.lbox + 6 * (int64_t)J, sh) < w.bx.rc2m;
                }
            }
            leaves(__ballot_sync(kFull, keep), base, b0, b1);
        };

        {
            const float4 r0 = s_lv.box[top][0], r1 = s_lv.box[top][1];
            bool in = false, all = false;
            if (lane < kShiftCodes) {  // the root at each image
                set_image((uint32_t)lane);
                in = gap2_f(alo, ahi, r0, r1) < thi;
                all = in && maxgap2_f(alo, ahi, r0, r1) < tlo;
            }
            unsigned images = __ballot_sync(kFull, in);
            const unsigned whole = __ballot_sync(kFull, all);
            while (images) {
                const int image = __ffs(images) - 1;
                images &= images - 1;
                set_image((uint32_t)image);
                if ((whole >> image) & 1u) {
                    range(0, nl - 1);
                    continue;
                }
                if (top <= 1) {
                    test_leaves(0);
                    continue;
                }
                // lane t: members of the open group of level t + 1 still to
                // be taken (todo), which of them are kept whole, the first's index
                unsigned todo = 0, kept = 0;
                int first = 0;
                auto test_group = [&](int t, int base) {  // the members of level t from `base` on
                    const int g = base + lane;
                    bool part = false, full = false;
                    if (g < (int)s_lv.n[t]) {
                        const float4 b0 = s_lv.box[t][2 * (int64_t)g], b1 = s_lv.box[t][2 * (int64_t)g + 1];
                        part = gap2_f(alo, ahi, b0, b1) < thi;
                        full = part && maxgap2_f(alo, ahi, b0, b1) < tlo;
                    }
                    const unsigned P = __ballot_sync(kFull, part), K = __ballot_sync(kFull, full);
                    if (lane == t) {
                        todo = P;
                        kept = K;
                        first = base;
                    }
                };
                int t = top - 1;
                test_group(t, 0);
                while (t < top) {
                    const unsigned m = __shfl_sync(kFull, todo, t);
                    if (!m) {
                        ++t;
                        continue;
                    }
                    const int bit = __ffs(m) - 1;
                    const int g = __shfl_sync(kFull, first, t) + bit;
                    const bool full = (__shfl_sync(kFull, kept, t) >> bit) & 1u;
                    if (lane == t) todo &= todo - 1;
                    if (full) {
                        const long long f = (long long)g << (5 * t), l = ((long long)(g + 1) << (5 * t)) - 1;
                        range((int)f, l < nl ? (int)l : nl - 1);
                    } else if (t == 1) {
                        test_leaves(32 * g);
                    } else {
                        --t;
                        test_group(t, 32 * g);
                    }
                }
            }
        }
        if (WRITE) {
            if ((at != end || (SPLIT && fat != fend)) && lane == 0) atomicOr(w.err, 4u);
        } else {
            for (int o = 16; o > 0; o >>= 1) src += __shfl_xor_sync(kFull, src, o);
            if (lane == 0) {
                const long long cost = src * (w.lfirst[I + 1] - w.lfirst[I]);
                w.lcnt[I] = c;
                w.lcost[I] = cost;
                if (SPLIT) w.lfar[I] = cf;
                if (caching) {
                    const bool fits = nrun[0] + nrun[1] <= kslot;
                    w.lruns[I] = fits ? nrun[0] : -1;
                    if (SPLIT) {
                        w.lfruns[I] = nrun[1];
                        if (!fits) atomicAdd((unsigned long long*)&s_redo, 1ULL);
                    }
                    if (SPLIT ? nall > kslot : !fits) atomicAdd((unsigned long long*)&s_uncached, 1ULL);
                }
                atomicAdd((unsigned long long*)&s_pairs, (unsigned long long)c);
                atomicAdd((unsigned long long*)&s_eval, (unsigned long long)cost);
                if (SPLIT) atomicAdd((unsigned long long*)&s_far, (unsigned long long)cf);
                atomicMax(&s_cost, cost);
                atomicMax(&s_row, c);
            }
        }
    }
    if (WRITE) return;
    __syncthreads();
    if (threadIdx.x == 0) {  // one update per block
        atomicAdd((unsigned long long*)(w.cnt + kCntPairs), (unsigned long long)s_pairs);
        atomicAdd((unsigned long long*)(w.cnt + kCntEvaluated), (unsigned long long)s_eval);
        if (SPLIT) atomicAdd((unsigned long long*)(w.cnt + kCntFar), (unsigned long long)s_far);
        if (s_uncached) atomicAdd((unsigned long long*)(w.cnt + kCntUncached), (unsigned long long)s_uncached);
        if (SPLIT && s_redo) atomicAdd((unsigned long long*)(w.cnt + kCntRedo), (unsigned long long)s_redo);
        atomicMax(w.cnt + kCntMaxCost, s_cost);
        atomicMax(w.cnt + kCntMaxRow, s_row);
    }
}

// Writes the cached rows at rowptr, near runs from the start of each slot or, with
// lfruns, far runs from its end.  One warp per row: lane k loads run k of
// a group of 32 (one coalesced load), a warp scan of the run lengths gives
// each run's first entry, and the group's entries are written 32 at a time,
// entry e finding its run by a binary search over the lanes (shuffles).  A
// run list that does not add up to the row's length (a corrupt cache) sets
// error bit 4.
__global__ void __launch_bounds__(256) k_pairs_expand(int64_t nl, const int32_t* __restrict__ lruns,
                                                      const int32_t* __restrict__ lfruns,
                                                      const uint2* __restrict__ cache, int kslot,
                                                      const int64_t* __restrict__ rowptr,
                                                      uint32_t* __restrict__ pairs,
                                                      unsigned* __restrict__ err)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t I = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); I < nl; I += nw) {
        int nrun = lruns[I];
        if (nrun >= 0 && lfruns) nrun = lfruns[I];
        if (nrun <= 0) continue;  // empty, or walked by the write pass
        const uint2* slot = cache + I * (int64_t)kslot;
        const int64_t row0 = rowptr[I], len = rowptr[I + 1] - row0;
        int64_t done = 0;  // entries of the earlier groups
        bool bad = false;
        for (int r0 = 0; r0 < nrun; r0 += 32) {
            const int nv = nrun - r0 < 32 ? nrun - r0 : 32;
            const int r = r0 + lane;
            const uint2 run = lane < nv ? slot[lfruns ? kslot - 1 - r : r] : make_uint2(0u, 0u);
            int64_t inc = run.y;  // inclusive scan of the run lengths
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t v = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += v;
            }
            const int64_t tot = __shfl_sync(kFull, inc, 31);
            const int64_t exc = inc - run.y;
            if (done + tot > len) {
                bad = true;
                break;
            }
            for (int64_t e0 = 0; e0 < tot; e0 += 32) {
                const int64_t e = e0 + lane;
                int lo = 0;  // the last run whose first entry is <= e
                for (int step = 16; step > 0; step >>= 1) {
                    const int cand = lo + step;
                    const int64_t v = __shfl_sync(kFull, exc, cand & 31);
                    if (cand < nv && v <= e) lo = cand;
                }
                const uint32_t x = __shfl_sync(kFull, run.x, lo);
                const int64_t first = __shfl_sync(kFull, exc, lo);
                if (e < tot) pairs[row0 + done + e] = x + ((uint32_t)(e - first) << 5);
            }
            done += tot;
        }
        if ((bad || done != len) && lane == 0) atomicOr(err, 4u);
    }
}

// Expansion centre and radius of each leaf for the multipole split: the
// centre of its particle box and half the box diagonal; also the centre's
// offset from the leaf's cell centre (lcen, units of L / 2^22) in FP32, so
// that centre differences are an exact integer part plus a small FP32 one.
__global__ void k_fcen(const double* __restrict__ lbox, const int4* __restrict__ lcen,
                       double unit, int64_t nl, double4* __restrict__ fcen,
                       float4* __restrict__ fofs)
{
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= nl) return;
    const double* A = lbox + 6 * g;
    const int4 q = lcen[g];
    const int qc[3] = {q.x, q.y, q.z};
    double c[3], o[3], r2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double ea = __dmul_rn(0.5, __dsub_rn(A[3 + a], A[a]));
        c[a] = __dmul_rn(0.5, __dadd_rn(A[a], A[3 + a]));
        o[a] = __dsub_rn(c[a], __dmul_rn((double)qc[a], unit));
        r2 = __dadd_rn(r2, __dmul_rn(ea, ea));
    }
    const double r = __dsqrt_rn(r2);
    fcen[g] = make_double4(c[0], c[1], c[2], r);
    fofs[g] = make_float4((float)o[0], (float)o[1], (float)o[2], (float)r);
}

// --------------------------------------------------------------- payload --
// (float)x in integer arithmetic: the FP64 pipe's conversion takes as long as
// its arithmetic.  Round to nearest even; results outside the normal FP32 range
// (and 0) take the conversion itself.
__device__ __forceinline__ float to_float(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32), e = (hi >> 20) & 0x7ffu;
    if (e < 1023u - 126u || e > 1023u + 126u) return (float)x;
    // exponent rebiased, mantissa cut to 23 bits; a carry of the rounding runs into the exponent
    unsigned f = (unsigned)((b << 1) >> 30) - ((1023u - 127u) << 23);
    const unsigned rest = (unsigned)b & 0x1fffffffu;
    f += rest > 0x10000000u || (rest == 0x10000000u && (f & 1u));
    return __uint_as_float(f | (hi & 0x80000000u));
}

// The workspace arrays of one leaf: leaf record, integer cell centre (units
// L / 2^22), leaf-local FP32 coordinates in units of 2 r_s, FP64 copy, perm.
__global__ void k_payload(const int32_t* __restrict__ lfirst, const int32_t* __restrict__ llevel,
                          const uint64_t* __restrict__ lkey, int64_t nl, int64_t n, BoxK bx,
                          const double* __restrict__ wpos, const int32_t* __restrict__ idx,
                          float4* __restrict__ pf, double4* __restrict__ pd,
                          int32_t* __restrict__ perm, int4* __restrict__ leaf,
                          int4* __restrict__ lcen)
{
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;  // 8 lanes per leaf
    const int sub = threadIdx.x & 7;
    if (g >= nl) return;
    const int64_t f = lfirst[g], e = g + 1 < nl ? lfirst[g + 1] : n;
    const int L = llevel[g];
    const uint64_t k = lkey[g];
    const int sh = kMortonBits - L;
    const uint32_t sc = 1u << sh;
    const int32_t cx = (int32_t)((2 * (compact3_d(k >> 2) >> sh) + 1) * sc);
    const int32_t cy = (int32_t)((2 * (compact3_d(k >> 1) >> sh) + 1) * sc);
    const int32_t cz = (int32_t)((2 * (compact3_d(k) >> sh) + 1) * sc);
    if (sub == 0) {
        leaf[g] = make_int4((int)f, (int)(e - f), 0, 0);
        lcen[g] = make_int4(cx, cy, cz, L);
    }
    const double c[3] = {__dmul_rn((double)cx, bx.unit), __dmul_rn((double)cy, bx.unit),
                         __dmul_rn((double)cz, bx.unit)};
    for (int64_t q = f + sub; q < e; q += 8) {
        const int64_t p = idx[q];
        const double2* w = reinterpret_cast<const double2*>(wpos + 4 * p);
        const double2 xy = w[0], zm = w[1];
        pf[q] = make_float4(to_float(__dmul_rn(__dsub_rn(xy.x, c[0]), bx.inv2rs)),
                            to_float(__dmul_rn(__dsub_rn(xy.y, c[1]), bx.inv2rs)),
                            to_float(__dmul_rn(__dsub_rn(zm.x, c[2]), bx.inv2rs)), to_float(zm.y));
        if (pd) pd[q] = make_double4(xy.x, xy.y, zm.x, zm.y);
        perm[q] = (int32_t)p;
    }
}

// schedule keys: maxcost - cost ascending = cost descending; equal costs keep
// leaf order (stable sort); and the costs into the workspace
__global__ void k_sched_keys(const int64_t* __restrict__ lcost, int64_t nl, long long maxcost,
                             uint64_t* __restrict__ key, int32_t* __restrict__ val,
                             int64_t* __restrict__ cost)
{
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= nl) return;
    cost[g] = lcost[g];
    key[g] = (uint64_t)(maxcost - lcost[g]);
    val[g] = (int32_t)g;
}

// The sorted schedule into the workspace, and for each level the number of
// items whose work exceeds its line (the keys ascend, so they come first).
struct HeavyLines {
    long long cost[kHeavyLevels];
};
__global__ void k_sched_out(const uint64_t* __restrict__ key, const int32_t* __restrict__ val,
                            int64_t nl, long long maxcost, HeavyLines heavy,
                            int32_t* __restrict__ items, int* __restrict__ n_heavy)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= nl) return;
    items[i] = val[i];
    const long long mine = maxcost - (long long)key[i];
    const long long next = i + 1 < nl ? maxcost - (long long)key[i + 1] : -1;
    for (int l = 0; l < kHeavyLevels; ++l)
        if (mine > heavy.cost[l] && next <= heavy.cost[l]) n_heavy[l] = (int)(i + 1);
}

// blocks of a row walk: a warp per leaf (at most nl of them), up to one wave
unsigned walk_blocks(int64_t nl, int sms)
{
    return (unsigned)std::min<int64_t>((nl + kWalkWarps - 1) / kWalkWarps, kWalkBlocks * (int64_t)sms);
}

unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

int dfail(int code, const std::string& msg)
{
    set_last_error(msg);
    return code;
}

int dcuda(int e, const char* what)
{
    return dfail(PSR_E_CUDA, std::string(what) + ": " + cudaGetErrorString((cudaError_t)e));
}

// Bounded host wait for the stream, then a copy of `bytes` to the host.
// Waits (at most timeout_ms) for the work queued on st, then copies a
// small device block to the host.  The wait polls without sleeping for
// its first 2 ms (the build's steps between waits take about a millisecond,
// and a sleeping poll wakes up to tens of microseconds late), then every 20
// microseconds.
int read_back(void* dst, const void* src, size_t bytes, cudaStream_t st, int timeout_ms)
{
    auto t0 = std::chrono::steady_clock::now();
    for (;;) {
        cudaError_t e = cudaStreamQuery(st);
        if (e == cudaSuccess) break;
        if (e != cudaErrorNotReady) return dcuda(e, "cudaStreamQuery");
        double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        if (ms > timeout_ms) return dfail(PSR_E_TIMEOUT, "device build did not finish within the timeout");
        if (ms > 2.0) std::this_thread::sleep_for(std::chrono::microseconds(20));
    }
    cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? PSR_OK : dcuda(e, "cudaMemcpyAsync (device build counters)");
}

float float_at_least(double x)
{
    float f = (float)x;
    return (double)f < x ? std::nextafter(f, INFINITY) : f;
}

float float_at_most(double x)
{
    float f = (float)x;
    return (double)f > x ? std::nextafter(f, -INFINITY) : f;
}

BoxK box_k(const psr_box& b)
{
    BoxK k;
    k.L = b.L;
    k.scale = std::ldexp(1.0, kMortonBits) / b.L;
    k.unit = std::ldexp(b.L, -kCentreShift);
    k.inv2rs = 1.0 / (2.0 * b.r_s);
    k.rc2m = b.r_c * b.r_c * (1.0 + 1e-5);
    // the walk's thresholds: the FP32 gaps are within 2^-20 L (gap2_f), their
    // squares' sums within 1e-6
    const double g = std::sqrt(k.rc2m), slack = std::ldexp(b.L, -20), in = g > slack ? g - slack : 0.0;
    k.thi = float_at_least((g + slack) * (g + slack) * (1.0 + 1e-6));
    k.tlo = float_at_most(in * in * (1.0 - 1e-6));
    k.theta2 = 0.0f;
    k.gt2 = 0.0f;
    k.rc2far = float_at_most(b.r_c * b.r_c * (1.0 - 1e-6));
    return k;
}

}  // namespace
}  // namespace psr

using namespace psr;

extern "C" {

int psr_device_build_scratch_bytes(int64_t n, size_t* bytes)
{
    if (!bytes || n < 1 || n > kMaxN)
        return dfail(PSR_E_ARG, "need 1 <= n <= 2^28 and a non-null output");
    *bytes = scratch_layout(n).bytes;
    return PSR_OK;
}

}  // extern "C"

namespace {

int device_build(const double* d_pos, const double* d_mass, int64_t n, const psr_box* box,
                 int max_leaf, int flags, double theta, void* d_scratch, size_t scratch_bytes,
                 void* stream, int timeout_ms, psr_leaves** out)
{
    auto t0 = std::chrono::steady_clock::now();
    if (!out) return dfail(PSR_E_ARG, "null output");
    *out = nullptr;
    if (!d_pos || !box || n < 1 || n > kMaxN)
        return dfail(PSR_E_ARG, "null argument or n outside [1, 2^28]");
    if (max_leaf < 1 || max_leaf > kMaxLeaf) return dfail(PSR_E_ARG, "max_leaf must be in [1, 64]");
    if (flags & ~(PSR_BUILD_NO_FP64 | PSR_BUILD_UNPACKED | PSR_BUILD_SPLIT_GAUSSIAN))
        return dfail(PSR_E_ARG, "the device builder takes PSR_BUILD_NO_FP64, PSR_BUILD_UNPACKED "
                                "and PSR_BUILD_SPLIT_GAUSSIAN (no ORB)");
    if (!(std::isfinite(box->L) && box->L > 0) || !(std::isfinite(box->r_s) && box->r_s > 0) ||
        !std::isfinite(box->G))
        return dfail(PSR_E_ARG, "L, r_s must be finite and positive");
    if (!(box->r_c > 0) || !(box->r_c < box->L)) return dfail(PSR_E_CUTOFF, "need 0 < r_c < L");
    if (!(box->r_c >= 1e-10) || !(box->L <= 1e12))
        return dfail(PSR_E_ARG, "the device builder takes r_c >= 1e-10 and L <= 1e12");
    const Scratch S = scratch_layout(n);
    if (!d_scratch || scratch_bytes < S.bytes || (reinterpret_cast<uintptr_t>(d_scratch) & 255))
        return dfail(PSR_E_WORKSPACE, "scratch must be 256-byte aligned and at least " +
                                          std::to_string(S.bytes) + " bytes");
    if (timeout_ms <= 0) timeout_ms = kDefaultTimeoutMs;
    cudaStream_t st = (cudaStream_t)stream;
    char* s = static_cast<char*>(d_scratch);
    double* wpos = (double*)(s + S.wpos);
    uint64_t* k0 = (uint64_t*)(s + S.key0);
    uint64_t* k1 = (uint64_t*)(s + S.key1);
    int32_t* v0 = (int32_t*)(s + S.val0);
    int32_t* v1 = (int32_t*)(s + S.val1);
    int64_t* flag = (int64_t*)(s + S.flag);
    int64_t* lid = (int64_t*)(s + S.lid);
    int32_t* lfirst = (int32_t*)(s + S.lfirst);
    int32_t* llevel = (int32_t*)(s + S.llevel);
    uint64_t* lkey = (uint64_t*)(s + S.lkey);
    double* lbox = (double*)(s + S.lbox);
    float4* lout = (float4*)(s + S.lout);
    int64_t* lcnt = (int64_t*)(s + S.lcnt);
    int64_t* lcost = (int64_t*)(s + S.lcost);
    int64_t* sums = (int64_t*)(s + S.sums);
    long long* cnt = (long long*)(s + S.cnt);
    int64_t* const n_plain = (int64_t*)cnt + kCntLeaves;
    int64_t* const n_packed = (int64_t*)cnt + kCntPacked;
    BoxK bx = box_k(*box);
    bx.theta2 = (float)(theta * theta);
    bx.gt2 = (flags & PSR_BUILD_SPLIT_GAUSSIAN) ? (float)(theta * theta * 4.0 * std::pow(box->r_s, 4))
                                               : INFINITY;

    int e;
    unsigned* const err = (unsigned*)(cnt + kCntError);
    const SortCtl sctl{(unsigned*)(s + S.sort), sort_tiles(n)};
    const ScanCtl scan0{(unsigned*)(s + S.scan0), sums}, scan1{(unsigned*)(s + S.scan1), sums + 2 * scan_tiles(n)};
    if ((e = (int)cudaMemsetAsync(s + S.cnt, 0, S.zero_end - S.cnt, st))) return dcuda(e, "cudaMemsetAsync");
    k_keys<<<nblk(n, 256), 256, 0, st>>>(d_pos, d_mass, n, bx, 1.0 / (double)n, wpos, k0, v0, cnt);
    if ((e = (int)cudaGetLastError())) return dcuda(e, "key kernel");
    uint64_t* kr;  // (k0, v0): one launch or eight passes
    int32_t* vr;
    if ((e = radix_sort(k0, v0, k1, v1, n, 3 * kMortonBits, sctl, err, &kr, &vr, st)))
        return dcuda(e, "radix sort");
    k_leaf_level<<<nblk(n, kLevelTile), kLevelTile, 0, st>>>(k0, n, max_leaf, flag, v1);
    if ((e = (int)cudaGetLastError())) return dcuda(e, "leaf level kernel");
    if ((e = scan_exclusive(flag, lid, n, nullptr, n_plain, scan0, err, st))) return dcuda(e, "scan");
    k_leaf_fill<<<nblk(n, 256), 256, 0, st>>>(flag, lid, v1, k0, n, lfirst, llevel, lkey);
    if ((e = (int)cudaGetLastError())) return dcuda(e, "leaf fill kernel");
    // From here on the kernels take the number of leaves from the counters: the
    // host waits once, for all counts (two more waits, to size the launches,
    // left the GPU idle for about 50 us of a build).
    const bool pack = !(flags & PSR_BUILD_UNPACKED);
    if (pack) {
        // pack sibling leaves: marks, pack ids, the packed leaves' arrays
        int64_t* pstart = flag;
        int64_t* pid = lid;
        int32_t* psize = (int32_t*)(s + S.psize);
        k_pack_mark<<<nblk(n, 256), 256, 0, st>>>(lfirst, llevel, lkey, n_plain, max_leaf, pstart, psize);
        if ((e = scan_exclusive(pstart, pid, n, n_plain, n_packed, scan1, err, st))) return dcuda(e, "scan");
        k_pack_fill<<<nblk(n, 256), 256, 0, st>>>(pstart, pid, psize, lfirst, llevel, lkey, n_plain,
                                                  (int32_t*)(s + S.lfirst2), (int32_t*)(s + S.llevel2),
                                                  (uint64_t*)(s + S.lkey2));
        if ((e = (int)cudaGetLastError())) return dcuda(e, "leaf packing kernel");
        lfirst = (int32_t*)(s + S.lfirst2);
    } else if ((e = (int)cudaMemcpyAsync(n_packed, n_plain, 8, cudaMemcpyDeviceToDevice, st))) {
        return dcuda(e, "cudaMemcpyAsync");
    }
    int dev = 0, sms = 0;
    if ((e = (int)cudaGetDevice(&dev))) return dcuda(e, "cudaGetDevice");
    if ((e = (int)cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)))
        return dcuda(e, "cudaDeviceGetAttribute");
    const unsigned wave = 8 * (unsigned)sms;
    k_leaf_box<<<std::min(nblk(8 * n, 256), wave), 256, 0, st>>>(lfirst, n, wpos, v0, lbox, lout, cnt);
    float4* const groups = (float4*)(s + S.groups);
    Levels* const levels = (Levels*)(s + S.levels);
    k_groups<<<std::min(nblk(n, 256), wave), 256, 0, st>>>(1, cnt, lout, groups, levels);
    k_groups<<<1, 1024, 0, st>>>(2, cnt, lout, groups, levels);
    if ((e = (int)cudaGetLastError())) return dcuda(e, "group kernel");
    WalkArgs wa{};
    wa.bx = bx;
    wa.levels = levels;
    wa.lfirst = lfirst;
    wa.lbox = lbox;
    wa.lcnt = lcnt;
    wa.lcost = lcost;
    wa.lfar = (int64_t*)(s + S.lfar);
    wa.cnt = cnt;
    wa.err = err;
    wa.lruns = (int32_t*)(s + S.lruns);
    wa.lfruns = (int32_t*)(s + S.lfruns);
    wa.cache = (uint2*)(s + S.cache);
    wa.ncache = S.ncache;
    if (theta > 0.0) k_rows<false, true><<<walk_blocks(n, sms), 32 * kWalkWarps, 0, st>>>(wa);
    else k_rows<false, false><<<walk_blocks(n, sms), 32 * kWalkWarps, 0, st>>>(wa);
    if ((e = (int)cudaGetLastError())) return dcuda(e, "pair count kernel");
    long long c[kCntWords];
    if ((e = read_back(c, cnt, sizeof c, st, timeout_ms))) return e;
    if (c[kCntError] & 1) return dfail(PSR_E_ARG, "non-finite position or mass");
    if (c[kCntError] & kErrLookback) return dfail(PSR_E_DEVICE, "a look-back of the build's scans or sorts ran out");
    const int64_t np = c[kCntLeaves], nl = c[kCntPacked];
    if (np < 1 || np > n || nl >= (1 << 27)) return dfail(PSR_E_ARG, "leaf count out of range");
    if (nl < 1 || nl > np) return dfail(PSR_E_DEVICE, "leaf packing failed");
    const int kslot = cache_slot(S.ncache, nl);
    if (c[kCntPairs] >= ((int64_t)1 << 32) || c[kCntFar] >= ((int64_t)1 << 32))
        return dfail(PSR_E_ARG, "more than 2^32 leaf pairs");

    Leaves* h = new (std::nothrow) Leaves();
    if (!h) return dfail(PSR_E_NOMEM, "out of host memory");
    try {
        h->nbox = 1;
        h->boxes.assign(box, box + 1);
        h->box_first = {0, n};
        h->n = n;
        h->max_leaf_req = max_leaf;
        h->flags = flags;
        h->n_leaves = nl;
        h->n_pairs = c[kCntPairs];
        h->evaluated = c[kCntEvaluated];
        h->max_leaf = (int)c[kCntMaxLeaf];
        h->max_row = (int)c[kCntMaxRow];
        h->has_pd = !(flags & PSR_BUILD_NO_FP64);
        h->device_built = true;
        h->has_far = theta > 0.0;
        h->theta = theta;
        h->n_far = theta > 0.0 ? c[kCntFar] : 0;
        h->boxdev = {box_constants(*box)};
        h->equal_mass = c[kCntMassDiff] == 0;
        if (h->equal_mass) {
            double m0;
            std::memcpy(&m0, &c[kCntMass0], sizeof m0);
            h->boxdev[0].m_eq = (float)m0;
        }
        parts_rule(c[kCntMaxCost], h->evaluated, nl, h->max_leaf, &h->boxdev[0]);
        h->lay = make_layout(*h);
    } catch (const std::bad_alloc&) {
        delete h;
        return dfail(PSR_E_NOMEM, "out of host memory");
    }
    h->db_scratch = s;
    h->max_cost = c[kCntMaxCost];
    h->db_kslot = kslot;
    h->db_uncached = kslot ? c[kCntUncached] : nl;
    h->db_redo = !kslot ? nl : theta > 0.0 ? c[kCntRedo] : c[kCntUncached];
    h->build_seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    *out = reinterpret_cast<psr_leaves*>(h);
    return PSR_OK;
}

}  // namespace

extern "C" {

int psr_device_build(const double* d_pos, const double* d_mass, int64_t n, const psr_box* box,
                     int max_leaf, int flags, void* d_scratch, size_t scratch_bytes, void* stream,
                     int timeout_ms, psr_leaves** out)
{
    return device_build(d_pos, d_mass, n, box, max_leaf, flags, 0.0, d_scratch, scratch_bytes,
                        stream, timeout_ms, out);
}

int psr_device_build_split(const double* d_pos, const double* d_mass, int64_t n,
                           const psr_box* box, int max_leaf, int flags, double theta,
                           void* d_scratch, size_t scratch_bytes, void* stream, int timeout_ms,
                           psr_leaves** out)
{
    if (out) *out = nullptr;
    if (!(theta > 0.0 && theta <= 1.0)) return dfail(PSR_E_ARG, "theta must be in (0, 1]");
    return device_build(d_pos, d_mass, n, box, max_leaf, flags, theta, d_scratch, scratch_bytes,
                        stream, timeout_ms, out);
}

int psr_device_build_finish(psr_leaves* hh, void* d_ws, size_t bytes, void* stream)
{
    Leaves* h = reinterpret_cast<Leaves*>(hh);
    if (!h || !h->db_scratch) return dfail(PSR_E_STATE, "not a pending device build");
    if (!d_ws || bytes < h->lay.total || (reinterpret_cast<uintptr_t>(d_ws) & 255))
        return dfail(PSR_E_WORKSPACE, "workspace must be 256-byte aligned and at least " +
                                          std::to_string(h->lay.total) + " bytes");
    const int64_t n = h->n, nl = h->n_leaves;
    const Scratch S = scratch_layout(n);
    char* s = h->db_scratch;
    char* w = static_cast<char*>(d_ws);
    const Layout& L = h->lay;
    cudaStream_t st = (cudaStream_t)stream;
    const BoxK bx = box_k(h->boxes[0]);
    int e, dev = 0, sms = 0;
    if ((e = (int)cudaGetDevice(&dev))) return dcuda(e, "cudaGetDevice");
    if ((e = (int)cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)))
        return dcuda(e, "cudaDeviceGetAttribute");
    // the control words first: the pair write kernel reports into the error
    // word that psr_check reads
    if ((e = (int)cudaMemsetAsync(w + L.ctrl, 0, kCtrlWords * 4, st))) return dcuda(e, "cudaMemsetAsync");
    const bool pack = !(h->flags & PSR_BUILD_UNPACKED);
    const int32_t* lfirst = (const int32_t*)(s + (pack ? S.lfirst2 : S.lfirst));
    k_payload<<<nblk(8 * nl, 256), 256, 0, st>>>(
        lfirst, (const int32_t*)(s + (pack ? S.llevel2 : S.llevel)),
        (const uint64_t*)(s + (pack ? S.lkey2 : S.lkey)), nl, n, bx,
        (const double*)(s + S.wpos), (const int32_t*)(s + S.val0), (float4*)(w + L.pf),
        h->has_pd ? (double4*)(w + L.pd) : nullptr, (int32_t*)(w + L.perm), (int4*)(w + L.leaf),
        (int4*)(w + L.lcen));
    if ((e = (int)cudaGetLastError())) return dcuda(e, "payload kernel");
    // row pointers: exclusive scan of the row lengths, then the total
    int64_t* rowptr = (int64_t*)(w + L.rowptr);
    int64_t* sums = (int64_t*)(s + S.sums);
    unsigned* const err = (unsigned*)(w + L.ctrl) + kCtrlError;
    const SortCtl sctl{(unsigned*)(s + S.sort), sort_tiles(n)};
    const ScanCtl scan0{(unsigned*)(s + S.scan0), sums}, scan1{(unsigned*)(s + S.scan1), sums + 2 * scan_tiles(n)};
    if ((e = (int)cudaMemsetAsync(s + S.sort, 0, S.zero_end - S.sort, st))) return dcuda(e, "cudaMemsetAsync");
    if ((e = scan_exclusive((const int64_t*)(s + S.lcnt), rowptr, nl, nullptr, rowptr + nl, scan0, err, st)))
        return dcuda(e, "scan");
    const double* lbox = (const double*)(s + S.lbox);
    int64_t* frow = h->has_far ? (int64_t*)(w + L.frow) : nullptr;
    if (h->has_far) {
        if ((e = scan_exclusive((const int64_t*)(s + S.lfar), frow, nl, nullptr, frow + nl, scan1, err, st)))
            return dcuda(e, "scan");
        k_fcen<<<nblk(nl, 128), 128, 0, st>>>(lbox, (const int4*)(w + L.lcen), bx.unit, nl,
                                              (double4*)(w + L.fcen), (float4*)(w + L.fofs));
        if ((e = (int)cudaGetLastError())) return dcuda(e, "expansion centre kernel");
    }
    WalkArgs wa{};
    wa.bx = bx;
    wa.levels = (const Levels*)(s + S.levels);
    wa.lfirst = lfirst;
    wa.lbox = lbox;
    wa.rowptr = rowptr;
    wa.frowptr = frow;
    wa.pairs = (uint32_t*)(w + L.pairs);
    wa.err = err;
    wa.lruns = (int32_t*)(s + S.lruns);
    wa.cache = (uint2*)(s + S.cache);
    wa.ncache = S.ncache;
    if (h->has_far) {
        wa.fpairs = (uint32_t*)(w + L.fpairs);
        wa.bx.theta2 = (float)(h->theta * h->theta);
        wa.bx.gt2 = (h->flags & PSR_BUILD_SPLIT_GAUSSIAN)
                        ? (float)(h->theta * h->theta * 4.0 * std::pow(h->boxes[0].r_s, 4))
                        : INFINITY;
    }
    // rows the count walk cached are expanded; the rest are walked again
    if (h->db_kslot) {
        k_pairs_expand<<<nblk(nl, 8), 256, 0, st>>>(nl, wa.lruns, nullptr, wa.cache, h->db_kslot, rowptr, wa.pairs,
                                                    wa.err);
        if (h->has_far)
            k_pairs_expand<<<nblk(nl, 8), 256, 0, st>>>(nl, wa.lruns, (const int32_t*)(s + S.lfruns), wa.cache,
                                                        h->db_kslot, frow, wa.fpairs, wa.err);
        if ((e = (int)cudaGetLastError())) return dcuda(e, "pair expand kernel");
    }
    if (h->db_redo > 0) {
        if (h->has_far) k_rows<true, true><<<walk_blocks(nl, sms), 32 * kWalkWarps, 0, st>>>(wa);
        else k_rows<true, false><<<walk_blocks(nl, sms), 32 * kWalkWarps, 0, st>>>(wa);
    }
    if ((e = (int)cudaGetLastError())) return dcuda(e, "pair write kernel");
    // schedule: the particle sort buffers are free again (values in int32
    // views of the flag / lid regions, both >= 4 nl bytes)
    uint64_t* k0 = (uint64_t*)(s + S.key0);
    uint64_t* k1 = (uint64_t*)(s + S.key1);
    int32_t* v0 = (int32_t*)(s + S.flag);
    int32_t* v1 = (int32_t*)(s + S.lid);
    k_sched_keys<<<nblk(nl, 256), 256, 0, st>>>((const int64_t*)(s + S.lcost), nl,
                                                (long long)h->max_cost, k0, v0, (int64_t*)(w + L.cost));
    int bits = 1;
    while (bits < 63 && ((uint64_t)h->max_cost >> bits)) ++bits;
    uint64_t* kr;
    int32_t* vr;
    if ((e = radix_sort(k0, v0, k1, v1, nl, bits, sctl, err, &kr, &vr, st)))
        return dcuda(e, "schedule sort");
    HeavyLines heavy;
    for (int l = 0; l < kHeavyLevels; ++l) heavy.cost[l] = heavy_cost(l, h->evaluated);
    k_sched_out<<<nblk(nl, 256), 256, 0, st>>>(kr, vr, nl, (long long)h->max_cost, heavy,
                                               (int32_t*)(w + L.items), (int*)(w + L.ctrl) + kCtrlHeavy);
    if ((e = (int)cudaGetLastError())) return dcuda(e, "schedule kernel");
    if ((e = (int)cudaMemcpyAsync(w + L.boxes, h->boxdev.data(), sizeof(BoxDev),
                                  cudaMemcpyHostToDevice, st)))
        return dcuda(e, "cudaMemcpyAsync");
    h->d_ws = w;
    h->ws_bytes = bytes;
    h->uploaded = true;
    h->table = h->core = h->fine = h->t64 = TableState{};
    h->sm_count = sms;
    h->device = dev;
    h->db_scratch = nullptr;
    return PSR_OK;
}

}  // extern "C"
