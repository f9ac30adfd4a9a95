// Device helpers shared by the P2P kernels of libpsr.
#pragma once

#include <cuda_runtime.h>

#include "psr_internal.h"

namespace psr {

constexpr unsigned kFull = 0xffffffffu;
// rint by the 1.5 * 2^23 trick: for |t| < 2^22, (t + M) - M == rint(t) and the
// low mantissa bits of (t + M) hold rint(t) + 2^22.
constexpr float kMagic = 12582912.0f;
constexpr int kMagicBits = 0x4B400000;
// The FP32 kernels work in coordinates scaled by 1 / (2 r_s), so the pair
// distance is the paper's x = r / (2 r_s) directly.  A tiny constant is added
// to r^2 so that the self pair (d = 0 exactly) gives a finite 1/r and hence a
// zero term; it moves any pair farther than 1e-7 x-units by < 1e-6 relative.
constexpr float kEps2 = 1e-20f;
constexpr float kTwoOverSqrtPi = 1.1283791670955126f;
constexpr float kInf = __builtin_huge_valf();

__device__ __forceinline__ void set_error(unsigned* ctrl, unsigned bit)
{
    atomicOr(ctrl + kCtrlError, bit);
}

// Shift code (nx+1)*9 + (ny+1)*3 + (nz+1) -> n components.
__device__ __forceinline__ void decode_shift(unsigned code, int& nx, int& ny, int& nz)
{
    nx = (int)(code / 9u) - 1;
    ny = (int)((code / 3u) % 3u) - 1;
    nz = (int)(code % 3u) - 1;
}

// Two-sum (Knuth): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    float bp = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// Grid-wide end of a persistent launch: the last block to finish resets the
// work ticket and the done counter, so the next launch (or a graph replay)
// starts from zero without a memset.
__device__ __forceinline__ void persistent_exit(unsigned* ticket, unsigned* done)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned d = atomicAdd(done, 1u);
        if (d == gridDim.x - 1) {
            atomicExch(ticket, 0u);
            atomicExch(done, 0u);
            __threadfence();
        }
    }
}

// PTX rsqrt.approx.ftz.f32: one SFU instruction, max relative error 2^-22.9.
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 32-bit shared-window address of a shared-memory pointer.
__device__ __forceinline__ unsigned smem_u32(const void* p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

// Loads from read-only shared data (the interpolation table): no ordering.
__device__ __forceinline__ float lds_f1(unsigned a)
{
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float2 lds_f2(unsigned a)
{
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ float4 lds_f4(unsigned a)
{
    float4 v;
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
// Barrier of the calling warp's group of `warps` consecutive warps (the block
// holds a whole number of groups; barrier 0 is left to __syncthreads).
__device__ __forceinline__ void group_sync(int warps)
{
    const int id = 1 + (int)(threadIdx.x >> 5) / warps;
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(32 * warps) : "memory");
}

// How a row's sums are formed: over `parts` consecutive parts of its entries, each
// by itself from zero, added in order lane by lane.  Which rows have parts, and how
// many, is fixed by the row and its box alone (parts_rule), so that neither the
// other boxes, the launch's shape nor its shard move a bit of the result.  Who
// forms them is the launch's choice (FwdArgs::rows), and each choice has kernel
// instances of its own.  The FP32 pair loops have no register to spare, so what an
// item needs to know after its pair loop waits in one word of shared memory, the
// unused last word of the warp's target box.
__device__ __forceinline__ volatile unsigned* row_word(float4* box)
{
    return reinterpret_cast<volatile unsigned*>(box) + 7;
}

// no row has parts
struct WholeRow {
    __device__ __forceinline__ void park(float4*) const {}
    __device__ static __forceinline__ WholeRow at(float4*) { return WholeRow{}; }
    __device__ static constexpr bool joint() { return false; }
    __device__ static constexpr bool in_turn() { return false; }
    __device__ static constexpr int parts() { return 1; }
    __device__ static constexpr int part() { return 0; }
    __device__ static __forceinline__ int leaf(int I) { return I; }
    __device__ static constexpr bool last() { return true; }
    __device__ __forceinline__ void next(float4*) {}
};
// the warps of a group side by side, one part each (at least as many warps as
// parts); rows without parts also by single warps
struct JointRow {
    unsigned v;  // parts | warp << 4 | joint << 8
    __device__ __forceinline__ void park(float4* box) const
    {
        if ((threadIdx.x & 31) == 0) *row_word(box) = v;
        __syncwarp();
    }
    __device__ static __forceinline__ JointRow at(float4* box) { return JointRow{*row_word(box)}; }
    __device__ __forceinline__ bool joint() const { return v >> 8; }
    __device__ static constexpr bool in_turn() { return false; }
    __device__ __forceinline__ int parts() const { return (int)(v & 15u); }
    __device__ __forceinline__ int part() const { return (int)((v >> 4) & 15u); }
    __device__ static __forceinline__ int leaf(int I) { return I; }
    __device__ static constexpr bool last() { return true; }
    __device__ __forceinline__ void next(float4*) {}
};
// one warp all parts in turn
struct TurnRow {
    unsigned v;  // leaf << 5 | log2(parts) << 3 | part
    __device__ __forceinline__ void park(float4* box) const
    {
        if ((threadIdx.x & 31) == 0) *row_word(box) = v;
        __syncwarp();
    }
    __device__ static __forceinline__ TurnRow at(float4* box) { return TurnRow{*row_word(box)}; }
    __device__ static constexpr bool joint() { return false; }
    __device__ __forceinline__ bool in_turn() const { return v & 24u; }
    __device__ __forceinline__ int parts() const { return 1 << ((v >> 3) & 3u); }
    __device__ __forceinline__ int part() const { return (int)(v & 7u); }
    __device__ __forceinline__ int leaf(int) const { return (int)(v >> 5); }
    __device__ __forceinline__ bool last() const { return part() + 1 >= parts(); }
    __device__ __forceinline__ void next(float4* box)
    {
        ++v;
        __syncwarp();
        park(box);
    }
};

template <int ROWS>
__device__ __forceinline__ auto row_work(const FwdArgs& a, int I, int box, bool split)
{
    if constexpr (ROWS == kRowsWhole) {
        return WholeRow{};
    } else {
        const BoxDev& bx = a.boxes[box];
        int parts = a.cost[I] > bx.above[a.kind] ? bx.parts[a.kind] : 1;
        if (parts < 1 || parts > (ROWS == kRowsInTurn ? 8 : split ? a.group : 1)) {
            set_error(a.ctrl, kErrParts);
            parts = 1;
        }
        if constexpr (ROWS == kRowsJoint)
            return JointRow{split ? (unsigned)(parts | (int)(threadIdx.x >> 5) % a.group << 4 | 256) : (unsigned)parts};
        else
            return TurnRow{(unsigned)I << 5 | (unsigned)(31 - __clz(parts)) << 3};
    }
}

// The entries of this warp's present part of a row.
template <class Work>
__device__ __forceinline__ void row_part(const FwdArgs& a, int I, const Work& w, long long& e0, long long& re)
{
    I = w.leaf(I);
    e0 = a.rowptr[I];
    re = a.rowptr[I + 1];
    if (w.joint() || w.in_turn()) {
        const int len = (int)(re - e0), part = w.part(), parts = w.parts();
        re = part < parts ? e0 + (long long)len * (part + 1) / parts : e0;
        e0 += part < parts ? (long long)len * part / parts : 0;
    }
}

// A sum over parts, and the 8-byte word it is kept in: FP64, or a compensated
// FP32 pair.
template <int ACC>
struct PartSum {
    double v = 0.0;
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void load(const volatile char* p)
    {
        if (ACC == PSR_ACC_FP64) {
            v = *reinterpret_cast<const volatile double*>(p);
        } else {
            hi = reinterpret_cast<const volatile float*>(p)[0];
            lo = reinterpret_cast<const volatile float*>(p)[1];
        }
    }
    __device__ __forceinline__ void add(const PartSum& o)
    {
        if (ACC == PSR_ACC_FP64) {
            v += o.v;
        } else {
            float s, e;
            two_sum(hi, o.hi, s, e);
            hi = s;
            lo += o.lo + e;
        }
    }
    __device__ __forceinline__ float scaled(float g) const
    {
        return ACC == PSR_ACC_FP64 ? (float)(v * (double)g) : (hi + lo) * g;
    }
};

// The sums of the parts that one warp has formed so far.  In local memory, by
// volatile accesses: they are touched once a part, and in registers they push the
// pair loop's values out (batch of 64 boxes 7.01 -> 6.76 ms).
template <int ACC, int N>
struct PartTotals {
    volatile double v[ACC == PSR_ACC_FP64 ? N : 1];
    volatile float hi[ACC == PSR_ACC_FP64 ? 1 : N], lo[ACC == PSR_ACC_FP64 ? 1 : N];
    __device__ __forceinline__ PartSum<ACC> get(int i) const
    {
        PartSum<ACC> p;
        if (ACC == PSR_ACC_FP64) {
            p.v = v[i];
        } else {
            p.hi = hi[i];
            p.lo = lo[i];
        }
        return p;
    }
    __device__ __forceinline__ void put(int i, const PartSum<ACC>& p)
    {
        if (ACC == PSR_ACC_FP64) {
            v[i] = p.v;
        } else {
            hi[i] = p.hi;
            lo[i] = p.lo;
        }
    }
    // adds p to sum i (part 0: to zero) and returns it
    __device__ __forceinline__ PartSum<ACC> add(int i, int part, const PartSum<ACC>& p)
    {
        PartSum<ACC> t;
        if (part) t = get(i);
        t.add(p);
        put(i, t);
        return t;
    }
};

// End of a row that a group of warps shares: every lane of every warp has left the
// sums of its part (NC words a target; word(t, s, i): the byte offset of target t's
// component i in stream s) in the warp's region, `stride` bytes apart, `base` this
// warp's.  One thread a target and component adds each lane's over the parts, then
// the S streams, in the order in which one warp adds them, and hands the sum to
// write(t, i, sum).  next_item's barrier frees the regions.
template <int NC, int ACC, class Work, class Word, class Write>
__device__ __forceinline__ void join_parts(const FwdArgs& a, const Work& w, int n_targets, int S, const char* base,
                                           int stride, Word word, Write write)
{
    group_sync(a.group);
    const int gw = (int)(threadIdx.x >> 5) % a.group;
    base -= gw * stride;
    for (int u = 32 * gw + (int)(threadIdx.x & 31); u < NC * n_targets; u += 32 * a.group) {
        const int t = u / NC, i = u - NC * t;
        PartSum<ACC> sum;
        for (int s = 0; s < S; ++s) {
            PartSum<ACC> lane, part;
            for (int k = 0; k < w.parts(); ++k) {
                part.load(base + k * stride + word(t, s, i));
                lane.add(part);
            }
            if (s) sum.add(lane);
            else sum = lane;
        }
        write(t, i, sum);
    }
}

// The next item of a persistent launch.  The schedule's first *a.heavy items
// (their work is more than a fraction of what one warp of a full chip gets,
// see heavy_cost) are taken by groups of a.group warps, one ticket a group
// (split stays true; s_it: one word per group), the rest by single warps; the
// ticket on which a group leaves the first phase goes to its first warp.
// Returns false when no item is left.
template <int ROWS>
__device__ __forceinline__ bool next_item(const FwdArgs& a, unsigned* ticket, bool& split,
                                          int n_heavy, volatile int* s_it, int& it)
{
    if (ROWS == kRowsJoint && split) {
        const int g = (threadIdx.x >> 5) / a.group;
        const bool first = threadIdx.x - g * 32 * a.group < 32;
        group_sync(a.group);  // the group's last item is combined
        if (first && (threadIdx.x & 31) == 0)
            s_it[g] = (int)atomicAdd(ticket, 1u) * a.item_stride + a.item_offset;
        group_sync(a.group);
        it = s_it[g];
        if (it < n_heavy) return true;  // n_heavy <= n_items
        split = false;
        if (first) return it < a.n_items;
    }
    int t = 0;
    if ((threadIdx.x & 31) == 0) t = (int)atomicAdd(ticket, 1u) * a.item_stride + a.item_offset;
    it = __shfl_sync(kFull, t, 0);
    return it < a.n_items;
}

// Targets per lane for the scalar kernel, by cost per useful pair.  One
// iteration of a stream evaluates one staged source against the lane's R
// targets, kPairInstr instructions per target plus kSourceInstr for the
// source itself (its shared-memory load and the loop), and the warp's
// S_R = floor(32 / ceil(n_I / R)) streams serve n_I S_R pairs per iteration:
// the cost per pair is (kPairInstr R + kSourceInstr) / S_R, the cheapest R
// wins, ties going to the smaller.  The per-source term is set to 0, the
// measured best: with 3, 6 or 10 the rule moves leaves of 25-32 particles to
// R = 2 or 3 at equal lane fill, and whole launches ran 2-5 % slower.  So a
// larger R is taken only where it fills strictly more lanes: R = 3 for
// leaves of 3, 6, 9, 11-12, 17-18, 21-24 (24 = 8 lanes x 3 targets x 4
// streams) and 33-48 particles (11-16 lanes x 2 streams, against 17-24 lanes
// x 1 for R = 2; 6 % faster on leaves of up to 64); R = 2 for 19-20 and
// 49-64.  R = 1 needs n_I <= 32; R = 3 needs tiles of at least 128
// particles (its final reduction takes 3 x 768 B of the warp's staging
// buffer).
constexpr int kPairInstr = 20, kSourceInstr = 0;
__device__ __forceinline__ int targets_per_lane(int n, int cap)
{
    int best = 0, bnum = 0, bS = 1;
#pragma unroll
    for (int R = 1; R <= 3; ++R) {
        const int T = (n + R - 1) / R;
        if (T > 32 || (R == 3 && cap < 128)) continue;
        const int S = 32 / T, num = kPairInstr * R + kSourceInstr;
        if (best == 0 || num * bS < bnum * S) {
            best = R;
            bnum = num;
            bS = S;
        }
    }
    return best;
}

// Morton-order source payload of the cotangent: cs[k] = (c[perm[k]], 0).
template <typename T, typename T4>
__global__ void gather_cot_kernel(const T* __restrict__ cot, const int32_t* __restrict__ perm,
                                  T4* __restrict__ cs, long long n)
{
    long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= n) return;
    long long i = perm[k];
    T4 v;
    v.x = cot[3 * i];
    v.y = cot[3 * i + 1];
    v.z = cot[3 * i + 2];
    v.w = 0;
    cs[k] = v;
}

}  // namespace psr
