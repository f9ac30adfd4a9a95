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

// This warp's entries of a row: all of them, or with split its share among
// the warps of its group.
__device__ __forceinline__ void row_part(const FwdArgs& a, int I, bool split, long long& e0, long long& re)
{
    e0 = a.rowptr[I];
    re = a.rowptr[I + 1];
    if (split) {
        const int len = (int)(re - e0), W = a.group, w = (threadIdx.x >> 5) % W;
        re = e0 + (long long)len * (w + 1) / W;
        e0 += (long long)len * w / W;
    }
}

// The next item of a persistent launch.  The schedule's first *a.heavy items
// (their work is more than a fraction of what one warp of a full chip gets,
// see heavy_cost) are taken by groups of a.group warps, one ticket a group
// (split stays true; s_it: one word per group), the rest by single warps; the
// ticket on which a group leaves the first phase goes to its first warp.
// Returns false when no item is left.  Which items are split, and how, is
// fixed by the schedule alone, so results do not depend on the order in which
// blocks run.
template <bool SPLIT>
__device__ __forceinline__ bool next_item(const FwdArgs& a, unsigned* ticket, bool& split,
                                          int n_heavy, volatile int* s_it, int& it)
{
    if (SPLIT && split) {
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
