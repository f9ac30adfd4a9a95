// FP64 P2P kernels: what the forward (p2p_fwd_f64.cu) and the adjoint
// (p2p_adj_f64.cu) share.
//
// Bound.  The FP64 pipe issues one warp instruction in 16 cycles of an SM (1/64
// of the FP32 rate), so a launch's time is the FP64 instructions of its pair
// evaluations and nothing else; integer and FP32 work beside them is free up to
// some 60 instructions per FP64 one.  The kernels therefore
//  - stage a row's sources in shared memory, culled against the target leaf's
//    box as the FP32 kernels do (here in FP64, 9 instructions per 32 sources),
//    so that 88 % of the evaluated pairs of the 128^3 NFW set lie within the
//    cutoff instead of 74 %;
//  - fill the lanes with 1, 2 or 3 targets each (targets_per_lane): 92 % of
//    them busy on packed leaves, where a power-of-two stream width left 63 %
//    for a leaf of 20;
//  - take T(x) (and exp(-x^2)) from a Taylor table about the nearest of nodes
//    0.0044 apart, to fifth order, formed from erfc and exp in FP64: the first
//    term left out is below 2e-17, an eighth of T's last place;
//  - take 1/r from the FP64 rsqrt estimate (about 2^-20) and one third-order
//    step, y (1 + e/2 + 3 e^2/8) with e = 1 - r^2 y^2: five instructions, and
//    compare with the cutoff as integers (positive doubles order as their bits).
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "kcommon.cuh"

namespace psr {

constexpr double kMagic64 = 6755399441055744.0;  // 1.5 * 2^52: x + kMagic64 holds rint(x) in its low bits
constexpr int kT64Terms = 6;

__device__ __forceinline__ long long bits64(double x) { return __double_as_longlong(x); }

__device__ __forceinline__ double rsqrt64(double r2)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(r2));
    const double e = fma(-(r2 * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// 0 < r2 < rc2
__device__ __forceinline__ bool inside64(double r2, long long rc2m1)
{
    return (unsigned long long)(bits64(r2) - 1) < (unsigned long long)rc2m1;  // rc2m1 = bits(rc2) - 1
}

// entry (clamped to kmax) and offset from its node, in node spacings, of
// distance r (us nodes per unit of r)
__device__ __forceinline__ int node64(double r, double us, int kmax, double& f)
{
    const double fk = fma(r, us, kMagic64);
    f = fma(r, us, -(fk - kMagic64));
    return min(__double2loint(fk), kmax);
}

template <int DEG>
__device__ __forceinline__ double horner64(const double* __restrict__ c, double f)
{
    double v = c[DEG];
#pragma unroll
    for (int m = DEG - 1; m >= 0; --m) v = fma(f, v, c[m]);
    return v;
}

// A warp's shared memory: cap staged sources of NV double2 ({x, y}, {z, m} and
// for the adjoint {c_x, c_y}, {c_z, 0}), 32 entry records, and the target box
// (centre, half extents, squared cutoff).
constexpr int kMeta64Bytes = 32 * 8 + 8 * 8;
__host__ __device__ constexpr int warp64_bytes(int nv, int cap) { return 16 * nv * cap + kMeta64Bytes; }

// The target box of the lanes' R targets; the squared cutoff is widened by what
// the FP64 rounding of box and coordinates can move a distance.
template <int R>
__device__ __forceinline__ void cull_box64(const double4* xi, const bool* act, double r_c, double L,
                                           double* __restrict__ box)
{
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (act[r]) {
            lo[0] = fmin(lo[0], xi[r].x); hi[0] = fmax(hi[0], xi[r].x);
            lo[1] = fmin(lo[1], xi[r].y); hi[1] = fmax(hi[1], xi[r].y);
            lo[2] = fmin(lo[2], xi[r].z); hi[2] = fmax(hi[2], xi[r].z);
        }
    for (int o = 16; o > 0; o >>= 1)
        for (int i = 0; i < 3; ++i) {
            lo[i] = fmin(lo[i], __shfl_xor_sync(kFull, lo[i], o));
            hi[i] = fmax(hi[i], __shfl_xor_sync(kFull, hi[i], o));
        }
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        const double w = r_c * (1.0 + 1e-9) + 1e-14 * L;
        for (int i = 0; i < 3; ++i) {
            box[i] = 0.5 * (lo[i] + hi[i]);
            box[3 + i] = 0.5 * (hi[i] - lo[i]);
        }
        box[6] = w * w;
    }
    __syncwarp();
}

// Stages one chunk of the row from entry e0 on (the scheme of stage_chunk in
// fwd_f32_common.cuh): returns the entries taken, nst the staged sources, each
// at its periodic image.
template <int NV, bool CULL>
__device__ __forceinline__ int stage64(const FwdArgs& a, long long e0, long long re, double L, int cap,
                                       double2* __restrict__ stage, int2* __restrict__ meta,
                                       const double* __restrict__ box, int& nst)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const double4* __restrict__ pd = reinterpret_cast<const double4*>(a.pd);
    const double4* __restrict__ cs = reinterpret_cast<const double4*>(a.cot_sorted);
    const int4* __restrict__ leaf = reinterpret_cast<const int4*>(a.leaf);
    const unsigned* __restrict__ prow = a.pairs + e0;
    const int rem = (int)min(re - e0, (long long)0x7fffffff);
    int nk = 0, eb = 0;
    for (;;) {
        const int e = eb + lane;
        int cnt = 0, first = 0, code = 13;
        if (e < rem) {
            const unsigned ent = prow[e];
            const int J = (int)(ent >> 5);
            code = (int)(ent & 31u);
            unsigned bad = J >= a.n_leaves ? kErrLeafIndex : code >= kShiftCodes ? kErrShiftCode : 0u;
            if (!bad) {
                const int4 lj = leaf[J];
                cnt = lj.y;
                first = lj.x;
                if (lj.x < 0 || lj.y < 1 || lj.y > a.max_leaf || (long long)lj.x + lj.y > a.n)
                    bad = kErrParticleRange;
            }
            if (bad) {  // one particle that is dropped below
                set_error(a.ctrl, bad);
                cnt = 1;
                first = 0;
                code = -1;
            }
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        const int ntake = __popc(__ballot_sync(kFull, e < rem && incl <= cap - nk));
        if (ntake == 0) break;
        const int nraw = __shfl_sync(kFull, incl, ntake - 1), excl = incl - cnt;
        if (lane < ntake) meta[lane] = make_int2(first - excl, code);
        __syncwarp();
        int C = 0;  // entry starts before this round
        for (int p0 = 0; p0 < nraw; p0 += 32) {
            const int rel = excl - p0;
            const unsigned M =
                __reduce_or_sync(kFull, (lane < ntake && rel >= 0 && rel < 32) ? (1u << rel) : 0u);
            const int k = C + __popc(M & ((2u << lane) - 1u)) - 1;
            C += __popc(M);
            const int p = p0 + lane;
            bool keep = p < nraw;
            double4 v = make_double4(0.0, 0.0, 0.0, 0.0), c = v;
            if (keep) {
                const int2 m = meta[k];
                const int src = m.x + p;
                v = pd[src];
                if (NV == 4) c = cs[src];
                if (m.y != 13 && m.y >= 0) {
                    int nx, ny, nz;
                    decode_shift((unsigned)m.y, nx, ny, nz);
                    v.x = fma((double)nx, L, v.x);
                    v.y = fma((double)ny, L, v.y);
                    v.z = fma((double)nz, L, v.z);
                }
                keep = m.y >= 0;
                if (CULL) {
                    double g[3] = {fabs(v.x - box[0]) - box[3], fabs(v.y - box[1]) - box[4],
                                   fabs(v.z - box[2]) - box[5]};
#pragma unroll
                    for (int i = 0; i < 3; ++i) g[i] = bits64(g[i]) < 0 ? 0.0 : g[i];
                    keep = keep && bits64(fma(g[0], g[0], fma(g[1], g[1], g[2] * g[2]))) < bits64(box[6]);
                }
            }
            const unsigned K = __ballot_sync(kFull, keep);
            if (keep) {
                double2* d = stage + NV * (nk + __popc(K & lt));
                d[0] = make_double2(v.x, v.y);
                d[1] = make_double2(v.z, v.w);
                if (NV == 4) {
                    d[2] = make_double2(c.x, c.y);
                    d[NV - 1] = make_double2(c.z, 0.0);
                }
            }
            nk += __popc(K);
        }
        __syncwarp();
        eb += ntake;
        if (ntake < 32 || eb >= rem) break;
    }
    __syncwarp();
    nst = nk;
    return eb;
}

// Adds the S stream partials (NC components per target slot) of each target
// through the warp's staging buffer, in stream order, and hands each target's
// sums to write(target, sums); with split, the sums of the group's warps are
// added after that, in warp order (stride: bytes between the warps' buffers).
template <int NC, int R, class Write>
__device__ __forceinline__ void finish64(const FwdArgs& a, int4 li, const double (*acc)[NC], const bool* act,
                                         int lane, int s, int S, int T, double2* __restrict__ stage,
                                         bool split, int stride, Write write)
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        volatile double* red = reinterpret_cast<volatile double*>(stage) + 32 * NC * r;
#pragma unroll
        for (int i = 0; i < NC; ++i) red[NC * lane + i] = acc[r][i];
        __syncwarp();
        if (s == 0 && act[r]) {
            double v[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) v[i] = acc[r][i];
            for (int t = 1; t < S; ++t)
#pragma unroll
                for (int i = 0; i < NC; ++i) v[i] += red[NC * (lane + t * T) + i];
            if (split) {  // streams t >= 1 sit above the first T entries
#pragma unroll
                for (int i = 0; i < NC; ++i) red[NC * lane + i] = v[i];
            } else {
                write(li.x + lane + T * r, v);
            }
        }
        __syncwarp();
    }
    if (!split) return;
    group_sync(a.group);
    const int nw = a.group, gw = (threadIdx.x >> 5) % nw;
    const char* base = reinterpret_cast<const char*>(stage) - gw * stride;
    for (int t = 32 * gw + lane; t < li.y; t += 32 * nw) {
        double v[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) v[i] = 0.0;
        for (int w = 0; w < nw; ++w) {
            const volatile double* o = reinterpret_cast<const volatile double*>(base + w * stride) +
                                       32 * NC * (t / T) + NC * (t % T);
#pragma unroll
            for (int i = 0; i < NC; ++i) v[i] += o[i];
        }
        write(li.x + t, v);
    }
}

// a checked schedule entry; false (and the error word) if it is out of range
__device__ __forceinline__ bool item64(const FwdArgs& a, int it, int lane, int& I, int4& li)
{
    I = a.items[it];
    if (I < 0 || I >= a.n_leaves) {
        if (lane == 0) set_error(a.ctrl, kErrItemIndex);
        return false;
    }
    li = reinterpret_cast<const int4*>(a.leaf)[I];
    if (li.x < 0 || li.y <= 0 || li.y > a.max_leaf || li.y > 64 || (long long)li.x + li.y > a.n ||
        li.z < 0 || li.z >= a.nbox) {
        if (lane == 0) set_error(a.ctrl, kErrParticleRange);
        return false;
    }
    return true;
}

}  // namespace psr
