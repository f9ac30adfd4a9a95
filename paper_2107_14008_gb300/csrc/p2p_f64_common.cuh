// FP64 P2P kernels: what the forward (p2p_fwd_f64.cu) and the adjoint
// (p2p_adj_f64.cu) share.
//
// Bound.  The FP64 pipe issues one warp instruction in 16 cycles of an SM (1/64
// of the FP32 rate), so a launch's time is the FP64 instructions of its pair
// evaluations and nothing else; integer and FP32 work beside them is free up to
// some 60 instructions per FP64 one.  The kernels therefore
//  - stage a row's sources in shared memory, culled against the target leaf's
//    box as the FP32 kernels do (here in FP64, 9 instructions per 32 sources);
//  - find each lane's pairs within the cutoff by an FP32 test first (rounded
//    outward; a bit mask per lane), so that every lane then takes its own next
//    pair: of uniform sets, whose leaves are large against the cutoff, 42 % of
//    the lanes had a pair within it when all took the same source.  The
//    entries are staged in strides over the row, which evens out the lanes'
//    counts in a chunk (58 % against 49 % in row order);
//  - fill the lanes with 1, 2 or 3 targets each (targets_per_lane): 92 % of
//    them busy on packed leaves, where a power-of-two stream width left 63 %
//    for a leaf of 20;
//  - take T(x) (and exp(-x^2)) from a table of degree-5 polynomials about nodes
//    1/256 apart (plain64_kernel), the Taylor series formed from erfc and exp in
//    FP64 with its sixth and seventh terms folded into the lower ones: off by
//    4e-19 at most, relative to T by 3e-18 at x = 2.25, 1e-16 at 3.5 and 3e-15 at
//    the table's end, x = 5.32.  Pairs beyond it (instances with TAIL, for
//    cutoffs beyond it) take erfc and exp;
//  - take 1/r from the FP64 rsqrt estimate y (off by 9e-7) and the binomial series
//    of (1 - e)^(-1/2), e = 1 - r^2 y^2, to second order, and r from r^2 y the same
//    way: six instructions for both, 1/r within 0.75 of its last place (1/r^2 by a
//    series of its own, one instruction more, cost 1 % of the adjoint and made
//    sums no more exact), and compare with the cutoff as integers (positive
//    doubles order as their bits).
// Error against quad precision (3000 particles, uniform and clustered, relative
// RMS): forces 5.2e-16, dL/dx 7.0e-16, dL/dm 5.5e-16; with erfc, exp, a root and
// divisions per pair 1.0e-15, 1.1e-15 and 1.0e-15.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "kcommon.cuh"

namespace psr {

constexpr double kMagic64 = 6755399441055744.0;  // 1.5 * 2^52: x + kMagic64 holds rint(x) in its low bits
constexpr int kT64Terms = 6;

__device__ __forceinline__ long long bits64(double x) { return __double_as_longlong(x); }

// ri = 1 / sqrt(r2), r = sqrt(r2)
__device__ __forceinline__ void rsqrt64(double r2, double& ri, double& r)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(r2));
    const double g = r2 * y, e = fma(-g, y, 1.0), c = e * fma(e, 0.375, 0.5);
    ri = fma(y, c, y);
    r = fma(g, c, g);
}

// 0 < r2 < rc2
__device__ __forceinline__ bool inside64(double r2, long long rc2m1)
{
    return (unsigned long long)(bits64(r2) - 1) < (unsigned long long)rc2m1;  // rc2m1 = bits(rc2) - 1
}

// node and offset from it, in node spacings, of distance r >= 0 (us nodes per
// unit of r).  fk's low word is the node below 2^32, where its high word is
// kMagic64's; beyond (r_s far below r_c: x above 1.6e7), infinity included,
// INT_MAX.
__device__ __forceinline__ int node64(double r, double us, double& f)
{
    const double fk = fma(r, us, kMagic64);
    const bool low = __double2hiint(fk) == 0x43380000;
    f = low ? fma(r, us, -(fk - kMagic64)) : 0.0;
    return low ? (int)min((unsigned)__double2loint(fk), 0x7fffffffu) : 0x7fffffff;
}

// T(x) and exp(-x^2) beyond the table
static __device__ __noinline__ double2 tail64(double x)
{
    const double q = exp(-x * x);
    return make_double2(erfc(x) + 1.1283791670955126 * x * q, q);  // 2 / sqrt(pi)
}

template <int DEG>
__device__ __forceinline__ double horner64(const double* __restrict__ c, double f)
{
    double v = c[DEG];
#pragma unroll
    for (int m = DEG - 1; m >= 0; --m) v = fma(f, v, c[m]);
    return v;
}

// A warp's shared memory: kStage64 staged sources - FP32 coordinates from the
// target box's centre in units of 2^k, k the exponent of r_c, the particle's
// index, and its periodic steps (nx + 1) | (ny + 1) << 2 | (nz + 1) << 4 - then
// the lanes' targets at the three steps of each axis, 32 entry records, and the
// target box (centre, half extents, squared cutoff).  The FP64 coordinates are
// read from global memory (L1, L2) per pair: a load is nothing beside a pair's
// FP64 instructions, and the small buffers leave two blocks per SM.
constexpr int kStage64 = 256;
constexpr int kTarget64 = 17 * kStage64, kMeta64 = kTarget64 + 9 * 32 * 8, kBox64 = kMeta64 + 32 * 8;
constexpr int kWarp64Bytes = kBox64 + 8 * 8;
struct Warp64 {
    float4* near;
    unsigned char* steps;
    double* target;
    int2* meta;
    double* box;
    __device__ explicit Warp64(unsigned char* base)
        : near(reinterpret_cast<float4*>(base)), steps(base + 16 * kStage64),
          target(reinterpret_cast<double*>(base + kTarget64)), meta(reinterpret_cast<int2*>(base + kMeta64)),
          box(reinterpret_cast<double*>(base + kBox64))
    {
    }
    // the lane's target x at the steps n = -1, 0, 1 of each axis, x - n L: a pair's
    // difference is then x_j - (x_i - n L) with no FP64 instruction for the image
    // (images: some staged source is not in the box itself)
    __device__ void set_target(double4 x, double L, bool images) const
    {
        double* t = target + (threadIdx.x & 31);
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            if (n != 1 && !images) continue;
            const double s = (n - 1) * L;
            t[32 * n] = n == 1 ? x.x : x.x - s;
            t[32 * (3 + n)] = n == 1 ? x.y : x.y - s;
            t[32 * (6 + n)] = n == 1 ? x.z : x.z - s;
        }
    }
    // staged source k's difference from the target
    __device__ double3 diff(double4 p, int k) const
    {
        const double* t = target + (threadIdx.x & 31);
        const int c = steps[k];
        return make_double3(p.x - t[32 * (c & 3)], p.y - t[32 * (3 + ((c >> 2) & 3))], p.z - t[32 * (6 + (c >> 4))]);
    }
};

// d in units of 2^k as FP32, cut to 23 bits, in integer arithmetic (d below
// 2^(k - 126) gives 0, above 2^(k + 126) a value far beyond the cutoff)
__device__ __forceinline__ float near_float(double d, int k)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const int e = (int)((hi >> 20) & 0x7ffu) - 1023 - k;
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned f = e < -126 ? 0u : e > 126 ? 0x7e800000u : ((unsigned)(e + 127) << 23) | m;
    return __uint_as_float(f | (hi & 0x80000000u));
}
__device__ __forceinline__ int exponent_of(double x) { return (int)((__double2hiint(x) >> 20) & 0x7ff) - 1023; }

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

// Stages one chunk of the row part [e0, e0 + len) (the scheme of stage_chunk in
// fwd_f32_common.cuh), from its p-th entry on in strided order: 32 columns of
// consecutive entries, taken row by row.  Returns the entries taken, nst the
// staged sources, each at its periodic image.
template <bool CULL>
__device__ __forceinline__ int stage64(const FwdArgs& a, long long e0, int len, int p, double L, int kx,
                                       const Warp64& w, int& nst, bool& images)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const double4* __restrict__ pd = reinterpret_cast<const double4*>(a.pd);
    const int4* __restrict__ leaf = reinterpret_cast<const int4*>(a.leaf);
    const unsigned* __restrict__ prow = a.pairs + e0;
    const int col = len >> 5, more = len & 31;  // the first `more` columns have one more entry
    int nk = 0, eb = p;
    bool shifted = false;  // this lane staged a source at an image
    for (;;) {
        const int e = eb + lane;
        int cnt = 0, first = 0, code = 13;
        if (e < len) {
            const int c = e & 31;
            const unsigned ent = prow[c * col + min(c, more) + (e >> 5)];
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
        const int ntake = __popc(__ballot_sync(kFull, e < len && incl <= kStage64 - nk));
        if (ntake == 0) break;
        const int nraw = __shfl_sync(kFull, incl, ntake - 1), excl = incl - cnt;
        if (lane < ntake) w.meta[lane] = make_int2(first - excl, code);
        __syncwarp();
        int C = 0;  // entry starts before this round
        for (int p0 = 0; p0 < nraw; p0 += 32) {
            const int rel = excl - p0;
            const unsigned M =
                __reduce_or_sync(kFull, (lane < ntake && rel >= 0 && rel < 32) ? (1u << rel) : 0u);
            const int k = C + __popc(M & ((2u << lane) - 1u)) - 1;
            C += __popc(M);
            const int q = p0 + lane;
            bool keep = q < nraw;
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            int steps = 21;  // 1 | 1 << 2 | 1 << 4: no shift
            if (keep) {
                const int2 m = w.meta[k];
                const int src = m.x + q;
                double4 v = pd[src];
                if (m.y != 13 && m.y >= 0) {
                    int nx, ny, nz;
                    decode_shift((unsigned)m.y, nx, ny, nz);
                    if (nx) v.x = fma((double)nx, L, v.x);
                    if (ny) v.y = fma((double)ny, L, v.y);
                    if (nz) v.z = fma((double)nz, L, v.z);
                    steps = (nx + 1) | (ny + 1) << 2 | (nz + 1) << 4;
                }
                keep = m.y >= 0;
                const double d[3] = {v.x - w.box[0], v.y - w.box[1], v.z - w.box[2]};
                f = make_float4(near_float(d[0], kx), near_float(d[1], kx), near_float(d[2], kx), __int_as_float(src));
                if (CULL) {
                    double g[3];
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        g[i] = fabs(d[i]) - w.box[3 + i];
                        g[i] = bits64(g[i]) < 0 ? 0.0 : g[i];
                    }
                    keep = keep && bits64(fma(g[0], g[0], fma(g[1], g[1], g[2] * g[2]))) < bits64(w.box[6]);
                }
            }
            const unsigned K = __ballot_sync(kFull, keep);
            if (keep) {
                const int pos = nk + __popc(K & lt);
                w.near[pos] = f;
                w.steps[pos] = (unsigned char)steps;
                shifted = shifted || steps != 21;
            }
            nk += __popc(K);
        }
        __syncwarp();
        eb += ntake;
        if (ntake < 32 || eb >= len) break;
    }
    images = __any_sync(kFull, shifted);
    nst = nk;
    return eb - p;
}

// A target in the same FP32 coordinates, and the squared distance below which a
// staged source may lie within the cutoff: coordinates are at most r_c plus
// twice the half extents, cut by 2^-23 of that, differences and squares by a few
// 2^-24 more, which 1e-6 of the sum covers.
__device__ __forceinline__ float3 target64(double4 x, const double* box, int kx)
{
    return make_float3(near_float(x.x - box[0], kx), near_float(x.y - box[1], kx), near_float(x.z - box[2], kx));
}
__device__ __forceinline__ float cut64(double r_c, const double* box, int kx)
{
    const double w = r_c + 1e-6 * (r_c + 2.0 * (box[3] + box[4] + box[5]));
    const float f = near_float(w, kx) * 1.000001f;
    return f * f;
}

// Calls pair(k) for each staged source k of the lane's stream (s, s + S, ...)
// that may lie within the cutoff of the lane's target t.
// Every lane takes its own next one, by a bit mask over its stream's sources.
template <class Pair>
__device__ __forceinline__ void near_pairs(const float4* __restrict__ near, int nst, int s, int S, float3 t,
                                           float cut, bool on, Pair pair)
{
    auto maybe = [&](int k) {
        const float4 v = near[k];
        const float dx = v.x - t.x, dy = v.y - t.y, dz = v.z - t.z;
        return fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < cut;
    };
    constexpr int kWords = kStage64 / 32;
    const int J = on && nst > s ? (nst - s + S - 1) / S : 0;  // sources of this lane's stream
    unsigned m[kWords];
#pragma unroll
    for (int w = 0; w < kWords; ++w) {
        m[w] = 0;
        const int jn = min(J - 32 * w, 32);
        for (int j = 0; j < jn; ++j) m[w] |= (maybe(s + (32 * w + j) * S) ? 1u : 0u) << j;
    }
    __syncwarp();
    for (;;) {
        int w = 0;  // the lane's next word with a bit left
        unsigned bits = 0;
#pragma unroll
        for (int i = kWords - 1; i >= 0; --i)
            if (m[i]) {
                w = i;
                bits = m[i];
            }
        if (!__any_sync(kFull, bits != 0)) break;
        if (bits) {
#pragma unroll
            for (int i = 0; i < kWords; ++i)
                if (i == w) m[i] &= m[i] - 1;
            pair(s + (32 * w + __ffs(bits) - 1) * S);
        }
    }
}

// Adds the S stream partials (NC components per target slot) of each target
// through the warp's staging buffer, in stream order, and hands each target's
// sums to write(target, component, sum); in a row that a group of warps shares each has the
// sums of its part (join_parts; stride: bytes between the warps' regions).
template <int NC, int R, class Work, class Write>
__device__ __forceinline__ void finish64(const FwdArgs& a, int4 li, const double (*acc)[NC], const bool* act, int lane, int s, int S,
                                         int T, float4* __restrict__ stage, const Work& rw, int stride,
                                         Write write)
{
    const bool joint = rw.joint();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        volatile double* red = reinterpret_cast<volatile double*>(stage) + 32 * NC * r;
#pragma unroll
        for (int i = 0; i < NC; ++i) red[NC * lane + i] = acc[r][i];
        __syncwarp();
        if (!joint && s == 0 && act[r]) {
            double v[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) v[i] = acc[r][i];
            for (int t = 1; t < S; ++t)
#pragma unroll
                for (int i = 0; i < NC; ++i) v[i] += red[NC * (lane + t * T) + i];
#pragma unroll
            for (int i = 0; i < NC; ++i) write(li.x + lane + T * r, i, v[i]);
        }
        __syncwarp();
    }
    if (joint)
        join_parts<NC, PSR_ACC_FP64>(
            a, rw, li.y, S, reinterpret_cast<const char*>(stage), stride,
            [T](int t, int s, int i) { return 8 * (32 * NC * (t / T) + NC * (t % T + s * T) + i); },
            [&](int t, int i, const PartSum<PSR_ACC_FP64>& p) { write(li.x + t, i, p.v); });
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
