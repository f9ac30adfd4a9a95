// FP64 forward P2P kernel: the plain double-precision path (paper, Section 2
// pair force, Eq. tr), or, with a Taylor interpolation level, the paper's
// double-precision table path (Section 3.3: the Eq. int expansion about the
// nearest of N + 1 nodes, level T_[4] for double precision).  Both evaluate T
// from a table in shared memory; the plain path's has nodes close enough that
// T is as near as erfc and exp give it.  p2p_f64_common.cuh says what bounds the kernel and
// what it does about it.  48^3 NFW set: 255 ms with erfc, exp, a square root and
// a division per tile pair and one warp per leaf.
#include <cuda_runtime.h>

#include "p2p_f64_common.cuh"

namespace psr {

// Taylor tables of the levels T_[2] and T_[4] in FP64: node k = 0..N, x_k = k h,
// six doubles per node, the Eq. int coefficients of eps^m (eps = x - x_k) times
// h^m, so that the expansion is a polynomial in f = x/h - k (zero above the level).
__global__ void table64_kernel(int N, int level, double h, double* __restrict__ t)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > N) return;
    double* c = t + 6 * (int64_t)k;
    const double x = k * h, x2 = x * x;
    const double E = -2.0 * 1.1283791670955126 * exp(-x2);  // -4 exp(-x^2) / sqrt(pi)
    c[0] = erfc(x) - 0.5 * x * E;
    c[1] = x2 * E * h;
    c[2] = -x * (x2 - 1.0) * E * h * h;
    c[3] = level >= 4 ? (2.0 / 3.0 * x2 * x2 - 5.0 / 3.0 * x2 + 1.0 / 3.0) * E * h * h * h : 0.0;
    c[4] = level >= 4 ? -x * (x2 * x2 / 3.0 - 1.5 * x2 + 1.0) * E * h * h * h * h : 0.0;
    c[5] = 0.0;
}

// The plain path's tables of T (t) and, unless null, Q = exp(-x^2) (q): nodes
// x_k = k / 256, k = 0..N, six coefficients in f = 256 x - k.  Taylor coefficients
// about x_k: Q's by (m + 1) q_{m+1} = -2 (x q_m + q_{m-1}), T's from T' = -c x^2 Q,
// c = 4 / sqrt(pi).  The terms in f^6 and f^7 are replaced by the polynomials of
// degree 4 and 5 nearest to them on [-1/2, 1/2] (Chebyshev economisation), which
// divides the error of leaving them out by 32 and 64.
__global__ void plain64_kernel(int N, double* __restrict__ t, double* __restrict__ q)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > N) return;
    const double h = 1.0 / kPlain64PerX, x = k * h;
    const double c = 2.0 * 1.1283791670955126;  // 4 / sqrt(pi)
    double Q[8], T[8];
    Q[0] = exp(-x * x);
    Q[1] = -2.0 * x * Q[0];
    for (int m = 1; m < 7; ++m) Q[m + 1] = -2.0 * (x * Q[m] + Q[m - 1]) / (m + 1);
    T[0] = erfc(x) + 0.5 * c * x * Q[0];
    for (int m = 0; m < 7; ++m)
        T[m + 1] = -c * (x * x * Q[m] + (m > 0 ? 2.0 * x * Q[m - 1] : 0.0) + (m > 1 ? Q[m - 2] : 0.0)) / (m + 1);
    for (int i = 0; i < (q ? 2 : 1); ++i) {
        double* a = i ? Q : T;
        double hm = 1.0;
        for (int m = 1; m < 8; ++m) a[m] *= hm *= h;
        double* o = (i ? q : t) + 6 * (int64_t)k;
        o[0] = a[0] + a[6] / 2048.0;
        o[1] = a[1] + a[7] * (14.0 / 8192.0);
        o[2] = a[2] - a[6] * (72.0 / 2048.0);
        o[3] = a[3] - a[7] * (448.0 / 8192.0);
        o[4] = a[4] + a[6] * (768.0 / 2048.0);
        o[5] = a[5] + a[7] * (3584.0 / 8192.0);
    }
}

int launch_table64(int table_n, int interp, double x_c, void* d_out, void* stream)
{
    const int threads = 32, blocks = (table_n + 1 + threads - 1) / threads;
    table64_kernel<<<blocks, threads, 0, (cudaStream_t)stream>>>(
        table_n, interp == PSR_TAYLOR4 ? 4 : 2, x_c / table_n, reinterpret_cast<double*>(d_out));
    return (int)cudaGetLastError();
}

Plain64 plain64(double x_c)
{
    const double want = std::ceil(x_c * kPlain64PerX);
    return Plain64{want > kPlain64MaxN ? kPlain64MaxN : (int)want, want > kPlain64MaxN};
}

int launch_plain64(double x_c, void* d_t, void* d_q, void* stream)
{
    const int n = plain64(x_c).n;
    const int threads = 32, blocks = (n + 1 + threads - 1) / threads;
    plain64_kernel<<<blocks, threads, 0, (cudaStream_t)stream>>>(n, reinterpret_cast<double*>(d_t),
                                                                 reinterpret_cast<double*>(d_q));
    return (int)cudaGetLastError();
}

// One target leaf (rw: this warp's parts of its row).  EQM: every particle of
// the box has one mass, applied once per target.  COUNT: pairs
// within the cutoff and pairs evaluated are counted, over every tile pair (no
// cull).
template <bool COUNT, bool EQM, int DEG, bool TAIL, int R, class Work>
__device__ __forceinline__ void fwd64_item(const FwdArgs& a, int I, int4 li, const double* tab,
                                           const Warp64& w64, unsigned long long& npairs,
                                           unsigned long long& nev, Work rw,
                                           PartTotals<PSR_ACC_FP64, 9>& tot)
{
    const int lane = threadIdx.x & 31;
    const double4* __restrict__ pd = reinterpret_cast<const double4*>(a.pd);
    const int nI = li.y, T = (nI + R - 1) / R, S = 32 / T, s = lane / T, q = lane - s * T;
    const bool on = s < S;
    const BoxDev& bx = a.boxes[li.z];
    const long long rc2m1 = bits64(bx.rc2) - 1;
    const double us = DEG == 5 ? bx.inv_2rs * kPlain64PerX : (double)a.table_n / bx.r_c;
    const int kmax = a.t64_max;

    double4 xi[R];
    bool act[R];
    double acc[R][3];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = q + T * r;
        act[r] = on && t < nI;
        xi[r] = pd[li.x + (act[r] ? t : 0)];
        acc[r][0] = acc[r][1] = acc[r][2] = 0.0;
    }
    cull_box64<R>(xi, act, bx.r_c, bx.L, w64.box);
    const int kx = exponent_of(bx.r_c);
    const float cut = cut64(bx.r_c, w64.box, kx);
    float3 ti[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ti[r] = target64(xi[r], w64.box, kx);
    unsigned cnt = 0;
    long long e0, re;
    row_part(a, I, rw, e0, re);
    const int len = (int)(re - e0);
    for (int e = 0; e < len;) {
        int nst;
        bool images;
        e += stage64<!COUNT>(a, e0, len, e, bx.L, kx, w64, nst, images);
        if (COUNT && lane == 0) nev += (unsigned long long)nst * (unsigned)nI;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            w64.set_target(xi[r], bx.L, images);
            near_pairs(w64.near, nst, s, S, ti[r], cut, act[r], [&](int k) {
                const int j = __float_as_int(w64.near[k].w);
                const double4 p = pd[j];
                const double3 d = w64.diff(p, k);
                const double dx = d.x, dy = d.y, dz = d.z;
                const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                if (inside64(r2, rc2m1)) {
                    double ri, rr, f;
                    rsqrt64(r2, ri, rr);
                    const int kk = node64(rr, us, f);
                    const double Tv = TAIL && kk > kmax ? tail64(rr * bx.inv_2rs).x
                                                        : horner64<DEG>(tab + 6 * min(kk, kmax), f);
                    double w = ri * ri * ri * Tv;
                    if (!EQM) w *= p.w;
                    acc[r][0] = fma(w, dx, acc[r][0]);
                    acc[r][1] = fma(w, dy, acc[r][1]);
                    acc[r][2] = fma(w, dz, acc[r][2]);
                    if (COUNT) ++cnt;
                }
            });
        }
        __syncwarp();
    }
    if (COUNT) npairs += cnt;
    if (rw.in_turn()) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < 3; ++i) acc[r][i] = tot.add(3 * r + i, rw.part(), PartSum<PSR_ACC_FP64>{acc[r][i]}).v;
    }
    if (!rw.last()) return;
    const double g = EQM ? bx.G * pd[li.x].w : bx.G;
    finish64<3, R>(a, li, acc, act, lane, s, S, T, w64.near, rw, kWarp64Bytes,
                   [&](int target, int i, double v) {
                       reinterpret_cast<double*>(a.out)[3LL * a.perm[target] + i] = g * v;
                   });
}

// DEG 5: the plain path (TAIL: the cutoff lies beyond its table), 4: the Taylor levels.
template <bool COUNT, bool EQM, int DEG, bool TAIL, int ROWS>
__global__ void __launch_bounds__(256, 2) p2p_fwd_f64_kernel(const FwdArgs a)
{
    extern __shared__ __align__(16) unsigned char smem64[];
    __shared__ int s_it[8];
    double* tab = reinterpret_cast<double*>(smem64);
    const int words = 6 * (a.t64_max + 1);
    for (int i = threadIdx.x; i < words; i += blockDim.x) tab[i] = reinterpret_cast<const double*>(a.table)[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const Warp64 w64(smem64 + 8 * words + (threadIdx.x >> 5) * kWarp64Bytes);
    unsigned long long npairs = 0, nev = 0;
    const int n_heavy = ROWS != kRowsJoint ? 0 : a.heavy ? min(*a.heavy, a.n_items) : a.n_items;
    bool split = n_heavy > 0;
    int it;
    while (next_item<ROWS>(a, a.ctrl + kCtrlTicketFwd, split, n_heavy, s_it, it)) {
        int I;
        int4 li;
        if (!item64(a, it, lane, I, li)) continue;
        const int R = targets_per_lane(li.y, 128);
        auto rw = row_work<ROWS>(a, I, li.z, split);
        PartTotals<PSR_ACC_FP64, 9> tot;  // kRowsInTurn
        for (;;) {  // parts in turn
            if (R == 1) fwd64_item<COUNT, EQM, DEG, TAIL, 1>(a, I, li, tab, w64, npairs, nev, rw, tot);
            else if (R == 2) fwd64_item<COUNT, EQM, DEG, TAIL, 2>(a, I, li, tab, w64, npairs, nev, rw, tot);
            else fwd64_item<COUNT, EQM, DEG, TAIL, 3>(a, I, li, tab, w64, npairs, nev, rw, tot);
            if (rw.last()) break;
            if constexpr (ROWS == kRowsInTurn) ++rw.v;
        }
    }
    if (COUNT) {
        for (int off = 16; off > 0; off >>= 1) npairs += __shfl_xor_sync(kFull, npairs, off);
        if (lane == 0 && npairs)
            atomicAdd(reinterpret_cast<unsigned long long*>(a.ctrl + kCtrlPairsLo), npairs);
        if (lane == 0 && nev)  // lane 0 alone counted the warp's staged pairs
            atomicAdd(reinterpret_cast<unsigned long long*>(a.ctrl + kCtrlEvalLo), nev);
    }
    persistent_exit(a.ctrl + kCtrlTicketFwd, a.ctrl + kCtrlDoneFwd);
}

namespace {

bool taylor64(int interp) { return interp == PSR_TAYLOR2 || interp == PSR_TAYLOR4; }

template <int DEG, bool TAIL, int ROWS>
const void* pick64_r(bool count, bool eqm)
{
    return count ? (const void*)p2p_fwd_f64_kernel<true, false, DEG, TAIL, ROWS>
           : eqm ? (const void*)p2p_fwd_f64_kernel<false, true, DEG, TAIL, ROWS>
                 : (const void*)p2p_fwd_f64_kernel<false, false, DEG, TAIL, ROWS>;
}

template <int DEG, bool TAIL>
const void* pick64_t(int rows, bool count, bool eqm)
{
    return rows == kRowsJoint    ? pick64_r<DEG, TAIL, kRowsJoint>(count, eqm)
           : rows == kRowsInTurn ? pick64_r<DEG, TAIL, kRowsInTurn>(count, eqm)
                                 : pick64_r<DEG, TAIL, kRowsWhole>(count, eqm);
}

const void* pick64(int interp, double x_c, int rows, bool count, bool eqm)
{
    return taylor64(interp)    ? pick64_t<4, false>(rows, count, eqm)
           : plain64(x_c).tail ? pick64_t<5, true>(rows, count, eqm)
                               : pick64_t<5, false>(rows, count, eqm);
}

}  // namespace

size_t fwd_f64_smem(int interp, int table_n, double x_c, int warps)
{
    const int entries = 1 + (taylor64(interp) ? table_n : plain64(x_c).n);
    return (size_t)entries * 48 + (size_t)warps * kWarp64Bytes;
}

int launch_fwd_f64(const FwdArgs& args, double x_c, void* stream)
{
    FwdArgs a = args;
    a.t64_max = taylor64(a.interp) ? a.table_n : plain64(x_c).n;
    const size_t smem = fwd_f64_smem(a.interp, a.table_n, x_c, a.warps_per_block);
    const void* k = pick64(a.interp, x_c, a.rows, a.count_pairs, a.equal_mass);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    void* params[] = {&a};
    return (int)cudaLaunchKernel(k, dim3(a.blocks), dim3(a.warps_per_block * 32), params, smem,
                                 (cudaStream_t)stream);
}

int fwd_f64_occupancy(int warps, int interp, int table_n, double x_c, int* out)
{
    const void* f = pick64(interp, x_c, kRowsWhole, false, false);
    const size_t smem = fwd_f64_smem(interp, table_n, x_c, warps);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, f, warps * 32, smem);
}

}  // namespace psr
