// FP64 forward P2P kernel: the plain double-precision path (paper, Section 2
// pair force, Eq. tr), or, with a Taylor interpolation level, the paper's
// double-precision table path (Section 3.3: the Eq. int expansion about the
// nearest of N + 1 nodes, level T_[4] for double precision).  Both evaluate T
// from a table in shared memory; the plain path's has nodes close enough that
// T is exact to rounding.  p2p_f64_common.cuh says what bounds the kernel and
// what it does about it.  48^3 NFW set: 255 ms with erfc, exp, a square root and
// a division per tile pair and one warp per leaf.
#include <cuda_runtime.h>

#include "p2p_f64_common.cuh"

namespace psr {

// Taylor tables in FP64: node k = 0..N, x_k = k h, six doubles per node, the
// coefficients of eps^m (eps = x - x_k) times h^m, so that the expansion is a
// polynomial in f = x/h - k (zero above the level).  T's are those of Eq. int and
// the next, from T' = x^2 E, E = -4 exp(-x^2) / sqrt(pi); Q = exp(-x^2) likewise
// (levels: 2 or 4 as Eq. int's, 5).  Entry N + 1, written at level 5, is zero.
__global__ void table64_kernel(int N, int level, double h, double* __restrict__ t, double* __restrict__ q)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > N + (level == 5 ? 1 : 0)) return;
    double* c = t + 6 * (int64_t)k;
    const double x = k * h, x2 = x * x, Q = exp(-x2);
    const double E = -2.0 * 1.1283791670955126 * Q;  // -4 exp(-x^2) / sqrt(pi)
    const double h2 = h * h, h3 = h2 * h, h4 = h2 * h2, h5 = h4 * h;
    const double on = k <= N ? 1.0 : 0.0, four = level >= 4 ? on : 0.0, five = level >= 5 ? on : 0.0;
    c[0] = on * (erfc(x) - 0.5 * x * E);
    c[1] = on * (x2 * E * h);
    c[2] = on * (-x * (x2 - 1.0) * E * h2);
    c[3] = four * ((2.0 / 3.0 * x2 * x2 - 5.0 / 3.0 * x2 + 1.0 / 3.0) * E * h3);
    c[4] = four * (-x * (x2 * x2 / 3.0 - 1.5 * x2 + 1.0) * E * h4);
    c[5] = five * (((2.0 / 15.0 * x2 - 14.0 / 15.0) * x2 + 1.3) * x2 - 0.2) * E * h5;
    if (!q) return;
    c = q + 6 * (int64_t)k;
    c[0] = on * Q;
    c[1] = on * (-2.0 * x * Q * h);
    c[2] = on * ((2.0 * x2 - 1.0) * Q * h2);
    c[3] = on * (x * (2.0 - 4.0 / 3.0 * x2) * Q * h3);
    c[4] = on * (((2.0 / 3.0 * x2 - 2.0) * x2 + 0.5) * Q * h4);
    c[5] = on * (x * ((-4.0 / 15.0 * x2 + 4.0 / 3.0) * x2 - 1.0) * Q * h5);
}

int launch_table64(int table_n, int interp, double x_c, void* d_out, void* stream)
{
    const int threads = 32, blocks = (table_n + 1 + threads - 1) / threads;
    table64_kernel<<<blocks, threads, 0, (cudaStream_t)stream>>>(
        table_n, interp == PSR_TAYLOR4 ? 4 : 2, x_c / table_n, reinterpret_cast<double*>(d_out), nullptr);
    return (int)cudaGetLastError();
}

Plain64 plain64(double x_c)
{
    Plain64 p;
    // T(12) is below 1e-61: beyond, the zero entry
    p.x_top = x_c < 12.0 ? x_c : 12.0;
    const double want = std::ceil(p.x_top / 0.0044);
    p.n = want < 16.0 ? 16 : want > kPlain64MaxN ? kPlain64MaxN : (int)want;
    return p;
}

int launch_plain64(double x_c, void* d_t, void* d_q, void* stream)
{
    const Plain64 p = plain64(x_c);
    const int threads = 32, blocks = (p.n + 2 + threads - 1) / threads;
    table64_kernel<<<blocks, threads, 0, (cudaStream_t)stream>>>(
        p.n, 5, p.x_top / p.n, reinterpret_cast<double*>(d_t), reinterpret_cast<double*>(d_q));
    return (int)cudaGetLastError();
}

// One target leaf (or, with split, this warp's part of its row).  EQM: every
// particle of the box has one mass, applied once per target.  COUNT: pairs
// within the cutoff and pairs evaluated are counted, over every tile pair (no
// cull).
template <bool COUNT, bool EQM, int DEG, int R>
__device__ __forceinline__ void fwd64_item(const FwdArgs& a, int I, int4 li, const double* tab,
                                           const Warp64& w64, unsigned long long& npairs,
                                           unsigned long long& nev, bool split)
{
    const int lane = threadIdx.x & 31;
    const double4* __restrict__ pd = reinterpret_cast<const double4*>(a.pd);
    const int nI = li.y, T = (nI + R - 1) / R, S = 32 / T, s = lane / T, q = lane - s * T;
    const bool on = s < S;
    const BoxDev& bx = a.boxes[li.z];
    const long long rc2m1 = bits64(bx.rc2) - 1;
    const double us = DEG == 5 ? bx.inv_2rs * a.t64_scale : (double)a.table_n / bx.r_c;
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
    row_part(a, I, split, e0, re);
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
                    const double ri = rsqrt64(r2);
                    double f;
                    const int kk = node64(r2 * ri, us, kmax, f);
                    const double Tv = horner64<DEG>(tab + 6 * kk, f);
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
    const double g = EQM ? bx.G * pd[li.x].w : bx.G;
    finish64<3, R>(a, li, acc, act, lane, s, S, T, w64.near, split, kWarp64Bytes,
                   [&](int target, const double* v) {
                       double* out = reinterpret_cast<double*>(a.out) + 3LL * a.perm[target];
                       out[0] = g * v[0];
                       out[1] = g * v[1];
                       out[2] = g * v[2];
                   });
}

// DEG 5: the plain path, 4: the Taylor levels.
template <bool COUNT, bool EQM, int DEG>
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
    const int n_heavy = a.group <= 1 ? 0 : a.heavy ? min(*a.heavy, a.n_items) : a.n_items;
    bool split = n_heavy > 0;
    int it;
    while (next_item<true>(a, a.ctrl + kCtrlTicketFwd, split, n_heavy, s_it, it)) {
        int I;
        int4 li;
        if (!item64(a, it, lane, I, li)) continue;
        const int R = targets_per_lane(li.y, 128);
        if (R == 1) fwd64_item<COUNT, EQM, DEG, 1>(a, I, li, tab, w64, npairs, nev, split);
        else if (R == 2) fwd64_item<COUNT, EQM, DEG, 2>(a, I, li, tab, w64, npairs, nev, split);
        else fwd64_item<COUNT, EQM, DEG, 3>(a, I, li, tab, w64, npairs, nev, split);
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

template <int DEG>
const void* pick64(bool count, bool eqm)
{
    return count ? (const void*)p2p_fwd_f64_kernel<true, false, DEG>
           : eqm ? (const void*)p2p_fwd_f64_kernel<false, true, DEG>
                 : (const void*)p2p_fwd_f64_kernel<false, false, DEG>;
}

}  // namespace

size_t fwd_f64_smem(int interp, int table_n, double x_c, int warps)
{
    const int entries = taylor64(interp) ? table_n + 1 : plain64(x_c).n + 2;
    return (size_t)entries * 48 + (size_t)warps * kWarp64Bytes;
}

int launch_fwd_f64(const FwdArgs& args, double x_c, void* stream)
{
    FwdArgs a = args;
    const bool tay = taylor64(a.interp);
    const Plain64 p = plain64(x_c);
    a.t64_max = tay ? a.table_n : p.n + 1;
    a.t64_scale = p.n / p.x_top;
    const size_t smem = fwd_f64_smem(a.interp, a.table_n, x_c, a.warps_per_block);
    const void* k = tay ? pick64<4>(a.count_pairs, a.equal_mass) : pick64<5>(a.count_pairs, a.equal_mass);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    void* params[] = {&a};
    return (int)cudaLaunchKernel(k, dim3(a.blocks), dim3(a.warps_per_block * 32), params, smem,
                                 (cudaStream_t)stream);
}

int fwd_f64_occupancy(int warps, int interp, int table_n, double x_c, int* out)
{
    const void* f = taylor64(interp) ? pick64<4>(false, false) : pick64<5>(false, false);
    const size_t smem = fwd_f64_smem(interp, table_n, x_c, warps);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, f, warps * 32, smem);
}

}  // namespace psr
