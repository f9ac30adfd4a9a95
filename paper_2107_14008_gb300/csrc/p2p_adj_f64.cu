// FP64 adjoint P2P kernel: the sums of p2p_adj.cu in double precision (r, not
// x, units).  p2p_f64_common.cuh says what bounds it: about 47 FP64
// instructions per pair with one mass per box, T and exp(-x^2) from the plain
// path's tables.  32^3 uniform set: 36.7 ms with erfc, exp, a square root and
// divisions per tile pair and one warp per leaf.
#include <cuda_runtime.h>

#include "p2p_f64_common.cuh"

namespace psr {

template <bool EQM, bool TAIL, int R, class Work>
__device__ __forceinline__ void adj64_item(const FwdArgs& a, int I, int4 li, const double* tab,
                                           const double* tabq, const Warp64& w64, Work rw,
                                           PartTotals<PSR_ACC_FP64, 12>& tot)
{
    const int lane = threadIdx.x & 31;
    const double4* __restrict__ pd = reinterpret_cast<const double4*>(a.pd);
    const double4* __restrict__ cs = reinterpret_cast<const double4*>(a.cot_sorted);
    const int nI = li.y, T = (nI + R - 1) / R, S = 32 / T, s = lane / T, q = lane - s * T;
    const bool on = s < S;
    const BoxDev& bx = a.boxes[li.z];
    const long long rc2m1 = bits64(bx.rc2) - 1;
    const double us = bx.inv_2rs * kPlain64PerX;
    // exp(-x^2) / (2 sqrt(pi) r_s^3), the second part of -g'(r) r
    const double cq = 1.0 / (2.0 * 1.7724538509055160 * bx.r_s * bx.r_s * bx.r_s);

    double4 xi[R], ck[R];
    bool act[R];
    double g[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = q + T * r;
        act[r] = on && t < nI;
        xi[r] = pd[li.x + (act[r] ? t : 0)];
        ck[r] = cs[li.x + (act[r] ? t : 0)];
#pragma unroll
        for (int i = 0; i < 4; ++i) g[r][i] = 0.0;
    }
    cull_box64<R>(xi, act, bx.r_c, bx.L, w64.box);
    const int kx = exponent_of(bx.r_c);
    const float cut = cut64(bx.r_c, w64.box, kx);
    float3 ti[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ti[r] = target64(xi[r], w64.box, kx);
    long long e0, re;
    row_part(a, I, rw, e0, re);
    const int len = (int)(re - e0);
    for (int e = 0; e < len;) {
        int nst;
        bool images;
        e += stage64<true>(a, e0, len, e, bx.L, kx, w64, nst, images);
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
                    const double4 c = cs[j];
                    double ri, rr, f;
                    rsqrt64(r2, ri, rr);
                    const double ri2 = ri * ri;
                    const int node = node64(rr, us, f), kk = 6 * min(node, a.t64_max);
                    double Tv, Qv;
                    if (TAIL && node > a.t64_max) {
                        const double2 tq = tail64(rr * bx.inv_2rs);
                        Tv = tq.x;
                        Qv = tq.y;
                    } else {
                        Tv = horner64<5>(tab + kk, f);
                        Qv = horner64<5>(tabq + kk, f);
                    }
                    const double gg = Tv * (ri2 * ri);  // T / r^3
                    const double Q = cq * Qv;
                    const double hf = -ri2 * fma(3.0, gg, Q);  // g'(r)/r
                    // v = m_k c_j - m_j c_k (one mass: c_j - c_k, m applied at the end)
                    const double vx = EQM ? c.x - ck[r].x : fma(xi[r].w, c.x, -p.w * ck[r].x);
                    const double vy = EQM ? c.y - ck[r].y : fma(xi[r].w, c.y, -p.w * ck[r].y);
                    const double vz = EQM ? c.z - ck[r].z : fma(xi[r].w, c.z, -p.w * ck[r].z);
                    const double hd = hf * fma(dx, vx, fma(dy, vy, dz * vz));
                    g[r][0] = fma(gg, vx, fma(hd, dx, g[r][0]));
                    g[r][1] = fma(gg, vy, fma(hd, dy, g[r][1]));
                    g[r][2] = fma(gg, vz, fma(hd, dz, g[r][2]));
                    g[r][3] = fma(gg, fma(dx, c.x, fma(dy, c.y, dz * c.z)), g[r][3]);
                }
            });
        }
        __syncwarp();
    }
    if (rw.in_turn()) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < 4; ++i) g[r][i] = tot.add(4 * r + i, rw.part(), PartSum<PSR_ACC_FP64>{g[r][i]}).v;
    }
    if (!rw.last()) return;
    const double G = bx.G, gx = EQM ? G * pd[li.x].w : G;
    finish64<4, R>(a, li, g, act, lane, s, S, T, w64.near, rw, kWarp64Bytes,
                   [&](int target, int i, double v) {
                       const int idx = a.perm[target];
                       if (i < 3) reinterpret_cast<double*>(a.out)[3LL * idx + i] = gx * v;
                       else if (a.out_m) reinterpret_cast<double*>(a.out_m)[idx] = -G * v;
                   });
}

template <bool EQM, bool TAIL, int ROWS>
__global__ void __launch_bounds__(256, 2) p2p_adj_f64_kernel(const FwdArgs a)
{
    extern __shared__ __align__(16) unsigned char smem64[];
    __shared__ int s_it[8];
    double* tab = reinterpret_cast<double*>(smem64);
    const int words = 6 * (a.t64_max + 1);
    double* tabq = tab + words;
    for (int i = threadIdx.x; i < words; i += blockDim.x) {
        tab[i] = reinterpret_cast<const double*>(a.table)[i];
        tabq[i] = reinterpret_cast<const double*>(a.table)[6 * (kPlain64MaxN + 1) + i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const Warp64 w64(smem64 + 16 * words + (threadIdx.x >> 5) * kWarp64Bytes);
    const int n_heavy = ROWS != kRowsJoint ? 0 : a.heavy ? min(*a.heavy, a.n_items) : a.n_items;
    bool split = n_heavy > 0;
    int it;
    while (next_item<ROWS>(a, a.ctrl + kCtrlTicketAdj, split, n_heavy, s_it, it)) {
        int I;
        int4 li;
        if (!item64(a, it, lane, I, li)) continue;
        const int R = targets_per_lane(li.y, 128);
        auto rw = row_work<ROWS>(a, I, li.z, split);
        PartTotals<PSR_ACC_FP64, 12> tot;  // kRowsInTurn
        for (;;) {  // parts in turn
            if (R == 1) adj64_item<EQM, TAIL, 1>(a, I, li, tab, tabq, w64, rw, tot);
            else if (R == 2) adj64_item<EQM, TAIL, 2>(a, I, li, tab, tabq, w64, rw, tot);
            else adj64_item<EQM, TAIL, 3>(a, I, li, tab, tabq, w64, rw, tot);
            if (rw.last()) break;
            if constexpr (ROWS == kRowsInTurn) ++rw.v;
        }
    }
    persistent_exit(a.ctrl + kCtrlTicketAdj, a.ctrl + kCtrlDoneAdj);
}

namespace {

template <bool TAIL, int ROWS>
auto pick_adj64_r(bool eqm)
{
    return eqm ? p2p_adj_f64_kernel<true, TAIL, ROWS> : p2p_adj_f64_kernel<false, TAIL, ROWS>;
}

template <bool TAIL>
auto pick_adj64_t(int rows, bool eqm)
{
    return rows == kRowsJoint    ? pick_adj64_r<TAIL, kRowsJoint>(eqm)
           : rows == kRowsInTurn ? pick_adj64_r<TAIL, kRowsInTurn>(eqm)
                                 : pick_adj64_r<TAIL, kRowsWhole>(eqm);
}

auto pick_adj64(double x_c, int rows, bool eqm)
{
    return plain64(x_c).tail ? pick_adj64_t<true>(rows, eqm) : pick_adj64_t<false>(rows, eqm);
}

}  // namespace

size_t adj_f64_smem(double x_c, int warps)
{
    return (size_t)(plain64(x_c).n + 1) * 96 + (size_t)warps * kWarp64Bytes;
}

int launch_adj_f64(const FwdArgs& args, double x_c, void* stream)
{
    FwdArgs a = args;
    cudaStream_t st = (cudaStream_t)stream;
    gather_cot_kernel<double, double4><<<(unsigned)((a.n + 255) / 256), 256, 0, st>>>(
        reinterpret_cast<const double*>(a.cot), a.perm, reinterpret_cast<double4*>(a.cot_sorted), a.n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    a.t64_max = plain64(x_c).n;
    const size_t smem = adj_f64_smem(x_c, a.warps_per_block);
    auto k = pick_adj64(x_c, a.rows, a.equal_mass);
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    k<<<a.blocks, a.warps_per_block * 32, smem, st>>>(a);
    return (int)cudaGetLastError();
}

int adj_f64_occupancy(int warps, double x_c, int* out)
{
    const size_t smem = adj_f64_smem(x_c, warps);
    auto k = pick_adj64(x_c, kRowsWhole, false);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, warps * 32, smem);
}

}  // namespace psr
