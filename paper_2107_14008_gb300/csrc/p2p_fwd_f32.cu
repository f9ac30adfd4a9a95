// FP32 forward P2P: variant dispatch, shared-memory sizing, and the
// interpolation-table builder (paper, Section 3.3).
#include <cuda_runtime.h>

#include "kcommon.cuh"

namespace psr {

template <bool PK, int ROWS>
int launch_fwd_f32_variant(const FwdArgs& a, int precision, size_t smem, cudaStream_t st);
template <bool PK>
const void* fwd_f32_kernel_ptr(int precision, int interp, int accum, int core);

// ------------------------------------------------------------------ table --
// Entries k = 0..N-1 describe [x_k, x_{k+1}], x_k = k x_c / N, as functions of
// f = (x - x_k)/h - 1/2 in [-1/2, 1/2]; entry N is zero (beyond the cutoff).
// Linear entries are (M_k, D_k, A_k, 0): the chord is M_k + f D_k, or, with
// t = u - 1/2 = k + f (u = x/h), A_k + t D_k where A_k = M_k - k D_k, which
// the forward kernel evaluates in one FMA without forming f.
// Second half (offset N+1): the same for Q(x) = exp(-x^2), used by the adjoint.
// Taylor modes (Eq. int of Section 3.3): node k = 0..N, two float4 per node,
// the level-2 or level-4 expansion about x_k in powers of f = (x - x_k)/h:
//   T_k + x_k^2 E_k eps - x_k (x_k^2 - 1) E_k eps^2
//       + (2/3 x_k^4 - 5/3 x_k^2 + 1/3) E_k eps^3 - x_k (x_k^4/3 - 3/2 x_k^2 + 1) E_k eps^4,
// eps = f h, E_k = -4 exp(-x_k^2) / sqrt(pi), T_k = erfc(x_k) - x_k E_k / 2.
__global__ void table_kernel(int N, int interp, double x_c, float4* __restrict__ tT,
                             float4* __restrict__ tQ)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > N) return;
    if (interp == PSR_TAYLOR2 || interp == PSR_TAYLOR4) {
        const double h = x_c / N, x = k * h, x2 = x * x;
        const double E = -2.0 * 1.1283791670955126 * exp(-x2);
        const double c0 = erfc(x) - 0.5 * x * E;
        const double c1 = x2 * E * h;
        const double c2 = -x * (x2 - 1.0) * E * h * h;
        const bool four = interp == PSR_TAYLOR4;
        const double c3 = four ? (2.0 / 3.0 * x2 * x2 - 5.0 / 3.0 * x2 + 1.0 / 3.0) * E * h * h * h : 0.0;
        const double c4 = four ? -x * (x2 * x2 / 3.0 - 1.5 * x2 + 1.0) * E * h * h * h * h : 0.0;
        tT[2 * k] = make_float4((float)c0, (float)c1, (float)c2, (float)c3);
        tT[2 * k + 1] = make_float4((float)c4, 0.f, 0.f, 0.f);
        return;
    }
    if (k == N) {
        tT[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tQ) tQ[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const double h = x_c / N;
    const double c2 = 1.1283791670955126;  // 2 / sqrt(pi)
    double x0 = k * h, x1 = (k + 1) * h;
    double q0 = exp(-x0 * x0), q1 = exp(-x1 * x1);
    double T0 = erfc(x0) + c2 * x0 * q0, T1 = erfc(x1) + c2 * x1 * q1;
    // T' = x^2 E(x) = -(4/sqrt(pi)) x^2 exp(-x^2); Q' = -2 x exp(-x^2)
    double D0 = -2.0 * c2 * x0 * x0 * q0, D1 = -2.0 * c2 * x1 * x1 * q1;
    double P0 = -2.0 * x0 * q0, P1 = -2.0 * x1 * q1;
    auto make = [&](double f0, double f1, double d0, double d1) {
        if (interp == PSR_LINEAR) {
            const double m = 0.5 * (f0 + f1), d = f1 - f0;
            return make_float4((float)m, (float)d, (float)(m - k * d), 0.f);
        }
        // Hermite cubic in s = f + 1/2: a0 + a1 s + a2 s^2 + a3 s^3
        double a0 = f0, a1 = h * d0;
        double a2 = -3.0 * f0 - 2.0 * h * d0 + 3.0 * f1 - h * d1;
        double a3 = 2.0 * f0 + h * d0 - 2.0 * f1 + h * d1;
        return make_float4((float)(a0 + 0.5 * a1 + 0.25 * a2 + 0.125 * a3),
                           (float)(a1 + a2 + 0.75 * a3), (float)(a2 + 1.5 * a3), (float)a3);
    };
    tT[k] = make(T0, T1, D0, D1);
    if (tQ) tQ[k] = make(q0, q1, P0, P1);
}

int launch_table(int table_n, int interp, double x_c, void* d_out, void* d_q_out, void* stream)
{
    // one warp per block: FP64 work, one SM's FP64 pipe per warp (16 -> 4 us for 1024 intervals)
    int threads = 32, blocks = (table_n + 1 + threads - 1) / threads;
    table_kernel<<<blocks, threads, 0, (cudaStream_t)stream>>>(
        table_n, interp, x_c, reinterpret_cast<float4*>(d_out), reinterpret_cast<float4*>(d_q_out));
    return (int)cudaGetLastError();
}

// (1 - T(x)) / x^3, an entire function of x^2: its series
// (4 / sqrt(pi)) sum_n (-1)^n x^(2n) / (n! (2n + 3)) below x = 0.7 (where the
// difference would cancel; the first term left out is below 1e-18), the
// closed form above.
__device__ double core_h(double x)
{
    constexpr double c[16] = {
        0.7522527780636751, -0.45135166683820505, 0.16119702387078752, -0.0417918210035375,
        0.008548327023450852, -0.0014466399578147598, 0.00020895910501768752, -2.6339382985422794e-05,
        2.9458520444222863e-06, -2.961438563175843e-07, 2.703922166377944e-08, -2.2614621755160987e-09,
        1.7449553823426687e-10, -1.2497027937202137e-11, 8.350548621632764e-13, -5.2296365105174886e-14};
    const double x2 = x * x;
    if (x < 0.7) {
        double s = c[15];
#pragma unroll
        for (int n = 14; n >= 0; --n) s = fma(s, x2, c[n]);
        return s;
    }
    return (1.0 - (erfc(x) + 1.1283791670955126 * x * exp(-x2))) / (x2 * x);
}

// Core table (core_weight): entries k = 0..N-1 are minus the chord of H(q) =
// x_c^3 (1 - T) / x^3, q = (x / x_c)^2, over q N in [k, k + 1], moved by half
// its error at the interval's middle; entry N, met at and beyond the cutoff
// (q = 1, 1/r = 1), is -1.  Bound: the FP64 pipe; a step's leaf set builds its
// table anew, so the warps go to as many SMs (31 entries a warp, a block each;
// the next lane has the next node): 1024 intervals in blocks of 256 threads
// that evaluated three points each took 51 us.
constexpr int kCoreEntries = 31;
__global__ void core_table_kernel(int N, double x_c, float2* __restrict__ t)
{
    const int k = blockIdx.x * kCoreEntries + threadIdx.x;  // node; lane 31 is the next block's first
    const double s3 = x_c * x_c * x_c, step = 1.0 / N;      // N is a power of two
    const double q0 = k * step;
    const double h0 = s3 * core_h(x_c * sqrt(q0)), hm = s3 * core_h(x_c * sqrt(q0 + 0.5 * step));
    const double h1 = __shfl_down_sync(kFull, h0, 1);
    if (threadIdx.x == kCoreEntries || k > N) return;
    const double D = (h1 - h0) * N;
    t[k] = k == N ? make_float2(-1.0f, 0.0f)
                  : make_float2((float)(-(h0 - D * q0 + 0.5 * (hm - 0.5 * (h0 + h1)))), (float)-D);
}

int launch_core_table(int table_n, double x_c, void* d_out, void* stream)
{
    const int blocks = (table_n + 1 + kCoreEntries - 1) / kCoreEntries;
    core_table_kernel<<<blocks, 32, 0, (cudaStream_t)stream>>>(table_n, x_c,
                                                                    reinterpret_cast<float2*>(d_out));
    return (int)cudaGetLastError();
}

// The packed variant takes the core form of a linear table from 1024
// intervals on and for x_c <= 3.5: there its interpolation error in T
// (3.2e-7 at x_c = 2.25 and 1024 intervals, 1.9e-6 at 3.5, as x_c^4) is no
// larger than the chord table's (8.0e-7 and 1.9e-6, as x_c^2).  Coarser
// tables stay the chord in x that a caller of such a table asks for, and
// PSR_KERNEL_SCALAR stays the chord form with its order of sums throughout.
bool fwd_core(int precision, int interp, int table_n, int variant, double x_c)
{
    return precision == PSR_FP32_TABLE && interp == PSR_LINEAR && variant == PSR_KERNEL_PACKED &&
           table_n >= 1024 && x_c <= 3.5;
}

// bytes of one table entry in shared memory (and in global for Taylor)
size_t table_entry_bytes(int interp)
{
    return interp == PSR_LINEAR ? 8 : interp == PSR_CUBIC ? 16 : 32;
}

// ---------------------------------------------------------------- launch --
constexpr int kMetaPerWarpHost = 34;  // 32 entry records + 2 target-box slots

size_t fwd_f32_smem(int precision, int interp, int table_n, int warps, int cap)
{
    size_t tab = precision != PSR_FP32_TABLE ? 0 : (size_t)(table_n + 1) * table_entry_bytes(interp);
    return ((tab + 15) & ~(size_t)15) + (size_t)warps * (cap + kMetaPerWarpHost) * 16;
}

int launch_fwd_f32(const FwdArgs& a, int precision, void* stream)
{
    size_t smem = fwd_f32_smem(precision, a.interp, a.table_n, a.warps_per_block, a.stage_cap);
    cudaStream_t st = (cudaStream_t)stream;
    const bool pk = a.variant == PSR_KERNEL_PACKED;
    if (a.rows == kRowsJoint)
        return pk ? launch_fwd_f32_variant<true, kRowsJoint>(a, precision, smem, st)
                  : launch_fwd_f32_variant<false, kRowsJoint>(a, precision, smem, st);
    if (a.rows == kRowsInTurn)
        return pk ? launch_fwd_f32_variant<true, kRowsInTurn>(a, precision, smem, st)
                  : launch_fwd_f32_variant<false, kRowsInTurn>(a, precision, smem, st);
    return pk ? launch_fwd_f32_variant<true, kRowsWhole>(a, precision, smem, st)
              : launch_fwd_f32_variant<false, kRowsWhole>(a, precision, smem, st);
}

int fwd_f32_occupancy(int precision, int interp, int accum, int warps, int table_n, int cap,
                      int variant, int core, int* out)
{
    size_t smem = fwd_f32_smem(precision, interp, table_n, warps, cap);
    const void* f = variant == PSR_KERNEL_PACKED
                        ? fwd_f32_kernel_ptr<true>(precision, interp, accum, core)
                        : fwd_f32_kernel_ptr<false>(precision, interp, accum, 0);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return (int)e;
    }
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, f, warps * 32, smem);
}

}  // namespace psr
