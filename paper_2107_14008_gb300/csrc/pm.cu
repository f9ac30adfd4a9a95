// Long-range particle-mesh (PM) accelerations of the PM-FMM split (paper,
// Section 2: phi_long solves Poisson's equation on a mesh with a Gaussian-
// filtered Green's function; the split radius is r_s = 1.2 L / N_PM).
//
//   1. k_cic_deposit  cloud-in-cell assignment of the masses onto the N^3 mesh
//                     (points at g L/N), FP32 atomics, density m / Delta^3
//   2. cuFFT R2C
//   3. k_pm_field     times -4 pi G exp(-k^2 r_s^2) / k^2, divided by the
//                     squared CIC window (assignment and interpolation) unless
//                     PSR_PM_NO_DECONVOLVE, and by N^3 (cuFFT does not
//                     normalise), zero at k = 0; then -i k_c for each axis c
//                     (Nyquist plane of axis c zeroed), three spectra
//   4. cuFFT C2R, the three axes as one batch (from N = 896 on one by one)
//   5. k_cic_interp   CIC interpolation of the three component meshes at the
//                     particles, written to (or added into) the output
//
// Bound.  The particle kernels by scattered L2 traffic (mesh points of particles
// in input order); their FP64 part, which the FP64 pipe would otherwise
// dominate (a warp instruction in 16 SM cycles, fmod hundreds of them), is two
// instructions per coordinate.  The mesh work by launches and passes: the
// Green's function, gradient and batch of three make it one pass and two
// transforms instead of four passes and four.  128^3 mesh and 2.1 M particles:
// 430 -> 213 us.
//
// The filter is exp(-k^2 r_s^2), the Fourier complement of the short-range
// erfc(r/2 r_s) of Eq. tr (the paper prints exp(-k^2/4r_s^2), which is not).
// cuFFT plans are made once per mesh size with automatic work-area allocation
// off: psr_pm_forces runs the FFTs in the caller's scratch.
#include <cuda_runtime.h>
#include <cufft.h>

#include <cmath>
#include <new>
#include <string>

#include "kcommon.cuh"

namespace psr {
void set_last_error(const std::string& msg);
}

using namespace psr;

struct psr_pm {
    int n;
    cufftHandle r2c, c2r;
    int batch;    // axes that one inverse transform takes
    size_t work;  // bytes of the larger cuFFT work area
};

namespace {

struct Mesh {
    size_t rho, phik, ak, acc, work, bytes;
};

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

Mesh mesh_layout(int n, size_t work)
{
    Mesh m{};
    const size_t nr = (size_t)n * n * n, nc = (size_t)n * n * (n / 2 + 1);
    size_t o = 0;
    m.rho = o;  o = a256(o + 4 * nr);
    m.phik = o; o = a256(o + 8 * nc);
    m.ak = o;   o = a256(o + 3 * 8 * nc);   // the batch's spectra and meshes, axis after axis;
                                            // phik and ak together hold 16 N^3 bytes too
    m.acc = o;  o = a256(o + 3 * 4 * nr);
    m.work = o; o = a256(o + work);
    m.bytes = o;
    return m;
}

struct CicPoint {
    int i[3][2];
    float w[3][2];
};

// Finite position -> the two mesh points and weights per axis.  In the sum
// u + 2^20, u = x / Delta < 1024, the high word's low 20 bits are floor(u) and
// the low word is its fraction in units of 2^-32.
__device__ __forceinline__ CicPoint cic_point(const double* p, double L, double inv_delta, int n)
{
    CicPoint c;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double v = p[a];
        if ((unsigned long long)__double_as_longlong(v) >= (unsigned long long)__double_as_longlong(L)) {
            v = fmod(v, L);  // outside [0, L)
            if (v < 0) v += L;
            if (!(v < L)) v = 0.0;
        }
        const double t = __dadd_rn(__dmul_rn(v, inv_delta), 1048576.0);
        int i0 = __double2hiint(t) & 0xfffff;
        if (i0 >= n) i0 = 0;  // rounded up to n
        const float f = __uint2float_rn((unsigned)__double2loint(t)) * 2.3283064365386963e-10f;
        c.i[a][0] = i0;
        c.i[a][1] = i0 + 1 == n ? 0 : i0 + 1;
        c.w[a][0] = 1.0f - f;
        c.w[a][1] = f;
    }
    return c;
}

__device__ __forceinline__ bool finite3(const double* p)
{
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        ok = ok && ((unsigned long long)__double_as_longlong(p[a]) & 0x7fffffffffffffffULL) < 0x7ff0000000000000ULL;
    return ok;
}

// A particle with a non-finite coordinate deposits nothing (and is skipped
// by the interpolation).  The two z neighbours of each of the four rows take one
// 8-byte reduction, which wants the first at an even place: pairs that start at
// an odd z go to a second mesh, one place further along (rows of N + 2: cell z at
// z + 1, and cell 0 as the wrapped neighbour of N - 1 at N + 1), which
// k_cic_join adds to the first.  Four reductions per particle instead of
// eight; the L2 traffic of scattered reductions is what the kernel waits for.
__global__ void k_cic_deposit(const double* __restrict__ pos, const double* __restrict__ mass,
                              int64_t np, double L, double inv_delta, int n, float m_default,
                              float inv_vol, float* __restrict__ rho, float* __restrict__ odd)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= np) return;
    const double p[3] = {pos[3 * j], pos[3 * j + 1], pos[3 * j + 2]};
    if (!finite3(p)) return;
    const float m = (mass ? (float)mass[j] : m_default) * inv_vol;
    const CicPoint c = cic_point(p, L, inv_delta, n);
    const int z = c.i[2][0], stride = (z & 1) ? n + 2 : n;
    float* const mesh = (z & 1) ? odd + z + 1 : rho + z;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const float wab = m * c.w[0][a] * c.w[1][b];
            asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(
                             mesh + ((size_t)c.i[0][a] * n + c.i[1][b]) * stride),
                         "f"(wab * c.w[2][0]), "f"(wab * c.w[2][1])
                         : "memory");
        }
}

// rho += the mesh of the odd pairs; one thread per cell pair (z, z + 1), z even
__global__ void k_cic_join(float2* __restrict__ rho, const float* __restrict__ odd, int n)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int h = n / 2;
    if (t >= (int64_t)n * n * h) return;
    const int z = 2 * (int)(t % h);
    const float* row = odd + (t / h) * (n + 2);
    float2 v = rho[t];
    v.x += z ? row[z + 1] : row[n + 1];  // cell 0 is only ever a wrapped neighbour
    v.y += row[z + 2];
    rho[t] = v;
}

// the three component meshes as one mesh of float4
__global__ void k_pm_gather(const float* __restrict__ g, int64_t nr, float4* __restrict__ out)
{
    const int64_t i = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);  // nr is a multiple of 8
    if (i >= nr) return;
    const float4 x = *reinterpret_cast<const float4*>(g + i), y = *reinterpret_cast<const float4*>(g + nr + i),
                 z = *reinterpret_cast<const float4*>(g + 2 * nr + i);
    out[i] = make_float4(x.x, y.x, z.x, 0.f);
    out[i + 1] = make_float4(x.y, y.y, z.y, 0.f);
    out[i + 2] = make_float4(x.z, y.z, z.z, 0.f);
    out[i + 3] = make_float4(x.w, y.w, z.w, 0.f);
}

// signed frequency of FFT index i (index n/2 is the Nyquist frequency -n/2)
__device__ __forceinline__ int freq(int i, int n) { return i < n / 2 ? i : i - n; }

// ak[c] = -i k_c times the Green's function (and 1 / N^3) times phik, the
// Nyquist plane of axis c zeroed.  Filter and window are products over the
// axes, exp(-k_a^2 r_s^2) / sinc^4(k_a Delta / 2): each block forms the N/2 + 1
// values of one axis in shared memory and multiplies three of them per mode
// (an exponential, three sines and six divisions per mode before).
__global__ void __launch_bounds__(256) k_pm_field(const cufftComplex* __restrict__ phik,
                                                  cufftComplex* __restrict__ ak, int n, float kf, float r_s2,
                                                  float g4pi, float half_delta, int deconvolve, float inv_n3)
{
    __shared__ float s_axis[513];
    const int nz = n / 2 + 1;
    for (int i = threadIdx.x; i < nz; i += blockDim.x) {
        const float k = kf * i, y = k * half_delta;
        float w = expf(-k * k * r_s2);
        if (deconvolve && i) {
            const float s = sinf(y) / y, s2 = s * s;
            w /= s2 * s2;
        }
        s_axis[i] = w;
    }
    __syncthreads();
    const int nc = n * n * nz;  // at most 2^29 + 2^20
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nc; t += gridDim.x * blockDim.x) {
        const int iz = t % nz, row = t / nz, iy = row % n, ix = row / n;
        const int fx = freq(ix, n), fy = freq(iy, n);
        const float kx = kf * fx, ky = kf * fy, kz = kf * iz;
        const float k2 = kx * kx + ky * ky + kz * kz;
        float g = 0.0f;
        if (k2 > 0.0f) g = -g4pi / k2 * inv_n3 * (s_axis[abs(fx)] * s_axis[abs(fy)] * s_axis[iz]);
        const cufftComplex v = phik[t];
        const float re = v.x * g, im = v.y * g;
        const float k3[3] = {2 * abs(fx) == n ? 0.0f : kx, 2 * abs(fy) == n ? 0.0f : ky, 2 * iz == n ? 0.0f : kz};
#pragma unroll
        for (int c = 0; c < 3; ++c)  // -i k (x + i y) = k y - i k x
            ak[(size_t)c * nc + t] = make_float2(k3[c] * im, -k3[c] * re);
    }
}

// Bound: lines looked up per load of a warp's scattered lanes, so a particle's
// eight points are eight 16-byte loads of (a_x, a_y, a_z) instead of 24 of 4.
__global__ void k_cic_interp(const double* __restrict__ pos, int64_t np, double L,
                             double inv_delta, int n, const float4* __restrict__ g,
                             float* __restrict__ acc, int accumulate)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= np) return;
    const double p[3] = {pos[3 * j], pos[3 * j + 1], pos[3 * j + 2]};
    if (!finite3(p)) return;
    const CicPoint c = cic_point(p, L, inv_delta, n);
    float s[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const float4 v = g[((size_t)c.i[0][a] * n + c.i[1][b]) * n + c.i[2][d]];
                const float w = c.w[0][a] * c.w[1][b] * c.w[2][d];
                s[0] = fmaf(w, v.x, s[0]);
                s[1] = fmaf(w, v.y, s[1]);
                s[2] = fmaf(w, v.z, s[2]);
            }
    for (int a = 0; a < 3; ++a) acc[3 * j + a] = accumulate ? acc[3 * j + a] + s[a] : s[a];
}

int pfail(int code, const std::string& msg)
{
    set_last_error(msg);
    return code;
}

int cuda_err(cudaError_t e, const char* what)
{
    return pfail(PSR_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

int fft_err(cufftResult r, const char* what)
{
    return pfail(PSR_E_CUDA, std::string(what) + ": cuFFT status " + std::to_string((int)r));
}

unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

extern "C" {

int psr_pm_create(int n_pm, psr_pm** out)
{
    if (!out) return pfail(PSR_E_ARG, "null output");
    *out = nullptr;
    if (n_pm < 8 || n_pm > 1024 || (n_pm & 1))
        return pfail(PSR_E_ARG, "n_pm must be even and in [8, 1024]");
    psr_pm* pm = new (std::nothrow) psr_pm();
    if (!pm) return pfail(PSR_E_NOMEM, "out of host memory");
    pm->n = n_pm;
    // three axes at once while their 3 N^3 reals stay below 2^31 (N < 895), one by
    // one beyond: the plan's counts are 32-bit
    const int64_t cells = (int64_t)n_pm * n_pm * n_pm;
    pm->batch = 3 * cells < ((int64_t)1 << 31) ? 3 : 1;
    size_t w1 = 0, w2 = 0;
    int dims[3] = {n_pm, n_pm, n_pm}, spec[3] = {n_pm, n_pm, n_pm / 2 + 1};
    cufftResult r;
    if ((r = cufftCreate(&pm->r2c)) != CUFFT_SUCCESS) {
        delete pm;
        return fft_err(r, "cufftCreate");
    }
    if ((r = cufftCreate(&pm->c2r)) != CUFFT_SUCCESS) {
        cufftDestroy(pm->r2c);
        delete pm;
        return fft_err(r, "cufftCreate");
    }
    if ((r = cufftSetAutoAllocation(pm->r2c, 0)) != CUFFT_SUCCESS ||
        (r = cufftSetAutoAllocation(pm->c2r, 0)) != CUFFT_SUCCESS ||
        (r = cufftMakePlan3d(pm->r2c, n_pm, n_pm, n_pm, CUFFT_R2C, &w1)) != CUFFT_SUCCESS ||
        (r = cufftMakePlanMany(pm->c2r, 3, dims, spec, 1, n_pm * n_pm * (n_pm / 2 + 1), dims, 1,
                               n_pm * n_pm * n_pm, CUFFT_C2R, pm->batch, &w2)) != CUFFT_SUCCESS) {
        cufftDestroy(pm->r2c);
        cufftDestroy(pm->c2r);
        delete pm;
        return fft_err(r, "cuFFT plan");
    }
    pm->work = w1 > w2 ? w1 : w2;
    *out = pm;
    return PSR_OK;
}

int psr_pm_scratch_bytes(const psr_pm* pm, size_t* bytes)
{
    if (!pm || !bytes) return pfail(PSR_E_ARG, "null argument");
    *bytes = mesh_layout(pm->n, pm->work).bytes;
    return PSR_OK;
}

int psr_pm_forces(psr_pm* pm, const double* d_pos, const double* d_mass, int64_t n,
                  const psr_box* box, int flags, void* d_scratch, size_t scratch_bytes,
                  float* d_acc, void* stream)
{
    if (!pm || !box || ((!d_pos || !d_acc) && n > 0) || n < 0)
        return pfail(PSR_E_ARG, "null argument or n < 0");
    if (flags & ~(PSR_PM_ACCUMULATE | PSR_PM_NO_DECONVOLVE))
        return pfail(PSR_E_ARG, "unknown PM flags");
    if (!(std::isfinite(box->L) && box->L > 0) || !(std::isfinite(box->r_s) && box->r_s > 0) ||
        !std::isfinite(box->G))
        return pfail(PSR_E_ARG, "L, r_s must be finite and positive");
    const int N = pm->n;
    const Mesh M = mesh_layout(N, pm->work);
    if (!d_scratch || scratch_bytes < M.bytes || (reinterpret_cast<uintptr_t>(d_scratch) & 255))
        return pfail(PSR_E_WORKSPACE, "scratch must be 256-byte aligned and at least " +
                                          std::to_string(M.bytes) + " bytes");
    if (n == 0) return PSR_OK;
    cudaStream_t st = (cudaStream_t)stream;
    char* s = static_cast<char*>(d_scratch);
    float* rho = (float*)(s + M.rho);
    cufftComplex* phik = (cufftComplex*)(s + M.phik);
    cufftComplex* ak = (cufftComplex*)(s + M.ak);
    float* g = (float*)(s + M.acc);
    const double L = box->L, delta = L / N;
    const int64_t nr = (int64_t)N * N * N, nc = (int64_t)N * N * (N / 2 + 1);
    cudaError_t e;
    cufftResult r;
    // the deposit's second mesh, and later the float4 mesh, take the spectra's place
    float* odd = (float*)phik;
    float4* g4 = (float4*)phik;
    if ((e = cudaMemsetAsync(rho, 0, 4 * (size_t)nr, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(odd, 0, 8 * (size_t)nc, st)) != cudaSuccess)
        return cuda_err(e, "cudaMemsetAsync");
    k_cic_deposit<<<nblk(n, 256), 256, 0, st>>>(d_pos, d_mass, n, L, 1.0 / delta, N,
                                                (float)(1.0 / (double)n),
                                                (float)(1.0 / (delta * delta * delta)), rho, odd);
    k_cic_join<<<nblk(nr / 2, 256), 256, 0, st>>>((float2*)rho, odd, N);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_err(e, "deposit kernel");
    if ((r = cufftSetStream(pm->r2c, st)) != CUFFT_SUCCESS ||
        (r = cufftSetStream(pm->c2r, st)) != CUFFT_SUCCESS ||
        (r = cufftSetWorkArea(pm->r2c, s + M.work)) != CUFFT_SUCCESS ||
        (r = cufftSetWorkArea(pm->c2r, s + M.work)) != CUFFT_SUCCESS)
        return fft_err(r, "cuFFT stream / work area");
    if ((r = cufftExecR2C(pm->r2c, rho, phik)) != CUFFT_SUCCESS) return fft_err(r, "cufftExecR2C");
    const float kf = (float)(2.0 * M_PI / L);
    k_pm_field<<<(unsigned)(nc < 256 * 1216 ? nblk(nc, 256) : 1216), 256, 0, st>>>(
        phik, ak, N, kf, (float)(box->r_s * box->r_s), (float)(4.0 * M_PI * box->G),
        (float)(0.5 * delta), (flags & PSR_PM_NO_DECONVOLVE) ? 0 : 1, (float)(1.0 / (double)nr));
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_err(e, "field kernel");
    for (int c = 0; c < 3; c += pm->batch)
        if ((r = cufftExecC2R(pm->c2r, ak + c * nc, g + c * nr)) != CUFFT_SUCCESS)
            return fft_err(r, "cufftExecC2R");
    k_pm_gather<<<nblk(nr / 4, 256), 256, 0, st>>>(g, nr, g4);
    k_cic_interp<<<nblk(n, 256), 256, 0, st>>>(d_pos, n, L, 1.0 / delta, N, g4, d_acc,
                                               (flags & PSR_PM_ACCUMULATE) ? 1 : 0);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_err(e, "interpolation kernel");
    return PSR_OK;
}

void psr_pm_free(psr_pm* pm)
{
    if (!pm) return;
    cufftDestroy(pm->r2c);
    cufftDestroy(pm->c2r);
    delete pm;
}

}  // extern "C"
