// prs_generic.cu -- initial conditions and the any-shape leapfrog step.
//
//   init     : SplitMix64 random field (Sec. III initial conditions), dphi = 0
//   step     : Eqs. 3-5 with the damping of Eq. 6, one thread per site, any box
//              side >= 3 (used for PRS_REPRO and for FP32 3D boxes whose planes hold
//              2^32 sites or more)
//   copy     : both fields of a state in one launch
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>

#include "prs_arith.cuh"
#include "prs_chain.h"
#include "prs_internal.h"
#include "prs_ptx.cuh"
#include "prs_site.cuh"

namespace prs {

// ------------------------------------------------------------ initial field

__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t idx)
{
    // Output number idx of SplitMix64 started at state `seed` (Steele, Lea & Flood 2014).
    uint64_t z = seed + (idx + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

template <typename R>
__global__ void k_init_random(R* __restrict__ phi, R* __restrict__ dphi, int64_t S, uint64_t seed, bool zero_dphi)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S; s += (int64_t)gridDim.x * blockDim.x) {
        uint64_t k = splitmix64_at(seed, (uint64_t)s) >> 40;  // top 24 bits
        // (2k+1) 2^-24 - 1 is exact in both float and double
        double u = (double)(2ull * k + 1ull) * (1.0 / 16777216.0) - 1.0;
        phi[s] = (R)u;
        if (zero_dphi) dphi[s] = (R)0;
    }
}

static int grid_for(int64_t work, int block)
{
    int64_t b = (work + block - 1) / block;
    const int64_t cap = 152 * 64;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

cudaError_t launch_init_random(const Geo& g, int precision, uint64_t seed, void* phi, void* dphi, bool zero_dphi,
                               cudaStream_t st)
{
    const int block = 256;
    int grid = grid_for(g.S, block);
    if (precision == PRS_FP32)
        k_init_random<float><<<grid, block, 0, st>>>((float*)phi, (float*)dphi, g.S, seed, zero_dphi);
    else
        k_init_random<double><<<grid, block, 0, st>>>((double*)phi, (double*)dphi, g.S, seed, zero_dphi);
    return cudaGetLastError();
}

// Grid of the row-wise kernels: up to four x blocks per row (more where a few rows would leave SMs without
// one: 10^6 x 3 doubles 102 us a step, with four 1340), y blocks striding over the rows, at most cap blocks
// in all.
static dim3 rows_grid(const Geo& g, int cap)
{
    const int64_t rows = (int64_t)g.ny * g.nz;
    const int most = 4 * rows < cap ? (int)(cap / rows) : 4;
    const int gx = (g.nx + 255) / 256 < most ? (g.nx + 255) / 256 : most;
    int64_t gy = cap / gx;
    if (gy > rows) gy = rows;
    if (gy < 1) gy = 1;
    return dim3((unsigned)gx, (unsigned)gy, 1);
}

// --------------------------------------------------------- generic step

template <typename R, bool REPRO, int D>
__global__ void k_step_generic(const R* phi, R* phi_out, const R* dphi, R* dphi_out, Geo g, StepCoef<R> k,
                               RunConst<R> rc, KickD kd)
{
    chain_enter();
    const int64_t nx = g.nx, ny = g.ny, nz = g.nz;
    const int64_t plane = nx * ny;
    // rows of x: y blocks stride over the rows (y, z decoded once per row), x threads over a row
    for (int64_t r = blockIdx.y; r < ny * nz; r += gridDim.y) {
        const int64_t y = r % ny, z = r / ny;
        const int64_t row = r * nx;
        const int64_t ypo = ((y + 1 == ny ? 0 : y + 1) - y) * nx, ymo = ((y == 0 ? ny - 1 : y - 1) - y) * nx;
        const int64_t zpo = ((z + 1 == nz ? 0 : z + 1) - z) * plane, zmo = ((z == 0 ? nz - 1 : z - 1) - z) * plane;
        for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < nx; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = row + x;
        R c = phi[s];
        R xp = phi[row + (x + 1 == nx ? 0 : x + 1)];
        R xm = phi[row + (x == 0 ? nx - 1 : x - 1)];
        R yp = phi[s + ypo];
        R ym = phi[s + ymo];
        R zp = (R)0, zm = (R)0;
        if (D == 3) {
            zp = phi[s + zpo];
            zm = phi[s + zmo];
        }
        R v = dphi[s];
        R pn;
        if constexpr (sizeof(R) == 8 && !REPRO)
            site_update_folded<D>(c, xp, xm, yp, ym, zp, zm, v, pn, kd, rc.deta);
        else
            site_update<R, REPRO, D>(c, xp, xm, yp, ym, zp, zm, v, pn, k, rc);
        dphi_out[s] = v;
        phi_out[s] = pn;
        }
    }
}

template <typename R>
static RunConst<R> make_rc(const double rcd[6])
{
    return RunConst<R>{(R)rcd[0], (R)rcd[1], (R)rcd[2], (R)rcd[3], (R)rcd[4], (R)rcd[5]};
}

template <typename R, bool REPRO>
static cudaError_t step_generic_t(const Geo& g, const void* in, void* out, const void* dphi, void* dphi_out,
                                  const double coef[3], const double rcd[6], cudaStream_t st)
{
    const int block = 256;
    const dim3 grid = rows_grid(g, 152 * 16);
    StepCoef<R> k{(R)coef[0], (R)coef[1], (R)coef[2]};
    RunConst<R> rc = make_rc<R>(rcd);
    const KickD kd = kick_f64(coef, rcd);
    void (*kernel)(const R*, R*, const R*, R*, Geo, StepCoef<R>, RunConst<R>, KickD) = k_step_generic<R, REPRO, 3>;
    if (g.dims == 2) {
        if constexpr (sizeof(R) == 4) return cudaErrorNotSupported;  // FP32 2D boxes take the register march
        else kernel = k_step_generic<R, REPRO, 2>;
    }
    return launch_chained(kernel, grid, block, 0, st, (const R*)in, (R*)out, (const R*)dphi, (R*)dphi_out, g, k, rc, kd);
}

cudaError_t launch_step_generic(const Geo& g, int precision, bool repro, const void* in, void* out, const void* dphi,
                                void* dphi_out, const double coef[3], const double rcd[6], const MarchShape& shape,
                                cudaStream_t st)
{
    if (precision == PRS_FP32) return step_generic_t<float, false>(g, in, out, dphi, dphi_out, coef, rcd, st);
    if (repro) return step_generic_t<double, true>(g, in, out, dphi, dphi_out, coef, rcd, st);
    const cudaError_t e = launch_step_fix64(g, (const double*)in, (double*)out, (const double*)dphi, (double*)dphi_out,
                                            coef, rcd, shape, st);
    if (e != cudaErrorNotSupported) return e;
    return step_generic_t<double, false>(g, in, out, dphi, dphi_out, coef, rcd, st);
}

// ---------------------------------------------------------- state copies

// phi and dphi of a state in one launch, 64 bytes a thread and turn.  Bound by HBM for large boxes
// (1024^3: what two device-to-device copies take); for small ones by the launch, of which this
// saves one (256^2: 4 us of 81).
__global__ void __launch_bounds__(256) k_copy_state(const float4* p, float4* po, const float4* v, float4* vo, int64_t n)
{
    chain_enter();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * 4;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x * 4 + threadIdx.x; i < 2 * n; i += stride) {
        float4 a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t j = i + u * (int64_t)blockDim.x;
            if (j < 2 * n) a[u] = j < n ? __ldcs(p + j) : __ldcs(v + (j - n));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t j = i + u * (int64_t)blockDim.x;
            if (j < n) po[j] = a[u];
            else if (j < 2 * n) vo[j - n] = a[u];
        }
    }
}

// Whether the kernel may read bytes at p: memory of the current device, in one allocation.  (A copy
// by the driver finds out by itself and returns an error; a kernel would fault.)
static bool on_device(const void* p, size_t bytes)
{
    using Range = decltype(&cuMemGetAddressRange);
    static std::atomic<Range> fn{nullptr};
    Range range = fn.load(std::memory_order_acquire);
    if (!range) {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !f) {
            cudaGetLastError();
            return false;
        }
        range = reinterpret_cast<Range>(f);
        fn.store(range, std::memory_order_release);
    }
    cudaPointerAttributes attr;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    CUdeviceptr base = 0;
    size_t size = 0;
    return attr.type == cudaMemoryTypeDevice && attr.device == dev &&
           range(&base, &size, (CUdeviceptr)p) == CUDA_SUCCESS && (CUdeviceptr)p - base <= size &&
           bytes <= size - (size_t)((CUdeviceptr)p - base);
}

cudaError_t launch_copy_state(const void* phi, void* phi_out, const void* dphi, void* dphi_out, size_t bytes,
                              cudaStream_t st)
{
    const uintptr_t a = (uintptr_t)phi, b = (uintptr_t)phi_out, c = (uintptr_t)dphi, d = (uintptr_t)dphi_out;
    auto apart = [&](uintptr_t s, uintptr_t t) { return s + bytes <= t || t + bytes <= s; };
    if (((a | b | c | d | bytes) & 15u) || !apart(a, b) || !apart(a, d) || !apart(c, b) || !apart(c, d) ||
        !apart(b, d) || !on_device(phi, bytes) || !on_device(dphi, bytes)) {
        cudaError_t e = cudaSuccess;  // one after the other
        if (a != b) e = cudaMemcpyAsync(phi_out, phi, bytes, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess && c != d) e = cudaMemcpyAsync(dphi_out, dphi, bytes, cudaMemcpyDeviceToDevice, st);
        return e;
    }
    const int64_t n = (int64_t)(bytes / 16);
    return launch_chained(k_copy_state, dim3((unsigned)grid_for(2 * n, 1024)), 256, 0, st, (const float4*)phi,
                          (float4*)phi_out, (const float4*)dphi, (float4*)dphi_out, n);
}

}  // namespace prs
