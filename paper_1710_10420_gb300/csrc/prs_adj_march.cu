// prs_adj_march.cu -- launching the adjoint's register march.
#include <math.h>

#include <algorithm>
#include <atomic>

#include "prs_adj_march.cuh"
#include "prs_adj_march.h"
#include "prs_chain.h"

namespace prs {

cudaError_t launch_adj_march(const Geo& g, const float* phi, const float* v, const float coef[5], const float* lt_in,
                             float* lt_out, float* lphi, const double run_const[6], bool last, const DiagScratch& scr,
                             cudaStream_t st)
{
    using namespace march;
    if (g.dims != 3 || (int64_t)g.nx * g.ny >= ((int64_t)1 << 32)) return cudaErrorNotSupported;
    AdjArgs a;
    a.lt_in = lt_in;
    a.lt_out = lt_out;
    a.lphi = lphi;
    a.phi = phi;
    a.v = v;
    a.k = AdjStepF{coef[0], coef[1], coef[2], coef[3], coef[4]};
    const double* c = run_const;
    a.rc = RunConst<float>{(float)c[0], (float)c[1], (float)c[2], (float)c[3], (float)c[4], (float)c[5]};
    a.scr = scr;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nz = g.nz;
    a.last = last;
    a.nstrips = (g.nx + width(1, 2) - 1) / width(1, 2);
    a.ygroups = (g.ny + kAdjRows * kWarps - 1) / (kAdjRows * kWarps);
    // chunks: whole waves against the two planes each re-reads, one partial slot a block
    const int64_t tiles = (int64_t)a.nstrips * a.ygroups;
    if (tiles > scr.max_blocks) return cudaErrorNotSupported;
    const double slots = 3.0 * sm_count_current();
    double least = 1e300;
    a.cz = g.nz;
    for (int nc = 1; nc <= g.nz && tiles * nc <= scr.max_blocks; nc += nc < 32 ? 1 : nc / 16) {
        const int cz = (g.nz + nc - 1) / nc, n = (g.nz + cz - 1) / cz;
        const double w = (double)tiles * n / slots;
        const double cost = (w <= 1.0 ? 1.1 - 0.1 * w : 0.5 * (ceil(w) + w + 0.35)) * (cz + 2);
        if (cost < least * 0.999) least = cost, a.cz = cz;
    }
    const int64_t blocks = tiles * ((g.nz + a.cz - 1) / a.cz);
    const uintptr_t bits = (uintptr_t)lt_in | (uintptr_t)lt_out | (uintptr_t)lphi | (uintptr_t)phi | (uintptr_t)v;
    const bool vec = g.nx % 2 == 0 && bits % 8 == 0;
    constexpr size_t smem = (size_t)kWarps * kAdjRing * kAdjSlot * sizeof(float);
    static std::atomic<unsigned long long> attr[2];
    void (*kernel)(AdjArgs) = vec ? k_adj_march<true> : k_adj_march<false>;
    const cudaError_t e = smem_limit_once(attr[vec], (const void*)kernel, (int)smem);
    return e != cudaSuccess ? e : launch_chained(kernel, dim3((unsigned)blocks), kThreads, smem, st, a);
}

}  // namespace prs
