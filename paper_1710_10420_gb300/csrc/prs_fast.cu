// prs_fast.cu -- the FP32 leapfrog step (Eqs. 3-6), one step per pass, for 3D boxes whose x side is a multiple
// of 128 and at most 1024 (the single steps that the passes of several leave over).  One kernel
// applies Eqs. 3-5 in a single pass over HBM (read phi and dphi once, write them once: 16 B per
// site-update), where the paper's OpenCL code ran one kernel per equation.  The tile routines (bulk-async
// plane staging, shuffles, bounded waits) live in prs_tile.cuh; this file sizes
// the grids: one CTA per tile, two resident per SM.
#include <cuda_runtime.h>

#include "prs_arith.cuh"
#include "prs_chain.h"
#include "prs_internal.h"
#include "prs_ptx.cuh"
#include "prs_tile.cuh"

namespace prs {

template <int ITEMS>
__global__ void __launch_bounds__(kFastThreads, 2)
    k_step3d_f32(const float* __restrict__ phi_in, float* __restrict__ phi_out, const float* v, float* v_out, int nx,
                 int ny, int nz, int ty, int cz, KickF k, RunConst<float> rc, unsigned int* err)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    chain_enter();
    const int ytiles = ny / ty;
    Tile3D T{phi_in, phi_out, v, v_out, nx, ny, nz, ty, (int)(blockIdx.x % ytiles) * ty,
             (int)(blockIdx.x / ytiles) * cz, 0};
    T.zn = min(cz, nz - T.z0);
    tile3d<ITEMS>(T, k, rc, smem_raw, err);
}

// ------------------------------------------------------------------ dispatch

static constexpr int kItems = 4;  // float4 per thread per plane: 4096 sites per plane tile

static size_t smem3d(int nx, int ty) { return tile_smem3d(nx, ty); }

static constexpr size_t kFastSmemMax = 100 * 1024;

bool fast_step_ok(const Geo& g, int precision)
{
    if (precision != PRS_FP32) return false;
    if (g.nx % 128 != 0 || g.nx > kItems * 1024 || (kItems * 1024) % g.nx != 0) return false;
    const int t = kItems * 1024 / g.nx;  // rows per plane tile
    if (g.ny % t != 0) return false;
    return g.dims == 2 || smem3d(g.nx, t) <= kFastSmemMax;
}

// Shortest chunks the planner considers: 4 planes.  A small box must be
// cut into enough chunks to occupy the GPU, or each pass is bound by the latency of a few CTAs
// marching long chunks (128^3 22.1 us per step with at least 16 planes a chunk against 8.2; large
// boxes pick long chunks either way).
constexpr int kMinPlanes = 4;

// Number of z-chunks: balance whole waves of resident
// CTAs against the two halo planes each chunk re-reads.
static int pick_chunks(int tiles, int len, int min_len, int slots)
{
    int best = 1;
    double best_score = -1.0;
    for (int nc = 1; nc <= len / min_len || nc == 1; ++nc) {
        int c = (len + nc - 1) / nc;
        int n = (len + c - 1) / c;
        long long blocks = (long long)tiles * n;
        long long waves = (blocks + slots - 1) / slots;
        double fill = (double)blocks / (double)(waves * slots);
        double halo = (double)c / (double)(c + 2);
        double score = fill * halo * (waves >= 2 ? 1.0 : 0.9);
        if (score > best_score + 1e-9) {
            best_score = score;
            best = n;
        }
        if (nc > 4096) break;
    }
    return best;
}

cudaError_t launch_step_fast(const Geo& g, const float* in, float* out, const float* v, float* v_out,
                             KickF k, RunConst<float> rc, unsigned int* err, cudaStream_t st)
{
    if (g.dims != 3 || !fast_step_ok(g, PRS_FP32)) return cudaErrorNotSupported;
    static std::atomic<unsigned long long> attr{0};
    const int t = kItems * 1024 / g.nx;
    const int slots = 2 * sm_count_current();  // two resident CTAs per SM
    const size_t sm = smem3d(g.nx, t);
    const cudaError_t e = smem_limit_once(attr, (const void*)k_step3d_f32<kItems>, (int)kFastSmemMax);
    if (e != cudaSuccess) return e;
    const int ytiles = g.ny / t;
    int nchunks = pick_chunks(ytiles, g.nz, kMinPlanes, slots);
    const int cz = (g.nz + nchunks - 1) / nchunks;
    nchunks = (g.nz + cz - 1) / cz;
    return launch_chained(k_step3d_f32<kItems>, dim3((unsigned)(ytiles * nchunks)), kFastThreads, sm, st, in, out, v,
                          v_out, g.nx, g.ny, g.nz, t, cz, k, rc, err);
}

}  // namespace prs
