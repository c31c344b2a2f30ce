// prs_march2d_launch.cuh -- the launcher of one arithmetic of the 2D register march; each is
// compiled in a file of its own.
#pragma once

#include "prs_chain.h"
#include "prs_march2d.cuh"

namespace prs {

namespace march {

inline void set_kick(Fold32::K& k, const double c[3], const double rc[6])
{
    const KickP p = kick_packed(kick_f32(c, rc), (float)rc[0]);
    k = Fold32::K{p.c1, p.g, p.k1, p.nk2};
}
inline void set_kick(StepCoef<float>& k, const double c[3], const double*)
{
    k = StepCoef<float>{(float)c[0], (float)c[1], (float)c[2]};
}

template <class M, int T, int COLS, bool VEC, int NR>
cudaError_t launch_one(const Geo& g, int cy, int nruns, const MarchRun* runs, cudaStream_t st)
{
    Args<M, T, NR> a;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nruns = nruns;
    a.nstrips = (g.nx + width(T, COLS) - 1) / width(T, COLS);
    a.cy = cy;
    a.nchunks = (g.ny + cy - 1) / cy;
    for (int r = 0; r < nruns; ++r) {
        const MarchRun& q = runs[r];
        a.phi_in[r] = (const float*)q.phi_in;
        a.phi_out[r] = (float*)q.phi_out;
        a.v_in[r] = (const float*)q.v_in;
        a.v_out[r] = (float*)q.v_out;
        for (int l = 0; l < T; ++l) set_kick(a.k[r][l], q.coef[l], q.run_const);
        const double* c = q.run_const;
        a.rc[r] = RunConst<float>{(float)c[0], (float)c[1], (float)c[2], (float)c[3], (float)c[4], (float)c[5]};
    }
    const int64_t warps = (int64_t)a.nstrips * a.nchunks * nruns, blocks = (warps + kWarps - 1) / kWarps;
    if (warps > 0x7fffffff) return cudaErrorInvalidValue;
    return launch_chained(k_march2d<M, T, COLS, VEC, NR>, dim3((unsigned)blocks), kThreads, 0, st, a);
}

template <class M, int T, int COLS>
cudaError_t launch_cols(const Geo& g, int cy, int nruns, const MarchRun* runs, cudaStream_t st)
{
    uintptr_t bits = 0;
    for (int r = 0; r < nruns; ++r)
        bits |= (uintptr_t)runs[r].phi_in | (uintptr_t)runs[r].phi_out | (uintptr_t)runs[r].v_in |
                (uintptr_t)runs[r].v_out;
    const bool vec = g.nx % COLS == 0 && bits % (4 * COLS) == 0;
    if constexpr (M::kShared) {
        if (nruns > 1)
            return vec ? launch_one<M, T, COLS, true, kMarchMaxRuns>(g, cy, nruns, runs, st)
                       : launch_one<M, T, COLS, false, kMarchMaxRuns>(g, cy, nruns, runs, st);
    }
    return vec ? launch_one<M, T, COLS, true, 1>(g, cy, 1, runs, st)
               : launch_one<M, T, COLS, false, 1>(g, cy, 1, runs, st);
}

template <class M, int T>
cudaError_t launch_t(const Geo& g, const MarchShape& s, int nruns, const MarchRun* runs, cudaStream_t st)
{
    return s.cols == 4 ? launch_cols<M, T, 4>(g, s.cy, nruns, runs, st) : launch_cols<M, T, 2>(g, s.cy, nruns, runs, st);
}

template <class M>
cudaError_t launch(const Geo& g, int t, const MarchShape& s, int nruns, const MarchRun* runs, cudaStream_t st)
{
    switch (t) {
        case 1: return launch_t<M, 1>(g, s, nruns, runs, st);
        case 2: return launch_t<M, 2>(g, s, nruns, runs, st);
        case 3: return launch_t<M, 3>(g, s, nruns, runs, st);
        case 4: return launch_t<M, 4>(g, s, nruns, runs, st);
        case 5: return launch_t<M, 5>(g, s, nruns, runs, st);
        case 6: return launch_t<M, 6>(g, s, nruns, runs, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace march

cudaError_t launch_march_fold32(const Geo& g, int t, const MarchShape& s, int nruns, const MarchRun* runs,
                                cudaStream_t st);
cudaError_t launch_march_plain32(const Geo& g, int t, const MarchShape& s, int nruns, const MarchRun* runs,
                                 cudaStream_t st);

}  // namespace prs
