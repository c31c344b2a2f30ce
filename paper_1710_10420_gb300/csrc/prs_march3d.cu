// prs_march3d.cu -- launching the 3D register march.
#include <math.h>

#include <algorithm>
#include <atomic>

#include "prs_march2d_launch.cuh"
#include "prs_march3d.cuh"

namespace prs {

namespace march {

template <class M, int T, bool VEC, int NR>
cudaError_t launch3_one(const Geo& g, int nruns, const MarchRun* runs, cudaStream_t st, int cz)
{
    constexpr size_t smem = (size_t)kWarps * kRing3 * (2 * kRows + 4 * T - 2) * 64 * sizeof(float);
    static std::atomic<unsigned long long> attr{0};
    const cudaError_t e = smem_limit_once(attr, (const void*)k_march3d<M, T, VEC, NR>, (int)smem);
    if (e != cudaSuccess) return e;
    Args3<M, T, NR> a;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nz = g.nz;
    a.nruns = nruns;
    a.nstrips = (g.nx + width(T, 2) - 1) / width(T, 2);
    a.ygroups = (g.ny + kRows * kWarps - 1) / (kRows * kWarps);
    const int64_t tiles = (int64_t)a.nstrips * a.ygroups * nruns;
    a.cz = cz;
    a.nchunks = (g.nz + cz - 1) / cz;
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
    const int64_t blocks = tiles * a.nchunks;
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    return launch_chained(k_march3d<M, T, VEC, NR>, dim3((unsigned)blocks), kThreads, smem, st, a);
}

template <class M, int T>
cudaError_t launch3_t(const Geo& g, int nruns, const MarchRun* runs, cudaStream_t st, int cz)
{
    uintptr_t bits = 0;
    for (int r = 0; r < nruns; ++r)
        bits |= (uintptr_t)runs[r].phi_in | (uintptr_t)runs[r].phi_out | (uintptr_t)runs[r].v_in |
                (uintptr_t)runs[r].v_out;
    const bool vec = g.nx % 2 == 0 && bits % 8 == 0;
    if constexpr (M::kShared) {
        if (nruns > 1)
            return vec ? launch3_one<M, T, true, kMarchMaxRuns>(g, nruns, runs, st, cz) : cudaErrorNotSupported;
    }
    return vec ? launch3_one<M, T, true, 1>(g, 1, runs, st, cz) : launch3_one<M, T, false, 1>(g, 1, runs, st, cz);
}

template <class M>
cudaError_t launch3(const Geo& g, int t, int nruns, const MarchRun* runs, cudaStream_t st, int cz)
{
    switch (t) {
        case 1: return launch3_t<M, 1>(g, nruns, runs, st, cz);
        case 2: return launch3_t<M, 2>(g, nruns, runs, st, cz);
        case 3: return launch3_t<M, 3>(g, nruns, runs, st, cz);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace march

bool march3d_ok(const Geo& g) { return g.dims == 3 && (int64_t)g.nx * g.ny < ((int64_t)1 << 32); }

// As march_us in 2D: a warp's iteration takes its instructions' latency or its scheduler's turns for
// all its warps, a pass its iterations or its bytes (beyond L2 at 5.6 TB/s).  Waves of blocks count half
// as whole and half as they fill, as measured from 67^3 to 1024^3: long chunks waste fewer of their
// cz + 2t planes, short ones fill the GPU.
int march3d_planes(const Geo& g, int t, int nruns, double* us)
{
    const int u = march::width(t, 2);
    const double tiles = (double)((g.nx + u - 1) / u) *
                         ((g.ny + march::kRows * march::kWarps - 1) / (march::kRows * march::kWarps)) * nruns;
    const int sms = sm_count_current();
    const double slots = (double)sms * march::resident3(t);
    double rows = 0.0;  // updates of an iteration, in rows
    for (int l = 1; l <= t; ++l) rows += march::kRows + 2 * (t - l);
    const double base = 380.0 + 36.0 * rows;  // cycles at 1.9 GHz
    const double lone = (march_packed(g) ? 1.0 : 1.2) * base, turn = (march_packed(g) ? 0.72 : 0.95) * base;
    int best = 1;
    double least = 1e300;
    for (int nc = 1; nc <= g.nz && nc <= 4096; nc += nc < 32 ? 1 : nc / 16) {
        const int c = (g.nz + nc - 1) / nc, n = (g.nz + c - 1) / c;
        const double w = tiles * n / slots, at_once = w < 1.0 ? tiles * n : slots;
        const double waves = w <= 1.0 ? 1.1 - 0.1 * w : 0.5 * (ceil(w) + w + 0.35);
        const double cost = waves * (c + 2 * t) * std::max(lone, ceil(at_once / sms) * turn);
        if (cost < least * 0.999) least = cost, best = c;
    }
    if (us) {
        const double bytes = 16.0 * (double)g.S * nruns;
        *us = 3.5 + std::max(least / 1900.0, bytes / (bytes < 1e8 ? 9.0e6 : (t == 1 ? 6.2e6 : 5.6e6)));
    }
    return best;
}

// The staged passes stay where they are the faster: one step on the boxes they take (1024^3: 2.54 ms,
// HBM; the march 2.8), two steps on large boxes where the 256 x 8 tensor-copy tiles fit (us: 0.154 a
// MB of the state crossing HBM twice and a start of up to 93, that is 2740 at 1024^3, 424 at 512^3 and
// 65 at 256^3; the march 3100, 395 and 60; below 2^24 sites their few long tiles take 25 us whatever the box,
// the march 6 to 16: 20 steps of 256 x 64 x 64 254 and 81 us).  Three steps are the march's: 3620, 510 and
// 80, which is the least time a step from 1024^3 down to 100^3.
void march_plan_3d(const Geo& g, int nruns, MarchPlan* p)
{
    p->nruns = nruns;
    for (int t = 1; t <= kMarchMaxT; ++t) {
        p->shape[t] = MarchShape{2, 1};
        p->us[t] = 1e300;
        if (t <= kMarch3MaxT && march3d_ok(g)) p->shape[t].cy = march3d_planes(g, t, nruns, &p->us[t]);
    }
    if (nruns > 1) return;
    const double mb = 16e-6 * (double)g.S;
    const double one = 3.5 + std::max(6.5, mb * 0.15), two = 3.5 + 0.154 * mb + std::min(93.0, 0.09 * mb);
    if (fast_step_ok(g, PRS_FP32) || !march3d_ok(g)) p->shape[1].cols = 0, p->us[1] = one;
    if (t2tma_ok(g) && g.S >= (int64_t)1 << 24 && two < p->us[2]) p->shape[2].cols = 0, p->us[2] = two;
}

void march_counts_3d(const MarchPlan& p, int64_t n, bool home, int64_t cnt[kMarchMaxT + 1])
{
    double least = 1e300;
    std::fill(cnt, cnt + kMarchMaxT + 1, 0);
    cnt[1] = n;
    for (int64_t b = 0; b <= 5 && 2 * b <= n; ++b)  // pairs, then single steps; the rest in triples
        for (int64_t c = 0; c <= 3 && 2 * b + c <= n; ++c) {
            if ((n - 2 * b - c) % 3) continue;
            const int64_t a = (n - 2 * b - c) / 3;
            if (home && (a + b) % 2 && c == 0) continue;
            const double cost = (a ? (double)a * p.us[3] : 0.0) + (b ? (double)b * p.us[2] : 0.0) + (double)c * p.us[1];
            if (cost < least) least = cost, cnt[3] = a, cnt[2] = b, cnt[1] = c;
        }
    for (int64_t c = 0; c <= 2 && c <= n; ++c) {  // pairs and single steps alone
        if ((n - c) % 2) continue;
        const int64_t b = (n - c) / 2;
        if (home && b % 2 && c == 0) continue;
        const double cost = (b ? (double)b * p.us[2] : 0.0) + (double)c * p.us[1];
        if (cost < least) least = cost, cnt[3] = 0, cnt[2] = b, cnt[1] = c;
    }
    if ((double)n * p.us[1] < least) cnt[3] = cnt[2] = 0, cnt[1] = n;
}

cudaError_t launch_march3d(const Geo& g, int t, int cz, int nruns, const MarchRun* runs, cudaStream_t st)
{
    const bool packed = march_packed(g);
    if (!march3d_ok(g) || nruns < 1 || nruns > kMarchMaxRuns) return cudaErrorInvalidValue;
    if (nruns > 1 && !packed) return cudaErrorNotSupported;
    return packed ? march::launch3<march::Fold32>(g, t, nruns, runs, st, cz)
                  : march::launch3<march::Plain32>(g, t, nruns, runs, st, cz);
}

}  // namespace prs
