// prs_march2d.cu -- choosing the arithmetic, the shape and the length of the passes of the 2D
// register march.
#include <algorithm>

#include "prs_march2d_launch.cuh"

namespace prs {

bool march_packed(const Geo& g)
{
    return fast_step_ok(g, PRS_FP32) || default_fused_steps(g, PRS_FP32, false) > 1;
}

// A warp's iteration takes the chain of its levels, or its scheduler's turns for all its warps,
// whichever is longer; a pass takes its waves of iterations or its bytes, and a launch (2.3 us from
// one kernel's end to the next's start).  Cycles at 1.9 GHz, measured per level and iteration (256^2
// to 4096^2): a lone warp 100 (two columns a lane: 78), each warp of a busy scheduler 92 (60); a
// third more with the unpacked arithmetic.  So small boxes take pairs and short chunks, which make
// warps, and boxes of 512^2 and more take quads and chunks of 20 to 60 rows, which waste fewer of
// their rows and columns (2048^2, T = 4: 16.5 us with quads, 20.6 with pairs).
static double march_us(const Geo& g, int t, int nruns, MarchShape* best)
{
    const int sms = sm_count_current();
    const double plain = march_packed(g) ? 1.0 : 1.3;
    double least = 1e300;
    for (int cols = 2; cols <= 4; cols += 2) {
        const int u = march::width(t, cols);
        const int64_t strips = (int64_t)((g.nx + u - 1) / u) * nruns;
        const int64_t slots = (int64_t)sms * march::resident(t, cols) * march::kWarps;
        const double chain = plain * (cols == 4 ? 100.0 : 78.0) * t, turn = plain * (cols == 4 ? 92.0 : 60.0) * t;
        for (int cy = 1;; cy += cy < 16 ? 1 : cy / 8) {
            if (cy > g.ny) cy = g.ny;
            const int64_t warps = strips * ((g.ny + cy - 1) / cy), waves = (warps + slots - 1) / slots;
            const double most = (double)(waves > 1 ? slots : warps);  // warps at once
            const double cost = (double)waves * (cy + 2 * t) * std::max(chain, most / (4.0 * sms) * turn);
            if (cost < least * 0.999) least = cost, *best = MarchShape{cols, cy};
            if (cy == g.ny) break;
        }
    }
    const double bytes = 16.0 * (double)g.S * nruns;  // beyond L2: 5.4 TB/s
    return 2.3 + std::max(least / 1900.0, bytes > 1e8 ? bytes / 5.4e6 : bytes / 1.2e7);
}

void march_plan(const Geo& g, int nruns, MarchPlan* p)
{
    p->nruns = nruns;
    for (int t = 1; t <= kMarchMaxT; ++t) p->us[t] = march_us(g, t, nruns, &p->shape[t]);
}

void march_counts(const MarchPlan& p, int64_t n, bool home, int64_t cnt[kMarchMaxT + 1])
{
    double least = 1e300;
    for (int t = (int)std::min<int64_t>(n, kMarchMaxT); t >= 1; --t) {
        // passes that differ by a step at most
        int64_t passes = (n + t - 1) / t, hi = 0, many = 0;
        for (int extra = 0; extra < 2; ++extra, ++passes) {
            hi = (n + passes - 1) / passes;
            many = n - (hi - 1) * passes;  // passes of hi steps; the others take hi - 1
            const int64_t multi = hi >= 3 ? passes : (hi == 2 ? many : 0);
            if (!home || (multi & 1) == 0 || multi < passes) break;
        }
        const double cost = (double)many * p.us[hi] + (hi > 1 ? (double)(passes - many) * p.us[hi - 1] : 0.0);
        if (cost >= least) continue;
        least = cost;
        std::fill(cnt, cnt + kMarchMaxT + 1, 0);
        cnt[hi] = many;
        if (hi > 1) cnt[hi - 1] = passes - many;
    }
}

cudaError_t launch_march2d(const Geo& g, int t, const MarchShape& shape, int nruns, const MarchRun* runs,
                           cudaStream_t st)
{
    if (g.dims != 2 || nruns < 1 || nruns > kMarchMaxRuns) return cudaErrorInvalidValue;
    if (nruns > 1 && !march_packed(g)) return cudaErrorNotSupported;
    return march_packed(g) ? launch_march_fold32(g, t, shape, nruns, runs, st)
                     : launch_march_plain32(g, t, shape, nruns, runs, st);
}

}  // namespace prs
