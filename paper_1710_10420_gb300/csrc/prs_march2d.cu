// prs_march2d.cu -- choosing the arithmetic, the shape and the length of the passes of the 2D
// register march.
#include <algorithm>

#include "prs_march2d_launch.cuh"

namespace prs {

bool march_packed(const Geo& g)
{
    return fast_step_ok(g, PRS_FP32) || default_fused_steps(g, PRS_FP32, false) > 1;
}

// Every scheduler holds as many warps as its SM holds blocks (b), so a pass takes the iterations of a chunk
// times what an iteration takes among b warps, or its bytes, and a launch (1.7 us from one kernel's end
// to the next's start).  Cycles of an iteration at 1.9 GHz, measured from 256^2 to 4096^2: a lone
// warp with four columns a lane 185 + 43 T, b of them 0.76 b times that; with two columns 150 + 40 T,
// b of them 0.3 + 0.51 b; a fifth more with the unpacked arithmetic.  The last block decides, so the rows
// of a chunk are the fewest that fill every SM with b blocks and no SM with one more: 4096^2, T = 5, 128
// rows and b = 2 46.4 us, 229 rows and 1.1 blocks an SM on average 78; 2048^2 15.3 and 23.4.  Small boxes
// come out with pairs, which make warps, boxes of 512^2 and more with quads, which waste fewer of their
// columns.
static double march_us(const Geo& g, int t, int nruns, MarchShape* best)
{
    const int64_t per_b = (int64_t)sm_count_current() * march::kWarps;  // warps of a block an SM
    const double plain = march_packed(g) ? 1.0 : 1.2;
    double least = 1e300;
    for (int cols = 2; cols <= 4; cols += 2) {
        const int u = march::width(t, cols), r = march::resident(t, cols);
        const int64_t strips = (int64_t)((g.nx + u - 1) / u) * nruns;
        const double lone = plain * (cols == 4 ? 185.0 + 43.0 * t : 150.0 + 40.0 * t);
        const auto among = [&](int64_t b) { return std::max(1.0, cols == 4 ? 0.76 * b : 0.3 + 0.51 * b); };
        for (int64_t b = 1; b <= 4 * r || least == 1e300; b += b < 4 * r ? 1 : b) {
            const int64_t most = std::min<int64_t>(b * per_b / strips, g.ny);  // chunks
            if (most < 1) continue;
            const int cy = (int)((g.ny + most - 1) / most);
            const double waves = (double)(b / r) * among(r) + (b % r ? among(b % r) : 0.0);
            const double cost = waves * lone * (cy + 2 * t);
            if (cost < least * 0.999) least = cost, *best = MarchShape{cols, cy};
            if (most == g.ny) break;
        }
    }
    const double bytes = 16.0 * (double)g.S * nruns;  // beyond L2: 6.1 TB/s
    return 1.7 + std::max(least / 1900.0, bytes > 1e8 ? bytes / 6.1e6 : bytes / 1.2e7);
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
