// prs_march2d.h -- launching the 2D register march (prs_march2d.cuh).
#pragma once

#include "prs_internal.h"

namespace prs {

constexpr int kMarchMaxT = 6;      // steps per pass
constexpr int kMarchMaxRuns = 16;  // runs of one box per launch

// Whether an FP32 box steps by the folded kick of the staged passes (the boxes of the one-step tiles, and
// those of 2^24 sites and more, in 2D also smaller ones, of the two- and three-step passes), else by
// the generic step's arithmetic, whose rounding errors are a little smaller.
bool march_packed(const Geo& g);

// The state of one FP32 run and the steps of a pass over it: coefficients (c1, c2, cV) of each
// step and the run's constants (the layout of RunConst).
struct MarchRun {
    const void* phi_in;
    void* phi_out;
    const void* v_in;
    void* v_out;  // may be v_in when t == 1
    double coef[kMarchMaxT][3];
    const double* run_const;
};

// How a pass is cut: columns a lane owns (2 or 4; 3D: 2) and rows (3D: planes) a warp marches.  cols
// 0: the pass is not the march's (3D boxes of the staged passes).
struct MarchShape {
    int cols, cy;
};

// Shapes and modelled times (us, with the launch) of the passes of 1 .. kMarchMaxT (3D: kMarch3MaxT)
// steps over nruns FP32 runs of a box.
struct MarchPlan {
    int nruns;  // 0: not made yet
    MarchShape shape[kMarchMaxT + 1];
    double us[kMarchMaxT + 1];
};
void march_plan(const Geo& g, int nruns, MarchPlan* p);     // 2D
void march_plan_3d(const Geo& g, int nruns, MarchPlan* p);  // 3D

// The passes of a call of n steps (>= 1): cnt[t] of t steps each, the longest first.  home: dphi has
// to end in the buffer it started in, so that the passes of two steps and more, which alternate
// between two buffers, are even in number or leave a single step to bring it back.
void march_counts(const MarchPlan& p, int64_t n, bool home, int64_t cnt[kMarchMaxT + 1]);     // 2D
void march_counts_3d(const MarchPlan& p, int64_t n, bool home, int64_t cnt[kMarchMaxT + 1]);  // 3D

// One pass of t steps (1 .. kMarchMaxT) over nruns (1 .. kMarchMaxRuns) runs of the 2D box g, any
// sides (several runs: march_packed boxes).
cudaError_t launch_march2d(const Geo& g, int t, const MarchShape& shape, int nruns, const MarchRun* runs,
                           cudaStream_t st);

}  // namespace prs
