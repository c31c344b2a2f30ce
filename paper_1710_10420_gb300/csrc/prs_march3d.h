// prs_march3d.h -- launching the 3D register march (prs_march3d.cuh).
#pragma once

#include "prs_march2d.h"

namespace prs {

constexpr int kMarch3MaxT = 3;  // steps per pass

// 3D boxes the march takes: planes whose element offsets fit 32 bits.
bool march3d_ok(const Geo& g);

// Planes a warp marches in a pass of t steps over nruns runs, and the pass's modelled time (us).
int march3d_planes(const Geo& g, int t, int nruns, double* us);

// One pass of t steps (1 .. kMarch3MaxT) over nruns (1 .. kMarchMaxRuns) runs of the FP32 3D box g, any
// sides (several runs: march_packed boxes); cz from march3d_planes.
cudaError_t launch_march3d(const Geo& g, int t, int cz, int nruns, const MarchRun* runs, cudaStream_t st);

}  // namespace prs
