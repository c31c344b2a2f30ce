// prs_adj_march.h -- launching the adjoint's register march (prs_adj_march.cuh).
#pragma once

#include "prs_internal.h"

namespace prs {

// One reverse step over the FP32 3D box g with the forward state (phi, v) at the step and the
// coefficients c1, c2, cV, dc1/dalpha, dc2/dalpha: lphi in place, lt_in -> lt_out (lv when last), the
// dJ/dalpha term in scr.result's sum_w.  cudaErrorNotSupported where the box does not fit.
cudaError_t launch_adj_march(const Geo& g, const float* phi, const float* v, const float coef[5], const float* lt_in,
                             float* lt_out, float* lphi, const double run_const[6], bool last, const DiagScratch& scr,
                             cudaStream_t st);

}  // namespace prs
