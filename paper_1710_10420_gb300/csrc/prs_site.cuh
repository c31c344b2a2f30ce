// prs_site.cuh -- Eqs. 3-5 at one site, the forms that the one-thread-a-site kernels and the 2D
// register march share (the packed FP32 form of the staged kernels is update4, prs_tile.cuh).
#pragma once

#include <cuda_runtime.h>

#include "prs_arith.cuh"
#include "prs_internal.h"

namespace prs {

// One site of Eqs. 3-5 in the canonical evaluation order:
//   s2 = (x+ + x-) ; s2 += (y+ + y-) ; [s2 += (z+ + z-)]
//   lap = (s2 - 2D c) / dx^2 ; f = (cV c)(c c / phi0^2 - 1)
//   v' = c1 v + c2 (lap - f) ; phi' = c + deta v'
template <typename R, bool REPRO, int D>
__device__ __forceinline__ void site_update(R c, R xp, R xm, R yp, R ym, R zp, R zm, R& v, R& phi_new,
                                            const StepCoef<R>& k, const RunConst<R>& rc)
{
    using A = Arith<R, REPRO>;
    R s2 = A::add(xp, xm);
    s2 = A::add(s2, A::add(yp, ym));
    if (D == 3) s2 = A::add(s2, A::add(zp, zm));
    R lap = A::mul(A::sub(s2, A::mul(rc.twoD, c)), rc.inv_dx2);
    R f = A::mul(A::mul(k.cV, c), A::sub(A::mul(A::mul(c, c), rc.inv_phi0sq), (R)1));
    R vn = A::add(A::mul(k.c1, v), A::mul(k.c2, A::sub(lap, f)));
    v = vn;
    phi_new = A::add(c, A::mul(rc.deta, vn));
}

// The same step with the step's constants folded on the host (FP64 without PRS_REPRO):
//   v' = c1 v + g s2 + c (k1 - k2 c^2),  g = c2/dx^2, k1 = c2 cV - 2D g, k2 = c2 cV/phi0^2,
// which is Eq. 4 rearranged: 11 double operations a site instead of 15.  GB300 issues FP64
// at a small fraction of its FP32 rate and the generic step is bound by that rate, so the
// operation count sets its speed.  Every term is odd in phi, so Z2 symmetry stays exact.
template <int D>
__device__ __forceinline__ void site_update_folded(double c, double xp, double xm, double yp, double ym, double zp,
                                                   double zm, double& v, double& phi_new, const KickD& k, double deta)
{
    double s2 = xp + xm;
    s2 = s2 + (yp + ym);
    if (D == 3) s2 = s2 + (zp + zm);
    const double u = c * fma(-k.k2, c * c, k.k1);
    const double vn = fma(k.c1, v, fma(k.g, s2, u));
    v = vn;
    phi_new = fma(deta, vn, c);
}

}  // namespace prs
