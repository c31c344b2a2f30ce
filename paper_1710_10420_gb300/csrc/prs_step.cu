// prs_step.cu -- chooses the kernel for one pass of fused leapfrog steps.
#include "prs_internal.h"
#include "prs_march3d.h"

namespace prs {

cudaError_t launch_step_generic(const Geo& g, int precision, bool repro, const void* in, void* out, const void* dphi,
                                void* dphi_out, const double coef[3], const double rcd[6], const MarchShape& shape,
                                cudaStream_t st);
cudaError_t launch_step_fast(const Geo& g, const float* in, float* out, const float* v, float* v_out,
                             KickF k, RunConst<float> rc, unsigned int* err, cudaStream_t st);

KickF kick_f32(const double coef[3], const double run_const[6])
{
    const double g = coef[1] * run_const[1];
    const double h = coef[1] * coef[2];
    return KickF{(float)coef[0], (float)g, (float)(h - run_const[3] * g), (float)(h * run_const[2])};
}

// 2D boxes that a caller may step with tblock = 2 or 3 (the limit of the staged passes that the
// register march replaced; without a tblock the march takes any FP32 2D box, up to six steps a pass).
static bool rows_ok(const Geo& g) { return g.dims == 2 && g.nx % 128 == 0 && g.nx <= 4096; }

// The same for tblock = 3 on 3D boxes.
static bool t3_ok(const Geo& g) { return g.nx % 128 == 0 && g.ny % 8 == 0 && g.ny >= 16 && g.nz >= 3; }

// Steps one pass may fuse (params.tblock above this is clamped): three on the FP32 boxes the
// three-step passes take, two on the other boxes of the two-step passes.
int max_fused_steps(const Geo& g, int precision, bool repro)
{
    (void)repro;
    if (!tblock_ok(g, precision)) return 1;
    return (g.dims == 3 ? t3_ok(g) : rows_ok(g)) ? 3 : 2;
}

// The fixed number of steps per pass that suits a box, which prs_default_tblock reports.  A run without
// a tblock is stepped by a plan of passes of several lengths instead (march_counts in 2D,
// march_counts_3d), chosen by the time each length takes there.  What this decides still: how an
// ensemble reports a box, and which 2D and 3D boxes take the packed arithmetic (march_packed).
int default_fused_steps(const Geo& g, int precision, bool repro)
{
    (void)repro;
    if (precision != PRS_FP32 || !tblock_ok(g, precision)) return 1;
    if (g.dims == 2) {
        if (rows_ok(g) && (g.nx >= 2048 || g.ny <= 1024)) return 3;
        return g.S >= (int64_t)1 << 24 ? 2 : 1;
    }
    if (g.S < (int64_t)1 << 24) return 1;
    return tblock3_rows(g) >= 4 ? 2 : 1;
}

cudaError_t launch_step_io(const Geo& g, int precision, bool repro, const void* phi_in, void* phi_out,
                           const void* dphi_in, void* dphi_out, const double coef[3], const double run_const[6],
                           const MarchShape& shape, unsigned int* err, cudaStream_t st)
{
    const MarchRun r{phi_in, phi_out, dphi_in, dphi_out, {{coef[0], coef[1], coef[2]}}, run_const};
    if (g.dims == 2 && precision == PRS_FP32) return launch_march2d(g, 1, shape, 1, &r, st);
    if (fast_step_ok(g, precision)) {
        const KickF k = kick_f32(coef, run_const);
        RunConst<float> rc{(float)run_const[0], (float)run_const[1], (float)run_const[2], (float)run_const[3],
                           (float)run_const[4], (float)run_const[5]};
        return launch_step_fast(g, (const float*)phi_in, (float*)phi_out, (const float*)dphi_in, (float*)dphi_out, k,
                                rc, err, st);
    }
    if (precision == PRS_FP32 && march3d_ok(g)) return launch_march3d(g, 1, shape.cy, 1, &r, st);
    return launch_step_generic(g, precision, repro, phi_in, phi_out, dphi_in, dphi_out, coef, run_const, shape, st);
}

}  // namespace prs
