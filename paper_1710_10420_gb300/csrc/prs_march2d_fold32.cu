// prs_march2d_fold32.cu -- the 2D register march (prs_march2d.cuh), arithmetic Fold32.
#include "prs_march2d_launch.cuh"

namespace prs {

cudaError_t launch_march_fold32(const Geo& g, int t, const MarchShape& s, int nruns, const MarchRun* runs,
                                cudaStream_t st)
{
    return march::launch<march::Fold32>(g, t, s, nruns, runs, st);
}

}  // namespace prs
