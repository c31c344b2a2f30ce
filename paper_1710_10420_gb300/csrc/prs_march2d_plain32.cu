// prs_march2d_plain32.cu -- the 2D register march (prs_march2d.cuh), arithmetic Plain32.
#include "prs_march2d_launch.cuh"

namespace prs {

cudaError_t launch_march_plain32(const Geo& g, int t, const MarchShape& s, int nruns, const MarchRun* runs,
                                 cudaStream_t st)
{
    return march::launch<march::Plain32>(g, t, s, nruns, runs, st);
}

}  // namespace prs
