// prs_chain.h -- launching a kernel so that its start overlaps the end of the one before it.
//
// A run's passes are short on small boxes (3 to 20 us), and from one kernel's last block to the next
// one's first a stream takes about 2 us.  A kernel that begins with chain_enter() (prs_ptx.cuh) is placed
// on the SMs as the blocks of its predecessor leave them, and waits there: 128^2 FP64 78 -> 61 us for an
// interval of 12 launches, 2500 x 1701 126 -> 115, 128^3 177 -> 164.  (Letting it in as soon as the
// predecessor's blocks have all started, by griddepcontrol.launch_dependents, costs large boxes up to a
// third: 1024^3 31.4 -> 41.9 ms.)
#pragma once

#include <cuda_runtime.h>

namespace prs {

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A&&... args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // the runtime keeps it, and a later plain launch would report it
    return e;
}

}  // namespace prs
