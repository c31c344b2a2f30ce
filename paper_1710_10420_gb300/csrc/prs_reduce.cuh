// prs_reduce.cuh -- fixed-order reduction of the diagnostic sums (Eq. 7, Eq. 8):
// warp shuffles, then the warps of a block, then one partial per block; the last
// block to finish (an atomic completion counter, no waiting) adds the partials in
// index order.  Repeated launches on the same grid give bit-identical results.
#pragma once

#include <cuda_runtime.h>

#include "prs_internal.h"

namespace prs {

__device__ __forceinline__ void acc_add(DiagAcc& a, const DiagAcc& b)
{
    a.sum_w += b.sum_w;
    a.sum_ratio += b.sum_ratio;
    a.n_links += b.n_links;
    a.n_wall += b.n_wall;
    a.n_vzero += b.n_vzero;
    a.n_nonfinite += b.n_nonfinite;
}

__device__ __forceinline__ void acc_shfl_down(DiagAcc& a, int off)
{
    DiagAcc o;
    o.sum_w = __shfl_down_sync(0xffffffffu, a.sum_w, off);
    o.sum_ratio = __shfl_down_sync(0xffffffffu, a.sum_ratio, off);
    o.n_links = __shfl_down_sync(0xffffffffu, a.n_links, off);
    o.n_wall = __shfl_down_sync(0xffffffffu, a.n_wall, off);
    o.n_vzero = __shfl_down_sync(0xffffffffu, a.n_vzero, off);
    o.n_nonfinite = __shfl_down_sync(0xffffffffu, a.n_nonfinite, off);
    acc_add(a, o);
}

// Fixed-order warp reduction: lane 0 ends with the sum of the warp.
__device__ __forceinline__ void acc_warp_reduce(DiagAcc& a)
{
    for (int off = 16; off > 0; off >>= 1) acc_shfl_down(a, off);
}

// Every thread of the block calls this once with its own sums: block bid of the nblocks
// that reduce into scr; their total lands in *scr.result and the counter is reset for the
// next launch.  sums: shared memory for blockDim.x pairs, free for use.  The last block reads the
// partials with all its threads (one warp reading 456 of them took about 8 us of a small box's
// diagnostics).
__device__ __forceinline__ void block_reduce_and_finish_at(DiagAcc a, const DiagScratch& scr, unsigned int bid,
                                                           unsigned int nblocks, double2* sums)
{
    __shared__ uint4 counts[32];
    __shared__ DiagAcc warp_sums[32];
    __shared__ bool is_last;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    // The FP64 sums go through shared memory to one warp: an SM adds two doubles a clock, so 5
    // shuffle-and-add levels in each of its 24 warps took 2 us.  A thread's counts fit 26 bits (it
    // sees far fewer sites), so each is one warp-wide integer reduction.
    sums[tid] = make_double2(a.sum_w, a.sum_ratio);
    const uint4 c = make_uint4(
        __reduce_add_sync(0xffffffffu, (unsigned)a.n_links), __reduce_add_sync(0xffffffffu, (unsigned)a.n_wall),
        __reduce_add_sync(0xffffffffu, (unsigned)a.n_vzero), __reduce_add_sync(0xffffffffu, (unsigned)a.n_nonfinite));
    if (lane == 0) counts[wid] = c;
    __syncthreads();
    if (wid == 0) {
        DiagAcc b{0.0, 0.0, 0, 0, 0, 0};
        for (int i = lane; i < (int)blockDim.x; i += 32) b.sum_w += sums[i].x, b.sum_ratio += sums[i].y;
        if (lane < nw) b.n_links = counts[lane].x, b.n_wall = counts[lane].y, b.n_vzero = counts[lane].z,
                       b.n_nonfinite = counts[lane].w;
        acc_warp_reduce(b);
        if (lane == 0) {
            scr.partials[bid] = b;
            __threadfence();
            unsigned int done = atomicAdd(scr.counter, 1u);
            is_last = (done == nblocks - 1);
        }
    }
    __syncthreads();
    if (!is_last) return;
    // the last block to finish reduces every partial in a fixed order
    __threadfence();
    DiagAcc t{0.0, 0.0, 0, 0, 0, 0};
    for (int i = tid; i < (int)nblocks; i += blockDim.x) {
        // other blocks wrote these: read through L2, not a possibly stale L1 line
        const DiagAcc* q = scr.partials + i;
        DiagAcc p{__ldcg(&q->sum_w), __ldcg(&q->sum_ratio), __ldcg(&q->n_links),
                  __ldcg(&q->n_wall), __ldcg(&q->n_vzero), __ldcg(&q->n_nonfinite)};
        acc_add(t, p);
    }
    acc_warp_reduce(t);
    if (lane == 0) warp_sums[wid] = t;
    __syncthreads();
    if (wid == 0) {
        DiagAcc b = lane < nw ? warp_sums[lane] : DiagAcc{0.0, 0.0, 0, 0, 0, 0};
        acc_warp_reduce(b);
        if (lane == 0) {
            *scr.result = b;
            *scr.counter = 0u;  // ready for the next launch on this scratch
            if (scr.host) {
                scr.host->result = b;
                scr.host->error = __ldcg(scr.error);
            }
        }
    }
}

// The whole grid reduces into scr.
__device__ __forceinline__ void block_reduce_and_finish(DiagAcc a, const DiagScratch& scr, double2* sums)
{
    block_reduce_and_finish_at(a, scr, blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z),
                               gridDim.x * gridDim.y * gridDim.z, sums);
}

// The same for blocks of at most 256 threads without shared memory to spare for it.
__device__ __forceinline__ void block_reduce_and_finish(DiagAcc a, const DiagScratch& scr)
{
    __shared__ double2 sums[256];
    block_reduce_and_finish(a, scr, sums);
}

}  // namespace prs
