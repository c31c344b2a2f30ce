// prs_march3d.cuh -- T leapfrog steps (Eqs. 3-5) per pass over an FP32 3D box of any sides, in registers.
//
// The 2D register march (prs_march2d.cuh) with rows: a warp owns 64 columns (a pair a lane) of kRows
// output rows and marches its chunk of planes along z through T levels.  Level l lives on
// kRows + 2 (T - l) rows; a level's z neighbours are the planes it saw in the two iterations before,
// its y neighbours the warp's other rows, its x neighbours the neighbouring lanes, and dphi waits an
// iteration in registers between levels.  Planes come through a ring in shared memory that each lane
// fills ahead for itself.  The warps of a block own neighbouring rows, so that the halo rows of one
// are another's in L1.
//
// What bounds it: latency, with the 8 (T = 3) or 12 (T = 2) warps an SM that the registers leave, which keep
// 0.4 to 0.6 of the issue slots busy.  The outer rows of each level are computed twice (T = 2: 1.25
// updates an output and step and 64/60 for the columns; T = 3: 1.5 and 64/56), which is what lets a warp
// run without waiting for its neighbours at a barrier, on boxes whose rows have no alignment for
// tensor copies.
//
// Measured: 512^3, T = 3, 522 us a pass, 382 M warp instructions at 0.60 of the issue slots, 2.16 GB
// of DRAM traffic for 2.15 GB of fields in and out; 1024^3 1.21 ms a step (pairs of staged tiles 1.37);
// 450 x 421 x 380 112 us a step (one thread a site: 571); 128^3 6.7 us a step (staged, short chunks: 9.6).
#pragma once

#include "prs_march2d.cuh"
#include "prs_march3d.h"

namespace prs {

namespace march {

constexpr int kRows = 4;   // output rows of a warp
constexpr int kRing3 = 3;  // planes of phi and dphi in flight or in use

// Blocks an SM holds: registers enough that a level's rows are scheduled side by side (T = 2 with 128
// instead of 168 took 430 instead of 395 us at 512^3 and 1220 instead of 735 cycles a lone iteration).
constexpr int resident3(int t) { return t == 1 ? 5 : (t == 2 ? 3 : 2); }

template <class M, int T, int NR>
struct Args3 {
    const float* phi_in[NR];
    float* phi_out[NR];
    const float* v_in[NR];
    float* v_out[NR];
    typename M::K k[NR][T];
    RunConst<float> rc[NR];
    int nx, ny, nz, nstrips, ygroups, nchunks, cz, nruns;
};

// VEC: nx even and the fields aligned to a pair.
template <class M, int T, bool VEC, int NR>
__global__ void __launch_bounds__(kThreads, resident3(T)) k_march3d(const __grid_constant__ Args3<M, T, NR> a)
{
    using P = typename M::P;
    using K = typename M::K;
    constexpr int COLS = 2, HX = halo(T, COLS), U = width(T, COLS), kRow = 32 * COLS;
    constexpr int N0 = kRows + 2 * T, N1 = N0 - 2;  // rows of level 0 and of level 1
    constexpr int kPlane = (N0 + N1) * kRow;        // floats of a ring slot: phi rows, then dphi rows
    extern __shared__ __align__(16) float ring3[];
    chain_enter();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nx = a.nx, ny = a.ny, nz = a.nz;
    // blocks: x strips fastest, then groups of kWarps row tiles, then chunks, then runs
    int b = blockIdx.x;
    const int strip = b % a.nstrips;
    b /= a.nstrips;
    const int x0 = strip * U, y0 = (b % a.ygroups * kWarps + wid) * kRows;
    b /= a.ygroups;
    const int z0 = b % a.nchunks * a.cz, run = NR > 1 ? b / a.nchunks : 0;
    if (y0 >= ny) return;
    K kk[T];
#pragma unroll
    for (int l = 0; l < T; ++l) kk[l] = a.k[run][l];
    const RunConst<float>& rc = a.rc[run];
    const f2 dt = pk2(rc.deta, rc.deta);
    float* const rp = ring3 + wid * kRing3 * kPlane + lane * COLS;
    const int planes = min(a.cz, nz - z0), rows = min(kRows, ny - y0);
    int xa = (x0 - HX + COLS * lane) % nx;
    if (xa < 0) xa += nx;
    const int x[COLS] = {xa, xa + 1 == nx ? 0 : xa + 1};
    const int c0 = COLS * lane - HX;
    const int lo = c0 < 0 ? COLS : 0, hi = min(COLS, min(U, nx - x0) - c0);
    unsigned row[N0];  // element offsets of the level-0 rows in a plane, periodic
    int yr = (y0 - T) % ny;
    if (yr < 0) yr += ny;
#pragma unroll
    for (int r = 0; r < N0; ++r) {
        row[r] = (unsigned)yr * (unsigned)nx;
        if (++yr == ny) yr = 0;
    }
    const int64_t plane = (int64_t)nx * ny;
    const int64_t out0 = (int64_t)z0 * plane + (int64_t)y0 * nx;
    float* pout = a.phi_out[run] + out0;
    float* vout = a.v_out[run] + out0;

    const int iters = planes + 2 * T;  // level-0 planes z0-T .. z0+planes+T-1
    int z = (z0 - T) % nz, next = 0, fill = 0;
    if (z < 0) z += nz;
    const float* pin = a.phi_in[run] + (int64_t)z * plane;
    const float* vin = a.v_in[run] + (int64_t)z * plane;
    auto fetch = [&] {  // the next plane into its ring slot; a group of its own, also when empty
        if (next < iters) {
            float* d = rp + fill * kPlane;
#pragma unroll
            for (int r = 0; r < N0; ++r) stage<COLS, VEC>(d + r * kRow, pin + row[r], x);
#pragma unroll
            for (int r = 0; r < N1; ++r) stage<COLS, VEC>(d + (N0 + r) * kRow, vin + row[r + 1], x);
            ++next, ++z;
            fill = fill == kRing3 - 1 ? 0 : fill + 1;
            const int64_t step = z == nz ? plane * (1 - (int64_t)nz) : plane;
            if (z == nz) z = 0;
            pin += step;
            vin += step;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int u = 0; u < kRing3 - 1; ++u) fetch();
    // level l: m[l] (rows 1 .. N-2), c[l] (all N = N0 - 2l rows), and the dphi it hands on
    P m[T][N1], c[T][N0], vd[T][N1];
    const P zero = M::pair(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < T; ++l) {
#pragma unroll
        for (int r = 0; r < N1; ++r) m[l][r] = vd[l][r] = zero;
#pragma unroll
        for (int r = 0; r < N0; ++r) c[l][r] = zero;  // overwritten before a plane that is kept reads them
    }
    int use = 0;
    for (int i = 0; i < iters; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing3 - 2) : "memory");
        const float* s = rp + use * kPlane;
        P p[N0], v[N1], q[1];
#pragma unroll
        for (int r = 0; r < N0; ++r) unstage<M, COLS>(s + r * kRow, q), p[r] = q[0];
        // dphi of plane i-1 is read one iteration late, from the slot before
        const float* sv = rp + (use == 0 ? kRing3 - 1 : use - 1) * kPlane;
#pragma unroll
        for (int r = 0; r < N1; ++r) unstage<M, COLS>(sv + (N0 + r) * kRow, q), v[r] = q[0];
        fetch();  // into the slot of plane i-1
        use = use == kRing3 - 1 ? 0 : use + 1;
#pragma unroll
        for (int l = 0; l < T; ++l) {  // level l+1 at plane i-1-l
            const int n = N0 - 2 * (l + 1);
            const K k = M::kShared ? kk[l] : a.k[0][l];
            P out[N1];
#pragma unroll
            for (int r = 0; r < N1; ++r) {
                if (r >= n) continue;
                float f0, f1;
                M::split(c[l][r + 1], f0, f1);
                const float left = __shfl_up_sync(0xffffffffu, f1, 1), right = __shfl_down_sync(0xffffffffu, f0, 1);
                out[r] = M::template update<3>(c[l][r], c[l][r + 1], c[l][r + 2], m[l][r], p[r + 1], left, right, v[r],
                                               k, dt, rc);
            }
#pragma unroll
            for (int r = 0; r < N1; ++r)
                if (r < n) m[l][r] = c[l][r + 1];
#pragma unroll
            for (int r = 0; r < N0; ++r)
                if (r < n + 2) c[l][r] = p[r];
#pragma unroll
            for (int r = 0; r < N1; ++r)
                if (r < n) p[r] = out[r];
            if (l + 1 < T) {  // the next level's rows are this one's without the outer two
#pragma unroll
                for (int r = 0; r < N1; ++r) {
                    if (r < n) {
                        const P t = vd[l][r];
                        vd[l][r] = v[r];
                        v[r] = t;
                    }
                }
#pragma unroll
                for (int r = 0; r + 1 < N1; ++r)
                    if (r < n - 2) v[r] = v[r + 1];
            }
        }
        if (i >= 2 * T) {
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                if (r >= rows) break;
                const P po[1] = {p[r]}, vo[1] = {v[r]};
                store<M, COLS, VEC>(pout + (unsigned)r * (unsigned)nx, x[0], lo, hi, po);
                store<M, COLS, VEC>(vout + (unsigned)r * (unsigned)nx, x[0], lo, hi, vo);
            }
            pout += plane;
            vout += plane;
        }
    }
}

}  // namespace march

}  // namespace prs
