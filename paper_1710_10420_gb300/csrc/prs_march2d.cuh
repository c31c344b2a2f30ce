// prs_march2d.cuh -- T leapfrog steps (Eqs. 3-5) per pass over an FP32 2D box of any sides, in registers.
//
// A warp owns a strip of 64 or 128 columns (two or four adjacent ones a lane) and a chunk of rows and
// marches along y through T levels: at iteration i it takes level-0 row i, and level l (the state after l
// steps) reaches row i-l.  A level's y neighbours are the rows it saw in the two iterations before,
// its x neighbours come from the neighbouring lanes, and the dphi a level hands to the next waits
// one iteration in a register, so nothing but the rows that enter and leave touches memory (through
// a ring in shared memory that each lane fills ahead for itself): no barrier, and no alignment
// beyond the element's.  Each level loses a column and a
// row on every side, so a strip yields 2 HX columns less than its width and a chunk re-reads 2T rows.
//
// What bounds it: the latency of an iteration's chain on small boxes, HBM at 16 B per T site-updates on
// boxes larger than L2 and between the two instruction issue (6 to 8 instructions a site-update in
// FP32, against about 16 when each level's rows pass through shared memory).  Both sides of a row are
// recomputed instead of exchanged, which is what lets warps run without waiting for one another.  phi
// and dphi are read across sites, so both go out of place.
//
// Measured (an output interval of 10 steps and the diagnostics, us; with the one- to three-step passes
// over rows in shared memory, or one thread a site on ragged boxes, that this replaced): 256^2 42 (82),
// 2048^2 87 (158), 4096^2 215 (375), 2500 x 1701 94 (328).
#pragma once

#include <cuda_runtime.h>

#include "prs_f32x2.cuh"
#include "prs_internal.h"
#include "prs_march2d.h"
#include "prs_ptx.cuh"
#include "prs_site.cuh"

namespace prs {

namespace march {

constexpr int kThreads = 128, kWarps = kThreads / 32;
constexpr int kRing = 8;  // rows of phi and dphi in flight or in use, a power of two

// Halo columns of a strip on each side: T, rounded up to a lane's columns.
constexpr int halo(int t, int cols) { return (t + cols - 1) / cols * cols; }
constexpr int width(int t, int cols) { return 32 * cols - 2 * halo(t, cols); }

// CTAs an SM holds (registers).
constexpr int resident(int t, int cols)
{
    return cols == 2 ? (t <= 2 ? 8 : (t == 3 ? 7 : (t == 4 ? 6 : 5))) : (t == 1 ? 6 : (t == 2 ? 5 : (t == 3 ? 4 : (t <= 5 ? 3 : 2))));
}

// The arithmetic of a pair of sites: phi at its own row (c), at the rows before and after (m, p)
// and beyond its ends (left, right); v is kicked in place; returns the new phi.

// FP32, the staged kernels' folded kick in packed pairs: the same operations as update4, so the same
// bits whichever kernel steps a box.  The kicks lie in shared memory as pairs: in registers they take
// 10 a level (T = 5: 12 warps an SM instead of 20), and read from the parameters by run they keep the
// constant port busy (4096^2, T = 4: 73% busy, 62 us a pass).
struct Fold32 {
    static constexpr bool kShared = true;
    struct alignas(16) K {
        unsigned long long c1, g, k1, nk2;
    };
    struct P {
        f2 r;
    };
    static __device__ __forceinline__ P pair(float a, float b) { return P{pk2(a, b)}; }
    static __device__ __forceinline__ void split(P p, float& a, float& b) { upk2(p.r, a, b); }
    // D = 3: zp, zm are the neighbours along z
    template <int D>
    static __device__ __forceinline__ P update(P m, P c, P p, P zm, P zp, float left, float right, P& v, const K& k,
                                                f2 dt, const RunConst<float>&)
    {
        float x, y;
        upk2(c.r, x, y);
        f2 s = add2(pk2(__fadd_rn(y, left), __fadd_rn(right, x)), add2(p.r, m.r));
        if (D == 3) s = add2(s, add2(zp.r, zm.r));
        const f2 u = mul2(c.r, fma2(f2{k.nk2}, mul2(c.r, c.r), f2{k.k1}));
        v.r = fma2(f2{k.c1}, v.r, fma2(f2{k.g}, s, u));
        return P{fma2(dt, v.r, c.r)};
    }
};

// FP32 of the boxes that the staged kernels do not take: Eqs. 3-5 as the generic step evaluates them,
// the constants read by the instructions that use them.
struct Plain32 {
    static constexpr bool kShared = false;
    using K = StepCoef<float>;
    struct P {
        float a, b;
    };
    static __device__ __forceinline__ P pair(float a, float b) { return P{a, b}; }
    static __device__ __forceinline__ void split(P p, float& a, float& b) { a = p.a, b = p.b; }
    template <int D>
    static __device__ __forceinline__ P update(P m, P c, P p, P zm, P zp, float left, float right, P& v, const K& k,
                                                f2, const RunConst<float>& rc)
    {
        P n;
        site_update<float, false, D>(c.a, c.b, left, p.a, m.a, zp.a, zm.a, v.a, n.a, k, rc);
        site_update<float, false, D>(c.b, right, c.a, p.b, m.b, zp.b, zm.b, v.b, n.b, k, rc);
        return n;
    }
};

// One launch: up to NR runs of one box, T kicks each.
template <class M, int T, int NR>
struct Args {
    const float* phi_in[NR];
    float* phi_out[NR];
    const float* v_in[NR];
    float* v_out[NR];
    typename M::K k[NR][T];
    RunConst<float> rc[NR];
    int nx, ny, nstrips, nchunks, cy, nruns;
};

// A lane's columns of a row on their way into the lane's own slot of the ring.
template <int COLS, bool VEC>
__device__ __forceinline__ void stage(float* dst, const float* row, const int (&x)[COLS])
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (VEC && COLS == 4) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(row + x[0]) : "memory");
    } else if constexpr (VEC) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(row + x[0]) : "memory");
    } else {
#pragma unroll
        for (int j = 0; j < COLS; ++j)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * j), "l"(row + x[j]) : "memory");
    }
}

template <class M, int COLS>
__device__ __forceinline__ void unstage(const float* src, typename M::P (&p)[COLS / 2])
{
    if constexpr (COLS == 4) {
        const float4 f = *reinterpret_cast<const float4*>(src);
        p[0] = M::pair(f.x, f.y);
        p[1] = M::pair(f.z, f.w);
    } else {
        const float2 f = *reinterpret_cast<const float2*>(src);
        p[0] = M::pair(f.x, f.y);
    }
}

// The lane's columns lo .. hi-1 (all or none of them when VEC) from column x on.
template <class M, int COLS, bool VEC>
__device__ __forceinline__ void store(float* p, int x, int lo, int hi, const typename M::P (&w)[COLS / 2])
{
    float f[COLS];
#pragma unroll
    for (int j = 0; j < COLS / 2; ++j) M::split(w[j], f[2 * j], f[2 * j + 1]);
    if constexpr (VEC) {
        if (hi <= lo) return;
        if constexpr (COLS == 4) *reinterpret_cast<float4*>(p + x) = make_float4(f[0], f[1], f[2], f[3]);
        else *reinterpret_cast<float2*>(p + x) = make_float2(f[0], f[1]);
    } else {
#pragma unroll
        for (int j = 0; j < COLS; ++j)
            if (j >= lo && j < hi) p[x + j] = f[j];
    }
}

// VEC: nx a multiple of COLS and the fields aligned to COLS floats.
template <class M, int T, int COLS, bool VEC, int NR>
__global__ void __launch_bounds__(kThreads, resident(T, COLS)) k_march2d(const __grid_constant__ Args<M, T, NR> a)
{
    using P = typename M::P;
    using K = typename M::K;
    constexpr int HX = halo(T, COLS), U = width(T, COLS), NP = COLS / 2, kRow = 32 * COLS;
    __shared__ __align__(16) float ring[kWarps][2 * kRing][kRow];  // phi rows, then dphi rows; a lane reads its own slots
    __shared__ K kicks[M::kShared ? kWarps : 1][T];
    chain_enter();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nx = a.nx, ny = a.ny;
    int w = blockIdx.x * kWarps + wid, run = 0;
    if (NR > 1) {
        run = w / (a.nstrips * a.nchunks);
        w -= run * a.nstrips * a.nchunks;
    }
    if (NR > 1 ? run >= a.nruns : w >= a.nstrips * a.nchunks) return;
    if (M::kShared) {
        if (lane < T) kicks[wid][lane] = a.k[run][lane];
        __syncwarp();
    }
    K kk[T];  // COLS == 4: in registers
#pragma unroll
    for (int l = 0; l < T; ++l) kk[l] = a.k[run][l];
    const RunConst<float>& rc = a.rc[run];
    const f2 dt = pk2(rc.deta, rc.deta);
    float* const rp = &ring[wid][0][lane * COLS];
    float* const rv = rp + kRing * kRow;
    const int chunk = w / a.nstrips, x0 = (w - chunk * a.nstrips) * U, y0 = chunk * a.cy;
    const int rows = min(a.cy, ny - y0);
    int x[COLS];  // the lane's columns, periodic
    x[0] = (x0 - HX + COLS * lane) % nx;
    if (x[0] < 0) x[0] += nx;
#pragma unroll
    for (int j = 1; j < COLS; ++j) x[j] = x[j - 1] + 1 == nx ? 0 : x[j - 1] + 1;
    const int c0 = COLS * lane - HX;  // of the strip's columns 0 .. U-1 this lane keeps c0+lo .. c0+hi-1
    const int lo = c0 < 0 ? COLS : 0, hi = min(COLS, min(U, nx - x0) - c0);
    float* pout = a.phi_out[run] + (int64_t)y0 * nx;
    float* vout = a.v_out[run] + (int64_t)y0 * nx;

    const int iters = rows + 2 * T;  // level-0 rows y0-T .. y0+rows+T-1
    int y = (y0 - T) % ny, next = 0;
    if (y < 0) y += ny;
    const float* pin = a.phi_in[run] + (int64_t)y * nx;
    const float* vin = a.v_in[run] + (int64_t)y * nx;
    auto fetch = [&] {  // the next row of both fields into its ring slots; a group of its own, also when empty
        if (next < iters) {
            const int slot = (next & (kRing - 1)) * kRow;
            stage<COLS, VEC>(rp + slot, pin, x);
            stage<COLS, VEC>(rv + slot, vin, x);
            ++next, ++y;
            const int64_t step = y == ny ? (int64_t)nx * (1 - ny) : nx;
            if (y == ny) y = 0;
            pin += step;
            vin += step;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int u = 0; u < kRing - 1; ++u) fetch();
    P m[T][NP], c[T][NP], vd[T][NP], vlast[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        vlast[j] = M::pair(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < T; ++l) m[l][j] = c[l][j] = vd[l][j] = vlast[j];  // overwritten before a row that is kept reads them
    }
#pragma unroll 3
    for (int i = 0; i < iters; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
        const int slot = (i & (kRing - 1)) * kRow;
        P p[NP], v[NP], vr[NP];  // phi row i, dphi row i-1
        unstage<M, COLS>(rp + slot, p);
        unstage<M, COLS>(rv + slot, vr);
        fetch();  // into the slot of row i-1
#pragma unroll
        for (int j = 0; j < NP; ++j) v[j] = vlast[j], vlast[j] = vr[j];
#pragma unroll
        for (int l = 0; l < T; ++l) {  // level l+1 at row i-1-l
            float f[COLS];
#pragma unroll
            for (int j = 0; j < NP; ++j) M::split(c[l][j], f[2 * j], f[2 * j + 1]);
            const float left = __shfl_up_sync(0xffffffffu, f[COLS - 1], 1);
            const float right = __shfl_down_sync(0xffffffffu, f[0], 1);
            const K k = M::kShared ? (COLS == 2 ? kicks[wid][l] : kk[l]) : a.k[0][l];
            P n[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                n[j] = M::template update<2>(m[l][j], c[l][j], p[j], p[j], p[j], j == 0 ? left : f[2 * j - 1],
                                             j == NP - 1 ? right : f[2 * j + 2], v[j], k, dt, rc);
                m[l][j] = c[l][j];
                c[l][j] = p[j];
                p[j] = n[j];
                if (l + 1 < T) {
                    const P t = vd[l][j];
                    vd[l][j] = v[j];
                    v[j] = t;
                }
            }
        }
        if (i >= 2 * T) {
            store<M, COLS, VEC>(pout, x[0], lo, hi, p);
            store<M, COLS, VEC>(vout, x[0], lo, hi, v);
            pout += nx;
            vout += nx;
        }
    }
}

}  // namespace march

}  // namespace prs
