// prs_adj_march.cuh -- the reverse step of the adjoint over an FP32 3D box of any sides.
//
// The staged sweep (k_adjoint3d_f32) takes boxes whose rows and y side fit its tiles, at the copy
// bandwidth.  On other boxes one thread a site read lt and its neighbours, phi and its neighbours, dphi
// and lphi one by one (250^3: 304 us a step; here 84.  128 x 104 x 200: 84 and 19).  Here a warp owns 64
// columns (a pair a lane) of four rows and marches along z as the forward march does (prs_march3d.cuh):
// lt's z neighbours wait in registers, its y neighbours are the warp's other rows, x neighbours come by
// shuffle, and everything an iteration uses comes in one slot of a ring each lane fills ahead for itself.
// The dJ/dalpha term takes phi (L lt) for lt (L phi), as the staged sweep does, so phi is read at the
// site only.
//
// (Two steps a pass, 32 bytes a site instead of 48 with lt and lphi between them in registers, took 219
// us a pass at 256^3 against 128 for two staged steps: 32 rows staged for four, eight warps an SM.)
#pragma once

#include "prs_march2d.cuh"
#include "prs_reduce.cuh"

namespace prs {

namespace march {

constexpr int kAdjRows = 4, kAdjRing = 3;
constexpr int kAdjSlot = (kAdjRows + 2 + 3 * kAdjRows) * 64;  // floats: rows of lt, then of lphi, phi and dphi

struct AdjStepF {
    float c1, c2, cV, dc1, dc2;
};

struct AdjArgs {
    const float* lt_in;
    float* lt_out;  // lt of the step before, or lv when `last`
    float* lphi;    // in place
    const float* phi;
    const float* v;
    AdjStepF k;
    RunConst<float> rc;
    DiagScratch scr;
    int nx, ny, nz, nstrips, ygroups, cz;
    bool last;
};

// Kahan's sum.
struct AdjAcc {
    float s, comp;
    __device__ __forceinline__ void add(float term)
    {
        const float y = term - comp, t = s + y;
        comp = (t - s) - y;
        s = t;
    }
};

// One site of the reverse step: l = lt_n and sum its neighbours' pair sums, q = phi^n; returns lt_{n-1}
// (lv_n when last), lp becomes lphi_n; Llt and f for the dJ/dalpha term.
__device__ __forceinline__ float adj_site(float l, float sum, float q, float& lp, const AdjStepF& k,
                                          const RunConst<float>& rc, bool last, float& Llt)
{
    Llt = (sum - rc.twoD * l) * rc.inv_dx2;
    const float fprime = k.cV * (3.0f * (q * q) * rc.inv_phi0sq - 1.0f);
    lp = lp + k.c2 * (Llt - fprime * l);
    return last ? k.c1 * l : k.c1 * l + rc.deta * lp;
}

__device__ __forceinline__ float adj_term(float l, float q, float v, float Llt, const AdjStepF& k,
                                          const RunConst<float>& rc)
{
    const float f = (k.cV * q) * ((q * q) * rc.inv_phi0sq - 1.0f);
    return l * (k.dc1 * v - k.dc2 * f) + k.dc2 * (q * Llt);
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads, 3) k_adj_march(const __grid_constant__ AdjArgs a)
{
    constexpr int R = kAdjRows, COLS = 2, HX = halo(1, COLS), U = width(1, COLS), kRow = 32 * COLS, N = R + 2;
    constexpr int oL = N, oP = oL + R, oV = oP + R;  // rows of a ring slot
    extern __shared__ __align__(16) float ring3[];
    chain_enter();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nx = a.nx, ny = a.ny, nz = a.nz;
    int b = blockIdx.x;
    const int x0 = b % a.nstrips * U;
    b /= a.nstrips;
    const int y0 = (b % a.ygroups * kWarps + wid) * R, z0 = b / a.ygroups * a.cz;
    const int planes = y0 < ny ? min(a.cz, nz - z0) : 0, rows = min(R, ny - y0);
    float* const rp = ring3 + wid * kAdjRing * kAdjSlot + lane * COLS;
    int xa = (x0 - HX + COLS * lane) % nx;
    if (xa < 0) xa += nx;
    const int x[COLS] = {xa, xa + 1 == nx ? 0 : xa + 1};
    const int c0 = COLS * lane - HX;
    const int lo = c0 < 0 ? COLS : 0, hi = min(COLS, min(U, nx - x0) - c0);
    const bool use0 = 0 >= lo && 0 < hi, use1 = 1 >= lo && 1 < hi;  // the lane's columns of the strip
    unsigned row[N];
    int yr = y0 == 0 ? ny - 1 : (y0 - 1) % ny;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        row[r] = (unsigned)yr * (unsigned)nx;
        if (++yr >= ny) yr = 0;
    }
    const int64_t plane = (int64_t)nx * ny;
    const int64_t out0 = (int64_t)z0 * plane + (int64_t)y0 * nx;
    float* lpo = a.lphi + out0;
    float* lto = a.lt_out + out0;
    const int iters = planes > 0 ? planes + 2 : 0;  // lt planes z0-1 .. z0+planes
    int z = z0 == 0 ? nz - 1 : z0 - 1, next = 0, fill = 0;
    auto fetch = [&] {  // a plane of lt and the plane before it of the fields read at the site
        if (next < iters) {
            float* d = rp + fill * kAdjSlot;
            const int64_t p0 = (int64_t)z * plane, p1 = (int64_t)(z == 0 ? nz - 1 : z - 1) * plane;
#pragma unroll
            for (int r = 0; r < N; ++r) stage<COLS, VEC>(d + r * kRow, a.lt_in + p0 + row[r], x);
            if (next >= 2) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    stage<COLS, VEC>(d + (oL + r) * kRow, a.lphi + p1 + row[r + 1], x);
                    stage<COLS, VEC>(d + (oP + r) * kRow, a.phi + p1 + row[r + 1], x);
                    stage<COLS, VEC>(d + (oV + r) * kRow, a.v + p1 + row[r + 1], x);
                }
            }
            ++next;
            fill = fill == kAdjRing - 1 ? 0 : fill + 1;
            if (++z == nz) z = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int u = 0; u < kAdjRing - 1; ++u) fetch();
    const float2 zero = make_float2(0.f, 0.f);
    float2 m[R], c[N];
#pragma unroll
    for (int r = 0; r < R; ++r) m[r] = zero;
#pragma unroll
    for (int r = 0; r < N; ++r) c[r] = zero;
    double tot = 0.0;
    int use = 0;
    auto at = [&](const float* s, int r) { return *reinterpret_cast<const float2*>(s + r * kRow); };
    for (int i = 0; i < iters; ++i) {  // lt plane i arrives, plane i-1 is stepped
        asm volatile("cp.async.wait_group %0;" ::"n"(kAdjRing - 2) : "memory");
        const float* s = rp + use * kAdjSlot;
        use = use == kAdjRing - 1 ? 0 : use + 1;
        float2 p[N];
#pragma unroll
        for (int r = 0; r < N; ++r) p[r] = at(s, r);
        if (i >= 2) {
            AdjAcc da{0.f, 0.f};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 l = c[r + 1], q = at(s, oP + r), v = at(s, oV + r);
                const float left = __shfl_up_sync(0xffffffffu, l.y, 1), right = __shfl_down_sync(0xffffffffu, l.x, 1);
                const float sa = ((l.y + left) + (c[r + 2].x + c[r].x)) + (p[r + 1].x + m[r].x);
                const float sb = ((right + l.x) + (c[r + 2].y + c[r].y)) + (p[r + 1].y + m[r].y);
                float2 lp = at(s, oL + r), out;
                float La, Lb;
                out.x = adj_site(l.x, sa, q.x, lp.x, a.k, a.rc, a.last, La);
                out.y = adj_site(l.y, sb, q.y, lp.y, a.k, a.rc, a.last, Lb);
                if (r < rows) {
                    if (use0) da.add(adj_term(l.x, q.x, v.x, La, a.k, a.rc));
                    if (use1) da.add(adj_term(l.y, q.y, v.y, Lb, a.k, a.rc));
                    const unsigned o = (unsigned)r * (unsigned)nx + (unsigned)x[0];
                    if constexpr (VEC) {
                        if (use0) {
                            *reinterpret_cast<float2*>(lto + o) = out;
                            *reinterpret_cast<float2*>(lpo + o) = lp;
                        }
                    } else {
                        if (use0) lto[o] = out.x, lpo[o] = lp.x;
                        if (use1) lto[o + 1] = out.y, lpo[o + 1] = lp.y;
                    }
                }
            }
            tot += (double)da.s;
            lto += plane;
            lpo += plane;
        }
        fetch();  // into the slot of the iteration before
#pragma unroll
        for (int r = 0; r < R; ++r) m[r] = c[r + 1];
#pragma unroll
        for (int r = 0; r < N; ++r) c[r] = p[r];
    }
    __syncthreads();  // the ring is free
    block_reduce_and_finish(DiagAcc{tot, 0.0, 0, 0, 0, 0}, a.scr, reinterpret_cast<double2*>(ring3));
}

}  // namespace march

}  // namespace prs
