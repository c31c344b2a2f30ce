// prs_tile.cuh -- the FP32 update of Eqs. 3-5 in the forms the staged kernels share, and the one-step
// 3D tile (prs_fast.cu).
//
// A tile is a run of z-planes, ty whole x-rows of y per plane.  phi arrives through the TMA
// engine: cp.async.bulk copies of whole row runs into a 4-slot shared-memory ring, one mbarrier
// per slot; while plane z is used, planes z-1, z, z+1 are resident and z+2 is in flight.  x
// neighbours come from the neighbouring lane's float4 by warp shuffle (rows are whole, so the
// periodic wrap is a shared-memory read by lanes 0 and 31); y and z neighbours are 128-bit
// shared-memory reads; dphi is pointwise and loaded into registers one plane ahead.
//
// Shared memory of a tile: [128 B: 4 mbarriers][4 ring slots].  Every mbarrier wait is bounded; a
// tile that gives up returns false (the same value in every thread) after letting its issued
// copies land.
#pragma once

#include <cuda_runtime.h>

#include "prs_internal.h"
#include "prs_f32x2.cuh"
#include "prs_ptx.cuh"

namespace prs {

static constexpr int kFastThreads = 256;

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__device__ __forceinline__ float4 ldg_stream4(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }

__device__ __forceinline__ void stg4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// Eqs. 3-5 at one site, FP32: x neighbours (xp, xm), y neighbours (a, b), z neighbours
// (e, f).  Returns phi^{n+1}; vv becomes dphi^{n+1/2}.  The kick is KickF's
// folded form, 11 operations a site (the FP64 path keeps the canonical order of Eqs. 3-5
// as written); every term is odd in phi, so a negated field steps to the negated field
// exactly.  Each operation is pinned (round-to-nearest intrinsics, the three fused
// multiply-adds explicit), so update4's packed pairs give the same bits.
__device__ __forceinline__ float update1(float cc, float xp, float xm, float a, float b, float e, float f, float& vv,
                                         const KickF& k, const RunConst<float>& rc)
{
    float s2 = __fadd_rn(xp, xm);
    s2 = __fadd_rn(s2, __fadd_rn(a, b));
    s2 = __fadd_rn(s2, __fadd_rn(e, f));
    const float u = __fmul_rn(cc, __fmaf_rn(-k.k2, __fmul_rn(cc, cc), k.k1));
    const float vn = __fmaf_rn(k.c1, vv, __fmaf_rn(k.g, s2, u));
    vv = vn;
    return __fmaf_rn(rc.deta, vn, cc);
}

// Eqs. 3-5 for the four sites of one float4: update1's operations on two packed pairs
// of sites (x, y) and (z, w), one f32x2 instruction per pair and operation, except the
// x-neighbour sums, whose operands straddle the pairs.
__device__ __forceinline__ void update4(float4 c, float left, float right, float4 yp, float4 ym, float4 zp, float4 zm,
                                        float4& v, float4& pn, const KickF& k, const RunConst<float>& rc)
{
    const f2 kc1 = pk2(k.c1, k.c1), kg = pk2(k.g, k.g), kk1 = pk2(k.k1, k.k1), nk2 = pk2(-k.k2, -k.k2);
    const f2 dt = pk2(rc.deta, rc.deta);
    f2 s0 = pk2(__fadd_rn(c.y, left), __fadd_rn(c.z, c.x));
    f2 s1 = pk2(__fadd_rn(c.w, c.y), __fadd_rn(right, c.z));
    s0 = add2(s0, add2(pk2(yp.x, yp.y), pk2(ym.x, ym.y)));
    s1 = add2(s1, add2(pk2(yp.z, yp.w), pk2(ym.z, ym.w)));
    s0 = add2(s0, add2(pk2(zp.x, zp.y), pk2(zm.x, zm.y)));
    s1 = add2(s1, add2(pk2(zp.z, zp.w), pk2(zm.z, zm.w)));
    const f2 c0 = pk2(c.x, c.y), c1 = pk2(c.z, c.w);
    const f2 u0 = mul2(c0, fma2(nk2, mul2(c0, c0), kk1));
    const f2 u1 = mul2(c1, fma2(nk2, mul2(c1, c1), kk1));
    const f2 v0 = fma2(kc1, pk2(v.x, v.y), fma2(kg, s0, u0));
    const f2 v1 = fma2(kc1, pk2(v.z, v.w), fma2(kg, s1, u1));
    upk2(v0, v.x, v.y);
    upk2(v1, v.z, v.w);
    upk2(fma2(dt, v0, c0), pn.x, pn.y);
    upk2(fma2(dt, v1, c1), pn.z, pn.w);
}

// update4 with the constants already packed (KickP): the same operations in the same order,
// so the same bits.
__device__ __forceinline__ void update4p(float4 c, float left, float right, float4 yp, float4 ym, float4 zp,
                                         float4 zm, float4& v, float4& pn, const KickP& k)
{
    const f2 kc1{k.c1}, kg{k.g}, kk1{k.k1}, nk2{k.nk2}, dt{k.dt};
    f2 s0 = pk2(__fadd_rn(c.y, left), __fadd_rn(c.z, c.x));
    f2 s1 = pk2(__fadd_rn(c.w, c.y), __fadd_rn(right, c.z));
    s0 = add2(s0, add2(pk2(yp.x, yp.y), pk2(ym.x, ym.y)));
    s1 = add2(s1, add2(pk2(yp.z, yp.w), pk2(ym.z, ym.w)));
    s0 = add2(s0, add2(pk2(zp.x, zp.y), pk2(zm.x, zm.y)));
    s1 = add2(s1, add2(pk2(zp.z, zp.w), pk2(zm.z, zm.w)));
    const f2 c0 = pk2(c.x, c.y), c1 = pk2(c.z, c.w);
    const f2 u0 = mul2(c0, fma2(nk2, mul2(c0, c0), kk1));
    const f2 u1 = mul2(c1, fma2(nk2, mul2(c1, c1), kk1));
    const f2 v0 = fma2(kc1, pk2(v.x, v.y), fma2(kg, s0, u0));
    const f2 v1 = fma2(kc1, pk2(v.z, v.w), fma2(kg, s1, u1));
    upk2(v0, v.x, v.y);
    upk2(v1, v.z, v.w);
    upk2(fma2(dt, v0, c0), pn.x, pn.y);
    upk2(fma2(dt, v1, c1), pn.z, pn.w);
}

// The scalar kick constants and time step of a packed kick (the low halves), for update1.
__device__ __forceinline__ KickF kick_scalar(const KickP& k)
{
    return KickF{__uint_as_float((unsigned)k.c1), __uint_as_float((unsigned)k.g), __uint_as_float((unsigned)k.k1),
                 -__uint_as_float((unsigned)k.nk2)};
}

__device__ __forceinline__ RunConst<float> deta_only(const KickP& k)
{
    return RunConst<float>{__uint_as_float((unsigned)k.dt), 0.f, 0.f, 0.f, 0.f, 0.f};
}

// x-neighbours of a float4 at column `col` of a whole row in shared memory.
__device__ __forceinline__ void x_halo(const float* row, int col, int nq, int nx, int lane, float4 c, float& left,
                                       float& right)
{
    left = __shfl_up_sync(0xffffffffu, c.w, 1);
    right = __shfl_down_sync(0xffffffffu, c.x, 1);
    if (lane == 0) left = row[col == 0 ? nx - 1 : 4 * col - 1];
    if (lane == 31) right = row[col == nq - 1 ? 0 : 4 * col + 4];
}

// After a wait gave up: let the copies this CTA issued land (each wait again
// bounded) before the CTA exits and its shared memory is reused.  Slots are
// waited in issue order from local index `from`.
static __device__ __noinline__ void drain(uint64_t* bar, int from, int issued, unsigned int* err)
{
    for (int i = from; i <= issued; ++i) mbar_wait(&bar[i & 3], (i >> 2) & 1, err);
}


// --------------------------------------------------------------- diagnostics
//
// Eq. 7 weights with the hardware's fast roots (prs_measure.cu).

// |g| / sum_i |g_i| with the hardware reciprocal square root and reciprocal
// (a few ulp).  den > 0 because the link's own component is non-zero; when the
// squares underflow (|g| below ~1e-19) the components are first divided by den.
__device__ __forceinline__ float link_weight_from(float num, float den, float gx, float gy, float gz)
{
    if (num >= 1e-30f) return __fdividef(num * rsqrtf(num), den);
    const float a = gx / den, b = gy / den, c = gz / den;
    return sqrtf(a * a + b * b + c * c);
}

__device__ __forceinline__ float link_weight3(float gx, float gy, float gz)
{
    float num = gx * gx;
    num = num + gy * gy;
    num = num + gz * gz;
    float den = fabsf(gx);
    den = den + fabsf(gy);
    den = den + fabsf(gz);
    return link_weight_from(num, den, gx, gy, gz);
}

__device__ __forceinline__ float link_weight2(float gx, float gy)
{
    float num = gx * gx;
    num = num + gy * gy;
    float den = fabsf(gx);
    den = den + fabsf(gy);
    return link_weight_from(num, den, gx, gy, 0.0f);
}

// Make generic-proxy writes of global memory visible to this CTA's bulk copies.
__device__ __forceinline__ void fence_proxy_async_global()
{
    asm volatile("fence.proxy.async.global;" ::: "memory");
}

struct Tile3D {
    const float* phi_in;
    float* phi_out;
    const float* v_in;
    float* v_out;
    int nx, ny, nz, ty;  // box; ty rows of y per plane in a tile
    int y0, z0, zn;      // first row, first plane, number of planes of this tile
};

__host__ __device__ constexpr size_t tile_smem3d(int nx, int ty) { return 128 + 4 * (size_t)(ty + 2) * nx * sizeof(float); }

// One 3D tile: Eqs. 3-5 (phi_in -> phi_out, v_in -> v_out).
template <int ITEMS>
__device__ __forceinline__ bool tile3d(const Tile3D& T, const KickF& k, const RunConst<float>& rc,
                                       unsigned char* smem, unsigned int* err)
{
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    float* ring = reinterpret_cast<float*>(smem + 128);
    const int tid = threadIdx.x, lane = tid & 31;
    const int nx = T.nx, ty = T.ty;
    const int ny = T.ny, nz = T.nz, y0 = T.y0, z0 = T.z0, zn = T.zn;
    const int nq = nx >> 2;
    const int tile = (ty + 2) * nx;
    const size_t plane = (size_t)nx * ny;

    if (tid == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) mbar_init(&bar[i], 1);
        mbar_fence_init();
    }
    __syncthreads();

    const int ytop = (y0 == 0 ? ny : y0) - 1;
    const int ybot = (y0 + ty == ny) ? 0 : y0 + ty;
    const unsigned rowb = (unsigned)nx * 4u;
    const int nloc = zn + 2;  // local planes 0..zn+1 = global z0-1 .. z0+zn (periodic)
    auto issue = [&](int i) {
        int p = z0 - 1 + i;
        p = p < 0 ? p + nz : (p >= nz ? p - nz : p);
        float* dst = ring + (i & 3) * tile;
        const float* src = T.phi_in + (size_t)p * plane;
        uint64_t* b = &bar[i & 3];
        mbar_arrive_expect_tx(b, rowb * (unsigned)(ty + 2));
        bulk_g2s(dst, src + (size_t)ytop * nx, rowb, b);
        bulk_g2s(dst + nx, src + (size_t)y0 * nx, rowb * (unsigned)ty, b);
        bulk_g2s(dst + (size_t)(ty + 1) * nx, src + (size_t)ybot * nx, rowb, b);
    };
    int issued = -1;  // thread 0: highest local plane whose copy was issued
    if (tid == 0)
        for (int i = 0; i < 3 && i < nloc; ++i) issue(i), issued = i;

    int row[ITEMS], col[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        int q = tid + kFastThreads * j;
        row[j] = q / nq;
        col[j] = q - row[j] * nq;
    }
    float4 vc[ITEMS];
    {
        const float* vb = T.v_in + (size_t)z0 * plane + (size_t)y0 * nx;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) vc[j] = ldg_stream4(vb + (size_t)row[j] * nx + 4 * col[j]);
    }

    for (int zi = 0; zi < zn; ++zi) {
        // local planes zi, zi+1, zi+2 (= z-1, z, z+1) must be resident
        bool ok = true;
        if (zi == 0) ok = mbar_wait(&bar[0], 0, err) && mbar_wait(&bar[1], 0, err);
        ok = ok && mbar_wait(&bar[(zi + 2) & 3], ((zi + 2) >> 2) & 1, err);
        // block-wide decision; also: every thread is done with the previous plane
        if (__syncthreads_or(!ok)) {
            if (tid == 0) drain(bar, zi, issued, err);
            __syncthreads();
            return false;
        }
        if (tid == 0 && zi + 3 < nloc) issue(zi + 3), issued = zi + 3;  // into the slot of plane z-2

        const int z = z0 + zi;
        float4 vn[ITEMS];
        if (zi + 1 < zn) {
            const float* vb = T.v_in + (size_t)(z + 1) * plane + (size_t)y0 * nx;
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) vn[j] = ldg_stream4(vb + (size_t)row[j] * nx + 4 * col[j]);
        }
        const float* pm = ring + (zi & 3) * tile + nx;
        const float* pc = ring + ((zi + 1) & 3) * tile + nx;
        const float* pp = ring + ((zi + 2) & 3) * tile + nx;
        float* po = T.phi_out + (size_t)z * plane + (size_t)y0 * nx;
        float* vo = T.v_out + (size_t)z * plane + (size_t)y0 * nx;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const int r = row[j];
            const int off = r * nx + 4 * col[j];
            float4 c = lds4(pc + off);
            float4 ym = lds4(pc + off - nx);
            float4 yp = lds4(pc + off + nx);
            float4 zm = lds4(pm + off);
            float4 zp = lds4(pp + off);
            float left, right;
            x_halo(pc + r * nx, col[j], nq, nx, lane, c, left, right);
            float4 pn;
            update4(c, left, right, yp, ym, zp, zm, vc[j], pn, k, rc);
            stg4(po + off, pn);
            stg4(vo + off, vc[j]);
        }
        if (zi + 1 < zn) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) vc[j] = vn[j];
        }
    }
    __syncthreads();  // the ring may be reused by the caller's next tile
    return true;
}

}  // namespace prs
