// prs_measure.cu -- the wall diagnostics (Eq. 7 link area, Eq. 8 wall velocity) of any box.
//
// What bounds it: 2 to 8 per cent of the links cross a wall and 5 to 15 per cent of the sites
// touch one, scattered so that most warps of consecutive sites hold a few.  Evaluating Eq. 7 and
// Eq. 8 where such a site happens to lie runs the square roots and divisions with most lanes
// idle (in FP64, where an SM issues two lanes a clock, that alone took most of the pass), and
// comparing every site with each of its 2D neighbours costs more than the field's memory traffic.
// So the sites are reduced to sign bits first and the arithmetic runs on compacted lists:
//   1. a CTA stages a tile of 128 columns x rows (3D: x planes) and its one-site halo into
//      shared memory with asynchronous copies (16 bytes where rows allow it, else one element);
//   2. one ballot per 32 sites makes sign words; a lane then finds the crossing links and wall
//      sites of 32 sites at a time with a handful of bit operations, and counts them with popc;
//   3. each warp compacts its links (then its wall sites) into a list and evaluates 32 at a time,
//      neighbours from shared memory, dphi gathered (just read for the finite test, so from L2).
//      (Eq. 8 at every site as dphi passes, predicated: 1024^3 3.73 against 3.46 ms.)
// Tiles are whole blocks of the box, not a march: three barriers a tile of up to 8192 sites, and
// three CTAs an SM overlap one tile's copies with the others' arithmetic.  Halo rows come from L2.
// Measured (us, this pass; the pass it replaced): 1024^3 FP32 3150 (4200), 450 x 421 x 380 FP32
// 360 (1400, IEEE), 256^3 FP64 260 (2240), 2048^2 FP64 60 (435); 8.6 GB in 3.15 ms at 1024^3 is
// 0.40 of the copy bandwidth.  What bounds it now is instruction issue and latency (70 thread
// instructions a site, 0.5 of the issue slots; FP64: the pipe's divisions and roots).
// The arithmetic of one link or site is that of Eqs. 7 and 8 in a fixed order; only the order of
// the FP64 sums depends on the tiling, and that is fixed for a box.
#include <cuda_runtime.h>

#include <math.h>

#include <type_traits>

#include "prs_arith.cuh"
#include "prs_chain.h"
#include "prs_internal.h"
#include "prs_ptx.cuh"
#include "prs_reduce.cuh"
#include "prs_tile.cuh"
#include "prs_tmap.h"

namespace prs {

namespace {

constexpr int kMThreads = 256, kMWarps = kMThreads / 32;
constexpr int kMCols = 128;             // columns of a tile: four sign words

// A tile row in shared memory: the left halo column right before an aligned run of 128 columns,
// the right halo column after it.
template <typename R>
struct MRow {
    static constexpr int kOff = 16 / (int)sizeof(R), kLd = kMCols + 2 * kOff;
};

// Tiles of 128 columns x 2^lty rows x 2^ltz planes (2D: ltz = 0); x tiles fastest.
struct MTiling {
    int lty, ltz;
    unsigned ntx, nty, ntiles;
};

int halo_rows(int dims, const MTiling& T) { return ((1 << T.lty) + 2) * (dims == 3 ? (1 << T.ltz) + 2 : 1); }

// Sign words a warp works on (one a lane, so at most 32; whole rows): its list holds 32 entries
// for each.
__host__ __device__ constexpr int words_per_warp(int nrows) { return 4 * nrows / kMWarps; }

size_t measure_smem(int dims, size_t elem, const MTiling& T)
{
    const size_t rows = (size_t)halo_rows(dims, T), ld = kMCols + 2 * (16 / elem);
    return rows * ld * elem + rows * 16 + ((rows + 15) & ~(size_t)15) +
           (size_t)kMWarps * words_per_warp(1 << (T.lty + T.ltz)) * 32 * sizeof(unsigned short);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

template <int BYTES>
__device__ __forceinline__ void cp_async_elem(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}

// phi < 0: -0 and NaN are not.  FP64 by integers (the FP64 pipe would compare two lanes a clock):
// the bit patterns above that of -0 and up to that of -infinity.
__device__ __forceinline__ bool is_neg(float a) { return a < 0.0f; }
__device__ __forceinline__ bool is_neg(double a)
{
    return (unsigned long long)__double_as_longlong(a) - 0x8000000000000001ull <= 0x7FEFFFFFFFFFFFFFull;
}

// The finite test, accumulated over values: FP32 adds value * 0, which is NaN iff the value is
// not finite; FP64 keeps the largest high word of the magnitudes (integers again).
struct FiniteF {
    float acc = 0.0f;
    __device__ __forceinline__ void see(float a) { acc = __fmaf_rn(a, 0.0f, acc); }
    __device__ __forceinline__ bool bad() const { return !(acc == 0.0f); }
};
struct FiniteD {
    unsigned big = 0;
    __device__ __forceinline__ void see(double a) { big = max(big, (unsigned)__double2hiint(a) & 0x7fffffffu); }
    __device__ __forceinline__ bool bad() const { return big >= 0x7ff00000u; }
};
template <typename R>
using Finite = std::conditional_t<sizeof(R) == 4, FiniteF, FiniteD>;

// Four consecutive values, 16-byte aligned.
__device__ __forceinline__ void load4(const float* p, float (&a)[4])
{
    const float4 f = *reinterpret_cast<const float4*>(p);
    a[0] = f.x, a[1] = f.y, a[2] = f.z, a[3] = f.w;
}
__device__ __forceinline__ void load4(const double* p, double (&a)[4])
{
    const double2 f = *reinterpret_cast<const double2*>(p), h = *reinterpret_cast<const double2*>(p + 2);
    a[0] = f.x, a[1] = f.y, a[2] = h.x, a[3] = h.y;
}

__device__ __forceinline__ int top_bit(unsigned m)
{
    int b;
    asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(m));
    return b;
}

struct MSums {
    double sw, sr;
    float pw, pr;  // FAST: this tile's partial sums (a few terms a thread), folded into sw, sr
    int nl, nw, nv0, nnf;
};

// Eq. 7 weight |g| / sum_i |g_i| of the link from tile site s along axis d, IEEE operations:
// g_d the one-sided difference, the transverse components the centred differences averaged over
// the link's ends, added in axis order.  When the squares underflow the components are scaled
// by den (> 0: the link's own component is not zero) first.
template <typename R, int D>
__device__ __forceinline__ R weight_ieee(const R* s, int d, int sy, int sz)
{
    using A = Arith<R, true>;
    const R* t = s + (d == 0 ? 1 : (d == 1 ? sy : sz));
    const int p1 = d == 0 ? sy : 1, p2 = d == 2 ? sy : sz;  // the transverse axes
    auto across = [&](int p) {
        return A::mul((R)0.25, A::add(A::sub(s[p], s[-p]), A::sub(t[p], t[-p])));
    };
    const R gd = A::sub(*t, *s), g1 = across(p1), g2 = D == 3 ? across(p2) : (R)0;
    R g[3];
    g[0] = d == 0 ? gd : g1;
    g[1] = d == 0 ? g1 : (d == 1 ? gd : g2);
    g[2] = d == 2 ? gd : g2;
    R num = (R)0, den = (R)0;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        num = A::add(num, A::mul(g[e], g[e]));
        den = A::add(den, fabs(g[e]));
    }
    const R tiny = sizeof(R) == 4 ? (R)1e-30 : (R)1e-290;
    if (!(num >= tiny)) {
        R n2 = (R)0;
#pragma unroll
        for (int e = 0; e < D; ++e) {
            const R r = A::div(g[e], den);
            n2 = A::add(n2, A::mul(r, r));
        }
        return A::sqrt(n2);
    }
    return A::div(A::sqrt(num), den);
}

// The same with the hardware reciprocal square root and division (link_weight_from).
template <int D>
__device__ __forceinline__ float weight_fast(const float* s, int d, int sy, int sz)
{
    const int od = d == 0 ? 1 : (d == 1 ? sy : sz);
    const float* t = s + od;
    const float gd = *t - *s;
    if (D == 2) {
        const int p = d == 0 ? sy : 1;
        const float g1 = 0.25f * ((s[p] - s[-p]) + (t[p] - t[-p]));
        return link_weight2(d == 0 ? gd : g1, d == 0 ? g1 : gd);
    }
    const int p1 = d == 0 ? sy : 1, p2 = d == 2 ? sy : sz;
    const float g1 = 0.25f * ((s[p1] - s[-p1]) + (t[p1] - t[-p1]));
    const float g2 = 0.25f * ((s[p2] - s[-p2]) + (t[p2] - t[-p2]));
    return link_weight3(d == 0 ? gd : g1, d == 0 ? g1 : (d == 1 ? gd : g2), d == 2 ? gd : g2);
}

// Exclusive prefix sum of cnt over the warp; total in every lane.
__device__ __forceinline__ int warp_prefix(int cnt, int lane, int& total)
{
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - cnt;
}

// The runs of one launch: blocks (., r) take run r.
template <typename R, int NR>
struct MRuns {
    const R* phi[NR];
    const R* dphi[NR];
    RunConst<R> rc[NR];
    DiagScratch scr[NR];
};

// FAST: FP32 with the hardware reciprocal square root and division; else IEEE operations.
// vec: rows may be staged 16 bytes at a time (row length and base address multiples of 16 bytes).
// err: the run's error word when map describes phi in boxes of a tile with its halo (then one
// tensor copy stages each tile whose rows do not wrap, the wrapped columns patched in), or null.
template <typename R, int D, bool FAST, int NR>
__global__ void __launch_bounds__(kMThreads, D == 2 ? 4 : 3)
    k_measure(const __grid_constant__ CUtensorMap map, const __grid_constant__ MRuns<R, NR> runs, Geo g, MTiling T,
              bool vec, unsigned int* err)
{
    const int run = NR > 1 ? blockIdx.y : 0;
    const R* phi = runs.phi[run];
    const R* dphi = runs.dphi[run];
    chain_enter();
    const RunConst<R>& rc = runs.rc[run];
    using A = Arith<R, true>;
    constexpr int kOff = MRow<R>::kOff, kLd = MRow<R>::kLd;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int ty = 1 << T.lty, tz = 1 << T.ltz;
    const int hrows = (ty + 2) * (D == 3 ? tz + 2 : 1);  // rows with the halo
    R* tile = reinterpret_cast<R*>(smem_raw);
    unsigned* sgn = reinterpret_cast<unsigned*>(tile + (size_t)hrows * kLd);  // four words a halo row
    unsigned char* side = reinterpret_cast<unsigned char*>(sgn + 4 * hrows);  // bits 0, 1: left, right halo column
    const int nrows = ty << T.ltz;
    const int per = words_per_warp(nrows);
    unsigned short* list =
        reinterpret_cast<unsigned short*>(side + ((hrows + 15) & ~15)) + (threadIdx.x >> 5) * per * 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sy = kLd, sz = kLd * (ty + 2);
    const int64_t plane = (int64_t)g.nx * g.ny;
    const double rscale = FAST && rc.V0 > (R)0 ? 1.0 / (double)rc.V0 : 0.0;
    MSums a{0.0, 0.0, 0.0f, 0.0f, 0, 0, 0, 0};

    __shared__ __align__(8) uint64_t bar;
    unsigned phase = 0;
    if (err && tid == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();

    for (unsigned q = blockIdx.x; q < T.ntiles; q += gridDim.x) {
        const unsigned q1 = q / T.ntx, q2 = q1 / T.nty;
        const int x0 = (int)(q - q1 * T.ntx) * kMCols, y0 = (int)(q1 - q2 * T.nty) << T.lty, z0 = (int)q2 << T.ltz;
        const int w = min(kMCols, g.nx - x0), hy = min(ty, g.ny - y0), hz = D == 3 ? min(tz, g.nz - z0) : 1;
        const bool whole = hy == ty && (D == 2 || hz == tz);
        const bool tma = err && y0 > 0 && y0 + ty < g.ny && (D == 2 || (z0 > 0 && z0 + tz < g.nz));
        R patch = (R)0;
        R* patch_at = nullptr;
        if (tma) {
            if (tid == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the last tile's patches
                mbar_arrive_expect_tx(&bar, (unsigned)(hrows * kLd * sizeof(R)));
                tma_load3(tile, &map, x0 - kOff, y0 - 1, D == 3 ? z0 - 1 : 0, &bar);
            }
            // threads 2h, 2h+1: the wrapped halo columns of halo row h (zero-filled by the copy)
            const int h = tid >> 1, left = (tid & 1) ^ 1;
            for (int u = h; u < hrows; u = hrows) {
                if (left ? x0 > 0 : x0 + w < g.nx) break;
                const int hz1 = D == 3 ? u / (ty + 2) : 1, hy1 = D == 3 ? u - hz1 * (ty + 2) : u;
                patch_at = tile + u * kLd + kOff + (left ? -1 : w);
                patch = phi[(D == 3 ? (int64_t)(z0 + hz1 - 1) * plane : 0) + (int64_t)(y0 + hy1 - 1) * g.nx +
                            (left ? g.nx - 1 : 0)];
            }
        }
        // else stage the tile, a warp a halo row: row hy1 - 1 of plane hz1 - 1
        const int xside = lane == 0 ? (x0 == 0 ? g.nx - 1 : x0 - 1) : (x0 + w == g.nx ? 0 : x0 + w);
        const int side_at = lane == 0 ? -1 : w;  // lanes 0 and 1: the halo columns
        for (int h = tma ? hrows : wid, hy1 = wid, hz1 = D == 3 ? 0 : 1; h < hrows; h += kMWarps, hy1 += kMWarps) {
            while (D == 3 && hy1 >= ty + 2) hy1 -= ty + 2, ++hz1;
            if (hy1 > hy + 1 || hz1 > hz + 1) continue;
            int y = y0 + hy1 - 1, z = z0 + hz1 - 1;
            y = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
            if (D == 3) z = z < 0 ? z + g.nz : (z >= g.nz ? z - g.nz : z);
            const R* src = phi + (D == 3 ? (int64_t)z * plane : 0) + (int64_t)y * g.nx;
            R* dst = tile + h * kLd + kOff;
            if (vec) {
#pragma unroll
                for (int u = 0; u < 4 / kOff; ++u) {
                    const int x = (lane + 32 * u) * kOff;
                    if (x < w) cp_async16(dst + x, src + x0 + x);
                }
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int x = lane + 32 * u;
                    if (x < w) cp_async_elem<(int)sizeof(R)>(dst + x, src + x0 + x);
                }
            }
            if (lane < 2) cp_async_elem<(int)sizeof(R)>(dst + side_at, src + xside);
        }
        // meanwhile: dphi once, for the finite test
        Finite<R> fin;
#pragma unroll 4
        for (int r = wid; r < nrows; r += kMWarps) {
            const int ry = r & (ty - 1), rz = r >> T.lty;
            if (!whole && (ry >= hy || rz >= hz)) continue;
            const R* src = dphi + (int64_t)(z0 + rz) * plane + (int64_t)(y0 + ry) * g.nx + x0 + 4 * lane;
            R v[4] = {(R)0, (R)0, (R)0, (R)0};
            if (vec && 4 * lane + 4 <= w) {
                load4(src, v);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (4 * lane + e < w) v[e] = src[e];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) fin.see(v[e]);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (tma) {
            const bool ok = mbar_wait(&bar, phase, err);
            if (__syncthreads_or(!ok)) {  // let the copy land (again bounded) before leaving
                if (tid == 0) mbar_wait(&bar, phase, err);
                __syncthreads();
                break;
            }
            phase ^= 1u;
            if (patch_at) *patch_at = patch;
        }
        __syncthreads();
        // four sign words a halo row, word e holding columns e, e+4, ... (a lane's four values by
        // one 128-bit read), and the finite test of phi on the tile's own rows
#pragma unroll 2
        for (int h = wid, hy1 = wid, hz1 = D == 3 ? 0 : 1; h < hrows; h += kMWarps, hy1 += kMWarps) {
            while (D == 3 && hy1 >= ty + 2) hy1 -= ty + 2, ++hz1;
            if (!whole && (hy1 > hy + 1 || hz1 > hz + 1)) continue;
            const R* row = tile + h * kLd + kOff;
            R p[4];
            load4(row + 4 * lane, p);
            unsigned b[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) b[e] = __ballot_sync(0xffffffffu, is_neg(p[e]));
            const unsigned s = __ballot_sync(0xffffffffu, is_neg(row[lane < 2 ? side_at : 0]));
            if (lane == 0) {
                *reinterpret_cast<uint4*>(sgn + 4 * h) = make_uint4(b[0], b[1], b[2], b[3]);
                side[h] = (unsigned char)(s & 3u);
            }
            if (hy1 >= 1 && hy1 <= hy && hz1 >= 1 && hz1 <= hz) {
                if (w == kMCols) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) fin.see(p[e]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (4 * lane + e < w) fin.see(p[e]);
                }
            }
        }
        __syncthreads();
        // the links and wall sites of 32 sites a lane
        unsigned lx = 0, ly = 0, lz = 0, wall = 0;
        int at = 0;  // tile offset of the word's first site
        const int wi = wid * per + lane;  // this lane's sign word: row wi/4, columns wi%4 + 4 bit
        if (lane < per && wi < 4 * nrows) {
            const int r = wi >> 2, c = wi & 3, ry = r & (ty - 1), rz = r >> T.lty;
            const int nb = (w - c + 3) >> 2;
            if (ry < hy && rz < hz && nb > 0) {
                const int h = (D == 3 ? (rz + 1) * (ty + 2) : 0) + ry + 1;
                const unsigned valid = nb >= 32 ? 0xffffffffu : (1u << nb) - 1u;
                const unsigned s = sgn[4 * h + c], sd = side[h];
                const unsigned next = c < 3 ? sgn[4 * h + c + 1] : (sgn[4 * h] >> 1) | (sd >> 1) << 31;
                const unsigned prev = c > 0 ? sgn[4 * h + c - 1] : (sgn[4 * h + 3] << 1) | (sd & 1u);
                at = h * kLd + kOff + c;
                lx = (s ^ next) & valid;
                ly = (s ^ sgn[4 * (h + 1) + c]) & valid;
                wall = lx | ly | ((s ^ prev) & valid) | ((s ^ sgn[4 * (h - 1) + c]) & valid);
                if (D == 3) {
                    lz = (s ^ sgn[4 * (h + ty + 2) + c]) & valid;
                    wall |= lz | ((s ^ sgn[4 * (h - ty - 2) + c]) & valid);
                }
                a.nl += __popc(lx) + __popc(ly) + __popc(lz);
                a.nw += __popc(wall);
            }
        }
        const R* vt = dphi + (int64_t)z0 * plane + (int64_t)y0 * g.nx + x0;
        // Eq. 8 at a wall site.  u = phi^2/phi0^2 - 1.  FP64 keeps the order of Eq. 1; FP32 factors it as
        // (phi - phi0)(phi + phi0)/phi0^2, equal in exact arithmetic and free of the cancellation
        // of phi^2 - 1 next to the vacua.
        auto energy = [&](unsigned e) {
            const int r = (int)(e >> 7), x = (int)((e & 31u) << 2 | (e >> 5 & 3u));
            const int ry = r & (ty - 1), rz = r >> T.lty;
            const R p = tile[((D == 3 ? (rz + 1) * (ty + 2) : 0) + ry + 1) * kLd + kOff + x];
            const R v = vt[(D == 3 ? rz * plane : 0) + (int64_t)ry * g.nx + x];
            R u;
            if (sizeof(R) == 8)
                u = A::sub(A::mul(A::mul(p, p), rc.inv_phi0sq), (R)1);
            else
                u = A::mul(A::mul(A::sub(p, rc.phi0), A::add(p, rc.phi0)), rc.inv_phi0sq);
            if constexpr (FAST) {  // dphi^2 / V = (dphi/u)^2 / V0, 1/V0 applied once per tile
                const bool pos = rc.V0 > 0.0f && u != 0.0f;
                const float f = __fdividef(v, u);
                a.nv0 += pos ? 0 : 1;
                a.pr += pos ? f * f : 0.0f;
            } else {
                const R V = A::mul(A::mul(rc.V0, u), u);
                if (V > (R)0)
                    a.sr += (double)A::div(A::mul(v, v), V);
                else
                    a.nv0++;
            }
        };
        auto weight = [&](unsigned e, int d) {  // Eq. 7
            if constexpr (FAST)
                a.pw += weight_fast<D>(tile + e, d, sy, sz);
            else
                a.sw += (double)weight_ieee<R, D>(tile + e, d, sy, sz);
        };
        const int nx_ = __popc(lx), ny_ = __popc(ly), nz_ = __popc(lz), nw_ = __popc(wall);
        const int all = __reduce_add_sync(0xffffffffu, nx_ + ny_ + nz_ + nw_);
        if (all == 0) {
        } else if (all <= min(32 * per, 1000)) {
            // one list for the links of each axis and the wall sites: three prefix sums in one
            // word (each below 2^10) beside that of the wall sites, then four independent chains
            unsigned links = nx_ | ny_ << 10 | nz_ << 20, walls = nw_;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, links, o), u = __shfl_up_sync(0xffffffffu, walls, o);
                if (lane >= o) links += t, walls += u;
            }
            const unsigned tl = __shfl_sync(0xffffffffu, links, 31);
            const int t0 = tl & 1023u, t1 = t0 + (tl >> 10 & 1023u), t2 = t1 + (tl >> 20);
            unsigned short *px = list + (links & 1023u) - nx_, *py = list + t0 + (links >> 10 & 1023u) - ny_;
            unsigned short *pz = list + t1 + (links >> 20) - nz_, *pw = list + t2 + walls - nw_;
            while (wall) {  // a link's site is a wall site: the other words are empty first
                const int b = top_bit(wall);
                const unsigned m = 1u << b;
                const unsigned short at_b = (unsigned short)(at + 4 * b);
                *pw++ = (unsigned short)(wi << 5 | b);
                if (lx & m) *px++ = at_b;
                if (ly & m) *py++ = at_b;
                if (D == 3 && (lz & m)) *pz++ = at_b;
                wall ^= m;
            }
            __syncwarp();
            for (int i = lane; i < t2; i += 32) weight(list[i], i < t0 ? 0 : (i < t1 ? 1 : 2));
            for (int i = t2 + lane; i < all; i += 32) energy(list[i]);
            __syncwarp();
        } else {  // a list at a time
            auto compact = [&](unsigned m, auto entry) {
                int total, k = warp_prefix(__popc(m), lane, total);
                while (m) {
                    const int b = top_bit(m);
                    m ^= 1u << b;
                    list[k++] = (unsigned short)entry(b);
                }
                __syncwarp();
                return total;
            };
            for (int d = 0; d < D; ++d) {
                const int total = compact(d == 0 ? lx : (d == 1 ? ly : lz), [&](int b) { return at + 4 * b; });
                for (int i = lane; i < total; i += 32) weight(list[i], d);
                __syncwarp();
            }
            const int total = compact(wall, [&](int b) { return wi << 5 | b; });
            for (int i = lane; i < total; i += 32) energy(list[i]);
            __syncwarp();
        }
        if (FAST) {
            a.sw += (double)a.pw;
            a.sr += (double)a.pr * rscale;
            a.pw = a.pr = 0.0f;
        }
        if (__syncthreads_or(fin.bad())) {  // (the tile is done with) count the non-finite sites of this tile
            for (int i = tid; i < nrows * kMCols; i += kMThreads) {
                const int r = i / kMCols, x = i - r * kMCols, ry = r & (ty - 1), rz = r >> T.lty;
                if (ry >= hy || rz >= hz || x >= w) continue;
                const R p = tile[((D == 3 ? (rz + 1) * (ty + 2) : 0) + ry + 1) * kLd + kOff + x];
                const R v = dphi[(int64_t)(z0 + rz) * plane + (int64_t)(y0 + ry) * g.nx + x0 + x];
                a.nnf += isfinite(p) && isfinite(v) ? 0 : 1;
            }
            __syncthreads();
        }
    }
    __syncthreads();  // the tile's memory is free
    block_reduce_and_finish_at(DiagAcc{a.sw, a.sr, a.nl, a.nw, a.nv0, a.nnf}, runs.scr[run], blockIdx.x, gridDim.x,
                               reinterpret_cast<double2*>(tile));
}

// Resident CTAs: four by registers (three in 3D), fewer where shared memory holds fewer.
int ctas_per_sm(int dims, size_t elem, const MTiling& T)
{
    const int regs = dims == 2 ? 4 : 3;
    const int smem = (int)(228 * 1024 / (measure_smem(dims, elem, T) + 3 * 1024));
    return smem < regs ? smem : regs;
}

// The tiling with the least modelled time: waves of the resident CTAs, each a fixed latency plus
// its halo rows' staging and its rows' work (us, from 512^3, 2048^2 and 128^3 FP32; a wave that
// leaves SMs with fewer CTAs shares its SM less).  Large boxes take the largest tiles (1024^3:
// 8 x 8 rows), small ones give every SM a tile.
MTiling tiling(const Geo& g, size_t elem, int sms)
{
    MTiling best{};
    double best_cost = 1e300;
    const int ymax = g.dims == 3 ? 3 : (elem == 4 ? 6 : 5), zmax = g.dims == 3 ? (elem == 4 ? 3 : 2) : 0;
    for (int ly = ymax; ly >= 2; --ly)
        for (int lz = zmax; lz >= 0 && ly + lz >= 3; --lz) {  // whole rows to each of the eight warps
            MTiling T;
            T.lty = ly;
            T.ltz = lz;
            T.ntx = ((unsigned)g.nx + kMCols - 1) / kMCols;
            T.nty = ((unsigned)g.ny + (1u << ly) - 1) >> ly;
            T.ntiles = T.ntx * T.nty * (((unsigned)g.nz + (1u << lz) - 1) >> lz);
            const double tiles = (double)T.ntiles, slots = (double)ctas_per_sm(g.dims, elem, T) * sms;
            const double waves = ceil(tiles / slots);
            const double fill = waves > 1 ? 1.0 : (tiles > sms ? tiles / slots : 1.0 / 3.0);
            const double cost = waves * (3.0 + fill * (0.03 * halo_rows(g.dims, T) + 0.11 * (1 << (ly + lz))));
            if (cost < best_cost) best_cost = cost, best = T;
        }
    return best;
}

// phi as boxes of a tile with its halo (x from 16 bytes before the tile's first column); false
// when the driver refuses.
template <typename R>
bool phi_map(CUtensorMap* m, const R* phi, const Geo& g, const MTiling& T)
{
    const EncodeTiled f = tmap_encoder();
    if (!f) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
    const cuuint64_t strides[2] = {(cuuint64_t)g.nx * sizeof(R), (cuuint64_t)g.nx * g.ny * sizeof(R)};
    const cuuint32_t box[3] = {(cuuint32_t)MRow<R>::kLd, (1u << T.lty) + 2, g.dims == 3 ? (1u << T.ltz) + 2 : 1};
    const cuuint32_t es[3] = {1, 1, 1};
    return f(m, sizeof(R) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3,
             const_cast<R*>(phi), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename R, int D, bool FAST, int NR>
cudaError_t measure_t(const Geo& g, int nruns, const MeasureRun* q, unsigned int* err, cudaStream_t st)
{
    static std::atomic<unsigned long long> attr{0};
    const int sms = sm_count_current();
    // the tiling of a run alone: a tile's partial sums are FP32 (FAST), so the same tiles give the same
    // sums to FP64 rounding
    const MTiling T = tiling(g, sizeof(R), sms);
    const MTiling most{D == 3 ? 3 : 6, D == 3 ? 3 : 0, 0, 0, 0};
    cudaError_t e = smem_limit_once(attr, (const void*)k_measure<R, D, FAST, NR>,
                                    (int)(sizeof(R) == 4 ? measure_smem(D, 4, most) : 100 * 1024));
    if (e != cudaSuccess) return e;
    // the resident CTAs, shared by the runs; one partial slot each
    const int all = ctas_per_sm(D, sizeof(R), T) * sms / nruns;
    int grid = T.ntiles < (unsigned)all ? (int)T.ntiles : (all > 0 ? all : 1);
    if (grid > q[0].scr.max_blocks) grid = q[0].scr.max_blocks;
    MRuns<R, NR> runs;
    uintptr_t bits = 0;
    for (int r = 0; r < nruns; ++r) {
        const double* c = q[r].run_const;
        runs.phi[r] = (const R*)q[r].phi;
        runs.dphi[r] = (const R*)q[r].dphi;
        runs.rc[r] = RunConst<R>{(R)c[0], (R)c[1], (R)c[2], (R)c[3], (R)c[4], (R)c[5]};
        runs.scr[r] = q[r].scr;
        bits |= (uintptr_t)q[r].phi | (uintptr_t)q[r].dphi;
    }
    const bool vec = g.nx % MRow<R>::kOff == 0 && (bits & 15u) == 0;
    CUtensorMap map{};
    if (NR > 1 || !err || !vec || !phi_map(&map, (const R*)q[0].phi, g, T)) err = nullptr;
    return launch_chained(k_measure<R, D, FAST, NR>, dim3((unsigned)grid, (unsigned)nruns), kMThreads,
                          measure_smem(D, sizeof(R), T), st, map, runs, g, T, vec, err);
}

template <typename R, bool FAST, int NR>
cudaError_t measure_d(const Geo& g, int nruns, const MeasureRun* q, unsigned int* err, cudaStream_t st)
{
    return g.dims == 3 ? measure_t<R, 3, FAST, NR>(g, nruns, q, err, st)
                       : measure_t<R, 2, FAST, NR>(g, nruns, q, err, st);
}

}  // namespace

cudaError_t launch_measure(const Geo& g, int precision, bool fast, const MeasureRun& run, unsigned int* err,
                           cudaStream_t st)
{
    if (precision != PRS_FP32) return measure_d<double, false, 1>(g, 1, &run, err, st);
    return fast ? measure_d<float, true, 1>(g, 1, &run, err, st) : measure_d<float, false, 1>(g, 1, &run, err, st);
}

cudaError_t launch_measure_runs(const Geo& g, int nruns, const MeasureRun* runs, cudaStream_t st)
{
    if (nruns < 1 || nruns > kMeasureMaxRuns) return cudaErrorInvalidValue;
    return measure_d<float, true, kMeasureMaxRuns>(g, nruns, runs, nullptr, st);
}

}  // namespace prs
