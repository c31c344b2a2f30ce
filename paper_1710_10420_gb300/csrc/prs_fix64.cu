// prs_fix64.cu -- the FP64 leapfrog step (Eqs. 3-5, folded kick) with its force in 64-bit fixed point.
//
// What bounds the plain FP64 step: GB300 adds or multiplies two doubles a clock and SM, so its 11
// (2D: 9) double operations a site take 350 us at 256^3, where HBM would allow 79 us.  An SM issues 64
// integer instructions in the time of one double instruction of a warp.  So the force
//   A = g (sum of the 2D neighbours) + phi (k1 - k2 phi^2)
// is evaluated in integers, and only the kick c1 dphi + A and the drift phi + deta dphi' stay
// double operations (one fused multiply-add each).
//
// With S the power of two at or above phi0, a value |phi| < 2 S becomes the integer phi/S 2^59,
// whose neighbour sum is exact; high-half products evaluate k1 - k2 phi^2, and its product with phi and
// the neighbour term, whose constants are scaled alike (2^(60-ek) / S; ek: the exponent that bounds the
// constants), are added in 128 bits.  A is rounded to 2^(ek-61) S, then to double.  Products are whole or
// of magnitudes, so the step of a negated field is the negated step, bit for bit.
//
// The integers hold their precision absolutely, doubles relatively: a value of S/128 or more converts
// exactly, a smaller one to 2^-60 S.  So the integers serve a site only where it or one of its neighbours
// is at least S/16, larger where the neighbours' constant g is below 2^ek/32 (wide lattices, strong
// potentials; make_fix64): over random stencils whose largest value lies between that and twice that, with
// W0 from 1.2 to infinity and dx from 0.5 to 10, the force's rms error is 0.02 to 0.79 of the double form's,
// and at most 0.85 where one neighbour holds that value and all the others are 1e-6 of it.  A warp takes the
// integers where they serve all its sites and no value is at 2 S or beyond (blow-ups) or not finite; else
// it evaluates the double form.  So that this holds for fields of any size, each warp scales by an S of its
// own, S 2^-down: it is lowered when the three planes of an iteration hold no value of a quarter of it or
// more, and raised again when a plane needs it; the planes already held are then converted again.
//
// Measured (us a step of a network of walls ten sites wide; the double form): 256^3 194 (356), 512^3 1476
// (2805), 128^3 32 (52), 2048^2 44 (74), 128^2 3.4 (4.3: the launch).  Wide walls have more sites without a
// large neighbour: 40 sites wide, 256^3 takes 277.  Before the precision of small values was kept (128-bit
// sums, the vote): 161 at 256^3, 39 at 2048^2.  What sets the pace now: 250 warp instructions for 32 sites at
// 0.59 of the issue slots, with the 16 warps an SM that 128 registers leave.
//
// A warp owns 32 columns (30 outputs) of four rows, in 2D 32 or 64 columns (one or two a lane) of one row,
// and marches along z (2D: y): a value is converted once where it enters, its z neighbours wait in
// registers, x neighbours come by shuffle.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "prs_chain.h"
#include "prs_internal.h"
#include "prs_march2d.h"
#include "prs_ptx.cuh"
#include "prs_site.cuh"

namespace prs {

namespace {

typedef long long i64;
typedef unsigned long long u64;

constexpr int kFxThreads = 128, kFxWarps = kFxThreads / 32;
// By dimensions and columns a lane (3D: 1): output columns of a warp, CTAs an SM (registers).
constexpr int fx_width(int cols) { return 32 * cols - 2; }
constexpr int fx_blocks(int dims, int cols) { return dims == 3 ? 4 : (cols == 1 ? 8 : 5); }

// The force's constants: k1, k2 S^2 and g scaled by 2^(62-ek), 2^(66-ek), 2^(65-ek); e_base: what a
// value's exponent field is subtracted from for its shift; e_out: exponent field of an A of 2^63; served:
// the shift of the smallest values that serve their site and its neighbours.
struct Fix64 {
    i64 k1;
    u64 k2, g;
    int e_base, e_out, served;
};

struct FixArgs {
    const double* phi_in;
    double* phi_out;
    const double* v_in;
    double* v_out;
    Fix64 f;
    KickD k;
    double deta;
    Geo g;
    int nstrips, ygroups, cz;
};

// phi/S 2^59, rounded (halves away from zero); shift is 3 for S <= |phi| < 2 S and below 3 for larger
// or non-finite values.
__device__ __forceinline__ i64 to_fixed(double d, int e_base, int& shift)
{
    const int hi = __double2hiint(d);
    const unsigned lo = (unsigned)__double2loint(d);
    shift = e_base - ((hi >> 20) & 0x7ff);
    const u64 m = ((u64)((hi & 0xfffff) | 0x100000) << 32 | lo) << 10;
    const u64 a = shift > 63 ? 0ull : ((m >> ((shift - 1) & 63)) + 1) >> 1;
    const i64 s = (i64)(hi >> 31);
    return (i64)(a ^ (u64)s) - s;
}

// a times sign (0 or -1): its negation where sign is -1.
__device__ __forceinline__ i64 with_sign(u64 a, i64 sign) { return (i64)(a ^ (u64)sign) - sign; }

// A of one site: c its value, s2 the sum of its neighbours.
// k2, e_out: f's for the warp's scale.
__device__ __forceinline__ double force(i64 c, i64 s2, const Fix64& f, u64 k2, int e_out)
{
    const i64 x = c << 3;                                       // x 2^62
    const u64 b = (u64)with_sign((u64)x, x >> 63);
    const u64 t = __umul64hi(b, b);                             // x^2 2^60
    const i64 k = f.k1 - (i64)__umul64hi(t, k2);                // (k1 - k2 phi^2) 2^(62-ek)
    const __int128 a = (__int128)x * k + (__int128)s2 * (i64)f.g;  // A 2^(124-ek), below 2^126
    const i64 sa = (i64)(a >> 64) >> 63;
    const unsigned __int128 w = (unsigned __int128)(sa ? -a : a);
    const u64 m = ((u64)(w >> 62) + 1) >> 1;                    // |A| 2^(61-ek)
    const int lz = __clzll((i64)m);
    const u64 n = m << (lz & 63);
    // 53 bits and the next as rounding, added onto the exponent: a carry bumps it
    const u64 bits = (n >> 11) + ((n >> 10) & 1ull) + ((u64)(unsigned)(e_out - lz - 2) << 52);
    return m ? __longlong_as_double((i64)(bits | ((u64)sa & 0x8000000000000000ull))) : 0.0;
}

template <int D, int C>
__global__ void __launch_bounds__(kFxThreads, fx_blocks(D, C)) k_step_fix64(const __grid_constant__ FixArgs a)
{
    // a lane's outputs (3D: rows, 2D: columns) and values, their halo, outputs of a warp across x
    constexpr int R = D == 3 ? 4 : C, N = D == 3 ? R + 2 : R, H = D == 3 ? 1 : 0, U = fx_width(C);
    chain_enter();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nx = a.g.nx, ny = D == 3 ? a.g.ny : 1, nz = D == 3 ? a.g.nz : a.g.ny;
    int x0, y0, z0;
    if (D == 3) {
        int b = blockIdx.x;
        x0 = b % a.nstrips * U;
        b /= a.nstrips;
        y0 = (b % a.ygroups * kFxWarps + wid) * R;
        z0 = b / a.ygroups * a.cz;
        if (y0 >= ny) return;
    } else {
        const int w = blockIdx.x * kFxWarps + wid;
        x0 = w % a.nstrips * U;
        y0 = 0;
        z0 = w / a.nstrips * a.cz;
        if (z0 >= nz) return;
    }
    const int planes = min(a.cz, nz - z0), rows = D == 3 ? min(R, ny - y0) : R;
    int x = (x0 - 1 + C * lane) % nx;
    if (x < 0) x += nx;
    const int first = C * lane - 1, last = min(U, nx - x0);  // the lane's first column of the strip's 0 .. last-1
    unsigned row[N];  // element offsets of the lane's values in a plane, periodic
#pragma unroll
    for (int r = 0; r < N; ++r) {
        if (D == 2) {
            row[r] = (unsigned)(x + r >= nx ? x + r - nx : x + r);
            continue;
        }
        int y = (y0 - H + r) % ny;
        if (y < 0) y += ny;
        row[r] = (unsigned)y * (unsigned)nx + (unsigned)x;
    }
    const int64_t plane = (int64_t)nx * ny;
    int z = z0 == 0 ? nz - 1 : z0 - 1;
    const double* pin = a.phi_in + (int64_t)z * plane;
    const double* vin = a.v_in + (int64_t)z0 * plane;
    double* pout = a.phi_out + (int64_t)z0 * plane;
    double* vout = a.v_out + (int64_t)z0 * plane;
    double next[N], vnext[R];  // the plane on its way
    auto fetch = [&] {
#pragma unroll
        for (int r = 0; r < N; ++r) next[r] = pin[row[r]];
        ++z;
        pin += z == nz ? plane * (1 - (int64_t)nz) : plane;
        if (z == nz) z = 0;
    };
    // planes z-1 (output rows), z, z+1 as integers, the values of planes z-1 (2D) and z, the planes' smallest shifts
    i64 m[R], c[N], p[N];
    double dm[R], d[R], v[R];
    int sm = 4096, sc = 4096, sp, down = 0;
    // bit r: output r; value r of planes z-1 and z serves its site; one of plane z next to value r or it does
    unsigned outputs = 0, bm = 0, bc = 0, wc = 0;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (first + (D == 2 ? r : 0) >= 0 && first + (D == 2 ? r : 0) < last && r < rows) outputs |= 1u << (r + H);
    const int most = a.f.e_out - 192;  // exponents of A stay in range
    u64 k2 = a.f.k2;
    fetch();
#pragma unroll
    for (int r = 0; r < R; ++r) m[r] = 0, vnext[r] = dm[r] = d[r] = 0.0;
#pragma unroll
    for (int r = 0; r < N; ++r) c[r] = 0;
    // Plane z0 + i arrives, plane z0 + i - 1 is updated.  A warp that changes its scale goes back to the
    // planes it holds (those before `live` have been updated).
    for (int i = -1, live = -1; i <= planes; ++i) {
        sp = 4096;
        double dn[R];
        unsigned bp = 0;  // bit r: value r serves its site and its neighbours
#pragma unroll
        for (int r = 0; r < N; ++r) {
            int s;
            p[r] = to_fixed(next[r], a.f.e_base - down, s);
            if (s <= a.f.served) bp |= 1u << r;
            sp = min(sp, s);
            if (r >= H && r < R + H) dn[r - H] = next[r];
        }
        const bool served = __all_sync(0xffffffffu, ((wc | bm | bp) & outputs) == outputs);
        sp = __reduce_min_sync(0xffffffffu, sp);
        const int least = min(min(sm, sc), sp);  // the shift of the largest value
        if ((least < 3 || least > 5) && least < 1100 && i >= live) {
            const int by = max(min(least - 3, most - down), -down);
            if (by != 0) {  // (planes of zeros lower the scale to its limit)
                down += by;
                k2 = down > 31 ? 0ull : a.f.k2 >> 2 * down;
                sm = sc = 4096;
                live = i;
                i = i < 1 ? -1 : i - 2;
                z = z0 + i < 0 ? nz - 1 : z0 + i;
                pin = a.phi_in + (int64_t)z * plane;
                fetch();
                --i;
                continue;
            }
        }
        if (i < planes) fetch();
        if (i >= live) {
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = vnext[r];
            if (i >= 0 && i < planes) {
#pragma unroll
                for (int r = 0; r < R; ++r) vnext[r] = r < rows ? vin[row[r + H]] : 0.0;
                vin += plane;
            }
        }
        if (i >= 1 && i >= live) {
            const bool fixed = min(min(sm, sc), sp) >= 3 && served;
            double pn[R];
            if (fixed) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const i64 cc = c[r + H];
                    const i64 left =
                        D == 2 && r > 0 ? c[r - 1] : __shfl_up_sync(0xffffffffu, c[D == 2 ? R - 1 : r + H], 1);
                    const i64 right =
                        D == 2 && r < R - 1 ? c[r + 1] : __shfl_down_sync(0xffffffffu, c[D == 2 ? 0 : r + H], 1);
                    i64 s2 = (left + right) + (m[r] + p[r + H]);
                    if (D == 3) s2 += c[r] + c[r + 2 * H];
                    v[r] = fma(a.k.c1, v[r], force(cc, s2, a.f, k2, a.f.e_out - down));
                    pn[r] = fma(a.deta, v[r], d[r]);
                }
            } else if (D == 2) {  // the double form, from registers
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const double left = r > 0 ? d[r - 1] : __shfl_up_sync(0xffffffffu, d[R - 1], 1);
                    const double right = r < R - 1 ? d[r + 1] : __shfl_down_sync(0xffffffffu, d[0], 1);
                    site_update_folded<D>(d[r], right, left, dn[r], dm[r], 0.0, 0.0, v[r], pn[r], a.k, a.deta);
                }
            } else {  // from memory: the planes' doubles take more registers than four blocks an SM leave
                const int zc = z0 + i - 1, zm = zc == 0 ? nz - 1 : zc - 1, zp = zc + 1 == nz ? 0 : zc + 1;
                const double* q = a.phi_in + (int64_t)zc * plane;
                const double* qp = a.phi_in + (int64_t)zp * plane;
                const double* qm = a.phi_in + (int64_t)zm * plane;
#pragma unroll 1
                for (int r = 0; r < rows; ++r) {
                    const int y = y0 + r;
                    const int64_t o = (int64_t)y * nx + x, up = (int64_t)(y + 1 == ny ? 0 : y + 1) * nx + x;
                    const int64_t dn2 = (int64_t)(y == 0 ? ny - 1 : y - 1) * nx + x, row0 = o - x;
                    const double xp = q[row0 + (x + 1 == nx ? 0 : x + 1)], xm = q[row0 + (x == 0 ? nx - 1 : x - 1)];
                    const double cc = q[o], yp = q[up], ym = q[dn2], zpv = qp[o], zmv = qm[o];
                    double vv, pp;
#pragma unroll
                    for (int u = 0; u < R; ++u) vv = u == r ? v[u] : vv;
                    site_update_folded<D>(cc, xp, xm, yp, ym, zpv, zmv, vv, pp, a.k, a.deta);
#pragma unroll
                    for (int u = 0; u < R; ++u)
                        if (u == r) v[u] = vv, pn[u] = pp;
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (outputs >> (r + H) & 1u) {
                    pout[row[r + H]] = pn[r];
                    vout[row[r + H]] = v[r];
                }
            pout += plane;
            vout += plane;
        }
        sm = sc, sc = sp;
        const unsigned bl = __shfl_up_sync(0xffffffffu, bp, 1), br = __shfl_down_sync(0xffffffffu, bp, 1);
        wc = bp | bp << 1 | bp >> 1 | (D == 3 ? bl | br : bl >> (R - 1) | br << (R - 1));
        bm = bc, bc = bp;
#pragma unroll
        for (int r = 0; r < R; ++r) m[r] = c[r + H], dm[r] = d[r], d[r] = dn[r];
#pragma unroll
        for (int r = 0; r < N; ++r) c[r] = p[r];
    }
}

}  // namespace

// The constants of a step, or false where they do not fit or no integers would serve (the double form
// everywhere then).
static bool make_fix64(const KickD& k, const double coef[3], const double run_const[6], Fix64* f)
{
    const double phi0 = run_const[5];
    int es;  // S = 2^es >= phi0
    const double fr = frexp(phi0, &es);
    if (fr == 0.5) --es;
    const double k2s = ldexp(k.k2, 2 * es);
    const double bound = fabs(k.k1) + 8.0 * fabs(k2s) + 4.0 * fabs(k.g);
    if (!(bound > 0) || !isfinite(bound) || k2s < 0 || !(k.g > 0)) return false;
    int ek;
    frexp(bound, &ek);  // bound < 2^ek
    if (ek < -400 || ek > 400 || es < -400 || es > 400) return false;
    // k1 = c2 cV - 2D c2/dx^2 from its unrounded parts: as a double it is off by up to 2^-55 (at sides of one),
    // which every step would repeat, and which a 63-bit constant need not carry
    const double h = coef[1] * coef[2], h_lo = fma(coef[1], coef[2], -h), g_lo = fma(coef[1], run_const[1], -k.g);
    const auto fixed = [&](double x) { return (i64)llrint(ldexp(x, 62 - ek)); };
    f->k1 = fixed(h) + fixed(h_lo) - (i64)run_const[3] * (fixed(k.g) + fixed(g_lo));
    f->k2 = (u64)llrint(ldexp(k2s, 65 - ek)) << 1;
    f->g = (u64)llrint(ldexp(k.g, 65 - ek));
    f->e_base = 1026 + es;
    f->e_out = 1023 + 63 + ek - 60 + es;
    f->served = 7;
    for (double least = ldexp(1.0, ek - 5); k.g < least && f->served > 2; least *= 0.5) --f->served;
    return f->served > 2;
}

// Columns a lane owns and planes (2D: rows) a warp marches.
MarchShape fix64_shape(const Geo& g)
{
    // 2D: two columns a lane share a row's bookkeeping, one makes twice the warps (us a step, two and one:
    // 256^2 4.0 3.4, 400^2 4.6 4.3, 512^2 5.2 5.5, 1024^2 11.9 13.2, 2048^2 39 44)
    const int cols = g.dims == 3 || g.S < ((int64_t)1 << 18) ? 1 : 2, width = fx_width(cols);
    const int nstrips = (g.nx + width - 1) / width, len = g.dims == 3 ? g.nz : g.ny;
    const int ygroups = g.dims == 3 ? (g.ny + 4 * kFxWarps - 1) / (4 * kFxWarps) : 1;
    // warps (2D) or blocks of them (3D) against the two planes a chunk re-reads and the iteration
    // that fills it
    const double tiles = (double)nstrips * ygroups / (g.dims == 3 ? 1 : kFxWarps);
    const double slots = (double)fx_blocks(g.dims, cols) * sm_count_current();
    double least = 1e300;
    MarchShape best{cols, len};
    for (int nc = 1; nc <= len && nc <= 4096; nc += nc < 32 ? 1 : nc / 16) {
        const int c = (len + nc - 1) / nc, n = (len + c - 1) / c;
        const double w = tiles * n / slots;
        const double cost = (w <= 1.0 ? 0.7 + 0.3 * w : 0.5 * (ceil(w) + w + 0.35)) * (c + 2.0);
        if (cost < least * 0.999) least = cost, best.cy = c;
    }
    return best;
}

cudaError_t launch_step_fix64(const Geo& g, const double* in, double* out, const double* v, double* v_out,
                              const double coef[3], const double run_const[6], const MarchShape& shape,
                              cudaStream_t st)
{
    const KickD k = kick_f64(coef, run_const);
    FixArgs a;
    if (!make_fix64(k, coef, run_const, &a.f)) return cudaErrorNotSupported;
    // boxes of a few rows leave most of a block's warps without any (us a step, the integers and the double
    // form: 2000 x 3 x 2000 316 and 280, 2000 x 5 x 2000 533 and 468, 2000 x 8 x 1000
    // 292 and 375)
    if (g.dims == 3 && g.ny < 6) return cudaErrorNotSupported;
    if (g.dims == 3 && (int64_t)g.nx * g.ny >= ((int64_t)1 << 32)) return cudaErrorNotSupported;
    a.phi_in = in;
    a.phi_out = out;
    a.v_in = v;
    a.v_out = v_out;
    a.k = k;
    a.deta = run_const[0];
    a.g = g;
    a.nstrips = (g.nx + fx_width(shape.cols) - 1) / fx_width(shape.cols);
    a.ygroups = g.dims == 3 ? (g.ny + 4 * kFxWarps - 1) / (4 * kFxWarps) : 1;
    a.cz = shape.cy;
    const int64_t n = ((g.dims == 3 ? g.nz : g.ny) + a.cz - 1) / a.cz;
    const int64_t blocks = g.dims == 3 ? (int64_t)a.nstrips * a.ygroups * n
                                       : ((int64_t)a.nstrips * n + kFxWarps - 1) / kFxWarps;
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    void (*const flat)(const FixArgs) = shape.cols == 1 ? k_step_fix64<2, 1> : k_step_fix64<2, 2>;
    return launch_chained(g.dims == 3 ? k_step_fix64<3, 1> : flat, dim3((unsigned)blocks), kFxThreads, 0, st, a);
}

}  // namespace prs
