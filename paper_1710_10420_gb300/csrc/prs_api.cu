// prs_api.cu -- the C ABI of include/prs.h for single runs: parameter checks, the
// FP64 damping schedule (Eq. 6), buffer ownership, and the order of kernel launches.
// No exception crosses the ABI; every CUDA error becomes PRS_ECUDA.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>
#include <new>

#include "prs.h"
#include "prs_internal.h"
#include "prs_march3d.h"
#include "prs_sim.h"

using namespace prs;



// ------------------------------------------------------------------ errors

static thread_local char g_last_error[256] = "";

int prs::cuda_fail(cudaError_t e, const char* what)
{
    snprintf(g_last_error, sizeof g_last_error, "%s: %s", what, cudaGetErrorString(e));
    return PRS_ECUDA;
}

#define PRS_CUDA(call)                                     \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

extern "C" const char* prs_strerror(int status)
{
    switch (status) {
        case PRS_OK: return "ok";
        case PRS_EINVAL: return "invalid argument";
        case PRS_ENOMEM: return "out of memory";
        case PRS_ECUDA: return "CUDA error";
        case PRS_ETIMEOUT: return "device wait timed out";
        case PRS_ENONFINITE: return "non-finite field value";
        case PRS_ESTATE: return "call out of order";
        default: return "unknown status";
    }
}

extern "C" const char* prs_last_error(void) { return g_last_error; }

namespace prs {
void record_error(const char* msg) { snprintf(g_last_error, sizeof g_last_error, "%s", msg); }
}  // namespace prs

// ------------------------------------------------------------- parameters

static const double kPi = 3.14159265358979323846;

static double potential_height(const prs_params& p) { return kPi * kPi / (2.0 * p.W0 * p.W0); }

// Eq. 6 and the force prefactor of Eq. 2 at step n, in FP64 on the host.
void prs::step_coefficients(const prs_params& p, int64_t n, double out[5])
{
    double eta = p.eta0 + (double)n * p.deta;  // computed from n, never accumulated
    double delta = 0.5 * p.alpha * p.deta * p.era_m / eta;
    double a_beta = 1.0;
    if (p.beta != 0.0) a_beta = pow(pow(eta, p.era_m), p.beta);  // a = eta^m, a(1) = 1
    out[0] = (1.0 - delta) / (1.0 + delta);
    out[1] = p.deta / (1.0 + delta);
    out[2] = 4.0 * potential_height(p) * a_beta / (p.phi0 * p.phi0);
    out[3] = delta;
    out[4] = 0.5 * p.deta * p.era_m / eta;
}

// Leapfrog stability of Eqs. 3-5 at step n: deta^2 (4D/dx^2 + max|V''|)/4 < 1,
// with max|V''| = 2 cV over |phi| <= phi0.
bool prs::cfl_ok(const prs_params& p, int64_t n)
{
    double c[5];
    step_coefficients(p, n, c);
    double lam = 4.0 * p.dims / (p.dx * p.dx) + 2.0 * c[2] * p.phi0 * p.phi0;
    return p.deta * p.deta * lam < 4.0;
}

static int check_params(const prs_params* pp, Geo* g)
{
    if (!pp) return PRS_EINVAL;
    const prs_params& p = *pp;
    if (p.dims != 2 && p.dims != 3) return PRS_EINVAL;
    if (p.precision != PRS_FP32 && p.precision != PRS_FP64) return PRS_EINVAL;
    if ((p.flags & ~(PRS_REPRO | PRS_FP32_CR | PRS_DEBUG)) != 0) return PRS_EINVAL;
    int64_t nx = p.N, ny = p.Ny ? p.Ny : p.N, nz = p.dims == 3 ? (p.Nz ? p.Nz : p.N) : 1;
    if (nx < 3 || ny < 3 || (p.dims == 3 && nz < 3)) return PRS_EINVAL;
    if (nx > (1 << 30) || ny > (1 << 30) || nz > (1 << 30)) return PRS_EINVAL;
    if (!(p.dx > 0) || !(p.deta > 0) || !(p.eta0 > 0) || !(p.phi0 > 0) || !(p.W0 > 0)) return PRS_EINVAL;
    if (!isfinite(p.dx) || !isfinite(p.deta) || !isfinite(p.eta0) || !isfinite(p.phi0)) return PRS_EINVAL;
    if (!isfinite(p.alpha) || !isfinite(p.beta) || !isfinite(p.era_m)) return PRS_EINVAL;
    if (p.tblock < 0 || p.tblock > 8) return PRS_EINVAL;
    if (!cfl_ok(p, 0)) return PRS_EINVAL;
    // delta must stay below 1 or (1-delta)/(1+delta) flips the velocity's sign
    double c[5];
    step_coefficients(p, 0, c);
    if (!(c[3] < 1.0)) return PRS_EINVAL;
    g->dims = p.dims;
    g->nx = (int)nx;
    g->ny = (int)ny;
    g->nz = (int)nz;
    g->S = nx * ny * nz;
    return PRS_OK;
}

extern "C" int prs_coefficients(const prs_params* params, int64_t n, double out[5])
{
    if (!params || !out || n < 0) return PRS_EINVAL;
    step_coefficients(*params, n, out);
    return PRS_OK;
}

// Largest stable time step at conformal time eta: deta^2 (4D/dx^2 + 2 cV(eta) phi0^2) < 4.
extern "C" int prs_stable_deta(const prs_params* params, double eta, double* deta_max)
{
    if (!params || !deta_max || !(eta > 0) || !isfinite(eta)) return PRS_EINVAL;
    prs_params q = *params;
    q.eta0 = eta;  // step 0 of q is at eta
    double c[5];
    step_coefficients(q, 0, c);
    const double lam = 4.0 * q.dims / (q.dx * q.dx) + 2.0 * c[2] * q.phi0 * q.phi0;
    if (!(lam > 0) || !isfinite(lam)) return PRS_EINVAL;
    *deta_max = 2.0 / sqrt(lam);
    return PRS_OK;
}

extern "C" int prs_default_tblock(const prs_params* params)
{
    Geo g;
    int rc = check_params(params, &g);
    if (rc) return rc;
    int t = default_fused_steps(g, params->precision, (params->flags & PRS_REPRO) != 0);
    return t < 1 ? 1 : t;
}

extern "C" int prs_max_tblock(const prs_params* params)
{
    Geo g;
    int rc = check_params(params, &g);
    if (rc) return rc;
    int t = max_fused_steps(g, params->precision, (params->flags & PRS_REPRO) != 0);
    return t < 1 ? 1 : t;
}

// -------------------------------------------------------------- lifecycle

static const int kMeasureBlocks = 8192;  // partial slots: the fast kernels use one per tile

// FP32 runs step by the register marches (prs_march2d.cuh, prs_march3d.cuh; in 3D beside the staged
// passes); without a tblock their plan also sets the steps of the passes.  An FP64 run's plan is the shape of
// its one-step passes.  (Planned with every launch it took 1.5 us of 12 for a step of 64^2.)
static bool march_run(const prs_sim* s) { return s->p.precision == PRS_FP32; }
static bool march_plans(const prs_sim* s) { return march_run(s) && s->p.tblock == 0; }
static void make_plan(prs_sim* s, int nruns)
{
    if (s->march.nruns == nruns) return;
    if (!march_run(s)) s->march.nruns = nruns, s->march.shape[1] = fix64_shape(s->g);
    else if (s->g.dims == 2) march_plan(s->g, nruns, &s->march);
    else march_plan_3d(s->g, nruns, &s->march);
}

// Device memory that bound runs of small boxes gave back, for the next such run: from the driver 10 MB take 90 us
// to get and 60 to return, beside a first interval of 190 us at 128^3.  At most kKeptBytes of it while any
// run exists, none afterwards.  (A pool of the driver's serves as fast but takes 2.2 ms to make.)  A piece
// comes here when the stream of its run has passed all its work, and no caller ever held its address.
static const size_t kKeptBytes = (size_t)64 << 20, kKeptMost = (size_t)32 << 20;
struct Kept {
    void* p;
    size_t bytes;
    int dev;
};
static std::mutex g_kept_mutex;  // of the three below
static Kept g_kept[16];
static size_t g_kept_bytes;
static int g_runs;  // runs that exist

static int current_device()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
    return dev;
}

// A kept piece of at least `bytes` and not much more on device dev, and its size; or null.
static void* take_kept(size_t bytes, int dev, size_t* size)
{
    std::lock_guard<std::mutex> lock(g_kept_mutex);
    Kept* best = nullptr;
    for (Kept& k : g_kept)
        if (k.p && k.dev == dev && k.bytes >= bytes && k.bytes / 2 <= bytes && (!best || k.bytes < best->bytes))
            best = &k;
    if (!best) return nullptr;
    void* p = best->p;
    *size = best->bytes;
    g_kept_bytes -= best->bytes;
    *best = Kept{};
    return p;
}

// A run comes (1) or goes (-1), its bound device memory on device dev with it (or null).
static void count_run(int change, void* mem = nullptr, size_t bytes = 0, int dev = -1)
{
    std::lock_guard<std::mutex> lock(g_kept_mutex);
    g_runs += change;
    if (g_runs > 0 && mem && bytes <= kKeptMost && g_kept_bytes + bytes <= kKeptBytes)
        for (Kept& k : g_kept)
            if (!k.p) {
                k = Kept{mem, bytes, dev};
                g_kept_bytes += bytes;
                return;
            }
    cudaFree(mem);
    for (Kept& k : g_kept)
        if (g_runs == 0 && k.p) cudaFree(k.p), k = Kept{};
    if (g_runs == 0) g_kept_bytes = 0;
}

extern "C" int prs_create(const prs_params* params, void* stream, prs_sim** out)
{
    if (!out) return PRS_EINVAL;
    Geo g;
    int rc = check_params(params, &g);
    if (rc) return rc;
    prs_sim* s = new (std::nothrow) prs_sim();
    if (!s) return PRS_ENOMEM;
    s->p = *params;
    s->g = g;
    s->elem = params->precision == PRS_FP32 ? sizeof(float) : sizeof(double);
    s->stream = (cudaStream_t)stream;
    s->rc[0] = params->deta;
    s->rc[1] = 1.0 / (params->dx * params->dx);
    s->rc[2] = 1.0 / (params->phi0 * params->phi0);
    s->rc[3] = (double)(2 * params->dims);
    s->rc[4] = potential_height(*params);
    s->rc[5] = params->phi0;
    s->scr.max_blocks = kMeasureBlocks;
    make_plan(s, 1);
    if (cudaMallocHost((void**)&s->h_status, sizeof(DevStatus)) != cudaSuccess ||
        ((params->flags & PRS_DEBUG) && cudaMalloc((void**)&s->d_dbg, sizeof(DebugCheck)) != cudaSuccess)) {
        int r = cuda_fail(cudaGetLastError(), "prs_create");
        cudaFreeHost(s->h_status);
        delete s;
        return r;
    }
    count_run(1);
    *out = s;
    return PRS_OK;
}

// Steps per pass this run takes (params.tblock, or the library's choice, clamped).
static int run_tblock(const prs_sim* s)
{
    const bool repro = (s->p.flags & PRS_REPRO) != 0;
    int tmax = max_fused_steps(s->g, s->p.precision, repro);
    int tb = s->p.tblock > 0 ? s->p.tblock : default_fused_steps(s->g, s->p.precision, repro);
    if (tb > tmax) tb = tmax;
    return tb < 1 ? 1 : tb;
}

// Whether the run takes passes of several steps, which need a second dphi buffer.
static bool wants_alt(const prs_sim* s) { return run_tblock(s) >= 2 || march_plans(s); }

// stream: the run's, or null while it is captured.
static int alloc_run_on(prs_sim* s, int fields, const cudaStream_t* stream)
{
    const size_t fs = ((size_t)s->g.S * s->elem + 511) & ~(size_t)511;
    const size_t scratch = sizeof(DiagAcc) * kMeasureBlocks + sizeof(DevStatus);
    bool alt = wants_alt(s);
    size_t bytes = fs * (size_t)(fields + (alt ? 1 : 0)) + scratch, size = 0;
    const int dev = current_device();
    void* m = fields ? nullptr : take_kept(bytes, dev, &size);
    if (!m && cudaMalloc(&m, bytes) != cudaSuccess) {
        cudaGetLastError();
        if (!alt) return PRS_ENOMEM;
        alt = false;
        bytes = fs * (size_t)fields + scratch;
        if (cudaMalloc(&m, bytes) != cudaSuccess) {
            cudaGetLastError();
            return PRS_ENOMEM;
        }
    }
    char* c = (char*)m + fs * (size_t)(fields + (alt ? 1 : 0));
    cudaError_t e = cudaMemsetAsync(c, 0, scratch, stream ? *stream : cudaStreamPerThread);
    if (e == cudaSuccess && !stream) e = cudaStreamSynchronize(cudaStreamPerThread);
    if (e != cudaSuccess) {
        cudaFree(m);
        return cuda_fail(e, "scratch of the diagnostics");
    }
    s->mem = m;
    s->mem_bytes = size ? size : bytes;
    s->mem_dev = dev;
    s->scr.partials = (DiagAcc*)c;
    s->d_status = (DevStatus*)(s->scr.partials + kMeasureBlocks);
    s->scr.result = &s->d_status->result;
    s->scr.counter = &s->d_status->counter;
    if (alt) s->dphi_alt = (char*)m + fs * (size_t)fields;
    if (fields) {
        s->phi[0] = m;
        s->phi[1] = (char*)m + fs;
        s->dphi = (char*)m + 2 * fs;
    }
    return PRS_OK;
}

// One allocation of `fields` fields, the second dphi buffer and the diagnostics' scratch; without the
// buffer where it does not fit.  (Beyond 2 MB an allocation takes 30 to 100 us, and as long to free: a run of
// 128^3 with its own fields 493 us from creation to release, with an allocation each 812; bound 498 and 630.)
// Neither it nor the scratch's first contents become part of a graph that the run's stream is captured into.
static int alloc_run(prs_sim* s, int fields)
{
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s->stream, &status) != cudaSuccess) cudaGetLastError();
    const bool capturing = status != cudaStreamCaptureStatusNone;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (capturing) cudaThreadExchangeStreamCaptureMode(&mode);
    const int rc = alloc_run_on(s, fields, capturing ? nullptr : &s->stream);
    if (capturing) cudaThreadExchangeStreamCaptureMode(&mode);
    return rc;
}

extern "C" int prs_bind(prs_sim* s, void* d_phi_a, void* d_phi_b, void* d_dphi)
{
    if (!s || !d_phi_a || !d_phi_b || !d_dphi || d_phi_a == d_phi_b) return PRS_EINVAL;
    if (((uintptr_t)d_phi_a | (uintptr_t)d_phi_b | (uintptr_t)d_dphi) & 15u) return PRS_EINVAL;
    if (s->have_buffers) return PRS_ESTATE;
    const int rc = alloc_run(s, 0);
    if (rc) return rc;
    s->phi[0] = d_phi_a;
    s->phi[1] = d_phi_b;
    s->dphi = d_dphi;
    s->cur = 0;
    s->owned = false;
    s->have_buffers = true;
    return PRS_OK;
}

int prs::ensure_buffers(prs_sim* s)
{
    if (s->have_buffers) return PRS_OK;
    if (s->p.flags & PRS_DEBUG) {
        const size_t bytes = (size_t)s->g.S * s->elem;
        void* f[3] = {nullptr, nullptr, nullptr};
        int rc = PRS_OK;
        for (int i = 0; i < 3 && !rc; ++i) rc = debug_alloc_field(bytes, &s->guard_base[i], &f[i]);
        if (!rc) rc = alloc_run(s, 0);
        if (rc) {
            for (int k = 0; k < 3; ++k) cudaFree(s->guard_base[k]), s->guard_base[k] = nullptr;
            return rc;
        }
        s->phi[0] = f[0];
        s->phi[1] = f[1];
        s->dphi = f[2];
    } else {
        const int rc = alloc_run(s, 3);
        if (rc) return rc;
    }
    s->cur = 0;
    s->owned = true;
    s->have_buffers = true;
    return PRS_OK;
}

extern "C" int prs_destroy(prs_sim* s)
{
    if (!s) return PRS_EINVAL;
    cudaStreamSynchronize(s->stream);
    for (int i = 0; i < 3; ++i) cudaFree(s->guard_base[i]);
    cudaFree(s->alt_mem);
    cudaFree(s->d_dbg);
    cudaFree(s->adj_ws);
    for (cudaEvent_t e : s->adj_ev) cudaEventDestroy(e);
    cudaFreeHost(s->h_status);
    if (s->owned) cudaFree(s->mem), s->mem = nullptr;
    count_run(-1, s->mem, s->mem_bytes, s->mem_dev);
    delete s;
    return PRS_OK;
}

// ------------------------------------------------------------------ state

// The second dphi buffer where it did not fit beside the fields, tried again with every new state, so that
// prs_step itself never allocates; while there is no room the run steps one step per pass.
static void ensure_dphi_alt(prs_sim* s)
{
    if (s->dphi_alt || !wants_alt(s)) return;
    if (cudaMalloc(&s->alt_mem, (size_t)s->g.S * s->elem) != cudaSuccess) {
        cudaGetLastError();
        s->alt_mem = nullptr;
    }
    s->dphi_alt = s->alt_mem;
}

static int prs_init_impl(prs_sim* s, const void* h_phi, const void* h_dphi)
{
    if (!s) return PRS_EINVAL;
    int rc = ensure_buffers(s);
    if (rc) return rc;
    size_t bytes = (size_t)s->g.S * s->elem;
    s->cur = 0;
    if (h_phi) {
        PRS_CUDA(cudaMemcpyAsync(s->phi[0], h_phi, bytes, cudaMemcpyHostToDevice, s->stream));
        if (h_dphi)
            PRS_CUDA(cudaMemcpyAsync(s->dphi, h_dphi, bytes, cudaMemcpyHostToDevice, s->stream));
        else
            PRS_CUDA(cudaMemsetAsync(s->dphi, 0, bytes, s->stream));
    } else {
        PRS_CUDA(launch_init_random(s->g, s->p.precision, s->p.seed, s->phi[0], s->dphi, h_dphi == nullptr,
                                    s->stream));
        if (h_dphi) PRS_CUDA(cudaMemcpyAsync(s->dphi, h_dphi, bytes, cudaMemcpyHostToDevice, s->stream));
    }
    // host arrays may be pageable and reused by the caller right after return
    PRS_CUDA(cudaStreamSynchronize(s->stream));
    ensure_dphi_alt(s);
    s->n = 0;
    s->initialised = true;
    return PRS_OK;
}

static int set_state_queued(prs_sim* s, const void* h_phi, const void* h_dphi, int64_t n, bool wait)
{
    if (!s || !h_phi || !h_dphi || n < 0) return PRS_EINVAL;
    int rc = ensure_buffers(s);
    if (rc) return rc;
    size_t bytes = (size_t)s->g.S * s->elem;
    PRS_CUDA(cudaMemcpyAsync(s->phi[s->cur], h_phi, bytes, cudaMemcpyHostToDevice, s->stream));
    PRS_CUDA(cudaMemcpyAsync(s->dphi, h_dphi, bytes, cudaMemcpyHostToDevice, s->stream));
    if (wait) PRS_CUDA(cudaStreamSynchronize(s->stream));
    ensure_dphi_alt(s);
    s->n = n;
    s->initialised = true;
    return PRS_OK;
}

static int prs_set_state_impl(prs_sim* s, const void* h_phi, const void* h_dphi, int64_t n)
{
    return set_state_queued(s, h_phi, h_dphi, n, true);
}

extern "C" int prs_set_state_async(prs_sim* s, const void* h_phi, const void* h_dphi, int64_t n)
{
    return debug_after(s, set_state_queued(s, h_phi, h_dphi, n, false), "prs_set_state_async", true);
}

static int set_state_device(prs_sim* s, const void* d_phi, const void* d_dphi, int64_t n)
{
    if (!s || !d_phi || !d_dphi || n < 0) return PRS_EINVAL;
    int rc = ensure_buffers(s);
    if (rc) return rc;
    size_t bytes = (size_t)s->g.S * s->elem;
    PRS_CUDA(launch_copy_state(d_phi, s->phi[s->cur], d_dphi, s->dphi, bytes, s->stream));
    ensure_dphi_alt(s);
    s->n = n;
    s->initialised = true;
    return PRS_OK;
}

extern "C" int prs_set_state_device(prs_sim* s, const void* d_phi, const void* d_dphi, int64_t n)
{
    return debug_after(s, set_state_device(s, d_phi, d_dphi, n), "prs_set_state_device", true);
}

extern "C" int prs_get_state(prs_sim* s, void* h_phi, void* h_dphi, int64_t* n)
{
    if (!s) return PRS_EINVAL;
    if (!s->initialised) return PRS_ESTATE;
    size_t bytes = (size_t)s->g.S * s->elem;
    if (h_phi) PRS_CUDA(cudaMemcpyAsync(h_phi, s->phi[s->cur], bytes, cudaMemcpyDeviceToHost, s->stream));
    if (h_dphi) PRS_CUDA(cudaMemcpyAsync(h_dphi, s->dphi, bytes, cudaMemcpyDeviceToHost, s->stream));
    PRS_CUDA(cudaStreamSynchronize(s->stream));
    if (n) *n = s->n;
    return PRS_OK;
}

extern "C" int prs_device_state(prs_sim* s, void** d_phi, void** d_dphi, int64_t* n)
{
    if (!s) return PRS_EINVAL;
    if (!s->initialised) return PRS_ESTATE;
    if (d_phi) *d_phi = s->phi[s->cur];
    if (d_dphi) *d_dphi = s->dphi;
    if (n) *n = s->n;
    return PRS_OK;
}

// From the next step on, steps of size deta: eta continues from the current time,
// eta_m = eta_n + (m - n) deta for the current step n (eta0 is re-based to eta_n - n deta).
static int set_deta(prs_sim* s, double deta)
{
    if (!s || !(deta > 0) || !isfinite(deta)) return PRS_EINVAL;
    prs_params q = s->p;
    const double eta_n = s->p.eta0 + (double)s->n * s->p.deta;
    q.eta0 = eta_n - (double)s->n * deta;
    q.deta = deta;
    double c[5];
    step_coefficients(q, s->n, c);
    if (!cfl_ok(q, s->n) || !(c[3] < 1.0)) return PRS_EINVAL;
    s->p = q;
    s->rc[0] = deta;
    return PRS_OK;
}

extern "C" int prs_set_deta(prs_sim* s, double deta) { return set_deta(s, deta); }

// ------------------------------------------------------ launcher setup

int prs::sm_count_current()
{
    static std::atomic<int> cache[64];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 152;
    }
    if (dev >= 0 && dev < 64 && (n = cache[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        return 152;
    }
    if (dev >= 0 && dev < 64) cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

cudaError_t prs::smem_limit_once(std::atomic<unsigned long long>& done, const void* func, int bytes)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = (dev >= 0 && dev < 64) ? 1ull << dev : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// ------------------------------------------------------------------- step

bool prs::cfl_ok_over(const prs_params& p, int64_t n, int64_t nsteps)
{
    return cfl_ok(p, n) && cfl_ok(p, n + nsteps - 1);
}

// The passes of a call of nsteps (>= 1): cnt[t] of t steps, the longest first.
static void step_plan(const prs_sim* s, const MarchPlan* march, int64_t nsteps, int64_t cnt[kMarchMaxT + 1])
{
    const int tb = run_tblock(s);
    // Multi-step passes read dphi across sites, so they write it to a second buffer.  A call runs its
    // passes the longest first, single steps last: FP32 without a tblock what march_counts plans; else
    // with T = tblock = 3, nsteps / 3 triples and a pair or a single step for the remainder; with T = 2,
    // pairs, and for an odd count a single step.  After an odd number of multi-step passes dphi sits in the
    // second buffer.  A run whose buffers the library owns (no PRS_DEBUG guard bands) then swaps the
    // roles of its two dphi buffers.  A run with bound buffers keeps dphi in the bound buffer at the end
    // of every call: the first single step after an odd number of multi-step passes reads dphi in the
    // second buffer and writes the bound one; with no single step to do it, the last pair runs as two
    // single steps, else the last triple as a pair and a single step.  Single steps otherwise update dphi
    // in place.
    const bool swap_ok = s->owned && (s->p.flags & PRS_DEBUG) == 0;
    for (int t = 0; t <= kMarchMaxT; ++t) cnt[t] = 0;
    // no second buffer (no room at prs_init), or planes beyond the march's offsets
    if (!s->dphi_alt || (s->g.dims == 3 && !march3d_ok(s->g))) {
        cnt[1] = nsteps;
        return;
    }
    if (march_plans(s)) {
        if (s->g.dims == 2) march_counts(*march, nsteps, !swap_ok, cnt);
        else march_counts_3d(*march, nsteps, !swap_ok, cnt);
        return;
    }
    int64_t n3 = 0, n2 = 0, n1 = nsteps;
    if (tb == 3) {
        n3 = nsteps / 3;
        n2 = nsteps - 3 * n3 == 2 ? 1 : 0;
        n1 = nsteps - 3 * n3 - 2 * n2;
    } else if (tb == 2) {
        n2 = nsteps / 2;
        n1 = nsteps - 2 * n2;
    }
    if (((n3 + n2) & 1) && n1 == 0 && !swap_ok) {
        if (n2 > 0) n2 -= 1, n1 += 2;
        else n3 -= 1, n2 += 1, n1 += 1;
    }
    cnt[3] = n3, cnt[2] = n2, cnt[1] = n1;
}

// Queue one pass of t steps from step n: phi[cur] -> phi[1 - cur], dphi from v_in to v_out (equal only
// for t = 1).  Flips cur when the launch succeeds.
static cudaError_t queue_pass(prs_sim* s, int t, int64_t n, const void* v_in, void* v_out)
{
    const bool repro = (s->p.flags & PRS_REPRO) != 0;
    unsigned int* err = &s->d_status->error;
    const void* in = s->phi[s->cur];
    void* out = s->phi[1 - s->cur];
    double c[kMarchMaxT][5];
    for (int l = 0; l < t; ++l) step_coefficients(s->p, n + l, c[l]);
    cudaError_t e = cudaErrorNotSupported;
    if (t == 2 && s->g.dims == 3 && (s->march.shape[2].cols == 0 || !march3d_ok(s->g))) {
        const RunConst<float> rcf{(float)s->rc[0], (float)s->rc[1], (float)s->rc[2],
                                  (float)s->rc[3], (float)s->rc[4], (float)s->rc[5]};
        e = launch_step_t2(s->g, (const float*)in, (float*)out, (const float*)v_in, (float*)v_out,
                           kick_f32(c[0], s->rc), kick_f32(c[1], s->rc), rcf, err, s->stream);
        if (e == cudaSuccess) s->waits = true;
    }
    if (e == cudaErrorNotSupported && march_run(s) && (t > 1 || s->march.shape[1].cols)) {
        MarchRun r{in, out, v_in, v_out, {}, s->rc};
        for (int l = 0; l < t; ++l)
            for (int q = 0; q < 3; ++q) r.coef[l][q] = c[l][q];
        e = s->g.dims == 2 ? launch_march2d(s->g, t, s->march.shape[t], 1, &r, s->stream)
                           : launch_march3d(s->g, t, s->march.shape[t].cy, 1, &r, s->stream);
    } else if (e == cudaErrorNotSupported) {
        e = launch_step_io(s->g, s->p.precision, repro, in, out, v_in, v_out, c[0], s->rc, s->march.shape[1], err,
                           s->stream);
        if (fast_step_ok(s->g, s->p.precision)) s->waits = true;
    }
    if (e == cudaSuccess) s->cur = 1 - s->cur;
    return e;
}

static int prs_step_impl(prs_sim* s, int64_t nsteps)
{
    if (!s || nsteps < 0) return PRS_EINVAL;
    if (!s->initialised) return PRS_ESTATE;
    if (nsteps == 0) return PRS_OK;
    if (!cfl_ok_over(s->p, s->n, nsteps)) return PRS_EINVAL;
    make_plan(s, 1);
    int64_t cnt[kMarchMaxT + 1];
    step_plan(s, &s->march, nsteps, cnt);
    void* vbuf[2] = {s->dphi, s->dphi_alt};
    int vi = 0;  // vbuf[vi] holds dphi
    int64_t n = s->n;
    for (int t = kMarchMaxT; t >= 1; --t)
        for (int64_t k = 0; k < cnt[t]; ++k, n += t) {
            // the first single step brings dphi home
            const cudaError_t e = queue_pass(s, t, n, vbuf[vi], t > 1 ? vbuf[1 - vi] : s->dphi);
            if (e != cudaSuccess) return cuda_fail(e, "prs_step launch");
            vi = t > 1 ? 1 - vi : 0;
        }
    if (vi) {  // dphi now sits in the second buffer, which becomes the run's own (only when swap_ok)
        void* t = s->dphi;
        s->dphi = s->dphi_alt;
        s->dphi_alt = t;
    }
    s->n += nsteps;
    return PRS_OK;
}

// ---------------------------------------------------------------- measure

// After a synchronised read of h_status: a bounded device wait that gave up makes
// the state untrustworthy; report it once and clear the word.
int prs::check_device_error(prs_sim* s)
{
    if (s->h_status->error == 0) return PRS_OK;
    snprintf(g_last_error, sizeof g_last_error, "device wait timed out (code %u)", s->h_status->error);
    s->h_status->error = 0;
    cudaMemsetAsync(&s->d_status->error, 0, sizeof(unsigned int), s->stream);
    cudaStreamSynchronize(s->stream);
    return PRS_ETIMEOUT;
}

// The FP32 diagnostics may take the hardware's reciprocals and roots; PRS_FP32_CR asks for
// correctly rounded division and sqrt, as do boxes off the staged tiles.
static bool fast_diag_ok(const prs_sim* s)
{
    return fast_step_ok(s->g, s->p.precision) && (s->p.flags & PRS_FP32_CR) == 0;
}

// Queue the diagnostics of the current state.
static cudaError_t queue_measure(prs_sim* s, const DiagScratch& scr)
{
    return launch_measure(s->g, s->p.precision, fast_diag_ok(s), MeasureRun{s->phi[s->cur], s->dphi, s->rc, scr},
                          &s->d_status->error, s->stream);
}

// Fill a prs_diag from the device status copied to s->h_status (after a sync).
static void diag_from_status(const prs_sim* s, int64_t step, prs_diag* d)
{
    const DiagAcc& a = s->h_status->result;
    d->sum_w = a.sum_w;
    d->sum_ratio = a.sum_ratio;
    d->n_links = a.n_links;
    d->n_wall = a.n_wall;
    d->n_vzero = a.n_vzero;
    d->n_nonfinite = a.n_nonfinite;
    d->area_per_volume = a.sum_w / ((double)s->g.S * s->p.dx);  // dA/V = dx^(D-1)/(S dx^D)
    int64_t nw = a.n_wall - a.n_vzero;
    d->gamma_v = nw > 0 ? sqrt(a.sum_ratio / (2.0 * (double)nw)) : 0.0;
    d->step = step;
    d->eta = s->p.eta0 + (double)step * s->p.deta;
}

// The diagnostics of the current state, then nsteps steps queued behind them while the result
// travels to the host.  (A one-step pass that also evaluated the diagnostics of the state it read
// took 4.6 ms at 1024^3, against 3.5 ms for the diagnostics alone and 1.4 for the same step inside a
// multi-step pass: it paid for intervals of one or two steps on large aligned 3D boxes, by 3 to 12%.)
// Runs whose diagnostics are the IEEE ones first hear of earlier passes whose bounded waits gave up: their
// state is not stepped on.
static int prs_step_measure_impl(prs_sim* s, int64_t nsteps, prs_diag* out)
{
    if (!s || !out || nsteps < 0) return PRS_EINVAL;
    if (!s->initialised) return PRS_ESTATE;
    if (nsteps > 0 && !cfl_ok_over(s->p, s->n, nsteps)) return PRS_EINVAL;
    const int64_t n0 = s->n;
    DiagScratch scr = s->scr;
    scr.host = s->h_status;
    scr.error = &s->d_status->error;
    const cudaError_t e = queue_measure(s, scr);
    if (e != cudaSuccess) return cuda_fail(e, "prs_measure launch");
    const bool ask = nsteps > 0 && s->waits && !fast_diag_ok(s);
    s->waits = false;  // the diagnostics bring the error word of the passes before them
    if (ask) {
        PRS_CUDA(cudaStreamSynchronize(s->stream));
        const int err = check_device_error(s);
        if (err) return err;
    }
    if (nsteps > 0) {
        const int rs = prs_step(s, nsteps);
        if (rs) return rs;
    }
    PRS_CUDA(cudaStreamSynchronize(s->stream));
    int err = check_device_error(s);
    if (err) return err;
    diag_from_status(s, n0, out);
    return s->h_status->result.n_nonfinite ? PRS_ENONFINITE : PRS_OK;
}

static int measure_into(prs_sim* s, prs_diag* d) { return prs_step_measure_impl(s, 0, d); }

int prs::step_runs(prs_sim* const* runs, int nruns, int64_t nsteps)
{
    if (nruns < 0 || nsteps < 0) return PRS_EINVAL;
    if (nruns == 0 || nsteps == 0) return PRS_OK;
    bool together = nruns > 1 && nruns <= kMarchMaxRuns;
    for (int r = 0; r < nruns; ++r) {
        const prs_sim* s = runs[r];
        if (!s) return PRS_EINVAL;
        if (!s->initialised) return PRS_ESTATE;
        if (!cfl_ok_over(s->p, s->n, nsteps)) return PRS_EINVAL;
        const Geo &g = s->g, &g0 = runs[0]->g;
        together = together && march_plans(s) && g.dims == g0.dims && g.nx == g0.nx && g.ny == g0.ny &&
                   g.nz == g0.nz && march_packed(g) && (g.dims == 2 || march3d_ok(g)) &&
                   s->stream == runs[0]->stream && s->dphi_alt && s->owned == runs[0]->owned &&
                   (s->p.flags & PRS_DEBUG) == 0;
    }
    if (!together) {
        for (int r = 0; r < nruns; ++r) {
            const int rc = prs_step_impl(runs[r], nsteps);
            if (rc) return rc;
        }
        return PRS_OK;
    }
    make_plan(runs[0], nruns);
    const MarchPlan& plan = runs[0]->march;
    int64_t cnt[kMarchMaxT + 1], done = 0;
    step_plan(runs[0], &plan, nsteps, cnt);
    MarchRun q[kMarchMaxRuns];
    int vi = 0;  // which of each run's dphi and dphi_alt holds dphi
    for (int t = kMarchMaxT; t >= 1; --t)
        for (int64_t k = 0; k < cnt[t]; ++k, done += t) {
            for (int r = 0; r < nruns; ++r) {
                prs_sim* s = runs[r];
                void* vbuf[2] = {s->dphi, s->dphi_alt};
                q[r].phi_in = s->phi[s->cur];
                q[r].phi_out = s->phi[1 - s->cur];
                q[r].v_in = vbuf[vi];
                q[r].v_out = t > 1 ? vbuf[1 - vi] : s->dphi;
                q[r].run_const = s->rc;
                for (int l = 0; l < t; ++l) {
                    double c[5];
                    step_coefficients(s->p, s->n + done + l, c);
                    for (int u = 0; u < 3; ++u) q[r].coef[l][u] = c[u];
                }
            }
            const cudaError_t e =
                runs[0]->g.dims == 2 ? launch_march2d(runs[0]->g, t, plan.shape[t], nruns, q, runs[0]->stream)
                                     : launch_march3d(runs[0]->g, t, plan.shape[t].cy, nruns, q, runs[0]->stream);
            if (e != cudaSuccess) return cuda_fail(e, "step_runs launch");
            for (int r = 0; r < nruns; ++r) runs[r]->cur = 1 - runs[r]->cur;
            vi = t > 1 ? 1 - vi : 0;
        }
    for (int r = 0; r < nruns; ++r) {
        prs_sim* s = runs[r];
        if (vi) {  // as prs_step_impl: only where the run may swap its dphi buffers
            void* v = s->dphi;
            s->dphi = s->dphi_alt;
            s->dphi_alt = v;
        }
        s->n += nsteps;
    }
    return PRS_OK;
}

int prs::queue_diagnostics(prs_sim* const* runs, int nruns, DiagAcc* const* results)
{
    for (int r0 = 0; r0 < nruns; r0 += kMeasureMaxRuns) {
        const int n = nruns - r0 < kMeasureMaxRuns ? nruns - r0 : kMeasureMaxRuns;
        MeasureRun q[kMeasureMaxRuns];
        bool together = n > 1;
        for (int r = 0; r < n; ++r) {
            prs_sim* s = runs[r0 + r];
            if (!s || !results[r0 + r]) return PRS_EINVAL;
            if (!s->initialised) return PRS_ESTATE;
            const Geo &g = s->g, &g0 = runs[r0]->g;
            together = together && fast_diag_ok(s) && g.dims == g0.dims && g.nx == g0.nx && g.ny == g0.ny &&
                       g.nz == g0.nz && s->stream == runs[r0]->stream;
            q[r] = MeasureRun{s->phi[s->cur], s->dphi, s->rc, s->scr};
            q[r].scr.result = results[r0 + r];
        }
        cudaError_t e = cudaSuccess;
        if (together) e = launch_measure_runs(runs[r0]->g, n, q, runs[r0]->stream);
        for (int r = 0; r < n && !together && e == cudaSuccess; ++r) e = queue_measure(runs[r0 + r], q[r].scr);
        if (e != cudaSuccess) return cuda_fail(e, "measure launch");
    }
    return PRS_OK;
}

static int prs_measure_ex_impl(prs_sim* s, prs_diag* out)
{
    if (!s || !out) return PRS_EINVAL;
    return measure_into(s, out);
}

static int prs_measure_impl(prs_sim* s, double* area_per_volume, double* gamma_v, int64_t* n_links,
                           int64_t* n_wall_sites)
{
    if (!s) return PRS_EINVAL;
    prs_diag d;
    int rc = measure_into(s, &d);
    if (rc != PRS_OK && rc != PRS_ENONFINITE) return rc;
    if (area_per_volume) *area_per_volume = d.area_per_volume;
    if (gamma_v) *gamma_v = d.gamma_v;
    if (n_links) *n_links = d.n_links;
    if (n_wall_sites) *n_wall_sites = d.n_wall;
    return rc;
}

// ------------------------------------------------ entry points (PRS_DEBUG checks)

extern "C" int prs_init(prs_sim* s, const void* h_phi, const void* h_dphi)
{
    return debug_after(s, prs_init_impl(s, h_phi, h_dphi), "prs_init", true);
}

extern "C" int prs_set_state(prs_sim* s, const void* h_phi, const void* h_dphi, int64_t n)
{
    return debug_after(s, prs_set_state_impl(s, h_phi, h_dphi, n), "prs_set_state", true);
}

extern "C" int prs_step(prs_sim* s, int64_t nsteps)
{
    return debug_after(s, prs_step_impl(s, nsteps), "prs_step", true);
}

extern "C" int prs_step_measure(prs_sim* s, int64_t nsteps, prs_diag* out)
{
    return debug_after(s, prs_step_measure_impl(s, nsteps, out), "prs_step_measure", true);
}

extern "C" int prs_measure_ex(prs_sim* s, prs_diag* out)
{
    return debug_after(s, prs_measure_ex_impl(s, out), "prs_measure_ex", false);
}

extern "C" int prs_measure(prs_sim* s, double* area_per_volume, double* gamma_v, int64_t* n_links,
                           int64_t* n_wall_sites)
{
    const int rc = prs_measure_impl(s, area_per_volume, gamma_v, n_links, n_wall_sites);
    return debug_after(s, rc, "prs_measure", false);
}
