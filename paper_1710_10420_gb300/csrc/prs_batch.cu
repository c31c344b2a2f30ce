// prs_batch.cu -- ensembles of independent PRS runs (mixed 2D/3D sizes, seeds and expansion eras).
//
// The paper motivates large sets of production runs (Sec. I, Sec. IV: calibrating the one-scale model
// needs many realisations); it runs them one at a time.  A small box leaves most of the GPU idle, and
// its passes cost little more than their launches.  Here the runs of one box are stepped together, up to
// 16 to a launch: each of their passes (the register marches, up to six steps a pass in 2D and three in 3D)
// and each output's diagnostics is one launch over all of them, its shape chosen for the group.  Groups
// are independent, so each runs on a stream of its own between a fork and a join on the ensemble's
// stream, and the latencies of one group's passes hide behind another's.
//
// (A persistent kernel over (run, tile, step) items with waits between neighbouring tiles, one step an
// item, took 32 ms where this takes 10 ms: 16 runs of 256^2, 4 of 512^2 and 4 of 128 x 64 x 64,
// 800 steps, diagnostics every 20.)
//
// The marches give the same bits whatever their shape and steps per pass, so a run's fields are those of
// the run stepped alone; its diagnostic sums group differently, so they agree to FP64 rounding.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "prs.h"
#include "prs_internal.h"
#include "prs_march3d.h"
#include "prs_sim.h"

using namespace prs;

// Runs of one box that are stepped together.
struct Group {
    std::vector<int> runs;
    cudaStream_t stream;
    cudaEvent_t done;
};

struct prs_batch {
    std::vector<prs_sim*> sims;
    std::vector<char> alone;  // per run: prs_batch_tuning reports it as stepped alone
    std::vector<Group> groups;
    cudaStream_t stream;
    bool own_stream;
    cudaEvent_t fork;
    char* fields;         // one allocation for every run's fields
    DiagAcc* results;     // device: the outputs of a call, run after run
    size_t result_slots;
};

static int batch_cuda(cudaError_t e, const char* what)
{
    if (e == cudaSuccess) return PRS_OK;
    char msg[256];
    snprintf(msg, sizeof msg, "%s: %s", what, cudaGetErrorString(e));
    record_error(msg);
    return PRS_ECUDA;
}

static int64_t align256(int64_t x) { return (x + 255) & ~(int64_t)255; }

// Boxes that fill the GPU by themselves (2^22 sites or more, stepped by multi-step passes by default) or,
// in 2D, boxes of 2^20 sites or more with rows of at least 1024 columns among at least 8 runs of the box:
// what prs_batch_tuning reports as stepped alone.
static bool steps_alone(const Geo& g, int class_runs)
{
    if (default_fused_steps(g, PRS_FP32, false) < 2) return false;
    if (g.S >= ((int64_t)1 << 22)) return true;
    return g.dims == 2 && g.nx >= 1024 && g.S >= ((int64_t)1 << 20) && class_runs >= 8;
}

static bool same_box(const Geo& a, const Geo& b)
{
    return a.dims == b.dims && a.nx == b.nx && a.ny == b.ny && a.nz == b.nz;
}

extern "C" int prs_batch_destroy(prs_batch* b);

static int batch_setup(prs_batch* b, const prs_params* runs, int nruns, void* stream)
{
    int rc;
    b->own_stream = stream == nullptr;
    if (b->own_stream) {
        if ((rc = batch_cuda(cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking), "prs_batch_create")))
            return rc;
    } else {
        b->stream = (cudaStream_t)stream;
    }
    size_t total = 0;
    for (int r = 0; r < nruns; ++r) {
        prs_sim* s = nullptr;
        if ((rc = prs_create(&runs[r], b->stream, &s))) return rc;
        b->sims.push_back(s);
        s->p.tblock = 0;  // the steps of a pass are the group's: runs with a tblock share its launches (16 of
                          // 256^2, 200 steps: 0.6 ms; each by itself 6.8)
        if (!fast_step_ok(s->g, runs[r].precision) || (s->g.dims == 3 && s->g.nx > 1024) || runs[r].flags != 0) {
            record_error("prs_batch_create: runs must be FP32 with an x side that is a multiple of 128 and divides "
                         "4096 (3D: at most 1024), and 4096/nx dividing the y side");
            return PRS_EINVAL;
        }
        total += 3 * (size_t)align256((int64_t)s->g.S * 4);
    }
    if (cudaMalloc((void**)&b->fields, total) != cudaSuccess) {
        cudaGetLastError();
        return PRS_ENOMEM;
    }
    if ((rc = batch_cuda(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming), "prs_batch_create"))) return rc;
    // groups: runs of one box, in the caller's order, at most as many as a launch takes
    for (int r = 0; r < nruns; ++r) {
        const Geo& g = b->sims[r]->g;
        size_t k = 0;
        while (k < b->groups.size() && (!same_box(b->sims[b->groups[k].runs[0]]->g, g) ||
                                        (int)b->groups[k].runs.size() == kMarchMaxRuns))
            ++k;
        if (k == b->groups.size()) {
            b->groups.push_back(Group{});
            Group& q = b->groups.back();
            if ((rc = batch_cuda(cudaStreamCreateWithFlags(&q.stream, cudaStreamNonBlocking), "prs_batch_create")))
                return rc;
            if ((rc = batch_cuda(cudaEventCreateWithFlags(&q.done, cudaEventDisableTiming), "prs_batch_create")))
                return rc;
        }
        b->groups[k].runs.push_back(r);
        b->sims[r]->stream = b->groups[k].stream;
    }
    size_t off = 0;
    for (int r = 0; r < nruns; ++r) {
        prs_sim* s = b->sims[r];
        const size_t fb = (size_t)align256(s->g.S * 4);
        char* f = b->fields + off;
        off += 3 * fb;
        if ((rc = prs_bind(s, f, f + fb, f + 2 * fb))) return rc;
        if ((rc = prs_init(s, nullptr, nullptr))) return rc;
        int same = 0;
        for (const prs_sim* q : b->sims) same += same_box(q->g, s->g);
        b->alone.push_back(steps_alone(s->g, same));
    }
    return PRS_OK;
}

extern "C" int prs_batch_create(const prs_params* runs, int nruns, void* stream, prs_batch** out)
{
    if (!runs || nruns < 1 || !out) return PRS_EINVAL;
    prs_batch* b = new (std::nothrow) prs_batch();
    if (!b) return PRS_ENOMEM;
    const int rc = batch_setup(b, runs, nruns, stream);
    if (rc) {
        prs_batch_destroy(b);
        return rc;
    }
    *out = b;
    return PRS_OK;
}

// Queue one group's part of a call: the diagnostics of its runs at every output they reach, and the
// steps between.  Runs that have taken their steps leave the group.
static int group_queue(prs_batch* b, const Group& q, const int64_t* nsteps, int64_t every, const size_t* slot)
{
    prs_sim* sims[kMarchMaxRuns];
    DiagAcc* res[kMarchMaxRuns];
    for (int64_t done = 0;;) {
        int n = 0;
        if (every > 0 && done % every == 0) {
            for (int r : q.runs)
                if (nsteps[r] >= done) {
                    sims[n] = b->sims[r];
                    res[n++] = b->results + slot[r] + done / every;
                }
            const int rc = n ? queue_diagnostics(sims, n, res) : PRS_OK;
            if (rc) return rc;
        }
        int64_t m = every > 0 ? every - done % every : INT64_MAX;
        n = 0;
        for (int r : q.runs)
            if (nsteps[r] > done) {
                m = std::min(m, nsteps[r] - done);
                sims[n++] = b->sims[r];
            }
        if (n == 0) return PRS_OK;
        const int rc = step_runs(sims, n, m);
        if (rc) return rc;
        done += m;
    }
}

// Queue a call's work, each group on its stream between a fork and a join on the ensemble's, and wait for
// its results.
static int run_queue(prs_batch* b, const int64_t* nsteps, int64_t every, const size_t* slot, std::vector<DiagAcc>& res)
{
    cudaError_t e = cudaEventRecord(b->fork, b->stream);
    for (Group& q : b->groups) {
        if (e == cudaSuccess) e = cudaStreamWaitEvent(q.stream, b->fork, 0);
        if (e != cudaSuccess) return batch_cuda(e, "prs_batch_run");
        const int rc = group_queue(b, q, nsteps, every, slot);
        if (rc) return rc;
        for (int r : q.runs)  // the error words of the runs' bounded waits
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(&b->sims[r]->h_status->error, &b->sims[r]->d_status->error, sizeof(unsigned),
                                    cudaMemcpyDeviceToHost, q.stream);
        if (e == cudaSuccess) e = cudaEventRecord(q.done, q.stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, q.done, 0);
    }
    if (e == cudaSuccess && !res.empty())
        e = cudaMemcpyAsync(res.data(), b->results, res.size() * sizeof(DiagAcc), cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    return batch_cuda(e, "prs_batch_run");
}

extern "C" int prs_batch_run(prs_batch* b, const int64_t* nsteps_per_run, int64_t measure_every, double* out_series,
                             int64_t out_capacity)
{
    if (!b || !nsteps_per_run || measure_every < 0) return PRS_EINVAL;
    const int R = (int)b->sims.size();
    std::vector<int64_t> n0(R), nout(R, 0);
    std::vector<size_t> slot(R);
    size_t slots = 0;
    for (int r = 0; r < R; ++r) {
        const int64_t n = nsteps_per_run[r];
        if (n < 0) return PRS_EINVAL;
        if (n > 0 && !cfl_ok_over(b->sims[r]->p, b->sims[r]->n, n)) return PRS_EINVAL;
        if (measure_every > 0 && (!out_series || n / measure_every + 1 > out_capacity)) return PRS_EINVAL;
        n0[r] = b->sims[r]->n;
        if (measure_every > 0) nout[r] = n / measure_every + 1;
        slot[r] = slots;
        slots += (size_t)nout[r];
    }
    int rc;
    if (slots > b->result_slots) {
        cudaFree(b->results);
        b->results = nullptr;
        b->result_slots = 0;
        if (cudaMalloc((void**)&b->results, slots * sizeof(DiagAcc)) != cudaSuccess) {
            cudaGetLastError();
            return PRS_ENOMEM;
        }
        b->result_slots = slots;
    }
    std::vector<DiagAcc> res(slots);
    if ((rc = run_queue(b, nsteps_per_run, measure_every, slot.data(), res))) {
        // groups may be forked and not joined: nothing stays in flight behind an error
        for (Group& q : b->groups) cudaStreamSynchronize(q.stream);
        cudaStreamSynchronize(b->stream);
        cudaGetLastError();
        return rc;
    }
    for (prs_sim* s : b->sims)
        if ((rc = check_device_error(s))) return rc;
    for (int r = 0; r < R; ++r) {
        const prs_sim* s = b->sims[r];
        for (int64_t k = 0; k < nout[r]; ++k) {
            const DiagAcc& a = res[slot[r] + (size_t)k];
            double* o = out_series + ((size_t)r * out_capacity + (size_t)k) * 4;
            const int64_t nw = a.n_wall - a.n_vzero;
            o[0] = (double)(n0[r] + k * measure_every);
            o[1] = a.sum_w / ((double)s->g.S * s->p.dx);
            o[2] = nw > 0 ? sqrt(a.sum_ratio / (2.0 * (double)nw)) : 0.0;
            o[3] = (double)a.n_links;
        }
    }
    return PRS_OK;
}

// A run's copies are queued on its group's stream: behind what the caller queued on the ensemble's (which
// may still fill or read the host arrays).
static int follow_caller(prs_batch* b, int run)
{
    cudaError_t e = cudaEventRecord(b->fork, b->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->sims[run]->stream, b->fork, 0);
    return batch_cuda(e, "ensemble state");
}

extern "C" int prs_batch_get_state(prs_batch* b, int run, void* h_phi, void* h_dphi, int64_t* n)
{
    if (!b || run < 0 || run >= (int)b->sims.size()) return PRS_EINVAL;
    const int rc = follow_caller(b, run);
    return rc ? rc : prs_get_state(b->sims[run], h_phi, h_dphi, n);
}

extern "C" int prs_batch_set_state(prs_batch* b, int run, const void* h_phi, const void* h_dphi, int64_t n)
{
    if (!b || run < 0 || run >= (int)b->sims.size() || !h_phi || !h_dphi || n < 0) return PRS_EINVAL;
    const int rc = follow_caller(b, run);
    return rc ? rc : prs_set_state(b->sims[run], h_phi, h_dphi, n);
}

extern "C" int prs_batch_tuning(prs_batch* b, int run, int* tile_len, double* group_bytes)
{
    if (!b || run < 0 || run >= (int)b->sims.size()) return PRS_EINVAL;
    if (tile_len) *tile_len = b->alone[run] ? 0 : 16;
    if (group_bytes) {
        *group_bytes = 0.0;
        for (const Group& q : b->groups)
            if (std::find(q.runs.begin(), q.runs.end(), run) != q.runs.end())
                *group_bytes = 12.0 * (double)b->sims[run]->g.S * (double)q.runs.size();
    }
    return PRS_OK;
}

extern "C" int prs_batch_destroy(prs_batch* b)
{
    if (!b) return PRS_EINVAL;
    if (b->stream) cudaStreamSynchronize(b->stream);
    for (prs_sim* s : b->sims) prs_destroy(s);
    for (Group& q : b->groups) {
        if (q.stream) cudaStreamDestroy(q.stream);
        if (q.done) cudaEventDestroy(q.done);
    }
    if (b->fork) cudaEventDestroy(b->fork);
    cudaFree(b->results);
    cudaFree(b->fields);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return PRS_OK;
}
