// C-ABI of the pulse-noise lattice library: handles, parameter validation,
// the pulse/sample schedule of Eq. (ST-expansion), workspace layout and the
// CUDA-graph cache for whole noise intervals.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>

#include "../../include/spinpulse.h"
#include "pdl.cuh"
#include "spin_internal.h"

using namespace spin;

// Small lattices replay several intervals as one graph: the GPU idles for two to
// two and a half microseconds between two graph launches, and an interval of a
// few small kernels takes only tens.  To capture and instantiate a graph costs
// the host about 1.9 us a kernel, as long as the kernel takes the GPU or less; so
// a longer graph is captured only while the GPU still works on at least as many
// intervals of the same call, and holds at most kGraphSteps steps.
constexpr int kGraphLevels = 4;
constexpr int kGraphSteps = 32;
constexpr long long kLongGraphSites = 1LL << 20;
constexpr long long kLongGraphAfter = 8;

struct spin_lattice {
    spin_params p;
    Geom g;
    Tableau tab;
    int elt;                 // bytes per real
    void* buf[2][3];         // [0] caller arrays, [1] workspace copy
    const void* hs[3];       // per-site field or nulls
    int cur;                 // which buffer holds the current state
    cudaStream_t st;
    long long n;             // completed steps
    long long eager_intervals;
    // workspace carve-out
    void* tmp;
    double* partials;
    int nblocks_obs;
    double* out_sample;
    double* out_obs;
    long long* d_interval;
    long long* d_sample_count;
    int* d_status;           // bit 0: a bounded device wait gave up
    double* ring;
    long long samples_read;
    cudaGraphExec_t graph[kGraphLevels][2];  // 2^level noise intervals starting from buffer 0 / 1
    int graph_end[kGraphLevels][2];          // the buffer they end in
    long long replayed;        // intervals replayed from graphs
    cudaStream_t capture_stream;
    // trajectory recording for the adjoint
    bool rec_active;
    int rec_K;
    long long rec_n0, rec_max;
    void* rec_store;
    char err[512];
};

namespace {

constexpr size_t kAlign = 256;
size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

struct Layout {
    size_t alt[3];
    size_t tmp;
    size_t partials;
    size_t out_sample, out_obs, interval, sample_count, status, ring;
    size_t total;
};

int validate(const spin_params* p) {
    if (!p) return SPIN_EINVAL;
    if (p->nx < 1 || p->ny < 1 || p->nz < 1) return SPIN_EINVAL;
    const long long N = (long long)p->nx * p->ny * p->nz;
    if (N >= (1LL << 31)) return SPIN_EINVAL;
    if (p->precision != 32 && p->precision != 64) return SPIN_EINVAL;
    if (p->integrator < 0 || p->integrator > 3) return SPIN_EINVAL;
    if (p->steps_per_pulse < 1) return SPIN_EINVAL;
    if (!std::isfinite(p->dt) || p->dt == 0.0) return SPIN_EINVAL;
    if (!(p->lambda >= 0.0) || !(p->T >= 0.0) || !std::isfinite(p->lambda) || !std::isfinite(p->T)) return SPIN_EINVAL;
    if (!std::isfinite(p->J) || !std::isfinite(p->D)) return SPIN_EINVAL;
    for (int a = 0; a < 3; ++a)
        if (!std::isfinite(p->H[a])) return SPIN_EINVAL;
    if (p->path < 0 || p->path > 1 || p->bc < 0 || p->bc > 1) return SPIN_EINVAL;
    if (p->replica < 0) return SPIN_EINVAL;
    if (p->noise < 0 || p->noise > 2) return SPIN_EINVAL;
    if (p->noise == 2) return SPIN_EUNSUPPORTED;  // rectangular noise: single-spin calls only
    return SPIN_OK;
}

Layout layout_for(const spin_params* p) {
    Layout L{};
    const Geom g{p->nx, p->ny, p->nz};
    const size_t elt = p->precision == 64 ? 8 : 4;
    const size_t comp = align_up(elt * (size_t)g.N());
    size_t off = 0;
    for (int c = 0; c < 3; ++c) {
        L.alt[c] = off;
        off += comp;
    }
    const Tableau tb = tableau_for(p->integrator);
    const bool generic = !tb.chain || p->path == 1 || !(tb.stages == 2 || tb.stages == 4);
    L.tmp = off;
    if (generic) off += align_up(elt * (size_t)(tb.stages + 1) * 3 * (size_t)g.N());
    else if (elt == 8) off += align_up(elt * (size_t)stage64_scratch(tb.stages) * (size_t)g.N());
    // stage inputs of the small-lattice FP32 stage kernels, with site fields or
    // without (RK5, which does not take them, has the room too: callers may count
    // on its workspace being the RK4 one and its own stage arrays)
    if (elt == 4 && p->path != 1 && stage32_small(g, tb.stages == 4 ? 4 : 2, true, false)) {
        if (!generic) L.tmp = off;
        off += align_up(elt * (size_t)stage32_scratch(tb.stages) * (size_t)g.N());
    }
    L.partials = off;
    off += align_up(sizeof(double) * 5 * (size_t)observables_blocks(g));
    L.out_sample = off;
    off += align_up(sizeof(double) * 8);
    L.out_obs = off;
    off += align_up(sizeof(double) * 8);
    L.interval = off;
    off += align_up(sizeof(long long));
    L.sample_count = off;
    off += align_up(sizeof(long long));
    L.status = off;
    off += align_up(sizeof(int));
    L.ring = off;
    off += align_up(sizeof(double) * 5 * SPIN_SAMPLE_RING);
    L.total = off;
    return L;
}

int set_err(spin_lattice* h, int code, const char* fmt, ...) {
    if (h) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(h->err, sizeof(h->err), fmt, ap);
        va_end(ap);
    }
    return code;
}

#define SPIN_CUDA(h, call)                                                                          \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess) return set_err(h, SPIN_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

bool is_pulse_step(long long n, int R) { return (n % R) == (R / 2); }

template <typename real>
StepLaunch<real> make_launch(spin_lattice* h, int from, bool pulse) {
    StepLaunch<real> L{};
    for (int c = 0; c < 3; ++c) {
        L.in[c] = static_cast<const real*>(h->buf[from][c]);
        L.out[c] = static_cast<real*>(h->buf[from ^ 1][c]);
        L.hs[c] = static_cast<const real*>(h->hs[c]);
    }
    L.g = h->g;
    L.ph.J = (real)h->p.J;
    L.ph.twoD = (real)(2.0 * h->p.D);
    for (int a = 0; a < 3; ++a) L.ph.H[a] = (real)h->p.H[a];
    L.ph.lambda = (real)h->p.lambda;
    L.dt = h->p.dt;
    L.tab = &h->tab;
    L.precession = h->p.precession;
    L.renorm = h->p.renorm;
    L.pulse = pulse ? 1 : 0;
    L.seed = h->p.seed;
    L.replica = (uint64_t)h->p.replica;
    L.sigma = (real)std::sqrt(2.0 * h->p.lambda * h->p.T * h->p.steps_per_pulse * std::fabs(h->p.dt));
    L.d_interval = h->d_interval;
    L.d_status = h->d_status;
    L.tmp = static_cast<real*>(h->tmp);
    L.stream = h->st;
    L.force_generic = h->p.path == 1;
    L.bc = h->p.bc;
    return L;
}

Phys<double> phys64(const spin_lattice* h) {
    Phys<double> ph{};
    ph.J = h->p.J;
    ph.twoD = 2.0 * h->p.D;
    for (int a = 0; a < 3; ++a) ph.H[a] = h->p.H[a];
    ph.lambda = h->p.lambda;
    return ph;
}

// Launch observables of buffer b; sample=true records into the ring.
cudaError_t observe(spin_lattice* h, int b, bool sample, cudaStream_t st, int into) {
    if (h->elt == 4) {
        const float* s[3] = {(const float*)h->buf[b][0], (const float*)h->buf[b][1], (const float*)h->buf[b][2]};
        const float* hs[3] = {(const float*)h->hs[0], (const float*)h->hs[1], (const float*)h->hs[2]};
        return launch_observables<float>(s, hs, h->g, phys64(h), h->partials, h->nblocks_obs,
                                         sample ? h->out_sample : h->out_obs, sample ? h->ring : nullptr,
                                         SPIN_SAMPLE_RING, h->d_interval, h->d_sample_count, h->p.steps_per_pulse, st,
                                         h->p.bc, into);
    }
    const double* s[3] = {(const double*)h->buf[b][0], (const double*)h->buf[b][1], (const double*)h->buf[b][2]};
    const double* hs[3] = {(const double*)h->hs[0], (const double*)h->hs[1], (const double*)h->hs[2]};
    return launch_observables<double>(s, hs, h->g, phys64(h), h->partials, h->nblocks_obs,
                                      sample ? h->out_sample : h->out_obs, sample ? h->ring : nullptr,
                                      SPIN_SAMPLE_RING, h->d_interval, h->d_sample_count, h->p.steps_per_pulse, st,
                                      h->p.bc, into);
}

// One step n -> n+1 from buffer *buf on stream st, which becomes the buffer of
// the new state (no other host bookkeeping).  A step goes from one buffer to
// the other; with an odd number of steps per interval the pulse of the FP32
// fused paths, a kernel of its own, goes back, so that an interval ends where
// it began and the state needs no copy to the caller's arrays (256^3: 60 us).
cudaError_t launch_one_step(spin_lattice* h, int* buf, long long n_next, cudaStream_t st, int into) {
    const int R = h->p.steps_per_pulse;
    const bool pulse = h->p.noise && is_pulse_step(n_next, R);
    const int from = *buf;
    int to = from ^ 1;
    cudaError_t e;
    if (h->elt == 4) {
        StepLaunch<float> L = make_launch<float>(h, from, pulse);
        L.stream = st;
        L.into = into;
        if (pulse && (R & 1) && !L.force_generic && (h->tab.chain || rk5_fused_supports(L))) {
            to = from;
            for (int c = 0; c < 3; ++c) L.pulse_out[c] = static_cast<float*>(h->buf[to][c]);
        }
        e = launch_step<float>(L);
    } else {
        StepLaunch<double> L = make_launch<double>(h, from, pulse);
        L.stream = st;
        L.into = into;
        e = launch_step<double>(L);
    }
    if (e != cudaSuccess) return e;
    *buf = to;
    if (n_next % R == 0) e = observe(h, to, true, st, into);
    return e;
}

// Capture 2^level full intervals (R steps + sample) starting from buffer `from`.
int capture_interval(spin_lattice* h, int level, int from) {
    if (!h->capture_stream) SPIN_CUDA(h, cudaStreamCreateWithFlags(&h->capture_stream, cudaStreamNonBlocking));
    cudaStream_t cs = h->capture_stream;
    SPIN_CUDA(h, cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    const int R = h->p.steps_per_pulse;
    int b = from;
    cudaError_t e = cudaSuccess;
    // the graph covers steps mR+1 .. (m+2^level)R; pulse and sample positions
    // depend only on n mod R, so step numbers from 1 on describe every interval
    for (int q = 1; q <= (R << level) && e == cudaSuccess; ++q) {
        e = launch_one_step(h, &b, q, cs, kIntervalGraph);
    }
    h->graph_end[level][from] = b;
    cudaGraph_t graph = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(cs, &graph);
    if (e != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return set_err(h, SPIN_ECUDA, "interval capture: %s", cudaGetErrorString(e));
    }
    if (e2 != cudaSuccess) return set_err(h, SPIN_ECUDA, "cudaStreamEndCapture: %s", cudaGetErrorString(e2));
    cudaError_t e3 = cudaGraphInstantiate(&h->graph[level][from], graph, 0);
    cudaGraphDestroy(graph);
    if (e3 != cudaSuccess) {
        h->graph[level][from] = nullptr;
        return set_err(h, SPIN_ECUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e3));
    }
    return SPIN_OK;
}

// Replay 2^level intervals from the current state's buffer.
int replay(spin_lattice* h, int level) {
    if (!h->graph[level][h->cur]) {
        const int rc = capture_interval(h, level, h->cur);
        if (rc != SPIN_OK) return rc;
    }
    SPIN_CUDA(h, cudaGraphLaunch(h->graph[level][h->cur], h->st));
    h->n += (long long)h->p.steps_per_pulse << level;
    h->cur = h->graph_end[level][h->cur];
    h->replayed += 1LL << level;
    return SPIN_OK;
}

// The level of the longest graph that n steps fill.
int longest_level(const spin_lattice* h, long long n) {
    if (h->g.N() > kLongGraphSites || h->replayed < kLongGraphAfter) return 0;
    int level = 0;
    while (level + 1 < kGraphLevels && ((long long)h->p.steps_per_pulse << (level + 1)) <= std::min<long long>(n, kGraphSteps))
        ++level;
    return level;
}

// The graph for a call that has nsteps left and *ahead intervals queued behind
// which no graph has been captured yet: the longest that there is, or that can be
// captured behind them.
int next_level(const spin_lattice* h, long long nsteps, long long* ahead) {
    int level = longest_level(h, nsteps);
    for (; level > 0 && !h->graph[level][h->cur]; --level)
        if (*ahead >= (1LL << level)) {
            *ahead -= 1LL << level;
            break;
        }
    return level;
}

// While recording, copy the current state into checkpoint slot (n-n0)/K
// whenever n - n0 is a multiple of K within the recorded range.
int record_if_due(spin_lattice* h) {
    if (!h->rec_active) return SPIN_OK;
    const long long d = h->n - h->rec_n0;
    if (d < 0 || d > h->rec_max || d % h->rec_K != 0) return SPIN_OK;
    const size_t comp = (size_t)h->elt * (size_t)h->g.N();
    char* slot = static_cast<char*>(h->rec_store) + (size_t)(d / h->rec_K) * 3 * comp;
    for (int c = 0; c < 3; ++c)
        SPIN_CUDA(h, cudaMemcpyAsync(slot + c * comp, h->buf[h->cur][c], comp, cudaMemcpyDeviceToDevice, h->st));
    return SPIN_OK;
}

template <typename real>
int backward_t(spin_lattice* h, const double dLdM[3], double dLdE, void* ws, double* gJ, double* gD,
                      double gH[3], void* g_h_site, void* g_s0) {
    AdjointRun<real> A{};
    A.g = h->g;
    A.tab = &h->tab;
    A.K = h->rec_K;
    A.n0 = h->rec_n0;
    A.n_end = h->n;
    A.R = h->p.steps_per_pulse;
    A.noise = h->p.noise;
    A.precession = h->p.precession;
    A.renorm = h->p.renorm;
    A.bc = h->p.bc;
    A.store_stages = adjoint_stores_stages(h->g, (int)sizeof(real), h->tab, h->p.path, h->rec_K) ? 1 : 0;
    A.seed = h->p.seed;
    A.replica = (uint64_t)h->p.replica;
    A.sigma = std::sqrt(2.0 * h->p.lambda * h->p.T * h->p.steps_per_pulse * std::fabs(h->p.dt));
    A.J = h->p.J;
    A.D = h->p.D;
    for (int a = 0; a < 3; ++a) {
        A.H[a] = h->p.H[a];
        A.dLdM[a] = dLdM[a];
    }
    A.lambda = h->p.lambda;
    A.dt = h->p.dt;
    A.h_site = static_cast<const real*>(h->hs[0]);
    A.store = static_cast<const real*>(h->rec_store);
    for (int c = 0; c < 3; ++c) A.final_state[c] = static_cast<const real*>(h->buf[h->cur][c]);
    A.step_template = make_launch<real>(h, 0, false);
    A.workspace = ws;
    A.stream = h->st;
    A.dLdE = dLdE;
    A.gJ = gJ;
    A.gD = gD;
    A.gH = gH;
    A.g_h = static_cast<double*>(g_h_site);
    A.g_s0 = static_cast<real*>(g_s0);
    SPIN_CUDA(h, adjoint_run<real>(A));
    int status = 0;   // the recomputing steps' bounded waits (adjoint_run has synchronised)
    SPIN_CUDA(h, cudaMemcpy(&status, h->d_status, sizeof(int), cudaMemcpyDeviceToHost));
    if (status & 1) return set_err(h, SPIN_ETIMEOUT, "a bounded wait in the fused step gave up; the gradients are invalid");
    return SPIN_OK;
}

}  // namespace

extern "C" {

const char* spin_strerror(int status) {
    switch (status) {
        case SPIN_OK: return "ok";
        case SPIN_WARN_APPLICABILITY: return "pulse-noise applicability condition violated (Lambda_N Delta t or lambda H Delta t too large)";
        case SPIN_EINVAL: return "invalid argument";
        case SPIN_ECUDA: return "CUDA runtime error";
        case SPIN_ENONFINITE: return "non-finite spin (integration unstable)";
        case SPIN_ETIMEOUT: return "bounded device wait timed out";
        case SPIN_EUNSUPPORTED: return "unsupported request";
        case SPIN_ENOSPACE: return "workspace too small";
        default: return "unknown status";
    }
}

const char* spin_last_error(const spin_lattice* h) { return h ? h->err : "null handle"; }

int spin_workspace_size(const spin_params* p, size_t* bytes) {
    if (!bytes) return SPIN_EINVAL;
    int v = validate(p);
    if (v != SPIN_OK) return v;
    *bytes = layout_for(p).total;
    return SPIN_OK;
}

int spin_lattice_create(const spin_params* p, void* sx, void* sy, void* sz, const void* h_site, void* workspace,
                        size_t workspace_bytes, void* cuda_stream, spin_lattice** out) {
    if (!out) return SPIN_EINVAL;
    *out = nullptr;
    int v = validate(p);
    if (v != SPIN_OK) return v;
    if (!sx || !sy || !sz || !workspace) return SPIN_EINVAL;
    if (reinterpret_cast<uintptr_t>(workspace) % kAlign != 0) return SPIN_EINVAL;
    const Layout L = layout_for(p);
    if (workspace_bytes < L.total) return SPIN_ENOSPACE;

    spin_lattice* h = new (std::nothrow) spin_lattice();
    if (!h) return SPIN_EINVAL;
    h->p = *p;
    h->g = Geom{p->nx, p->ny, p->nz};
    h->tab = tableau_for(p->integrator);
    h->elt = p->precision == 64 ? 8 : 4;
    h->buf[0][0] = sx;
    h->buf[0][1] = sy;
    h->buf[0][2] = sz;
    char* ws = static_cast<char*>(workspace);
    for (int c = 0; c < 3; ++c) h->buf[1][c] = ws + L.alt[c];
    const size_t comp_bytes = (size_t)h->elt * (size_t)h->g.N();
    for (int c = 0; c < 3; ++c) h->hs[c] = h_site ? static_cast<const char*>(h_site) + c * comp_bytes : nullptr;
    h->cur = 0;
    h->st = static_cast<cudaStream_t>(cuda_stream);
    h->n = 0;
    h->tmp = ws + L.tmp;
    h->partials = reinterpret_cast<double*>(ws + L.partials);
    h->nblocks_obs = observables_blocks(h->g);
    h->out_sample = reinterpret_cast<double*>(ws + L.out_sample);
    h->out_obs = reinterpret_cast<double*>(ws + L.out_obs);
    h->d_interval = reinterpret_cast<long long*>(ws + L.interval);
    h->d_sample_count = reinterpret_cast<long long*>(ws + L.sample_count);
    h->d_status = reinterpret_cast<int*>(ws + L.status);
    h->ring = reinterpret_cast<double*>(ws + L.ring);
    h->err[0] = 0;

    cudaError_t e = h->elt == 4 ? prepare_step_kernels<float>() : prepare_step_kernels<double>();
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_interval, 0, sizeof(long long), h->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_sample_count, 0, sizeof(long long), h->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_status, 0, sizeof(int), h->st);
    if (e != cudaSuccess) {
        delete h;
        return SPIN_ECUDA;
    }
    *out = h;

    // Applicability of the pulse-noise approximation, Eqs. (phi_condition)
    // and (non-thermal_condition).
    const double Dt = p->steps_per_pulse * std::fabs(p->dt);
    const double LN_Dt = 2.0 * p->lambda * p->T * Dt;
    const double Hmax = 6.0 * std::fabs(p->J) + 2.0 * std::fabs(p->D) +
                        std::sqrt(p->H[0] * p->H[0] + p->H[1] * p->H[1] + p->H[2] * p->H[2]);
    if (p->noise && (LN_Dt > 0.2 || p->lambda * Hmax * Dt > 1.0)) {
        set_err(h, SPIN_WARN_APPLICABILITY, "Lambda_N*Dt = %g, lambda*Hmax*Dt = %g", LN_Dt, p->lambda * Hmax * Dt);
        return SPIN_WARN_APPLICABILITY;
    }
    return SPIN_OK;
}

int spin_step_pulse(spin_lattice* h, int64_t nsteps) {
    if (!h || nsteps < 0) return SPIN_EINVAL;
    const int R = h->p.steps_per_pulse;
    // a caller's capture gets the steps' kernels themselves
    const int into = launch_into(h->st);
    const bool replays = into == kStream;
    long long intervals = 0, ahead = 0;   // replayed by this call; of those, not yet captured behind
    while (nsteps > 0) {
        if (h->rec_active) {
            // recording: a whole noise interval is replayed from the graph when
            // no checkpoint falls strictly inside it (one at its end is taken
            // after the replay); otherwise single eager steps, so that every
            // checkpoint step is seen
            const long long d0 = h->n - h->rec_n0;
            const long long next_ckpt = (d0 / h->rec_K + 1) * h->rec_K;
            if (replays && h->n % R == 0 && nsteps >= R && h->eager_intervals > 0 && d0 >= 0 && next_ckpt >= d0 + R) {
                int rc = replay(h, 0);
                if (rc != SPIN_OK) return rc;
                nsteps -= R;
                rc = record_if_due(h);
                if (rc != SPIN_OK) return rc;
                continue;
            }
            if (h->n % R == 0 && nsteps >= R) h->eager_intervals++;
            SPIN_CUDA(h, launch_one_step(h, &h->cur, h->n + 1, h->st, into));
            h->n += 1;
            nsteps -= 1;
            int rc = record_if_due(h);
            if (rc != SPIN_OK) return rc;
            continue;
        }
        if (replays && h->n % R == 0 && nsteps >= R && h->eager_intervals > 0) {
            const int level = next_level(h, nsteps, &ahead);
            const int rc = replay(h, level);
            if (rc != SPIN_OK) return rc;
            nsteps -= (int64_t)R << level;
            intervals += 1LL << level;
            ahead += 1LL << level;
            continue;
        }
        const bool interval_start = h->n % R == 0 && nsteps >= R;
        const int steps = interval_start ? R : 1;
        for (int q = 0; q < steps; ++q) {
            SPIN_CUDA(h, launch_one_step(h, &h->cur, h->n + 1, h->st, into));
            h->n += 1;
        }
        nsteps -= steps;
        if (interval_start) h->eager_intervals++;
    }
    if (h->cur == 1) {
        const size_t bytes = (size_t)h->elt * (size_t)h->g.N();
        for (int c = 0; c < 3; ++c)
            SPIN_CUDA(h, cudaMemcpyAsync(h->buf[0][c], h->buf[1][c], bytes, cudaMemcpyDeviceToDevice, h->st));
        h->cur = 0;
    }
    // the graph that a call like this one would begin with
    const int level = longest_level(h, intervals * R);
    if (level > 0 && !h->graph[level][0] && ahead >= (1LL << level)) return capture_interval(h, level, 0);
    return SPIN_OK;
}

int spin_observables(spin_lattice* h, double M[3], double* E) {
    if (!h || !M || !E) return SPIN_EINVAL;
    SPIN_CUDA(h, observe(h, h->cur, false, h->st, launch_into(h->st)));
    // one copy from the observables to the status word (neighbours in the
    // workspace): a small copy to the host costs 5 us or more
    char host[1024];
    const size_t span = reinterpret_cast<char*>(h->d_status) - reinterpret_cast<char*>(h->out_obs) + sizeof(int);
    static_assert(4 * kAlign <= sizeof(host), "observables, interval, sample count and status");
    if (span > sizeof(host)) return set_err(h, SPIN_EINVAL, "workspace layout");
    SPIN_CUDA(h, cudaMemcpyAsync(host, h->out_obs, span, cudaMemcpyDeviceToHost, h->st));
    SPIN_CUDA(h, cudaStreamSynchronize(h->st));
    double o[5];
    int status;
    memcpy(o, host, sizeof(o));
    memcpy(&status, host + span - sizeof(int), sizeof(int));
    if (status & 1) return set_err(h, SPIN_ETIMEOUT, "a bounded wait in the fused step gave up; the state is invalid");
    M[0] = o[0];
    M[1] = o[1];
    M[2] = o[2];
    *E = o[3];
    if (o[4] != 0.0) return set_err(h, SPIN_ENONFINITE, "%.0f non-finite spins", o[4]);
    return SPIN_OK;
}

int spin_samples(spin_lattice* h, double* out, int64_t max_records, int64_t* count) {
    if (!h || !count || (max_records > 0 && !out) || max_records < 0) return SPIN_EINVAL;
    // the count and the status word in one copy, then the records in one, or two
    // where the ring wraps (one per record before: 10 records 80 us)
    char host[2 * kAlign];
    const size_t span = reinterpret_cast<char*>(h->d_status) - reinterpret_cast<char*>(h->d_sample_count) + sizeof(int);
    if (span > sizeof(host)) return set_err(h, SPIN_EINVAL, "workspace layout");
    SPIN_CUDA(h, cudaMemcpyAsync(host, h->d_sample_count, span, cudaMemcpyDeviceToHost, h->st));
    SPIN_CUDA(h, cudaStreamSynchronize(h->st));
    long long total;
    int status;
    memcpy(&total, host, sizeof(total));
    memcpy(&status, host + span - sizeof(int), sizeof(int));
    if (status & 1) return set_err(h, SPIN_ETIMEOUT, "a bounded wait in the fused step gave up; the state is invalid");
    long long first = h->samples_read;
    if (total - first > SPIN_SAMPLE_RING) first = total - SPIN_SAMPLE_RING;
    if (total - first > max_records) first = total - max_records;
    const long long n = total - first;
    for (long long q = 0; q < n;) {
        const long long slot = (first + q) % SPIN_SAMPLE_RING;
        const long long m = std::min<long long>(n - q, SPIN_SAMPLE_RING - slot);
        SPIN_CUDA(h, cudaMemcpyAsync(out + 5 * q, h->ring + 5 * slot, (size_t)m * 5 * sizeof(double),
                                     cudaMemcpyDeviceToHost, h->st));
        q += m;
    }
    if (n > 0) SPIN_CUDA(h, cudaStreamSynchronize(h->st));
    h->samples_read = total;
    *count = n;
    return SPIN_OK;
}

int spin_get_step(const spin_lattice* h, int64_t* n) {
    if (!h || !n) return SPIN_EINVAL;
    *n = h->n;
    return SPIN_OK;
}

int spin_set_step(spin_lattice* h, int64_t n) {
    if (!h || n < 0) return SPIN_EINVAL;
    h->n = n;
    SPIN_CUDA(h, launch_set_counter(h->d_interval, n / h->p.steps_per_pulse, h->st));
    return SPIN_OK;
}

int spin_record_store_size(const spin_params* p, int32_t K, int64_t nsteps, size_t* bytes) {
    if (!bytes || K < 1 || nsteps < 1) return SPIN_EINVAL;
    int v = validate(p);
    if (v != SPIN_OK) return v;
    const size_t comp = (size_t)(p->precision == 64 ? 8 : 4) * (size_t)p->nx * p->ny * p->nz;
    *bytes = (size_t)((nsteps + K - 1) / K + 1) * 3 * comp;
    return SPIN_OK;
}

int spin_record_begin(spin_lattice* h, int32_t K, int64_t nsteps, void* store, size_t store_bytes) {
    if (!h || !store || K < 1 || nsteps < 1) return SPIN_EINVAL;
    size_t need = 0;
    spin_record_store_size(&h->p, K, nsteps, &need);
    if (store_bytes < need) return SPIN_ENOSPACE;
    h->rec_active = true;
    h->rec_K = K;
    h->rec_n0 = h->n;
    h->rec_max = nsteps;
    h->rec_store = store;
    return record_if_due(h);
}

int spin_backward_workspace_size(const spin_params* p, int32_t K, size_t* bytes) {
    if (!bytes || K < 1) return SPIN_EINVAL;
    int v = validate(p);
    if (v != SPIN_OK) return v;
    const Tableau tb = tableau_for(p->integrator);
    *bytes = adjoint_workspace_bytes(Geom{p->nx, p->ny, p->nz}, p->precision == 64 ? 8 : 4, tb, p->path, K);
    return SPIN_OK;
}

int spin_backward(spin_lattice* h, const double dLdM[3], double dLdE, void* workspace, size_t workspace_bytes,
                  double* gJ, double* gD, double gH[3], void* g_h_site, void* g_s0) {
    if (!h || !dLdM || !gJ || !gD || !gH || !workspace) return SPIN_EINVAL;
    if (!h->rec_active) return set_err(h, SPIN_EINVAL, "no recorded trajectory (call spin_record_begin first)");
    if (h->n <= h->rec_n0 || h->n - h->rec_n0 > h->rec_max)
        return set_err(h, SPIN_EINVAL, "recorded range %lld..%lld does not end at the current step %lld",
                       h->rec_n0, h->rec_n0 + h->rec_max, h->n);
    if (reinterpret_cast<uintptr_t>(workspace) % kAlign != 0) return SPIN_EINVAL;
    size_t need = 0;
    spin_backward_workspace_size(&h->p, h->rec_K, &need);
    if (workspace_bytes < need) return SPIN_ENOSPACE;
    if (h->elt == 4) return backward_t<float>(h, dLdM, dLdE, workspace, gJ, gD, gH, g_h_site, g_s0);
    return backward_t<double>(h, dLdM, dLdE, workspace, gJ, gD, gH, g_h_site, g_s0);
}

int spin_record_end(spin_lattice* h) {
    if (!h) return SPIN_EINVAL;
    h->rec_active = false;
    return SPIN_OK;
}

int spin_lattice_destroy(spin_lattice* h) {
    if (!h) return SPIN_EINVAL;
    for (auto& level : h->graph)
        for (cudaGraphExec_t g : level)
            if (g) cudaGraphExecDestroy(g);
    if (h->capture_stream) cudaStreamDestroy(h->capture_stream);
    delete h;
    return SPIN_OK;
}

int spin_noise_draw(uint64_t seed, int64_t k, int64_t replica, int64_t n_sites, int32_t precision, uint64_t* words,
                    void* gauss, void* cuda_stream) {
    if (n_sites < 0 || k < 0 || replica < 0 || (precision != 32 && precision != 64)) return SPIN_EINVAL;
    if (n_sites == 0) return SPIN_OK;
    if (!words && !gauss) return SPIN_EINVAL;
    cudaError_t e = launch_noise_draw(seed, k, replica, n_sites, precision, words, gauss,
                                      static_cast<cudaStream_t>(cuda_stream));
    return e == cudaSuccess ? SPIN_OK : SPIN_ECUDA;
}

}  // extern "C"
