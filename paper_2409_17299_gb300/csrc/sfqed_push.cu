// K2 / K3: the per-particle QED step (arXiv:2409.17299 Sec. 3, Algorithms 1-2).
//
// One pass kernel per particle kind (sfqed_pass.cuh): the photons, then the
// leptons with everything born in the step (Algorithm 2).
#include <math.h>
#include <string.h>

#include <chrono>

#include "sfqed_device.cuh"
#include "sfqed_internal.h"

namespace sfq {
namespace {

// Gridded field: [6][nodes] (caller's layout) -> [nodes][8] (two pads)
template <class T>
__global__ void k_grid_interleave(const T *src, T *dst, long long nodes) {
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nodes) return;
#pragma unroll
    for (int c = 0; c < 6; ++c) dst[8 * n + c] = src[c * nodes + n];
    dst[8 * n + 6] = (T)0;
    dst[8 * n + 7] = (T)0;
}

// Generations of newborns in one step after which the step gives up
// (QED_ERR_TIMEOUT), unless the configuration sets another limit.
constexpr unsigned long long PASS_LIMIT = 100000;
static unsigned long long pass_limit_of(const qed_ctx *ctx) {
    return ctx->cfg.pass_limit > 0 ? (unsigned long long)ctx->cfg.pass_limit : PASS_LIMIT;
}

__device__ __forceinline__ bool ctl_stopped(const DevCtl *ctl) {
    return ctl->overflow || ctl->timeout || ctl->bad_index;
}

// Opens the next step (index ctl->step_next): its time t_n = step dt and the
// phase reduced mod 2 pi (the pass kernels read both from the control block),
// and the pass ranges: every particle present.  After an overflow or a failed
// device check the ranges are empty, so the rest of the enqueued work does
// nothing.
__global__ void k_step_begin(DevCtl *ctl, double dt) {
    const unsigned long long step = ctl->step_next;
    ctl->step_next = step + 1;
    const double t_n = (double)step * dt;
    ctl->sv_t_n = t_n;
    ctl->sv_t_red_f = (float)fmod(t_n, 2.0 * 3.14159265358979323846);
    ctl->sv_step = (unsigned)step;
    ctl->step_passes = 0;
    const bool stop = ctl_stopped(ctl);
    for (int s = 0; s < 3; ++s) {
        ctl->begin[s] = 0;
        ctl->end[s] = stop ? 0 : min(ctl->count[s], ctl->capacity[s]);
        if (s < 2) ctl->born[s] = ctl->end[s];
    }
    ctl->arrive = 0;
    ctl->spilled = 0;
}

// Opens nsteps steps taken by one launch: the leptons' ranges as in
// k_step_begin, the control block as it is after the last step.
__global__ void k_advance_step(DevCtl *ctl, double dt, unsigned long long nsteps) {
    ctl->step_next += nsteps;
    ctl->sv_step = (unsigned)(ctl->step_next - 1);
    ctl->sv_t_n = (double)(ctl->step_next - 1) * dt;
    const bool stop = ctl_stopped(ctl);
    for (int s = 0; s < 2; ++s) ctl->end[s] = stop ? 0 : min(ctl->count[s], ctl->capacity[s]);
}

__global__ void k_set_step(DevCtl *ctl, unsigned long long step) { ctl->step_next = step; }

// Copies of several arrays, one per row of blocks.  Sizes are multiples of 4
// bytes; 16 bytes at a time where both ends allow it (an optical-depth array
// is only aligned to its elements).
constexpr int COPY_MAX = 30;
struct CopyList {
    const void *src[COPY_MAX];
    void *dst[COPY_MAX];
    unsigned long long bytes[COPY_MAX];
};
__global__ void __launch_bounds__(256) k_copy_arrays(const __grid_constant__ CopyList c) {
    const int k = blockIdx.y;
    const unsigned long long t = (unsigned long long)blockIdx.x * 256 + threadIdx.x, stride = (unsigned long long)gridDim.x * 256;
    const unsigned long long words = c.bytes[k] / 4;
    unsigned long long done = 0;
    if (((reinterpret_cast<uintptr_t>(c.src[k]) | reinterpret_cast<uintptr_t>(c.dst[k])) & 15u) == 0) {
        const uint4 *s = static_cast<const uint4 *>(c.src[k]);
        uint4 *d = static_cast<uint4 *>(c.dst[k]);
        const unsigned long long n = words / 4;
        unsigned long long i = t;
        for (; i + 3 * stride < n; i += 4 * stride) {          // four 16-byte loads in flight
            const uint4 v0 = s[i], v1 = s[i + stride], v2 = s[i + 2 * stride], v3 = s[i + 3 * stride];
            d[i] = v0; d[i + stride] = v1; d[i + 2 * stride] = v2; d[i + 3 * stride] = v3;
        }
        for (; i < n; i += stride) d[i] = s[i];
        done = n * 4;
    }
    const unsigned *s = static_cast<const unsigned *>(c.src[k]);
    unsigned *d = static_cast<unsigned *>(c.dst[k]);
    for (unsigned long long i = done + t; i < words; i += stride) d[i] = s[i];
}

// ---- component kernels for the parity tests ----
__global__ void k_philox(const uint4 *ctr, long long n, uint2 key, uint4 *out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = philox4x32_10(ctr[i], key);
}

template <class T>
__global__ void k_eval_rate(const T *coef, int is_photon, const double *chi, long long n, double *F) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T c = (T)chi[i];
    F[i] = (double)(is_photon ? rate_pair<T>(coef, c) : rate_em<T>(coef, c));
}

// chi of n particles (p, E, B as n x 3 doubles) in the mode's precision
template <class T>
__global__ void k_eval_chi(int is_photon, const double *p, const double *E, const double *B, long long n,
                           double *chi, unsigned long long *n64_out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T pv[3] = {(T)p[3 * i], (T)p[3 * i + 1], (T)p[3 * i + 2]};
    const T Ev[3] = {(T)E[3 * i], (T)E[3 * i + 1], (T)E[3 * i + 2]};
    const T Bv[3] = {(T)B[3 * i], (T)B[3 * i + 1], (T)B[3 * i + 2]};
    unsigned n64 = 0;
    T c;
    if (is_photon) {
        const T k0 = m_sqrt(pv[0] * pv[0] + pv[1] * pv[1] + pv[2] * pv[2]);
        c = photon_chi<T>(k0, pv, Ev, Bv, n64);
    } else {
        T gam, p2;
        lepton_chi<T>(pv, Ev, Bv, gam, c, p2, n64);
    }
    chi[i] = (double)c;
    if (n64) atomicAdd(n64_out, (unsigned long long)n64);
}

template <class T>
__global__ void k_sample(const T *tab, int is_photon, const double *chi, const double *u, long long n,
                         double *delta, double *om) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T o;
    const T uu = (T)u[i], vv = (T)(1.0 - u[i]);
    const T d = is_photon ? sample_pair<T>(tab, (T)chi[i], uu, vv, &o) : sample_emission<T>(tab, (T)chi[i], uu, vv, &o);
    delta[i] = (double)d;
    if (om) om[i] = (double)o;
}

}  // namespace
}  // namespace sfq

using namespace sfq;

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static qed_status check_species(const qed_species &s) {
    const void *ptrs[] = {s.x, s.y, s.z, s.px, s.py, s.pz, s.w, s.id, s.nevents};
    if (s.capacity < 0 || s.count < 0 || s.count > s.capacity) return QED_ERR_INVALID;
    if (s.capacity >= (int64_t)1 << 31) return QED_ERR_INVALID;   // the pass kernels index in 31 bits
    if (s.capacity == 0) return QED_OK;
    for (const void *q : ptrs)
        if (!q || !aligned16(q)) return QED_ERR_INVALID;
    return QED_OK;
}

static qed_status ensure_tau(qed_ctx *ctx, int s, int64_t cap) {
    if (ctx->tau_cap[s] >= cap) return QED_OK;
    if (ctx->tau[s]) SFQ_CUDA(cudaFreeAsync(ctx->tau[s], ctx->stream));
    ctx->tau[s] = nullptr;
    ctx->tau_cap[s] = 0;
    if (cudaMallocAsync(&ctx->tau[s], sizeof(double) * (size_t)(cap > 0 ? cap : 1), ctx->stream) != cudaSuccess)
        return QED_ERR_NOMEM;
    ctx->tau_cap[s] = cap;
    return QED_OK;
}

static size_t elem_bytes(const qed_ctx *ctx) { return ctx->cfg.precision == QED_FP32 ? 4 : 8; }

// Save / restore the particle state at the start of a call (overflow replay):
// all arrays of all species in one launch (a copy each took 9 to 30 calls of
// a few microseconds, a third of a one-step call with 1000 electrons).
static qed_status snapshot(qed_ctx *ctx, qed_particles *p, bool restore) {
    const size_t eb = elem_bytes(ctx);
    auto room = [](size_t bytes) { return (bytes + 15) / 16 * 16; };
    size_t need = 0;
    for (int s = 0; s < 3; ++s) {
        const size_t n = (size_t)p->s[s].count;
        need += 7 * room(n * eb) + room(n * 8) + room(n * 4) + (ctx->od[s] ? room(n * eb) : 0);
    }
    if (!restore && (int64_t)need > ctx->snap_bytes) {
        if (ctx->snap) SFQ_CUDA(cudaFreeAsync(ctx->snap, ctx->stream));
        ctx->snap = nullptr;
        ctx->snap_bytes = 0;
        if (cudaMallocAsync(&ctx->snap, need + 16, ctx->stream) != cudaSuccess) return QED_ERR_NOMEM;
        ctx->snap_bytes = (int64_t)need;
    }
    if (need == 0) return QED_OK;
    char *b = static_cast<char *>(ctx->snap);
    CopyList c;
    int k = 0;
    size_t most = 0;
    auto add = [&](void *q, size_t bytes) {
        c.src[k] = restore ? b : q;
        c.dst[k] = restore ? q : b;
        c.bytes[k] = bytes;
        ++k;
        b += room(bytes);
        most = bytes > most ? bytes : most;
    };
    for (int s = 0; s < 3; ++s) {
        const qed_species &S = p->s[s];
        const size_t n = (size_t)S.count;
        if (!n) continue;
        void *arr[] = {S.x, S.y, S.z, S.px, S.py, S.pz, S.w};
        for (void *q : arr) add(q, n * eb);
        add(S.id, n * 8);
        add(S.nevents, n * 4);
        if (ctx->od[s]) add(ctx->od[s], n * eb);
    }
    // 64 bytes per thread at first, at most one wave per array
    size_t blocks = (most + 256 * 64 - 1) / (256 * 64);
    const size_t wave = (size_t)ctx->sm_count * 8;
    k_copy_arrays<<<dim3((unsigned)(blocks < wave ? blocks : wave), (unsigned)k), 256, 0, ctx->stream>>>(c);
    SFQ_LAUNCHED(ctx, 1);
    SFQ_CUDA(cudaGetLastError());
    return QED_OK;
}

static qed_status read_ctl(qed_ctx *ctx) {
    SFQ_CUDA(cudaMemcpyAsync(ctx->ctl_host, ctx->ctl, sizeof(DevCtl), cudaMemcpyDeviceToHost, ctx->stream));
    const auto t0 = std::chrono::steady_clock::now();
    SFQ_CUDA(cudaStreamSynchronize(ctx->stream));
    ctx->sync_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return QED_OK;
}

// Profiling: event pairs around the push kernels, drained into kernel_ms.
qed_status sfq_drain_events(qed_ctx *ctx) {
    for (int k = 0; k < 4; ++k) {
        for (int i = 0; i < ctx->ev_used[k]; ++i) {
            float ms = 0.f;
            SFQ_CUDA(cudaEventSynchronize(ctx->ev[k][i][1]));
            SFQ_CUDA(cudaEventElapsedTime(&ms, ctx->ev[k][i][0], ctx->ev[k][i][1]));
            ctx->kernel_ms[k] += ms;
        }
        ctx->ev_used[k] = 0;
    }
    return QED_OK;
}

static qed_status ensure_events(qed_ctx *ctx) {
    if (ctx->ev_ready) return QED_OK;
    for (int k = 0; k < 4; ++k)
        for (int i = 0; i < qed_ctx::EVN; ++i)
            for (int j = 0; j < 2; ++j) SFQ_CUDA(cudaEventCreate(&ctx->ev[k][i][j]));
    ctx->ev_ready = true;
    return QED_OK;
}

// a group of launches timed as one (compaction, leveling)
template <class F> static qed_status timed_block(qed_ctx *ctx, int which, F body) {
    if (!ctx->cfg.profile) return body();
    if (ctx->ev_used[which] == qed_ctx::EVN) {
        qed_status e = sfq_drain_events(ctx);
        if (e != QED_OK) return e;
    }
    const int i = ctx->ev_used[which]++;
    SFQ_CUDA(cudaEventRecord(ctx->ev[which][i][0], ctx->stream));
    qed_status e = body();
    SFQ_CUDA(cudaEventRecord(ctx->ev[which][i][1], ctx->stream));
    return e;
}

// the pass kernels of the field's variant (analytic descriptors or grid)
template <class T>
static qed_status launch_pass(qed_ctx *ctx, PassArgs &a, bool photons, cudaGraphConditionalHandle h = 0, int loop = 0) {
    if (a.field_kind == QED_FIELD_GRID) return pass_grid::launch_pass<T>(ctx, a, photons, h, loop);
    return pass_analytic::launch_pass<T>(ctx, a, photons, h, loop);
}

template <class T>
static qed_status launch_od(qed_ctx *ctx, PassArgs &a, bool photons) {
    if (a.field_kind == QED_FIELD_GRID) return pass_grid::launch_od<T>(ctx, a, photons);
    return pass_analytic::launch_od<T>(ctx, a, photons);
}

// ---- the captured PIC step ----
// One step as a CUDA graph: the step-begin kernel, the photon pass and the
// lepton pass (a cascade: with a while node for newborns that a full block
// list left behind, Algorithm 2), then each species' merge step (leveling and
// removal of dead entries) decided on the device.  Every kernel reads its ranges and
// the step's time from the control block, so one graph serves every step and
// no step needs the host: a batch of steps is a run of graph launches.  The
// graph is rebuilt when the bound arrays, capacities, field or step change.
struct StepGraph {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    PassArgs args;           // the kernel arguments captured (compared byte-wise)
    int64_t cap[3];
    double dt;
    int top_kernels;         // kernel nodes outside the conditional bodies
};

void sfq_step_graph_free(qed_ctx *ctx) {
    StepGraph *G = static_cast<StepGraph *>(ctx->step_graph);
    if (!G) return;
    if (G->exec) cudaGraphExecDestroy(G->exec);
    if (G->g) cudaGraphDestroy(G->g);
    delete G;
    ctx->step_graph = nullptr;
}

template <class T>
static qed_status build_step_graph(qed_ctx *ctx, const PassArgs &args, qed_particles *p, double dt, StepGraph *G) {
    const bool cascade = ctx->cfg.push_photons != 0;
    const bool od_method = ctx->cfg.event_method == QED_METHOD_OPTICAL_DEPTH;
    const bool loop = cascade && !od_method;
    GraphBuild gb;
    if (cudaGraphCreate(&gb.g, 0) != cudaSuccess) return QED_ERR_CUDA;
    gb.st = ctx->cap_stream;
    const cudaStream_t saved = ctx->stream;
    const int64_t launches = ctx->launches;
    ctx->stream = gb.st;                   // the launchers issue on ctx->stream
    PassArgs a = args;
    qed_status rc = QED_OK;
    cudaGraphConditionalHandle h_pass = 0;
    do {
        if (loop && cudaGraphConditionalHandleCreate(&h_pass, gb.g, 0, cudaGraphCondAssignDefault) != cudaSuccess) {
            rc = QED_ERR_CUDA;
            break;
        }
        cudaError_t e = gb.capture(gb.g, [&] {
            k_step_begin<<<1, 1, 0, ctx->stream>>>(ctx->ctl, dt);
            a.pass = 0;
            const qed_status q = od_method ? launch_od<T>(ctx, a, cascade)
                                           : launch_pass<T>(ctx, a, cascade, h_pass, loop ? 1 : 0);
            if (q != QED_OK) return q;
            return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
        });
        if (e != cudaSuccess) {
            rc = QED_ERR_CUDA;
            break;
        }
        gb.top_kernels = 2 + (cascade ? 1 : 0);
        if (loop) {
            cudaGraph_t body;
            if (gb.conditional(h_pass, cudaGraphCondTypeWhile, &body) != cudaSuccess) {
                rc = QED_ERR_CUDA;
                break;
            }
            e = gb.capture(body, [&] {
                a.pass = 1;
                const qed_status q = launch_pass<T>(ctx, a, true, h_pass, 1);
                if (q != QED_OK) return q;
                return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
            });
            if (e != cudaSuccess) {
                rc = QED_ERR_CUDA;
                break;
            }
        }
        // merge step (Sec. 4.2): converted photons removed, each species
        // leveled when its count exceeds the cap
        if (cascade || ctx->cfg.thin_cap > 0) {
            const int64_t bound[3] = {p->s[0].capacity, p->s[1].capacity, p->s[2].capacity};
            const int64_t before = ctx->launches;
            e = gb.capture(gb.g, [&] {
                return sfq_merge(ctx, p, bound, ctx->cfg.thin_cap > 0 ? 7 : 0, cascade ? 4 : 0, 0, true, true);
            });
            if (e != cudaSuccess) {
                rc = QED_ERR_CUDA;
                break;
            }
            gb.top_kernels += (int)(ctx->launches - before);
        }
    } while (0);
    ctx->stream = saved;
    ctx->launches = launches;
    if (rc == QED_OK && cudaGraphInstantiate(&G->exec, gb.g, 0) != cudaSuccess) rc = QED_ERR_CUDA;
    if (rc != QED_OK) {
        cudaGraphDestroy(gb.g);
        cudaGetLastError();                        // clear a failed call's error
        return rc;
    }
    G->g = gb.g;
    G->args = args;
    for (int s = 0; s < 3; ++s) G->cap[s] = p->s[s].capacity;
    G->dt = dt;
    G->top_kernels = gb.top_kernels;
    return QED_OK;
}

// The step graph for these arguments (built or rebuilt when needed), or null
// when graphs with conditional nodes are not available (host-driven steps).
template <class T>
static StepGraph *step_graph_for(qed_ctx *ctx, const PassArgs &a, qed_particles *p, double dt) {
    if (ctx->step_graph_failed) return nullptr;
    StepGraph *G = static_cast<StepGraph *>(ctx->step_graph);
    bool same = G && G->dt == dt && memcmp(&G->args, &a, sizeof(PassArgs)) == 0;
    for (int s = 0; same && s < 3; ++s) same = G->cap[s] == p->s[s].capacity;
    if (same) return G;
    sfq_step_graph_free(ctx);
    G = new StepGraph;
    if (build_step_graph<T>(ctx, a, p, dt, G) != QED_OK) {
        delete G;
        ctx->step_graph_failed = 1;
        return nullptr;
    }
    ctx->step_graph = G;
    return G;
}

// Host-driven steps: the same kernels launched one by one, the host reading
// the control block after the passes, before the merge step.
// Used to time the kernels individually (cfg.profile: CUDA events around
// each launch) and where graphs with conditional nodes are unavailable.
template <class T>
static qed_status host_steps(qed_ctx *ctx, qed_particles *pw, PassArgs &a, double dt, int nsteps) {
    const bool cascade = ctx->cfg.push_photons != 0;
    const bool od_method = ctx->cfg.event_method == QED_METHOD_OPTICAL_DEPTH;
    qed_particles P = *pw;                         // counts below: bounds read back from the device
    for (int it = 0; it < nsteps; ++it) {
        a.pass = 0;
        k_step_begin<<<1, 1, 0, ctx->stream>>>(ctx->ctl, dt);
        SFQ_LAUNCHED(ctx, 1);
        qed_status e = od_method ? launch_od<T>(ctx, a, cascade) : launch_pass<T>(ctx, a, cascade);
        if (e != QED_OK) return e;
        if (cascade && !od_method) {
            // newborns left behind by a full block list take further launches
            for (a.pass = 1;; ++a.pass) {
                e = read_ctl(ctx);
                if (e != QED_OK) return e;
                if (!ctx->ctl_host->more) break;
                e = launch_pass<T>(ctx, a, true);
                if (e != QED_OK) return e;
            }
        }
        if (cascade || ctx->cfg.thin_cap > 0) {
            // merge step (Sec. 4.2): drop dead photons, then level
            if (!cascade || od_method) {
                e = read_ctl(ctx);
                if (e != QED_OK) return e;
            }
            const DevCtl &c = *ctx->ctl_host;
            if (c.overflow || c.timeout || c.bad_index) break;
            bool level = false;
            int64_t bound[3];
            for (int s = 0; s < 3; ++s) {
                bound[s] = P.s[s].capacity;
                level = level || (ctx->cfg.thin_cap > 0 && (int64_t)c.count[s] > ctx->cfg.thin_cap);
            }
            qed_status e2 = timed_block(ctx, level ? 3 : 2, [&] {
                return sfq_merge(ctx, &P, bound, ctx->cfg.thin_cap > 0 ? 7 : 0, cascade ? 4 : 0, 0, true, true);
            });
            if (e2 != QED_OK) return e2;
        }
    }
    return QED_OK;
}

// Opens a batch of steps: the counts and capacities of *p go to the device
// control block (staged in pinned memory), the context's per-particle work
// buffers grow to the capacities, and with restore_on_overflow the particle
// state is copied aside.
static qed_status open_batch(qed_ctx *ctx, qed_particles *p, int64_t step0) {
    ctx->launches = 0;
    ctx->sync_ms = 0.0;
    for (int k = 0; k < 4; ++k) ctx->kernel_ms[k] = 0.0;
    ctx->async_t0_ms = std::chrono::duration<double, std::milli>(
        std::chrono::steady_clock::now().time_since_epoch()).count();
    if (ctx->cfg.profile) {
        qed_status e = ensure_events(ctx);
        if (e != QED_OK) return e;
    }
    DevCtl &h = *ctx->ctl_up;
    memset(&h, 0, sizeof(DevCtl));
    for (int s = 0; s < 3; ++s) {
        h.count[s] = (unsigned long long)p->s[s].count;
        h.capacity[s] = (unsigned long long)p->s[s].capacity;
    }
    h.step_next = (unsigned long long)step0;
    h.pass_limit = pass_limit_of(ctx);
    SFQ_CUDA(cudaMemcpyAsync(ctx->ctl, &h, sizeof(DevCtl), cudaMemcpyHostToDevice, ctx->stream));
    int64_t bound[3];
    for (int s = 0; s < 3; ++s) {
        qed_status e = s < 2 ? ensure_tau(ctx, s, p->s[s].capacity) : QED_OK;
        if (e != QED_OK) return e;
        bound[s] = p->s[s].capacity;
    }
    // compaction work buffers sized once for the capacities
    qed_status e = sfq_ensure_merge(ctx, bound);
    if (e != QED_OK) return e;
    if (ctx->cfg.restore_on_overflow) {
        e = snapshot(ctx, p, false);
        if (e != QED_OK) return e;
    }
    ctx->async_p = *p;
    ctx->async_deferred = 0;
    for (int s = 0; s < 3; ++s) ctx->async_count0[s] = p->s[s].count;
    ctx->async_next_step = step0;
    ctx->async_open = 1;
    return QED_OK;
}

static bool same_binding(const qed_particles &a, const qed_particles &b) {
    for (int s = 0; s < 3; ++s) {
        const qed_species &x = a.s[s], &y = b.s[s];
        if (x.x != y.x || x.y != y.y || x.z != y.z || x.px != y.px || x.py != y.py || x.pz != y.pz || x.w != y.w ||
            x.id != y.id || x.nevents != y.nevents || x.capacity != y.capacity)
            return false;
    }
    return true;
}

// Enqueue nsteps steps of the open batch (no host wait on the graph path).
template <class T>
static qed_status enqueue_steps(qed_ctx *ctx, const qed_field_desc *field, double dt, int nsteps, int64_t step0) {
    qed_particles *p = &ctx->async_p;
    const bool cascade = ctx->cfg.push_photons != 0;
    if (step0 != ctx->async_next_step) {
        k_set_step<<<1, 1, 0, ctx->stream>>>(ctx->ctl, (unsigned long long)step0);
        SFQ_LAUNCHED(ctx, 1);
    }
    ctx->async_next_step = step0 + nsteps;
    if (nsteps == 0) return QED_OK;
    PassArgs a;
    memset(&a, 0, sizeof a);                       // padding included: the graph key compares bytes
    for (int s = 0; s < 3; ++s) {
        const qed_species &S = p->s[s];
        a.sp[s] = SpeciesDev{S.x, S.y, S.z, S.px, S.py, S.pz, S.w,
                             reinterpret_cast<unsigned long long *>(S.id), S.nevents, s < 2 ? ctx->tau[s] : nullptr,
                             ctx->od[s]};
    }
    const int64_t bound[3] = {p->s[0].capacity, p->s[1].capacity, p->s[2].capacity};
    for (int s = 0; s < 2; ++s) a.gen[s] = sfq_entry_words(ctx, bound, s);
    a.ctl = ctx->ctl;
    const bool f32 = sizeof(T) == 4;
    a.coef = f32 ? (const void *)ctx->coef32 : (const void *)ctx->coef64;
    a.coef32 = ctx->coef32;
    a.icdf_em = f32 ? (const void *)ctx->icdf_em32 : (const void *)ctx->icdf_em64;
    a.icdf_pair = f32 ? (const void *)ctx->icdf_pair32 : (const void *)ctx->icdf_pair64;
    a.mlp_w16 = ctx->cfg.sampler == QED_SAMPLER_MLP ? ctx->mlp_w16 : nullptr;
    a.field_kind = field->kind;
    if (field->kind == QED_FIELD_GRID) {
        long long nodes = 1;
        for (int d = 0; d < 3; ++d) {
            a.gn[d] = (int)field->params[d];
            a.ginv[d] = (double)a.gn[d] / field->params[3 + d];
            a.ginv_f[d] = (float)a.ginv[d];
            nodes *= a.gn[d];
        }
        // the caller's [component][node] values, interleaved per node for the
        // kernels (the grid is constant during the call)
        const size_t bytes = (size_t)nodes * 8 * sizeof(T);
        if (ctx->grid_il_bytes < bytes) {
            if (ctx->grid_il) SFQ_CUDA(cudaFreeAsync(ctx->grid_il, ctx->stream));
            ctx->grid_il = nullptr;
            ctx->grid_il_bytes = 0;
            if (cudaMallocAsync(&ctx->grid_il, bytes, ctx->stream) != cudaSuccess) return QED_ERR_NOMEM;
            ctx->grid_il_bytes = bytes;
        }
        k_grid_interleave<T><<<(unsigned)((nodes + 255) / 256), 256, 0, ctx->stream>>>(
            reinterpret_cast<const T *>(ctx->field_grid), reinterpret_cast<T *>(ctx->grid_il), nodes);
        SFQ_LAUNCHED(ctx, 1);
        SFQ_CUDA(cudaGetLastError());
        a.grid_il = ctx->grid_il;
    }
    a.field_zero = field_zero_of(*field);      // chi without its cancellation guard where allowed
    for (int i = 0; i < 6; ++i) {
        a.prm[i] = field->params[i];
        a.prm_f[i] = (float)field->params[i];
    }
    a.dt = dt;
    a.dt_f = (float)dt;
    a.lam_skip = ldexp(1.0, -54) / dt;
    a.lam_skip_f = (float)a.lam_skip;
    a.dt_f_gt = (double)a.dt_f > dt ? a.dt_f : nextafterf(a.dt_f, INFINITY);
    a.seed = ctx->cfg.seed;
    a.keys = philox_keys(ctx->cfg.seed);
    a.child_keys = philox_keys(ctx->cfg.seed ^ CHILD_KEY_XOR);
    a.soft_filter = ctx->cfg.soft_photon_filter;
    a.fly_newborns = cascade && ctx->cfg.event_method == QED_METHOD_SUBSTEP ? 1 : 0;

    ctx->async_deferred = 1;
    if (!cascade && ctx->cfg.thin_cap == 0 && ctx->cfg.event_method == QED_METHOD_SUBSTEP && !a.mlp_w16 && nsteps > 1 &&
        ctx->cfg.restore_on_overflow) {
        // An emission run of several steps: one launch for all of them, where
        // the leptons (their count does not change) are few enough for that to
        // pay.  Its blocks cannot stop at the step in which the photons run
        // out of room, so it is taken where the state goes back to the batch's
        // start then; the demand it counts is that of all its steps.
        const bool grid = field->kind == QED_FIELD_GRID;
        const int64_t n = p->s[0].count + p->s[1].count;
        const int blocks = grid ? pass_grid::steps_blocks<T>(ctx, n, nsteps) : pass_analytic::steps_blocks<T>(ctx, n, nsteps);
        if (blocks > 0) {
            a.pass = 0;
            k_advance_step<<<1, 1, 0, ctx->stream>>>(ctx->ctl, dt, (unsigned long long)nsteps);
            SFQ_LAUNCHED(ctx, 1);
            return grid ? pass_grid::launch_steps<T>(ctx, a, step0, nsteps, blocks)
                        : pass_analytic::launch_steps<T>(ctx, a, step0, nsteps, blocks);
        }
    }
    StepGraph *G = ctx->cfg.profile ? nullptr : step_graph_for<T>(ctx, a, p, dt);
    if (!G) return host_steps<T>(ctx, p, a, dt, nsteps);
    for (int it = 0; it < nsteps; ++it) SFQ_CUDA(cudaGraphLaunch(G->exec, ctx->stream));
    SFQ_LAUNCHED(ctx, (int64_t)nsteps * G->top_kernels);
    return QED_OK;
}

// Ends the open batch: reads the control block back (the one wait), fills the
// statistics, updates the counts of *p (or restores the state at the batch's
// start after an overflow, with restore_on_overflow).
static qed_status wait_batch(qed_ctx *ctx, qed_particles *p, qed_stats *out) {
    if (ctx->async_deferred) {
        // the steps may have left dead entries in place: remove them, so the
        // counts returned hold live particles only (after a step that ran out
        // of capacity nothing is moved)
        ctx->async_deferred = 0;
        const qed_particles &B = ctx->async_p;
        const int64_t bound[3] = {B.s[0].capacity, B.s[1].capacity, B.s[2].capacity};
        qed_status e = sfq_merge(ctx, &B, bound, 0, 7, 0, false, false);
        if (e != QED_OK) {
            ctx->async_open = 0;
            return e;
        }
    }
    qed_status e = read_ctl(ctx);
    ctx->async_open = 0;
    if (e != QED_OK) return e;
    DevCtl &c = *ctx->ctl_host;
    qed_status rc = QED_OK;
    if (c.overflow) rc = QED_ERR_CAPACITY;
    if (c.timeout) rc = QED_ERR_TIMEOUT;
    if (c.bad_index) rc = QED_ERR_STATE;
    qed_stats st{};
    st.particle_steps = (int64_t)c.particle_steps;
    st.emit_events = (int64_t)c.emit_events;
    st.pair_events = (int64_t)c.pair_events;
    for (int s = 0; s < 3; ++s) st.needed_capacity[s] = (int64_t)c.needed[s];
    st.max_subevents = (int64_t)c.max_subevents;
    st.overflow = (int64_t)c.overflow;
    st.passes = (int64_t)c.passes;
    st.thinned = (int64_t)c.thinned;
    st.moved = (int64_t)c.moved;
    st.lepton_steps = (int64_t)c.lepton_steps;
    st.chi_fp64 = (int64_t)c.chi_fp64;
    st.photon_steps = (int64_t)c.photon_steps;
    if (ctx->cfg.profile) {
        e = sfq_drain_events(ctx);
        if (e != QED_OK) return e;
    }
    for (int k = 0; k < 4; ++k) st.kernel_ms[k] = ctx->kernel_ms[k];
    st.launches = ctx->launches + (int64_t)c.graph_kernels;
    st.sync_ms = ctx->sync_ms;
    st.call_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now().time_since_epoch())
                     .count() - ctx->async_t0_ms;
    qed_particles &B = ctx->async_p;
    if (rc == QED_ERR_CAPACITY && ctx->cfg.restore_on_overflow) {
        for (int s = 0; s < 3; ++s) B.s[s].count = ctx->async_count0[s];
        e = snapshot(ctx, &B, true);
        if (e != QED_OK) return e;
        SFQ_CUDA(cudaStreamSynchronize(ctx->stream));
    } else {
        for (int s = 0; s < 3; ++s) B.s[s].count = (int64_t)min(c.count[s], c.capacity[s]);
    }
    for (int s = 0; s < 3; ++s) p->s[s].count = B.s[s].count;
    if (out) *out = st;
    ctx->acc.particle_steps += st.particle_steps;
    ctx->acc.emit_events += st.emit_events;
    ctx->acc.pair_events += st.pair_events;
    ctx->acc.passes += st.passes;
    ctx->acc.thinned += st.thinned;
    ctx->acc.moved += st.moved;
    ctx->acc.lepton_steps += st.lepton_steps;
    ctx->acc.chi_fp64 += st.chi_fp64;
    ctx->acc.photon_steps += st.photon_steps;
    ctx->acc.launches += st.launches;
    for (int k = 0; k < 4; ++k) ctx->acc.kernel_ms[k] += st.kernel_ms[k];
    ctx->acc.sync_ms += st.sync_ms;
    ctx->acc.call_ms += st.call_ms;
    if (st.max_subevents > ctx->acc.max_subevents) ctx->acc.max_subevents = st.max_subevents;
    return rc;
}

static qed_status check_push_args(qed_ctx *ctx, qed_particles *p, const qed_field_desc *field, double dt, int nsteps,
                                  int64_t step0) {
    if (!ctx || !p || !field || nsteps < 0 || !(dt > 0.0) || step0 < 0 || step0 + nsteps > 0xFFFFFFFFll)
        return QED_ERR_INVALID;
    if (ctx->cfg.sampler == QED_SAMPLER_MLP && !ctx->mlp_ready) return QED_ERR_STATE;
    if (field->kind < QED_FIELD_UNIFORM || field->kind > QED_FIELD_GRID) return QED_ERR_INVALID;
    if (ctx->cfg.event_method == QED_METHOD_OPTICAL_DEPTH) {
        for (int s = 0; s < 3; ++s)
            if (p->s[s].capacity > 0 && !ctx->od[s]) return QED_ERR_STATE;   // qed_set_optical_depth first
        if (ctx->cfg.sampler == QED_SAMPLER_MLP) return QED_ERR_INVALID;     // the table sampler only
    } else if (ctx->cfg.event_method != QED_METHOD_SUBSTEP) {
        return QED_ERR_INVALID;
    }
    if (field->kind == QED_FIELD_GRID) {
        if (!ctx->field_grid) return QED_ERR_STATE;
        for (int d = 0; d < 3; ++d) {
            const double n = field->params[d], len = field->params[3 + d];
            if (!(n >= 1.0 && n <= 65536.0 && n == floor(n)) || !(len > 0.0)) return QED_ERR_INVALID;
        }
    }
    if (ctx->async_open) return same_binding(ctx->async_p, *p) ? QED_OK : QED_ERR_STATE;
    for (int s = 0; s < 3; ++s) {
        qed_status e = check_species(p->s[s]);
        if (e != QED_OK) return e;
    }
    return QED_OK;
}

qed_status sfq_push_async(qed_ctx *ctx, qed_particles *p, const qed_field_desc *field, double dt, int nsteps,
                          int64_t step0) {
    qed_status e = check_push_args(ctx, p, field, dt, nsteps, step0);
    if (e != QED_OK) return e;
    if (!ctx->async_open) {
        e = open_batch(ctx, p, step0);
        if (e != QED_OK) return e;
    }
    if (ctx->cfg.precision == QED_FP32) return enqueue_steps<float>(ctx, field, dt, nsteps, step0);
    return enqueue_steps<double>(ctx, field, dt, nsteps, step0);
}

qed_status sfq_push_wait(qed_ctx *ctx, qed_particles *p, qed_stats *out) {
    if (!ctx || !p) return QED_ERR_INVALID;
    if (!ctx->async_open) return QED_ERR_STATE;
    if (!same_binding(ctx->async_p, *p)) return QED_ERR_STATE;
    return wait_batch(ctx, p, out);
}

qed_status sfq_push(qed_ctx *ctx, qed_particles *p, const qed_field_desc *field, double dt, int nsteps,
                    int64_t step0, qed_stats *out) {
    const bool opened = ctx && !ctx->async_open;
    qed_status e = sfq_push_async(ctx, p, field, dt, nsteps, step0);
    if (e != QED_OK) {
        // a batch this call opened is closed again (its work is drained)
        if (opened && ctx->async_open) {
            qed_stats tmp;
            wait_batch(ctx, p, &tmp);
        }
        return e;
    }
    return wait_batch(ctx, p, out);
}

qed_status sfq_philox(const uint32_t *ctr, int64_t n, uint64_t key, uint32_t *out, cudaStream_t s) {
    if (n < 0 || (n > 0 && (!ctr || !out))) return QED_ERR_INVALID;
    if (!aligned16(ctr) || !aligned16(out)) return QED_ERR_INVALID;
    if (n == 0) return QED_OK;
    k_philox<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(reinterpret_cast<const uint4 *>(ctr), n,
                                                         make_uint2((uint32_t)key, (uint32_t)(key >> 32)),
                                                         reinterpret_cast<uint4 *>(out));
    SFQ_CUDA(cudaGetLastError());
    SFQ_CUDA(cudaStreamSynchronize(s));
    return QED_OK;
}

qed_status sfq_eval_rate(qed_ctx *ctx, int is_photon, const double *chi, int64_t n, double *F) {
    if (!ctx || n < 0 || (n > 0 && (!chi || !F))) return QED_ERR_INVALID;
    if (n == 0) return QED_OK;
    const unsigned g = (unsigned)((n + 255) / 256);
    if (ctx->cfg.precision == QED_FP32) k_eval_rate<float><<<g, 256, 0, ctx->stream>>>(ctx->coef32, is_photon, chi, n, F);
    else k_eval_rate<double><<<g, 256, 0, ctx->stream>>>(ctx->coef64, is_photon, chi, n, F);
    SFQ_CUDA(cudaGetLastError());
    SFQ_CUDA(cudaStreamSynchronize(ctx->stream));
    return QED_OK;
}

qed_status sfq_eval_chi(qed_ctx *ctx, int is_photon, const double *p, const double *E, const double *B, int64_t n,
                        double *chi, int64_t *n_fp64) {
    if (!ctx || n < 0 || (n > 0 && (!p || !E || !B || !chi))) return QED_ERR_INVALID;
    if (n_fp64) *n_fp64 = 0;
    if (n == 0) return QED_OK;
    const unsigned g = (unsigned)((n + 255) / 256);
    unsigned long long *cnt = &ctx->ctl->chi_fp64;
    SFQ_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), ctx->stream));
    if (ctx->cfg.precision == QED_FP32) k_eval_chi<float><<<g, 256, 0, ctx->stream>>>(is_photon, p, E, B, n, chi, cnt);
    else k_eval_chi<double><<<g, 256, 0, ctx->stream>>>(is_photon, p, E, B, n, chi, cnt);
    SFQ_CUDA(cudaGetLastError());
    unsigned long long h = 0;
    SFQ_CUDA(cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    SFQ_CUDA(cudaStreamSynchronize(ctx->stream));
    if (n_fp64) *n_fp64 = (int64_t)h;
    return QED_OK;
}

qed_status sfq_sample(qed_ctx *ctx, int is_photon, const double *chi, const double *u, int64_t n, double *delta,
                      double *one_minus) {
    if (!ctx || n < 0 || (n > 0 && (!chi || !u || !delta))) return QED_ERR_INVALID;
    if (n == 0) return QED_OK;
    const unsigned g = (unsigned)((n + 255) / 256);
    if (ctx->cfg.precision == QED_FP32)
        k_sample<float><<<g, 256, 0, ctx->stream>>>(is_photon ? ctx->icdf_pair32 : ctx->icdf_em32, is_photon, chi, u,
                                                    n, delta, one_minus);
    else
        k_sample<double><<<g, 256, 0, ctx->stream>>>(is_photon ? ctx->icdf_pair64 : ctx->icdf_em64, is_photon, chi,
                                                     u, n, delta, one_minus);
    SFQ_CUDA(cudaGetLastError());
    SFQ_CUDA(cudaStreamSynchronize(ctx->stream));
    return QED_OK;
}
