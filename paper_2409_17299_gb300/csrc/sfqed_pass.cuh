// The pass kernels of the per-particle QED step (arXiv:2409.17299 Sec. 3,
// Algorithms 1-2) and their launcher, compiled twice: once for the analytic
// field descriptors (SFQ_GRID 0) and once for the gridded field (SFQ_GRID 1),
// each into its own namespace (SFQ_PASS_NS), so neither variant carries the
// other's field code or registers.
//
// One pass kernel per particle kind.  Each thread takes one particle of the
// pass range (grid-stride), runs Algorithm 1 for it to the end of the step
// (rate -> waiting time -> Boris push -> event), and appends every particle
// it creates with a warp-aggregated atomic.
//
// Algorithm 2 (newborns are pushed to the end of their birth step) takes no
// sweeps of its own: draws are keyed by id, so the order in which newborns
// are pushed does not matter.  The photon pass runs first; the pairs it
// creates carry their birth clock and are taken up by the lepton pass behind
// the step-start leptons.  In the lepton pass a new photon flies to the step
// end at once, in the thread that emitted it (the field at the emission point
// is at hand, and the photon's record is written once, at its final place),
// and the leptons of a pair it creates go to the block's queue.  Sweeping the
// newborns in passes of their own took 3 to 5 further passes over each
// species per step, each two or three launches and a read and a write of
// every newborn (standing-wave cascade, 1e7 particles per species: 0.26 of
// 1.9 ms per step; at 5e5 photons 44 of 145 us).  20 steps at the start of a
// cascade (1e5 leptons) 3.36 -> 2.86 ms, 40 steps with the network sampler at
// 1e7 photons 34.3 -> 30.0 ms, with the table at 5e7 88.8 -> 87.0 ms, of the
// standing wave at 1e7 per species 89.6 -> 88.2 ms.  Only when a block's queue
// is full do newborn leptons wait for a further launch of the lepton pass.
#pragma once

#include <math.h>
#include <string.h>

#include "sfqed_device.cuh"
#include "sfqed_internal.h"
#include "sfqed_mma.cuh"

#if !defined(SFQ_GRID) || !defined(SFQ_PASS_NS)
#error "define SFQ_GRID and SFQ_PASS_NS before including sfqed_pass.cuh"
#endif

namespace sfq {
namespace SFQ_PASS_NS {

// the field at a particle: the gridded field in the grid variant, the
// analytic descriptor otherwise
template <class T>
__device__ __forceinline__ void field_at(const PassArgs &a, const T x[3], const Phase<T> &ph, T E[3], T B[3]) {
#if SFQ_GRID
    (void)ph;
    eval_grid<T, PassArgs>(a, x, E, B);
#else
    eval_field_at<T, PassArgs>(a, x, ph, E, B);
#endif
}

template <class T>
__device__ __forceinline__ void field_tau(const PassArgs &a, const StepTime &tm, const T x[3], double tau, T E[3],
                                          T B[3]) {
#if SFQ_GRID
    (void)tau;
    (void)tm;
    eval_grid<T, PassArgs>(a, x, E, B);
#else
    eval_field_at<T, PassArgs>(a, x, time_phase<T, StepTime>(tm, tau), E, B);
#endif
}

// The current step's time and index, written into the control block by the
// step-begin kernel (so a step captured in a CUDA graph takes no per-step
// kernel arguments)
__device__ __forceinline__ StepTime load_step_time(const PassArgs &a) {
    const DevCtl *c = a.ctl;
    StepTime t;
    t.field_kind = a.field_kind;
    t.t_n = c->sv_t_n;
    t.t_n_red_f = c->sv_t_red_f;
    t.step = c->sv_step;
    return t;
}

// tau < dt for the clock's non-negative doubles, as an integer comparison of
// their bit patterns (which order like the values): no FP64 instruction
__device__ __forceinline__ bool before_step_end(double tau, double dt) {
    return __double_as_longlong(tau) < __double_as_longlong(dt);
}

// the step in the working precision (FP32: rounded once on the host)
template <class T> __device__ __forceinline__ T dt_of(const PassArgs &a);
template <> __device__ __forceinline__ float dt_of<float>(const PassArgs &a) { return a.dt_f; }
template <> __device__ __forceinline__ double dt_of<double>(const PassArgs &a) { return a.dt; }

template <class T> __device__ __forceinline__ T t_inf();
template <> __device__ __forceinline__ double t_inf<double>() { return __longlong_as_double(0x7ff0000000000000ll); }
template <> __device__ __forceinline__ float t_inf<float>() { return __int_as_float(0x7f800000); }

// Statistics of one thread: particles pushed and events of each kind.
struct PassStats {
    unsigned long long lep = 0, ph = 0, em = 0, pr = 0;
    unsigned mx = 0, n64 = 0, gen = 0;
};

__device__ __forceinline__ void flush_stats(DevCtl *ctl, PassStats s) {
    // called by every lane of the warp after the grid-stride loop
    for (int o = 16; o > 0; o >>= 1) {
        s.lep += __shfl_down_sync(0xffffffffu, s.lep, o);
        s.ph += __shfl_down_sync(0xffffffffu, s.ph, o);
        s.em += __shfl_down_sync(0xffffffffu, s.em, o);
        s.pr += __shfl_down_sync(0xffffffffu, s.pr, o);
        s.mx = max(s.mx, __shfl_down_sync(0xffffffffu, s.mx, o));
        s.n64 += __shfl_down_sync(0xffffffffu, s.n64, o);
        s.gen = max(s.gen, __shfl_down_sync(0xffffffffu, s.gen, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (s.n64) atomicAdd(&ctl->chi_fp64, (unsigned long long)s.n64);
        if (s.lep + s.ph) atomicAdd(&ctl->particle_steps, s.lep + s.ph);
        if (s.lep) atomicAdd(&ctl->lepton_steps, s.lep);
        if (s.ph) atomicAdd(&ctl->photon_steps, s.ph);
        if (s.em) atomicAdd(&ctl->emit_events, s.em);
        if (s.pr) atomicAdd(&ctl->pair_events, s.pr);
        if (s.mx) atomicMax(&ctl->max_subevents, (unsigned long long)s.mx);
        if (s.gen) atomicMax(&ctl->step_passes, (unsigned long long)s.gen);
    }
}

// True in every thread of the block that finishes last in its launch; what
// the other blocks wrote is then visible.  Called once per block, by all its
// threads.
__device__ __forceinline__ bool last_block(DevCtl *ctl) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(&ctl->arrive, 1ull) == gridDim.x - 1;
        if (s_last) ctl->arrive = 0;
        __threadfence();
    }
    __syncthreads();
    return s_last != 0;
}

__device__ __forceinline__ unsigned long long count_now(DevCtl *ctl, int s) {
    const unsigned long long c = __ldcg(&ctl->count[s]);
    return c < ctl->capacity[s] ? c : ctl->capacity[s];
}

// chi and energy of a lepton / photon in the mode's precision: FP64 mode uses
// the direct FP64 form; FP32 mode the guarded form with FP64 fallback.
__device__ __forceinline__ void note_overflow(DevCtl *ctl, int s, unsigned long long slot) {
    atomicMax(&ctl->needed[s], slot + 1);
    atomicExch(&ctl->overflow, 1ull);
}

// Algorithm 1 for electrons and positrons (both species of one pass).
//
// Divergence control (the GPU form of Algorithm 3's "sort handled particles
// to the front"): phase 1 pushes every particle of a tile (one per thread) to
// its first event or to the end of the step; particles at an event go to
// a per-block stack in shared memory.  Whenever the stack holds a full round,
// the block pops one item per thread and processes it densely: the event
// (chi at the point, energy draw, recoil, the photon's flight), then the next
// waiting time, ending either at the step end (state stored) or at the next
// event (pushed back).  The stack is drained after the last tile.  Newborn
// leptons enter the stack at their birth clock, without an event pending.
//
// Threads per block of the lepton pass: 256 in FP32, three blocks per SM (four
// would spill the photon's flight: 2.5% slower at 5e7 photons).  In FP64 128:
// the pass is bound by the FP64 pipe, which a few warps keep busy, and
// smaller blocks spread a small ensemble over more SMs (16384 electrons, one
// step: 87 us at 256 threads, 79 us at 128).
template <class T> constexpr int LB = sizeof(T) == 4 ? 256 : 128;
constexpr unsigned RESUME = 0x80000000u;   // stack item flag: no event pending (a newborn at its birth clock)
constexpr unsigned START = 0x40000000u;    // with it: a lepton at the step start (its first waiting time to be drawn)

template <class T> struct LeptonStack {
    static constexpr int Q = 2 * LB<T>;    // items: < LB left + LB pushed
    T x[3][Q], p[3][Q];
    double tau[Q];
    unsigned long long id[Q];
    T w[Q];
    unsigned idx[Q];               // index | species << 31
    unsigned k[Q];                 // events so far in this step (the pending one not counted)
    unsigned gen[Q];               // generation within the step (0: present at its start) | RESUME
    uint2 r[Q];                    // the pending event's energy draw words
    // newborn leptons of this block's photons, not on the stack yet (their
    // state is in the species arrays)
    unsigned nb_idx[LB<T>], nb_gen[LB<T>];
    // items pushed in iteration i of the block's loop are counted in
    // pushed[i mod 3]: the stack's size is then a uniform register value, no
    // thread reads a counter that another may already be adding to, and the
    // counter of iteration i + 1 is cleared in iteration i
    int pushed[3], nb_pushed[3];
};

// the block's view of its stack in one iteration
struct StackPos {
    int n;        // stack items below this iteration's pushes
    int nb;       // waiting newborns
    int it;       // iteration mod 3
};

template <class T> struct LeptonCtx {
    const PassArgs &a;
    DevCtl *ctl;
    const T *coef;
    const float *coef32;    // FP64 mode: the FP32 rate pieces (surely_flies)
    const T *icdf;
    unsigned long long cap_ph;
    unsigned gen_limit;     // generations a step may run (then it is marked as timed out)
    T alpha_r;
    const StepTime &tm;     // the step's time and index (block's shared copy)
    Phase<T> ph0;           // time phase at the step start (tau = 0)
};

// A rate below 2^-54 / dt cannot give an event in a step: the waiting time
// -ln u / lambda is at least 2^-53 / lambda > 2 dt, because 1 - u is never
// below 2^-53 (FP64 and FP32 draws alike).  Such particles skip the draw (no
// draw is consumed without an event, so the counter sequence is unchanged);
// in the cascades this is most photons with chi below ~0.1.
template <class T> __device__ __forceinline__ T lam_skip(const PassArgs &a);
template <> __device__ __forceinline__ float lam_skip<float>(const PassArgs &a) { return a.lam_skip_f; }
template <> __device__ __forceinline__ double lam_skip<double>(const PassArgs &a) { return a.lam_skip; }

// One waiting-time iteration from (x, p, tau).  Returns true and leaves the
// particle at its event point (tau advanced, draw words in rz) if an event
// happens before the step end, else pushes it to the end and returns false.
// FRESH: tau == 0 (first iteration of a particle present at the step start);
// then the event test "0 + dt_hat > dt" and the push length need no FP64
// instruction in FP32 mode (the smallest float above dt decides exactly).
template <class T, bool FRESH>
__device__ __forceinline__ bool advance(const LeptonCtx<T> &c, T x[3], T p[3], T q, double &tau,
                                        unsigned long long id, unsigned k, uint2 &rz, unsigned &n64) {
    const PassArgs &a = c.a;
    T E[3], B[3];
    if constexpr (FRESH) field_at<T>(a, x, c.ph0, E, B);
    else field_tau<T>(a, c.tm, x, tau, E, B);
    T gam, chi, p2;
    // in a round the copy of this code depends on what surrounds it: its sums
    // are rounded explicitly
    lepton_chi<T, !FRESH || sizeof(T) == 8>(p, E, B, gam, chi, p2, n64, a.field_zero);
    const T lam = p2 > (T)0 ? f_div(c.alpha_r, gam) * rate_em<T>(c.coef, chi) : (T)0;
    T dth = t_inf<T>();
    if (lam > lam_skip<T>(a)) {
        const uint4 r = event_draw(a.keys, id, c.tm.step, k);
        T uw, vw;
        Uniform<T>::draw(r.x, r.y, uw, vw);
        dth = f_div(Uniform<T>::neglog(uw, vw), lam);
        rz = make_uint2(r.z, r.w);
    }
    bool no_event;
    T h;
    if constexpr (FRESH && sizeof(T) == 4) { no_event = dth >= a.dt_f_gt; h = a.dt_f; }
    else if constexpr (FRESH) { no_event = dth > a.dt; h = a.dt; }
    else if constexpr (sizeof(T) == 4) {
        // FP32 mode after a particle's first event: the FP64 test
        // tau + dth > dt decided in FP32 wherever dth lies outside a margin
        // around the remaining time rem = dt - tau (rounded once to float);
        // the margin (2^-20 rem + 2^-40 dt) exceeds every rounding involved,
        // so the decision is the FP64 one, and within it the FP64 test runs
        const float rf = __double2float_rn(a.dt - tau);
        const float marg = fmaf(rf, 0x1p-20f, a.dt_f * 0x1p-40f);
        if (dth > rf + marg) no_event = true;
        else if (dth < rf - marg) no_event = false;
        else no_event = tau + (double)dth > a.dt;
        h = rf;
    } else { no_event = tau + (double)dth > a.dt; h = (T)(a.dt - tau); }
    if (no_event) {
        boris<T>(x, p, q, E, B, h, a.field_zero == 1, id, c.tm.step, k);
        tau = a.dt;
        return false;
    }
    boris<T>(x, p, q, E, B, dth, a.field_zero == 1, id, c.tm.step, k);
    if constexpr (FRESH) tau = (double)dth;
    else tau += (double)dth;
    return true;
}

// Kinematics of an emission with photon fraction delta (and 1 - delta) from a
// lepton of energy gam and momentum p: collinear, energy-conserving recoil.
// Returns whether the photon is kept, its momentum in kv.
template <class T>
__device__ __forceinline__ bool recoil(const PassArgs &a, T p[3], T gam, T p2, T delta, T om, T kv[3]) {
    T g_after = om * gam, k0 = delta * gam;
    if (g_after < (T)1) { g_after = (T)1; k0 = gam - (T)1; }
    const T inv = f_rsqrt(p2);
    const T nx = p[0] * inv, ny = p[1] * inv, nz = p[2] * inv;
    const T pa = f_sqrt((g_after - (T)1) * (g_after + (T)1));
    kv[0] = k0 * nx; kv[1] = k0 * ny; kv[2] = k0 * nz;
    p[0] = pa * nx; p[1] = pa * ny; p[2] = pa * nz;
    return !(a.soft_filter && k0 < (T)2);
}

template <class T>
__device__ __forceinline__ void append_photon(const PassArgs &a, DevCtl *ctl, unsigned long long cap, const T x[3],
                                              const T kv[3], T w, uint4 rid) {
    const unsigned long long slot = warp_append(&ctl->count[2], 1);
    if (slot < cap) {
        const SpeciesDev &P = a.sp[2];
        st<T>(P.x, slot, x[0]); st<T>(P.y, slot, x[1]); st<T>(P.z, slot, x[2]);
        st<T>(P.px, slot, kv[0]); st<T>(P.py, slot, kv[1]); st<T>(P.pz, slot, kv[2]);
        st<T>(P.w, slot, w);
        P.id[slot] = (unsigned long long)rid.x | ((unsigned long long)rid.y << 32);
        P.nev[slot] = 0u;
        if (P.od) st<T>(P.od, slot, (T)0);       // optical depth not drawn yet
    } else {
        note_overflow(ctl, 2, slot);
    }
}

// Pair creation at a photon's event point x at clock tau (Sec. 3): chi there,
// electron fraction from the inverse CDF with the draw words rz, both leptons
// along the photon's direction with energy-conserving momenta, appended with
// their ids.  born(species, slot) is called for each lepton that got a place.
// The caller removes the photon.
template <class T, class F>
__device__ __forceinline__ void pair_create(const PassArgs &a, const StepTime &tm, const T *icdf, const T x[3],
                                            const T kv[3], T k0, T nx, T ny, T nz, double tau, T w,
                                            unsigned long long id, unsigned k, uint2 rz, unsigned &n64, F born) {
    DevCtl *ctl = a.ctl;
    T E[3], B[3];
    field_tau<T>(a, tm, x, tau, E, B);
    const T chi = photon_chi<T>(k0, kv, E, B, n64, a.field_zero);
    T om, ue, ve;
    Uniform<T>::draw(rz.x, rz.y, ue, ve);
    const T delta = sample_pair<T>(icdf, chi, ue, ve, &om);
    T em = delta * k0, ep = om * k0;
    em = em < (T)1 ? (T)1 : em;
    ep = ep < (T)1 ? (T)1 : ep;
    const T pm = f_sqrt((em - (T)1) * (em + (T)1)), pp = f_sqrt((ep - (T)1) * (ep + (T)1));
    const uint4 rid = event_draw(a.child_keys, id, tm.step, k);
    const unsigned long long se = warp_append(&ctl->count[0], 1);
    const unsigned long long sp = warp_append(&ctl->count[1], 1);
    if (se < ctl->capacity[0]) {
        const SpeciesDev &P = a.sp[0];
        st<T>(P.x, se, x[0]); st<T>(P.y, se, x[1]); st<T>(P.z, se, x[2]);
        st<T>(P.px, se, pm * nx); st<T>(P.py, se, pm * ny); st<T>(P.pz, se, pm * nz);
        st<T>(P.w, se, w);
        P.id[se] = (unsigned long long)rid.x | ((unsigned long long)rid.y << 32);
        P.nev[se] = 0u;
        P.tau[se] = tau;
        if (P.od) st<T>(P.od, se, (T)0);
        born(0, (unsigned)se);
    } else {
        note_overflow(ctl, 0, se);
    }
    if (sp < ctl->capacity[1]) {
        const SpeciesDev &P = a.sp[1];
        st<T>(P.x, sp, x[0]); st<T>(P.y, sp, x[1]); st<T>(P.z, sp, x[2]);
        st<T>(P.px, sp, pp * nx); st<T>(P.py, sp, pp * ny); st<T>(P.pz, sp, pp * nz);
        st<T>(P.w, sp, w);
        P.id[sp] = (unsigned long long)rid.z | ((unsigned long long)rid.w << 32);
        P.nev[sp] = 0u;
        P.tau[sp] = tau;
        if (P.od) st<T>(P.od, sp, (T)0);
        born(1, (unsigned)sp);
    } else {
        note_overflow(ctl, 1, sp);
    }
}

// FP64 mode, a lepton at the step start: whether it surely has no event in the
// step, decided in FP32 as for photons (surely_flies below).  The lepton is
// then only pushed; the others go to the stack, where their waiting times are
// drawn in FP64, densely.  The emission rate grows with chi too.  (One
// emission in seven lepton-steps: 20 steps of the paper's test problem at
// 5e5 photons 15.4 -> 12.5 ms, 200 steps of 16384 electrons 9.8 -> 8.8 ms.)
__device__ __forceinline__ bool surely_calm(const LeptonCtx<double> &c, const double p[3], const double E[3],
                                            const double B[3], unsigned long long id) {
    const PassArgs &a = c.a;
    const float k[3] = {(float)p[0], (float)p[1], (float)p[2]};
    const float Ef[3] = {(float)E[0], (float)E[1], (float)E[2]}, Bf[3] = {(float)B[0], (float)B[1], (float)B[2]};
    const float p2 = k[0] * k[0] + k[1] * k[1] + k[2] * k[2], gam = sqrtf(1.0f + p2);
    // chi R <= |gamma E_perp| + |E along p| + |p x B|, each bounded with its rounding
    const float ax = k[1] * Ef[2] - k[2] * Ef[1], ay = k[2] * Ef[0] - k[0] * Ef[2], az = k[0] * Ef[1] - k[1] * Ef[0];
    const float bx = k[1] * Bf[2] - k[2] * Bf[1], by = k[2] * Bf[0] - k[0] * Bf[2], bz = k[0] * Bf[1] - k[1] * Bf[0];
    const float e2 = Ef[0] * Ef[0] + Ef[1] * Ef[1] + Ef[2] * Ef[2];
    const float sum = (fabsf(k[0]) + fabsf(k[1]) + fabsf(k[2])) *
                      (fabsf(Ef[0]) + fabsf(Ef[1]) + fabsf(Ef[2]) + fabsf(Bf[0]) + fabsf(Bf[1]) + fabsf(Bf[2]));
    float chi;
    if (a.field_zero) chi = sqrtf(e2 + ax * ax + ay * ay + az * az + bx * bx + by * by + bz * bz);     // E.(p x B) = 0
    else chi = sqrtf(e2 + ax * ax + ay * ay + az * az) + sqrtf(bx * bx + by * by + bz * bz);
    chi = (chi + sum * 0x1p-21f) * (float)(1.0 / RS) * 1.0001f;
    // beyond FP32's range (an infinity, or a NaN from the difference of two) nothing is decided
    if (!(chi < t_inf<float>() && gam < t_inf<float>())) return false;
    const float lam = (float)(ALPHA * RS) / gam * rate_em<float>(c.coef32, chi);
    const uint4 r = event_draw(a.keys, id, c.tm.step, 0u);
    float u, v;
    Uniform<float>::draw(r.x, r.y, u, v);
    // -ln u to 1e-6 in FP32, the rate bound's 1% aside
    return Uniform<float>::neglog(u, v) > lam * a.dt_f * 1.01f;
}

// A copy of v that the compiler does not see through.  Sub-expressions shared
// with other code may be fused into multiply-adds differently than alone; a
// photon's flight from such copies is rounded as in a kernel of its own, and
// does not change how the surrounding lepton arithmetic is rounded.
__device__ __forceinline__ float own(float v) { asm volatile("" : "+f"(v)); return v; }
__device__ __forceinline__ double own(double v) { asm volatile("" : "+d"(v)); return v; }

// FP64 mode: whether a photon surely reaches the step end, decided in FP32.
// Converting takes -ln u <= lambda h, and -ln u >= v = 1 - u; with a bound of
// lambda from above (chi bounded without cancellation, the FP32 rate form,
// monotonic in chi, 1% on top, far above every rounding and the arguments'
// own) v > lambda h decides, and neither chi, rate nor logarithm is needed in
// FP64.  Photons it does not decide (those that convert and about as many
// others) take the FP64 path, so what is computed is unchanged.  On GB300 an
// FP64 instruction occupies its pipe 16 times as long as an FP32 one: the
// photon pass at 5e5 photons in the standing wave took 265 us of a step, and 20 steps 18.6 ms; 15.4 ms with the bound.
// chi_ub: an upper bound of chi; tab32: the FP32 rate pieces.
__device__ __forceinline__ bool surely_flies(const PassArgs &a, const float *tab32, float chi_ub, float inv_k0, float h,
                                             unsigned long long id, unsigned step) {
    if (!(chi_ub < t_inf<float>())) return false;      // beyond FP32's range, or a NaN: not decided
    const float lam = (float)(ALPHA * RS) * inv_k0 * rate_pair<float>(tab32, chi_ub * 1.0001f);
    const uint4 r = event_draw(a.keys, id, step, 0u);
    float u, v;
    Uniform<float>::draw(r.x, r.y, u, v);
    return v > lam * h * 1.01f;
}

// chi R = |k0 E + k x B| without the part along k: at most |k x E| + |k x B|
__device__ __forceinline__ float chi_bound(const float k[3], const float E[3], const float B[3]) {
    const float ax = k[1] * E[2] - k[2] * E[1], ay = k[2] * E[0] - k[0] * E[2], az = k[0] * E[1] - k[1] * E[0];
    const float bx = k[1] * B[2] - k[2] * B[1], by = k[2] * B[0] - k[0] * B[2], bz = k[0] * B[1] - k[1] * B[0];
    const float e = fabsf(k[0]) + fabsf(k[1]) + fabsf(k[2]);      // the products' rounding: 2^-22 of their sizes
    const float f = fabsf(E[0]) + fabsf(E[1]) + fabsf(E[2]) + fabsf(B[0]) + fabsf(B[1]) + fabsf(B[2]);
    return (sqrtf(ax * ax + ay * ay + az * az) + sqrtf(bx * bx + by * by + bz * bz) + e * f * 0x1p-21f) * (float)(1.0 / RS);
}

// The same at the step start from the field's descriptor alone: in the
// standing wave E and B lie along (0, cos t, sin t) with E^2 + B^2 = a0^2
// everywhere, so chi R = a0 |k x (0, cos t, sin t)|, whatever x; a0 |k x
// (cos t, sin t, 0)| in the rotating field.  The step's phase is taken from
// the FP64 sine and cosine.
__device__ __forceinline__ float chi_bound_start(const PassArgs &a, const Phase<double> &ph, const float k[3]) {
    const float zero[3] = {0.f, 0.f, 0.f};
    const float c = (float)ph.c, s = (float)ph.s, a0 = a.prm_f[0];
    if (a.field_kind == QED_FIELD_ROTATING_E) {
        const float E[3] = {a0 * c, a0 * s, 0.f};
        return chi_bound(k, E, zero);
    }
    if (a.field_kind == QED_FIELD_STANDING_CP) {
        const float E[3] = {0.f, a0 * c, a0 * s};
        return chi_bound(k, E, zero);
    }
    const float E[3] = {a.prm_f[0], a.prm_f[1], a.prm_f[2]}, B[3] = {a.prm_f[3], a.prm_f[4], a.prm_f[5]};
    return chi_bound(k, E, B);
}

// One waiting time of a photon of energy k0 and direction n at x, where the
// field is (E, B), at clock tau (FRESH: the step start, tau = 0): the photon
// flies to the step end (returns false) or to the point where it converts
// (returns true: tau there, the pair's draw words in rz).
template <class T, bool FRESH>
__device__ __forceinline__ bool photon_flight(const PassArgs &a, const StepTime &tm, const T *s_coef, const T E[3],
                                              const T B[3], T x[3], const T kv[3], T k0, T inv, T nx, T ny, T nz,
                                              double &tau, unsigned long long id, uint2 &rz, unsigned &n64) {
    const T alpha_r = (T)(ALPHA * RS);
    T chi = photon_chi<T, !FRESH>(k0, kv, E, B, n64, a.field_zero);
    T lam;
    if constexpr (sizeof(T) == 4) lam = alpha_r * inv * rate_pair<T>(s_coef, chi);
    else lam = alpha_r / k0 * rate_pair<T>(s_coef, chi);     // the oracle's rounding
    // the remaining time of the step, and with FP32 clocks inside a step the
    // margin within which the FP64 test decides (as in the lepton pass)
    T h, marg = (T)0;
    if constexpr (FRESH) h = dt_of<T>(a);
    else {
        h = (T)(a.dt - tau);
        if constexpr (sizeof(T) == 4) marg = fmaf(h, 0x1p-20f, a.dt_f * 0x1p-40f);
    }
    uint4 r = make_uint4(0, 0, 0, 0);
    T dth = t_inf<T>();
    if (lam > lam_skip<T>(a)) {
        r = event_draw(a.keys, id, tm.step, 0u);
        T uw, vw;
        Uniform<T>::draw(r.x, r.y, uw, vw);
        // -ln u >= 1 - u = v: with v above lambda h (by a margin far above every
        // rounding involved) the photon reaches the step end, and neither the
        // logarithm nor the division is needed.  About one photon in a
        // thousand converts per step, so nearly every warp ends here.
        if (!(vw > lam * ((h + marg) * (T)(1.0 + 1e-4)))) dth = f_div(Uniform<T>::neglog(uw, vw), lam);
    }
    bool no_event;
    if constexpr (FRESH && sizeof(T) == 4) no_event = dth >= a.dt_f_gt;
    else if constexpr (FRESH) no_event = dth > a.dt;
    else if constexpr (sizeof(T) == 4) {
        if (dth > h + marg) no_event = true;
        else if (dth < h - marg) no_event = false;
        else no_event = tau + (double)dth > a.dt;
    } else no_event = tau + (double)dth > a.dt;
    if (no_event) {
        x[0] += nx * h; x[1] += ny * h; x[2] += nz * h;
        return false;
    }
    x[0] += nx * dth; x[1] += ny * dth; x[2] += nz * dth;
    if constexpr (FRESH) tau = (double)dth;
    else tau += (double)dth;
    rz = make_uint2(r.z, r.w);
    return true;
}

// A photon emitted in this step (momentum kv, field (E, B) at its birth point
// x, generation gen): its flight to the step end, then its record; or the
// pair it creates, whose leptons wait in the block's newborn list, or, when
// that is full, in the species arrays for a further launch.
template <class T>
__device__ __forceinline__ void fly_newborn(const LeptonCtx<T> &c, LeptonStack<T> &q, const StackPos &pos,
                                            const T Ee[3], const T Be[3], const T xe[3], const T ke[3], double tau,
                                            T w, uint4 rid, unsigned gen, PassStats &ps) {
    const PassArgs &a = c.a;
    const unsigned long long id = (unsigned long long)rid.x | ((unsigned long long)rid.y << 32);
    T x[3] = {own(xe[0]), own(xe[1]), own(xe[2])};
    const T E[3] = {own(Ee[0]), own(Ee[1]), own(Ee[2])}, B[3] = {own(Be[0]), own(Be[1]), own(Be[2])};
    const T kv[3] = {own(ke[0]), own(ke[1]), own(ke[2])};
    const T k0 = f_sqrt(kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2]);
    bool alive = true;
    ++ps.ph;
    ps.gen = max(ps.gen, gen);
    if (gen > c.gen_limit) atomicExch(&c.ctl->timeout, 1ull);
    else if (k0 > (T)0 && before_step_end(tau, a.dt)) {
        const T inv = f_div((T)1, k0);
        const T nx = kv[0] * inv, ny = kv[1] * inv, nz = kv[2] * inv;
        uint2 rz = make_uint2(0, 0);
        bool flies = false;
        if constexpr (sizeof(T) == 8) {
            const float kf[3] = {(float)kv[0], (float)kv[1], (float)kv[2]}, Ef[3] = {(float)E[0], (float)E[1], (float)E[2]},
                        Bf[3] = {(float)B[0], (float)B[1], (float)B[2]};
            const double h = a.dt - tau;
            flies = surely_flies(a, c.coef32, chi_bound(kf, Ef, Bf), (float)inv, (float)h, id, c.tm.step);
            if (flies) { x[0] += nx * h; x[1] += ny * h; x[2] += nz * h; }
        }
        if (!flies && photon_flight<T, false>(a, c.tm, c.coef, E, B, x, kv, k0, inv, nx, ny, nz, tau, id, rz, ps.n64)) {
            alive = false;
            ++ps.pr;
            ps.mx = max(ps.mx, 1u);
            pair_create<T>(a, c.tm, reinterpret_cast<const T *>(a.icdf_pair), x, kv, k0, nx, ny, nz, tau, w, id, 0u, rz,
                           ps.n64, [&](int s, unsigned i) {
                const int at = pos.nb + atomicAdd(&q.nb_pushed[pos.it], 1);
                if (at < LB<T>) {
                    q.nb_idx[at] = i | ((unsigned)s << 31);
                    q.nb_gen[at] = gen + 1u;
                } else {
                    // left at its birth clock for a further launch, with its
                    // generation; the sign bit marks it (those taken up here
                    // stay unmarked)
                    a.sp[s].tau[i] = -tau;
                    a.gen[s][i] = gen + 1u;
                    atomicAdd(&c.ctl->spilled, 1ull);
                }
            });
        }
    }
    if (alive) append_photon<T>(a, c.ctl, c.cap_ph, x, kv, w, rid);
}

// Network sampler of a block: the staged network (dynamic shared memory)
constexpr int MLP_SMEM_BYTES = MLP_INF_BYTES;

template <class T>
__device__ __forceinline__ void finish(const PassArgs &a, unsigned idx, const T x[3], const T p[3], unsigned k) {
    const SpeciesDev &S = a.sp[idx >> 31];
    const unsigned i = idx & 0x7FFFFFFFu;
    st<T>(S.x, i, x[0]); st<T>(S.y, i, x[1]); st<T>(S.z, i, x[2]);
    st<T>(S.px, i, p[0]); st<T>(S.py, i, p[1]); st<T>(S.pz, i, p[2]);
    if (k) S.nev[i] += k;
}

template <class T>
__device__ __forceinline__ void stack_push(LeptonStack<T> &q, const StackPos &pos, const T x[3], const T p[3],
                                           double tau, unsigned long long id, T w, unsigned idx, unsigned k,
                                           unsigned gen, uint2 rz) {
    const int slot = pos.n + atomicAdd(&q.pushed[pos.it], 1);
    q.x[0][slot] = x[0]; q.x[1][slot] = x[1]; q.x[2][slot] = x[2];
    q.p[0][slot] = p[0]; q.p[1][slot] = p[1]; q.p[2][slot] = p[2];
    q.tau[slot] = tau; q.id[slot] = id; q.w[slot] = w; q.idx[slot] = idx; q.k[slot] = k; q.gen[slot] = gen;
    q.r[slot] = rz;
}

// Pop min(n, LB) items, one per thread, and process each to its next event
// or the step end.  Every thread of the block calls this; pos.n is the
// stack's size and becomes the size below the round's pushes.
template <class T, bool MLP>
__device__ __forceinline__ void stack_round(const LeptonCtx<T> &c, LeptonStack<T> &q, StackPos &pos, PassStats &ps,
                                            const MlpInf &ms) {
    const int take = pos.n < LB<T> ? pos.n : LB<T>;
    const int t = threadIdx.x;
    T x[3], p[3], w = 0;
    double tau = 0.0;
    unsigned long long id = 0;
    unsigned idx = 0, k = 0, gen = RESUME;
    uint2 rz = make_uint2(0, 0);
    const bool mine = t < take;
    pos.n -= take;
    if (mine) {
        const int s = pos.n + t;
        x[0] = q.x[0][s]; x[1] = q.x[1][s]; x[2] = q.x[2][s];
        p[0] = q.p[0][s]; p[1] = q.p[1][s]; p[2] = q.p[2][s];
        tau = q.tau[s]; id = q.id[s]; w = q.w[s]; idx = q.idx[s]; k = q.k[s]; gen = q.gen[s]; rz = q.r[s];
    }
    __syncthreads();                                // the popped places may now be pushed to
    const bool event = !(gen & RESUME);
    const bool start = sizeof(T) == 8 && mine && (gen & START);
    gen &= ~(RESUME | START);
    // the event at the particle's current point: chi there, energy fraction
    // from the inverse CDF (or the network: the whole warp evaluates it for
    // its 32 items on the tensor cores), then the kinematics
    T E[3], B[3], gam = (T)1, chi = (T)0, p2 = (T)0, ue = (T)0.5, ve = (T)0.5, delta = (T)0, om = (T)1;
    if (event) {
        field_tau<T>(c.a, c.tm, x, tau, E, B);
        lepton_chi<T>(p, E, B, gam, chi, p2, ps.n64, c.a.field_zero);
        Uniform<T>::draw(rz.x, rz.y, ue, ve);
    }
    if constexpr (MLP) {
        float f0 = 0.f, f1 = 0.f;
        bool use_net = false;
        if (event) {
            const float sl = (float)logit(ue, ve);
            const float cf = (float)chi;
            use_net = cf >= 1e-3f && cf <= 1e3f && fabsf(sl) < 16.0f;
            if (use_net) { f0 = log10f(cf) / 3.0f; f1 = sl / 16.0f; }
        }
        const float y = mlp_forward_warp(f0, f1, ms);
        if (event) {
            if (use_net) {
                const T aa = (T)3 * chi * (T)__expf(16.0f * (y - 0.5f));
                om = (T)2 / ((T)2 + aa);
                delta = aa / ((T)2 + aa);
            } else {
                delta = sample_emission<T>(c.icdf, chi, ue, ve, &om);
            }
        }
    } else {
        if (event) delta = sample_emission<T>(c.icdf, chi, ue, ve, &om);
    }
    if (event) {
        T kv[3];
        if (recoil<T>(c.a, p, gam, p2, delta, om, kv)) {
            const uint4 rid = event_draw(c.a.child_keys, id, c.tm.step, k);
            if (c.a.fly_newborns) fly_newborn<T>(c, q, pos, E, B, x, kv, tau, w, rid, gen + 1u, ps);
            else append_photon<T>(c.a, c.ctl, c.cap_ph, x, kv, w, rid);
        }
        ++k;
        ++ps.em;
    }
    if (mine) {
        const T qch = (idx >> 31) ? (T)1 : (T)-1;
        bool again;
        if (start) again = advance<T, true>(c, x, p, qch, tau, id, 0u, rz, ps.n64);
        else again = before_step_end(tau, c.a.dt) && advance<T, false>(c, x, p, qch, tau, id, k, rz, ps.n64);
        if (again) {
            stack_push<T>(q, pos, x, p, tau, id, w, idx, k, gen, rz);
        } else {
            finish<T>(c.a, idx, x, p, k);
            ps.mx = max(ps.mx, k);
        }
    }
}

// One step's leptons.  FRESH: those present at the step start, then the
// newborns of the photon pass; else the newborns that a full block list left
// behind in the previous launch.  The last block to finish opens the next
// such launch (`loop`: through the step graph's while node `h`).
template <class T, bool FRESH, bool MLP>
__global__ void __launch_bounds__(LB<T>, (sizeof(T) == 4 && !MLP ? 3 : 2))
    k_lepton_pass(const __grid_constant__ PassArgs a, cudaGraphConditionalHandle h, int loop) {
    DevCtl *ctl = a.ctl;
    // 32-bit indices (a species holds fewer than 2^31 entries: bit 31 of idx names the species)
    const unsigned n0 = FRESH ? (unsigned)ctl->end[0] : 0u, n1 = FRESH ? (unsigned)ctl->end[1] : 0u;
    const unsigned n = n0 + n1;
    const unsigned nb0 = (unsigned)(FRESH ? ctl->end[0] : ctl->begin[0]);
    const unsigned nb1 = (unsigned)(FRESH ? ctl->end[1] : ctl->begin[1]);
    const unsigned m0 = (unsigned)(FRESH ? ctl->born[0] : ctl->end[0]) - nb0;
    const unsigned m = m0 + (unsigned)(FRESH ? ctl->born[1] : ctl->end[1]) - nb1;
    const unsigned nb_blk = gridDim.x - 1 - blockIdx.x;      // newborn tiles from the far end: few steps have many
    constexpr int NT = LB<T>;
    __shared__ __align__(16) T s_coef[RateWords<T>::N];
    __shared__ LeptonStack<T> q;
    __shared__ StepTime s_tm;
    extern __shared__ __align__(16) unsigned char dyn[];
    PassStats ps;
    // blocks past the pass's ranges stage nothing
    if (blockIdx.x * NT < n || nb_blk * NT < m) {
        MlpInf ms{nullptr, nullptr, nullptr};
        if constexpr (MLP) ms = mlp_stage(dyn, a.mlp_w16);
        for (int i = threadIdx.x; i < RateWords<T>::N; i += NT) s_coef[i] = reinterpret_cast<const T *>(a.coef)[i];
        if (threadIdx.x < 3) q.pushed[threadIdx.x] = q.nb_pushed[threadIdx.x] = 0;
        if (threadIdx.x == 0) s_tm = load_step_time(a);
        __syncthreads();
        const unsigned gen_limit = (unsigned)ctl->pass_limit;
        const LeptonCtx<T> c{a, ctl, s_coef, a.coef32, reinterpret_cast<const T *>(a.icdf_em), ctl->capacity[2], gen_limit,
                             (T)(ALPHA * RS), s_tm, time_phase<T, StepTime>(s_tm, 0.0)};
        // FP32 step-start pass: each thread stages its particle of the block's
        // next tile in shared memory while the block works on the current tile
        constexpr bool STAGE = FRESH && sizeof(T) == 4;
        constexpr int NF = STAGE ? 9 : 1, NS = STAGE ? NT : 1;
        __shared__ __align__(16) float stg[NF][NS];            // w x y z px py pz id(2 words)
        const unsigned stride = gridDim.x * NT;
        auto stage = [&](unsigned jj) {
            if constexpr (STAGE) {
                const int sp = jj < n0 ? 0 : 1;
                const unsigned ii = sp == 0 ? jj : jj - n0;
                const SpeciesDev &P = a.sp[sp];
                const int t = threadIdx.x;
                cp_async4(&stg[0][t], reinterpret_cast<const float *>(P.w) + ii);
                cp_async4(&stg[1][t], reinterpret_cast<const float *>(P.x) + ii);
                cp_async4(&stg[2][t], reinterpret_cast<const float *>(P.y) + ii);
                cp_async4(&stg[3][t], reinterpret_cast<const float *>(P.z) + ii);
                cp_async4(&stg[4][t], reinterpret_cast<const float *>(P.px) + ii);
                cp_async4(&stg[5][t], reinterpret_cast<const float *>(P.py) + ii);
                cp_async4(&stg[6][t], reinterpret_cast<const float *>(P.pz) + ii);
                cp_async4(&stg[7][t], P.id + ii);
                cp_async4(&stg[8][t], reinterpret_cast<const unsigned *>(P.id + ii) + 1);
            }
        };
        unsigned base = blockIdx.x * NT, nb_base = nb_blk * NT;
        if constexpr (STAGE) {
            if (base + threadIdx.x < n) stage(base + threadIdx.x);
            cp_async_commit();
        }

        // One loop with one call of stack_round: the next tile is taken while the
        // stack holds less than a round, the stack is drained at the end.  The
        // round (and the event arithmetic in it) then has a single inlined copy,
        // so which round processes a particle, which depends on the order of the
        // arrays, cannot change how its results are rounded.
        StackPos pos{0, 0, 0};
        for (;;) {
            const bool fresh = base < n && pos.nb < NT / 2;
            if (pos.n < NT && fresh) {
                const unsigned j = base + threadIdx.x;
                T w = (T)0, x[3], p[3];
                unsigned long long id = 0;
                if constexpr (STAGE) {
                    // this thread's staged particle, then the next tile's copies in
                    // flight (the slots are free once read)
                    cp_async_wait_all();
                    if (j < n) {
                        const int t = threadIdx.x;
                        w = stg[0][t];
                        x[0] = stg[1][t]; x[1] = stg[2][t]; x[2] = stg[3][t];
                        p[0] = stg[4][t]; p[1] = stg[5][t]; p[2] = stg[6][t];
                        id = (unsigned long long)__float_as_uint(stg[7][t]) |
                             ((unsigned long long)__float_as_uint(stg[8][t]) << 32);
                    }
                    if (j + stride < n) stage(j + stride);
                    cp_async_commit();
                }
                if (j < n) {
                    const int s = j < n0 ? 0 : 1;
                    const unsigned i = s == 0 ? j : j - n0;
                    const SpeciesDev &S = a.sp[s];
                    if constexpr (!STAGE) {
                        w = ld<T>(S.w, i);
                        x[0] = ld<T>(S.x, i); x[1] = ld<T>(S.y, i); x[2] = ld<T>(S.z, i);
                        p[0] = ld<T>(S.px, i); p[1] = ld<T>(S.py, i); p[2] = ld<T>(S.pz, i);
                        id = __ldg(S.id + i);
                    }
                    if (w > (T)0) {
                        double tau = 0.0;
                        const unsigned idx = i | ((unsigned)s << 31);
                        ++ps.lep;
                        uint2 rz = make_uint2(0, 0);
                        const T qch = s == 0 ? (T)-1 : (T)1;
                        if constexpr (sizeof(T) == 8) {
                            T E[3], B[3];
                            field_at<T>(a, x, c.ph0, E, B);
                            if (surely_calm(c, p, E, B, id)) {
                                boris<T, true>(x, p, qch, E, B, a.dt, a.field_zero == 1, id, c.tm.step, 0u);
                                finish<T>(a, idx, x, p, 0u);
                            } else {
                                stack_push<T>(q, pos, x, p, tau, id, w, idx, 0u, RESUME | START, rz);
                            }
                        } else if (advance<T, true>(c, x, p, qch, tau, id, 0u, rz, ps.n64)) {
                            stack_push<T>(q, pos, x, p, tau, id, w, idx, 0u, 0u, rz);
                        } else {
                            finish<T>(a, idx, x, p, 0u);
                        }
                    }
                }
                base += stride;
            } else if (pos.n < NT && (pos.nb > 0 || nb_base < m)) {
                // newborn leptons onto the stack: this block's own first, else a
                // tile of those waiting in the species arrays
                const bool own = pos.nb > 0;
                const unsigned t = threadIdx.x;
                unsigned idx = 0, gen = 1u;               // pairs of the photons present at the step start
                bool have = false;
                if (own) {
                    have = t < (unsigned)pos.nb;
                    if (have) { idx = q.nb_idx[t]; gen = q.nb_gen[t]; }
                } else {
                    const unsigned j = nb_base + t;
                    have = j < m;
                    if (have) idx = j < m0 ? nb0 + j : (nb1 + (j - m0)) | 0x80000000u;
                    nb_base += stride;
                }
                if (have) {
                    const SpeciesDev &S = a.sp[idx >> 31];
                    const unsigned i = idx & 0x7FFFFFFFu;
                    double tau = S.tau[i];
                    const T w = ld<T>(S.w, i);
                    if constexpr (!FRESH) {
                        // among those appended since, only the ones left behind carry the mark
                        if (!own) {
                            have = __double_as_longlong(tau) < 0;
                            tau = -tau;
                            if (have) gen = a.gen[idx >> 31][i];
                        }
                    }
                    if (have && gen > gen_limit) {
                        atomicExch(&ctl->timeout, 1ull);
                        have = false;
                    }
                    if (have && w > (T)0) {
                        ++ps.lep;
                        ps.gen = max(ps.gen, gen);
                        const T x[3] = {ld<T>(S.x, i), ld<T>(S.y, i), ld<T>(S.z, i)};
                        const T p[3] = {ld<T>(S.px, i), ld<T>(S.py, i), ld<T>(S.pz, i)};
                        stack_push<T>(q, pos, x, p, tau, S.id[i], w, idx, 0u, gen | RESUME, make_uint2(0, 0));
                    }
                }
                if (own) pos.nb = 0;
            } else {
                if (pos.n == 0) break;
                stack_round<T, MLP>(c, q, pos, ps, ms);
            }
            // the sizes after this iteration's pushes; the next iteration's
            // counters were last read an iteration ago
            const int nx = pos.it == 2 ? 0 : pos.it + 1;
            if (threadIdx.x == 0) q.pushed[nx] = q.nb_pushed[nx] = 0;
            __syncthreads();
            pos.n += q.pushed[pos.it];
            pos.nb = min(pos.nb + q.nb_pushed[pos.it], NT);
            pos.it = nx;
        }
        __syncwarp();
        flush_stats(ctl, ps);
    }
    if (!a.fly_newborns) return;
    if (last_block(ctl) && threadIdx.x == 0) {
        const bool more = __ldcg(&ctl->spilled) != 0 && !__ldcg(&ctl->overflow) && !__ldcg(&ctl->timeout);
        for (int s = 0; s < 2; ++s) {
            ctl->begin[s] = FRESH ? ctl->born[s] : ctl->end[s];
            ctl->end[s] = count_now(ctl, s);
        }
        ctl->more = more;
        if (!more) ctl->passes += __ldcg(&ctl->step_passes);
        ctl->spilled = 0;
        if (!FRESH && loop) ctl->graph_kernels += 1;
        if (loop) cudaGraphSetConditional(h, more ? 1u : 0u);
    }
}

// Several steps of an emission run (photons recorded, no leveling): nothing
// couples the leptons between steps, so one launch carries them through all
// steps of a call.  A block holds a lepton per thread in registers; per step
// those without an event are pushed to the step end, the others go through
// the stack as in the pass above and come back through the species arrays.
// The arithmetic per particle and step is that of the pass, as are the draws.
// Photons past the capacity are counted, not written, and every block takes
// all steps: the demand and the statistics do not depend on their timing.
//
// A launch per step is bound by its latency where the ensemble is small: the
// step-begin kernel, the tables' staging and the block's last, partly filled
// rounds took 80 us per step for 16384 electrons in FP64 (44 us here).
template <class T>
__global__ void __launch_bounds__(LB<T>, 2) k_lepton_steps(const __grid_constant__ PassArgs a, unsigned long long step0,
                                                           int nsteps) {
    constexpr int NT = LB<T>;
    DevCtl *ctl = a.ctl;
    __shared__ __align__(16) T s_coef[RateWords<T>::N];
    __shared__ LeptonStack<T> q;
    __shared__ StepTime s_tm;
    __shared__ Phase<T> s_ph;
    const unsigned n0 = (unsigned)ctl->end[0], n1 = (unsigned)ctl->end[1];
    const unsigned n = n0 + n1;
    if (blockIdx.x * NT >= n) return;
    for (int i = threadIdx.x; i < RateWords<T>::N; i += NT) s_coef[i] = reinterpret_cast<const T *>(a.coef)[i];
    if (threadIdx.x < 3) q.pushed[threadIdx.x] = 0;
    PassStats ps;
    MlpInf ms{nullptr, nullptr, nullptr};
    StackPos pos{0, 0, 0};
    auto next_iteration = [&] {                  // as in the pass: sizes after this iteration's pushes
        const int nx = pos.it == 2 ? 0 : pos.it + 1;
        if (threadIdx.x == 0) q.pushed[nx] = 0;
        __syncthreads();
        pos.n += q.pushed[pos.it];
        pos.it = nx;
    };
    for (unsigned base = blockIdx.x * NT; base < n; base += gridDim.x * NT) {
        const unsigned j = base + threadIdx.x;
        const int s = j < n0 ? 0 : 1;
        const unsigned i = s == 0 ? j : j - n0;
        const SpeciesDev &S = a.sp[s];
        const unsigned idx = i | ((unsigned)s << 31);
        T w = (T)0, x[3], p[3];
        unsigned long long id = 0;
        if (j < n) {
            w = ld<T>(S.w, i);
            x[0] = ld<T>(S.x, i); x[1] = ld<T>(S.y, i); x[2] = ld<T>(S.z, i);
            p[0] = ld<T>(S.px, i); p[1] = ld<T>(S.py, i); p[2] = ld<T>(S.pz, i);
            id = __ldg(S.id + i);
        }
        const T qch = s == 0 ? (T)-1 : (T)1;
        for (int it = 0; it < nsteps; ++it) {
            if (threadIdx.x == 0) {
                // the step's time and index as the step-begin kernel writes them
                const double t_n = (double)(step0 + it) * a.dt;
                s_tm.field_kind = a.field_kind;
                s_tm.t_n = t_n;
                s_tm.t_n_red_f = (float)fmod(t_n, 2.0 * 3.14159265358979323846);
                s_tm.step = (unsigned)(step0 + it);
                s_ph = time_phase<T, StepTime>(s_tm, 0.0);
            }
            __syncthreads();
            const LeptonCtx<T> c{a, ctl, s_coef, a.coef32, reinterpret_cast<const T *>(a.icdf_em), ctl->capacity[2], 0u,
                                 (T)(ALPHA * RS), s_tm, s_ph};
            bool away = false;
            if (w > (T)0) {
                double tau = 0.0;
                ++ps.lep;
                uint2 rz = make_uint2(0, 0);
                if constexpr (sizeof(T) == 8) {
                    T E[3], B[3];
                    field_at<T>(a, x, c.ph0, E, B);
                    away = !surely_calm(c, p, E, B, id);
                    if (away) stack_push<T>(q, pos, x, p, tau, id, w, idx, 0u, RESUME | START, rz);
                    else boris<T, true>(x, p, qch, E, B, a.dt, a.field_zero == 1, id, c.tm.step, 0u);
                } else {
                    away = advance<T, true>(c, x, p, qch, tau, id, 0u, rz, ps.n64);
                    if (away) stack_push<T>(q, pos, x, p, tau, id, w, idx, 0u, 0u, rz);
                }
            }
            next_iteration();
            while (pos.n > 0) {
                stack_round<T, false>(c, q, pos, ps, ms);
                next_iteration();
            }
            if (away) {                          // written by the thread that finished it, before the barrier
                x[0] = ld<T>(S.x, i); x[1] = ld<T>(S.y, i); x[2] = ld<T>(S.z, i);
                p[0] = ld<T>(S.px, i); p[1] = ld<T>(S.py, i); p[2] = ld<T>(S.pz, i);
            }
        }
        if (w > (T)0) finish<T>(a, idx, x, p, 0u);
        __syncthreads();                         // s_tm is rewritten by the next tile's first step
    }
    __syncwarp();
    flush_stats(ctl, ps);
}

// Photon push: straight flight, pair creation at the event, the photon is
// removed (weight 0) and the pair appended, its leptons left to the lepton
// pass of the same step (the last block to finish closes their range).
template <class T>
__global__ void __launch_bounds__(256, (sizeof(T) == 4 ? 4 : 1)) k_photon_pass(PassArgs a) {
    DevCtl *ctl = a.ctl;
    constexpr int NT = 256;
    // 32-bit indices (a species holds fewer than 2^31 entries)
    const unsigned n = (unsigned)ctl->end[2];
    __shared__ __align__(16) T s_coef[RateWords<T>::N];
    __shared__ StepTime s_tm;
    if (blockIdx.x * NT < n) {
        for (int i = threadIdx.x; i < RateWords<T>::N; i += NT) s_coef[i] = reinterpret_cast<const T *>(a.coef)[i];
        constexpr bool BOUND = sizeof(T) == 8 && !SFQ_GRID;
        __shared__ __align__(16) float s_coef32[BOUND ? NRATE32 : 4];
        if constexpr (BOUND)
            for (int i = threadIdx.x; i < NRATE32; i += NT) s_coef32[i] = a.coef32[i];
        if (threadIdx.x == 0) s_tm = load_step_time(a);
        __syncthreads();
        const StepTime &tm = s_tm;
        const T *icdf = reinterpret_cast<const T *>(a.icdf_pair);
        const SpeciesDev &S = a.sp[2];
        PassStats ps;
        const Phase<T> ph0 = time_phase<T, StepTime>(tm, 0.0);
        // FP32: each thread stages its next photon in shared memory (two
        // buffers) while it works on the current one
        constexpr bool STAGE = sizeof(T) == 4;
        constexpr int NB = STAGE ? 2 : 1, NF = STAGE ? 9 : 1, NS = STAGE ? NT : 1;
        __shared__ __align__(16) float stg[NB][NF][NS];       // w x y z kx ky kz id(2 words)
        const unsigned stride = gridDim.x * NT;
        auto stage = [&](unsigned i, int buf) {
            if constexpr (STAGE) {
                const int t = threadIdx.x;
                cp_async4(&stg[buf][0][t], reinterpret_cast<const float *>(S.w) + i);
                cp_async4(&stg[buf][1][t], reinterpret_cast<const float *>(S.x) + i);
                cp_async4(&stg[buf][2][t], reinterpret_cast<const float *>(S.y) + i);
                cp_async4(&stg[buf][3][t], reinterpret_cast<const float *>(S.z) + i);
                cp_async4(&stg[buf][4][t], reinterpret_cast<const float *>(S.px) + i);
                cp_async4(&stg[buf][5][t], reinterpret_cast<const float *>(S.py) + i);
                cp_async4(&stg[buf][6][t], reinterpret_cast<const float *>(S.pz) + i);
                cp_async4(&stg[buf][7][t], S.id + i);          // id: two 4-byte halves
                cp_async4(&stg[buf][8][t], reinterpret_cast<const unsigned *>(S.id + i) + 1);
            }
        };
        const unsigned j0 = blockIdx.x * NT + threadIdx.x;
        if constexpr (STAGE) {
            if (j0 < n) stage(j0, 0);
            cp_async_commit();
        }
        int buf = 0;
        for (unsigned i = j0; i < n; i += stride, buf ^= 1) {
            T w, x[3], kv[3];
            unsigned long long id;
            if constexpr (STAGE) {
                if (i + stride < n) stage(i + stride, buf ^ 1);
                cp_async_commit();
                cp_async_wait_prev();                // this thread's copies of photon i have landed
                const int t = threadIdx.x;
                w = stg[buf][0][t];
                x[0] = stg[buf][1][t]; x[1] = stg[buf][2][t]; x[2] = stg[buf][3][t];
                kv[0] = stg[buf][4][t]; kv[1] = stg[buf][5][t]; kv[2] = stg[buf][6][t];
                id = (unsigned long long)__float_as_uint(stg[buf][7][t]) |
                     ((unsigned long long)__float_as_uint(stg[buf][8][t]) << 32);
            } else {
                // all loads issued together (live photons are the rule)
                w = ld<T>(S.w, i);
                x[0] = ld<T>(S.x, i); x[1] = ld<T>(S.y, i); x[2] = ld<T>(S.z, i);
                kv[0] = ld<T>(S.px, i); kv[1] = ld<T>(S.py, i); kv[2] = ld<T>(S.pz, i);
                id = __ldg(S.id + i);
            }
            if (!(w > (T)0)) continue;
            ++ps.ph;
            const T k0 = f_sqrt(kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2]);
            if (k0 > (T)0) {
                const T inv = f_div((T)1, k0);
                const T nx = kv[0] * inv, ny = kv[1] * inv, nz = kv[2] * inv;
                bool flies = false;
#if !SFQ_GRID
                if constexpr (sizeof(T) == 8) {
                    const float kf[3] = {(float)kv[0], (float)kv[1], (float)kv[2]};
                    flies = surely_flies(a, s_coef32, chi_bound_start(a, ph0, kf), (float)inv, a.dt_f, id, tm.step);
                }
#endif
                T E[3], B[3];
                double tau = 0.0;
                uint2 rz = make_uint2(0, 0);
                if (flies) {
                    const T h = dt_of<T>(a);
                    x[0] += nx * h; x[1] += ny * h; x[2] += nz * h;
                } else if (field_at<T>(a, x, ph0, E, B);
                           photon_flight<T, true>(a, tm, s_coef, E, B, x, kv, k0, inv, nx, ny, nz, tau, id, rz, ps.n64)) {
                    pair_create<T>(a, tm, icdf, x, kv, k0, nx, ny, nz, tau, w, id, 0u, rz, ps.n64,
                                   [](int, unsigned) {});
                    st<T>(S.w, i, (T)0);       // the photon is eliminated
                    S.nev[i] += 1u;
                    ++ps.pr;
                    ps.mx = 1u;
                }
            }
            st<T>(S.x, i, x[0]); st<T>(S.y, i, x[1]); st<T>(S.z, i, x[2]);
        }
        __syncwarp();
        flush_stats(ctl, ps);
    }
    // No photon pushed, no pair born: the step-begin kernel's empty range stands.
    // In particular a step opened after an overflow or a timeout has empty
    // ranges while the counts are not zero, and must stay empty.
    if (n == 0) return;
    if (last_block(ctl) && threadIdx.x < 2) ctl->born[threadIdx.x] = count_now(ctl, threadIdx.x);
}


#if !SFQ_GRID
// The FP32 photon pass in a field that does not depend on the position and
// where chi is a sum of squares (rotating E, uniform E or B), two consecutive
// photons per thread.  A photon is a
// chain of some 250 dependent instructions (a scheduler issued in 65% of the
// cycles with one photon per thread and 32 warps per SM); the chains of two
// photons interleave, and copies, shared-memory reads and stores move two
// photons at a time.  Both photons' arithmetic is written out with explicit
// rounding where the compiler could fuse either way.  5e7 photons, rotating E:
// 40 steps of its cascade 82.2 -> 77.1 ms; two blocks per SM (105 registers) as fast as three (spills).
// The pass, one photon per thread -> two, in us (rotating E, uniform E, uniform B):
// 219 -> 173, 219 -> 183, 221 -> 184 at 2e7 photons, 22.1 -> 18.0, 22.7 -> 18.0,
// 22.5 -> 19.8 at 1e6, 8.8 -> 7.8, 7.9 -> 7.6, 8.4 -> 7.6 at 2e4.  With E and B
// both (field_zero 0) chi's FP64 fallback branches photon by photon and nothing
// interleaves: 1734 -> 1723 at 2e7, 98 -> 102 at 1e6, 11.7 -> 15.8 at 2e4;
// one photon per thread is the rule there.
// In the standing wave the two sine and cosine evaluations do not interleave
// (their argument reduction branches): 40 steps took 72.1 ms against 71.6 with
// one photon per thread, which stays the rule there and on the grid.
__device__ __forceinline__ void cp_async8z(void *smem, const void *gmem, unsigned bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(gmem), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16z(void *smem, const void *gmem, unsigned bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(gmem), "r"(bytes) : "memory");
}

__global__ void __launch_bounds__(256, 2) k_photon_pass2(const __grid_constant__ PassArgs a) {
    DevCtl *ctl = a.ctl;
    constexpr int NT = 256;
    const unsigned n = (unsigned)ctl->end[2];
    const unsigned pairs = (n + 1) / 2;
    __shared__ __align__(16) float s_coef[RateWords<float>::N];
    __shared__ StepTime s_tm;
    if (blockIdx.x * NT < pairs) {
        for (int i = threadIdx.x; i < RateWords<float>::N; i += NT) s_coef[i] = reinterpret_cast<const float *>(a.coef)[i];
        if (threadIdx.x == 0) s_tm = load_step_time(a);
        __syncthreads();
        const StepTime &tm = s_tm;
        const unsigned step = tm.step;
        const float *icdf = reinterpret_cast<const float *>(a.icdf_pair);
        const SpeciesDev &S = a.sp[2];
        PassStats ps;
        const Phase<float> ph0 = time_phase<float, StepTime>(tm, 0.0);
        const float *tab = s_coef + 4 * EM_NSEG;
        const float skip = a.lam_skip_f, h = a.dt_f;
        const float alpha_r = (float)(ALPHA * RS);
        // two buffers per thread: the next pair's copies run under this pair's work
        __shared__ __align__(16) float2 stg[2][7][NT];         // w x y z kx ky kz
        __shared__ __align__(16) ulonglong2 sid[2][NT];
        const unsigned stride = gridDim.x * NT;
        const int t = threadIdx.x;
        auto stage = [&](unsigned j, int buf) {
            const unsigned i = 2 * j, b = i + 1 < n ? 8u : 4u;     // an odd last photon: nothing read past the count
            cp_async8z(&stg[buf][0][t], reinterpret_cast<const float *>(S.w) + i, b);
            cp_async8z(&stg[buf][1][t], reinterpret_cast<const float *>(S.x) + i, b);
            cp_async8z(&stg[buf][2][t], reinterpret_cast<const float *>(S.y) + i, b);
            cp_async8z(&stg[buf][3][t], reinterpret_cast<const float *>(S.z) + i, b);
            cp_async8z(&stg[buf][4][t], reinterpret_cast<const float *>(S.px) + i, b);
            cp_async8z(&stg[buf][5][t], reinterpret_cast<const float *>(S.py) + i, b);
            cp_async8z(&stg[buf][6][t], reinterpret_cast<const float *>(S.pz) + i, b);
            cp_async16z(&sid[buf][t], S.id + i, 2 * b);
        };
        const unsigned j0 = blockIdx.x * NT + threadIdx.x;
        if (j0 < pairs) stage(j0, 0);
        cp_async_commit();
        int buf = 0;
        for (unsigned j = j0; j < pairs; j += stride, buf ^= 1) {
            if (j + stride < pairs) stage(j + stride, buf ^ 1);
            cp_async_commit();
            cp_async_wait_prev();                // this thread's copies of pair j have landed
            float w[2], x[3][2], k[3][2];
            unsigned long long id[2];
            {
                float2 v;
                v = stg[buf][0][t]; w[0] = v.x; w[1] = v.y;              // zero-filled past the count: dead
                for (int c = 0; c < 3; ++c) { v = stg[buf][1 + c][t]; x[c][0] = v.x; x[c][1] = v.y; }
                for (int c = 0; c < 3; ++c) { v = stg[buf][4 + c][t]; k[c][0] = v.x; k[c][1] = v.y; }
                const ulonglong2 u = sid[buf][t];
                id[0] = u.x; id[1] = u.y;
            }
            float k0[2], inv[2], nd[3][2], chi[2], lam[2];
            bool fly[2], due[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                k0[q] = f_sqrt(sum_sq<true>(k[0][q], k[1][q], k[2][q]));
                inv[q] = f_div(1.0f, k0[q]);
                fly[q] = w[q] > 0.f && k0[q] > 0.f;
                for (int c = 0; c < 3; ++c) nd[c][q] = __fmul_rn(k[c][q], inv[q]);
            }
            // chi of both photons, case by case
            if (a.field_zero == 1 && a.field_kind == QED_FIELD_ROTATING_E) {
                const float e0 = a.prm_f[0] * ph0.c, e1 = a.prm_f[0] * ph0.s;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float ax = diff_of_products(k[1][q], 0.f, k[2][q], e1);
                    const float ay = diff_of_products(k[2][q], e0, k[0][q], 0.f);
                    const float az = diff_of_products(k[0][q], e1, k[1][q], e0);
                    chi[q] = f_sqrt(sum_sq<true>(ax, ay, az)) * (float)(1.0 / RS);
                }
            } else {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float xq[3] = {x[0][q], x[1][q], x[2][q]}, kq[3] = {k[0][q], k[1][q], k[2][q]};
                    float E[3], B[3];
                    field_at<float>(a, xq, ph0, E, B);
                    unsigned n64 = 0;                 // a sum of squares: no evaluation in FP64
                    chi[q] = photon_chi<float, true>(k0[q], kq, E, B, n64, a.field_zero == 1 ? 1 : 2);
                }
            }
            // rates (rate_pair<float>, its last piece's continuation apart)
            bool beyond = false;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float u = piece_coord(chi[q], 2 * RSEG);
                beyond = beyond || u >= (float)PAIR_NSEG;
                const int i = u > 0.f ? min((int)u, PAIR_NSEG - 1) : 0;
                const float F = f_exp(__fsub_rn(piece_eval(tab, i, __fsub_rn(u, (float)i)), f_div(8.0f / 3.0f, chi[q])));
                lam[q] = __fmul_rn(__fmul_rn(alpha_r, inv[q]), chi[q] >= (float)PAIR_CHI_MIN ? F : 0.f);
            }
            if (beyond)
                for (int q = 0; q < 2; ++q) lam[q] = __fmul_rn(__fmul_rn(alpha_r, inv[q]), rate_pair<float>(s_coef, chi[q]));
            due[0] = fly[0] && lam[0] > skip;
            due[1] = fly[1] && lam[1] > skip;
            float uw[2], vw[2];
            uint4 r[2];
            if (due[0] || due[1]) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    r[q] = event_draw(a.keys, id[q], step, 0u);
                    Uniform<float>::draw(r[q].x, r[q].y, uw[q], vw[q]);
                    // as in photon_flight: above this the photon reaches the step end
                    due[q] = due[q] && !(vw[q] > lam[q] * (h * (float)(1.0 + 1e-4)));
                }
            }
            if (due[0] || due[1]) {
                for (int q = 0; q < 2; ++q) {
                    if (!due[q]) continue;
                    const float dth = f_div(Uniform<float>::neglog(q ? uw[1] : uw[0], q ? vw[1] : vw[0]), q ? lam[1] : lam[0]);
                    if (dth >= a.dt_f_gt) {
                        due[q] = false;
                        continue;
                    }
                    const float kq[3] = {q ? k[0][1] : k[0][0], q ? k[1][1] : k[1][0], q ? k[2][1] : k[2][0]};
                    const float nq[3] = {q ? nd[0][1] : nd[0][0], q ? nd[1][1] : nd[1][0], q ? nd[2][1] : nd[2][0]};
                    float xq[3] = {q ? x[0][1] : x[0][0], q ? x[1][1] : x[1][0], q ? x[2][1] : x[2][0]};
                    for (int c = 0; c < 3; ++c) xq[c] = __fmaf_rn(nq[c], dth, xq[c]);
                    const uint4 rq = q ? r[1] : r[0];
                    pair_create<float>(a, tm, icdf, xq, kq, q ? k0[1] : k0[0], nq[0], nq[1], nq[2], (double)dth,
                                       q ? w[1] : w[0], q ? id[1] : id[0], 0u, make_uint2(rq.z, rq.w), ps.n64,
                                       [](int, unsigned) {});
                    const unsigned i = 2 * j + q;
                    st<float>(S.w, i, 0.f);       // the photon is eliminated
                    S.nev[i] += 1u;
                    ++ps.pr;
                    ps.mx = 1u;
                    for (int c = 0; c < 3; ++c) { if (q) x[c][1] = xq[c]; else x[c][0] = xq[c]; }
                }
            } else {
                due[0] = due[1] = false;
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                ps.ph += w[q] > 0.f ? 1 : 0;
                if (fly[q] && !due[q])
                    for (int c = 0; c < 3; ++c) x[c][q] = __fmaf_rn(nd[c][q], h, x[c][q]);
            }
            // a dead photon's place is written back as it was read
            if (2 * j + 1 < n) {
                if (w[0] > 0.f || w[1] > 0.f) {
                    reinterpret_cast<float2 *>(S.x)[j] = make_float2(x[0][0], x[0][1]);
                    reinterpret_cast<float2 *>(S.y)[j] = make_float2(x[1][0], x[1][1]);
                    reinterpret_cast<float2 *>(S.z)[j] = make_float2(x[2][0], x[2][1]);
                }
            } else if (w[0] > 0.f) {
                st<float>(S.x, 2 * j, x[0][0]); st<float>(S.y, 2 * j, x[1][0]); st<float>(S.z, 2 * j, x[2][0]);
            }
        }
        __syncwarp();
        flush_stats(ctl, ps);
    }
    if (n == 0) return;                          // as in k_photon_pass
    if (last_block(ctl) && threadIdx.x < 2) ctl->born[threadIdx.x] = count_now(ctl, threadIdx.x);
}
#endif

// ---- the accumulated-optical-depth method (QED_METHOD_OPTICAL_DEPTH) ----
// Per particle and step: the rate at the step start; an optical depth not
// drawn yet (od <= 0) is drawn as -ln u from Philox(id, step, OD_DRAW); od
// decreases by lambda dt; the particle is pushed by dt; if od <= 0 the event
// happens at the end of the step (chi at the end point, energy from
// Philox(id, step, 0) words 2-3) and a fresh od = -ln u from words 0-1.  At
// most one event per particle and step; the children start at the next step.
// od is held in the context's precision: a particle that does not convert
// draws no random number and does no FP64 arithmetic in FP32 mode.
constexpr unsigned OD_DRAW = 0xFFFFFFFEu;

// -ln u from words 0-1 of a draw (the FP32 form keeps full relative precision
// for u near 1)
template <class T> __device__ __forceinline__ T od_exp1(const uint4 &r) {
    T u, v;
    Uniform<T>::draw(r.x, r.y, u, v);
    return Uniform<T>::neglog(u, v);
}

// od after this step's decrement, drawn first when not drawn yet.  The
// product is rounded on its own (no contraction), as in the oracle.
template <class T>
__device__ __forceinline__ T od_advance(const PassArgs &a, unsigned step, unsigned long long id, T od, T lam) {
    if (!(od > (T)0)) od = od_exp1<T>(event_draw(a.keys, id, step, OD_DRAW));
    return od - mul_rn<T>(lam, dt_of<T>(a));
}

template <class T>
__global__ void __launch_bounds__(256, (sizeof(T) == 4 ? 4 : 1)) k_lepton_od(PassArgs a) {
    __shared__ __align__(16) T s_coef[RateWords<T>::N];
    __shared__ StepTime s_tm;
    for (int i = threadIdx.x; i < RateWords<T>::N; i += blockDim.x) s_coef[i] = reinterpret_cast<const T *>(a.coef)[i];
    if (threadIdx.x == 0) s_tm = load_step_time(a);
    __syncthreads();
    const StepTime &tm = s_tm;
    DevCtl *ctl = a.ctl;
    const unsigned long long b0 = ctl->begin[0], n0 = ctl->end[0] - b0;
    const unsigned long long b1 = ctl->begin[1], n1 = ctl->end[1] - b1;
    const unsigned long long n = n0 + n1;
    const LeptonCtx<T> c{a, ctl, s_coef, a.coef32, reinterpret_cast<const T *>(a.icdf_em), ctl->capacity[2], 0u, (T)(ALPHA * RS),
                         tm, time_phase<T, StepTime>(tm, 0.0)};
    PassStats ps;
    for (unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (unsigned long long)gridDim.x * blockDim.x) {
        const int s = j < n0 ? 0 : 1;
        const unsigned long long i = s == 0 ? b0 + j : b1 + (j - n0);
        const SpeciesDev &S = a.sp[s];
        const T w = ld<T>(S.w, i);
        if (!(w > (T)0)) continue;
        T x[3] = {ld<T>(S.x, i), ld<T>(S.y, i), ld<T>(S.z, i)};
        T p[3] = {ld<T>(S.px, i), ld<T>(S.py, i), ld<T>(S.pz, i)};
        const unsigned long long id = __ldg(S.id + i);
        T od = ld<T>(S.od, i);
        ++ps.lep;
        T E[3], B[3];
        field_at<T>(a, x, c.ph0, E, B);
        T gam, chi, p2;
        lepton_chi<T>(p, E, B, gam, chi, p2, ps.n64, a.field_zero);
        const T lam = p2 > (T)0 ? c.alpha_r / gam * rate_em<T>(c.coef, chi) : (T)0;
        od = od_advance<T>(a, tm.step, id, od, lam);
        const T qch = s == 0 ? (T)-1 : (T)1;
        boris<T>(x, p, qch, E, B, dt_of<T>(a), a.field_zero == 1, id, tm.step, 0u);
        unsigned k = 0;
        if (od <= (T)0) {
            // the event at the end of the step
            field_tau<T>(a, tm, x, a.dt, E, B);
            lepton_chi<T>(p, E, B, gam, chi, p2, ps.n64, a.field_zero);
            const uint4 r = event_draw(a.keys, id, tm.step, 0u);
            T om, ue, ve;
            Uniform<T>::draw(r.z, r.w, ue, ve);
            const T delta = sample_emission<T>(c.icdf, chi, ue, ve, &om);
            T kv[3];
            if (recoil<T>(a, p, gam, p2, delta, om, kv))
                append_photon<T>(a, ctl, c.cap_ph, x, kv, w, event_draw(a.child_keys, id, tm.step, 0u));
            od = od_exp1<T>(r);
            k = 1;
        }
        st<T>(S.x, i, x[0]); st<T>(S.y, i, x[1]); st<T>(S.z, i, x[2]);
        st<T>(S.px, i, p[0]); st<T>(S.py, i, p[1]); st<T>(S.pz, i, p[2]);
        st<T>(S.od, i, od);
        if (k) S.nev[i] += 1u;
        ps.em += k;
        ps.mx = max(ps.mx, k);
    }
    __syncwarp();
    flush_stats(ctl, ps);
}

template <class T>
__global__ void __launch_bounds__(256, (sizeof(T) == 4 ? 4 : 1)) k_photon_od(PassArgs a) {
    __shared__ __align__(16) T s_coef[RateWords<T>::N];
    __shared__ StepTime s_tm;
    for (int i = threadIdx.x; i < RateWords<T>::N; i += blockDim.x) s_coef[i] = reinterpret_cast<const T *>(a.coef)[i];
    if (threadIdx.x == 0) s_tm = load_step_time(a);
    __syncthreads();
    const StepTime &tm = s_tm;
    DevCtl *ctl = a.ctl;
    const unsigned long long b = ctl->begin[2], n = ctl->end[2] - b;
    const unsigned long long cap_e = ctl->capacity[0], cap_p = ctl->capacity[1];
    const T *icdf = reinterpret_cast<const T *>(a.icdf_pair);
    const T alpha_r = (T)(ALPHA * RS);
    const SpeciesDev &S = a.sp[2];
    PassStats ps;
    const Phase<T> ph0 = time_phase<T, StepTime>(tm, 0.0);
    // FP32: each thread stages its next photon in shared memory (two
    // buffers) while it works on the current one, as in the step-start pass
    constexpr bool STAGE = sizeof(T) == 4;
    constexpr int NB = STAGE ? 2 : 1, NF = STAGE ? 10 : 1, NT = STAGE ? 256 : 1;
    __shared__ __align__(16) float stg[NB][NF][NT];       // w x y z kx ky kz id(2 words) od
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    auto stage = [&](unsigned long long jj, int buf) {
        if constexpr (STAGE) {
            const unsigned long long ii = b + jj;
            const int t = threadIdx.x;
            cp_async4(&stg[buf][0][t], reinterpret_cast<const float *>(S.w) + ii);
            cp_async4(&stg[buf][1][t], reinterpret_cast<const float *>(S.x) + ii);
            cp_async4(&stg[buf][2][t], reinterpret_cast<const float *>(S.y) + ii);
            cp_async4(&stg[buf][3][t], reinterpret_cast<const float *>(S.z) + ii);
            cp_async4(&stg[buf][4][t], reinterpret_cast<const float *>(S.px) + ii);
            cp_async4(&stg[buf][5][t], reinterpret_cast<const float *>(S.py) + ii);
            cp_async4(&stg[buf][6][t], reinterpret_cast<const float *>(S.pz) + ii);
            cp_async4(&stg[buf][7][t], S.id + ii);
            cp_async4(&stg[buf][8][t], reinterpret_cast<const unsigned *>(S.id + ii) + 1);
            cp_async4(&stg[buf][9][t], reinterpret_cast<const float *>(S.od) + ii);
        }
    };
    const unsigned long long j0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (STAGE) {
        if (j0 < n) stage(j0, 0);
        cp_async_commit();
    }
    int buf = 0;
    for (unsigned long long j = j0; j < n; j += stride, buf ^= 1) {
        const unsigned long long i = b + j;
        T w, x[3], kv[3], od;
        unsigned long long id;
        if constexpr (STAGE) {
            if (j + stride < n) stage(j + stride, buf ^ 1);
            cp_async_commit();
            cp_async_wait_prev();                // this thread's copies of photon j have landed
            const int t = threadIdx.x;
            w = stg[buf][0][t];
            x[0] = stg[buf][1][t]; x[1] = stg[buf][2][t]; x[2] = stg[buf][3][t];
            kv[0] = stg[buf][4][t]; kv[1] = stg[buf][5][t]; kv[2] = stg[buf][6][t];
            id = (unsigned long long)__float_as_uint(stg[buf][7][t]) |
                 ((unsigned long long)__float_as_uint(stg[buf][8][t]) << 32);
            od = stg[buf][9][t];
        } else {
            w = ld<T>(S.w, i);
            x[0] = ld<T>(S.x, i); x[1] = ld<T>(S.y, i); x[2] = ld<T>(S.z, i);
            kv[0] = ld<T>(S.px, i); kv[1] = ld<T>(S.py, i); kv[2] = ld<T>(S.pz, i);
            id = __ldg(S.id + i);
            od = ld<T>(S.od, i);
        }
        if (!(w > (T)0)) continue;
        ++ps.ph;
        const T k0 = f_sqrt(kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2]);
        unsigned k = 0;
        if (k0 > (T)0) {
            const T inv = f_div((T)1, k0);
            const T nx = kv[0] * inv, ny = kv[1] * inv, nz = kv[2] * inv;
            T E[3], B[3];
            field_at<T>(a, x, ph0, E, B);
            T chi = photon_chi<T>(k0, kv, E, B, ps.n64, a.field_zero);
            const T lam = alpha_r / k0 * rate_pair<T>(s_coef, chi);
            od = od_advance<T>(a, tm.step, id, od, lam);
            const T h = dt_of<T>(a);
            x[0] += nx * h; x[1] += ny * h; x[2] += nz * h;
            if (od <= (T)0) {
                // pair creation at the end of the step
                field_tau<T>(a, tm, x, a.dt, E, B);
                chi = photon_chi<T>(k0, kv, E, B, ps.n64, a.field_zero);
                const uint4 r = event_draw(a.keys, id, tm.step, 0u);
                T om, ue, ve;
                Uniform<T>::draw(r.z, r.w, ue, ve);
                const T delta = sample_pair<T>(icdf, chi, ue, ve, &om);
                T em = delta * k0, ep = om * k0;
                em = em < (T)1 ? (T)1 : em;
                ep = ep < (T)1 ? (T)1 : ep;
                const T pm = f_sqrt((em - (T)1) * (em + (T)1)), pp = f_sqrt((ep - (T)1) * (ep + (T)1));
                const uint4 rid = event_draw(a.child_keys, id, tm.step, 0u);
                const unsigned long long se = warp_append(&ctl->count[0], 1);
                const unsigned long long sp = warp_append(&ctl->count[1], 1);
                if (se < cap_e) {
                    const SpeciesDev &P = a.sp[0];
                    st<T>(P.x, se, x[0]); st<T>(P.y, se, x[1]); st<T>(P.z, se, x[2]);
                    st<T>(P.px, se, pm * nx); st<T>(P.py, se, pm * ny); st<T>(P.pz, se, pm * nz);
                    st<T>(P.w, se, w);
                    P.id[se] = (unsigned long long)rid.x | ((unsigned long long)rid.y << 32);
                    P.nev[se] = 0u;
                    st<T>(P.od, se, (T)0);
                } else {
                    note_overflow(ctl, 0, se);
                }
                if (sp < cap_p) {
                    const SpeciesDev &P = a.sp[1];
                    st<T>(P.x, sp, x[0]); st<T>(P.y, sp, x[1]); st<T>(P.z, sp, x[2]);
                    st<T>(P.px, sp, pp * nx); st<T>(P.py, sp, pp * ny); st<T>(P.pz, sp, pp * nz);
                    st<T>(P.w, sp, w);
                    P.id[sp] = (unsigned long long)rid.z | ((unsigned long long)rid.w << 32);
                    P.nev[sp] = 0u;
                    st<T>(P.od, sp, (T)0);
                } else {
                    note_overflow(ctl, 1, sp);
                }
                w = (T)0;
                k = 1;
            }
        }
        st<T>(S.x, i, x[0]); st<T>(S.y, i, x[1]); st<T>(S.z, i, x[2]);
        st<T>(S.od, i, od);
        if (k) { st<T>(S.w, i, w); S.nev[i] += 1u; }
        ps.pr += k;
        ps.mx = max(ps.mx, k);
    }
    __syncwarp();
    flush_stats(ctl, ps);
}

// ---- host side ----
template <class K>
inline qed_status timed_launch(qed_ctx *ctx, int which, K launch) {
    if (!ctx->cfg.profile) {
        launch();
        return QED_OK;
    }
    if (ctx->ev_used[which] == qed_ctx::EVN) {
        qed_status e = sfq_drain_events(ctx);
        if (e != QED_OK) return e;
    }
    const int i = ctx->ev_used[which]++;
    SFQ_CUDA(cudaEventRecord(ctx->ev[which][i][0], ctx->stream));
    launch();
    SFQ_CUDA(cudaEventRecord(ctx->ev[which][i][1], ctx->stream));
    return QED_OK;
}

// Persistent grids: one wave of resident blocks (SM count x blocks per SM
// from the occupancy calculator unless the configuration fixes it).
template <class K> inline int resident_blocks(const qed_ctx *ctx, K kernel, int threads) {
    int per_sm = ctx->cfg.blocks_per_sm;
    if (per_sm <= 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
            per_sm = 1;
    }
    return ctx->sm_count * per_sm;
}

template <class K> inline int resident_blocks_smem(const qed_ctx *ctx, K kernel, int threads, size_t smem) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return ctx->sm_count * per_sm;
}

template <class T, bool FRESH, bool MLP>
qed_status launch_leptons(qed_ctx *ctx, PassArgs &a, cudaGraphConditionalHandle h, int loop) {
    const int threads = LB<T>, smem = MLP ? MLP_SMEM_BYTES : 0;
    if constexpr (MLP) {
        static bool attr_set = false;   // the attribute is per function, set once
        if (!attr_set) {
            SFQ_CUDA(cudaFuncSetAttribute(k_lepton_pass<T, FRESH, MLP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            attr_set = true;
        }
    }
    const int bl = MLP ? resident_blocks_smem(ctx, k_lepton_pass<T, FRESH, MLP>, threads, smem)
                       : resident_blocks(ctx, k_lepton_pass<T, FRESH, MLP>, threads);
    qed_status e =
        timed_launch(ctx, 0, [&] { k_lepton_pass<T, FRESH, MLP><<<bl, threads, smem, ctx->stream>>>(a, h, loop); });
    SFQ_LAUNCHED(ctx, 1);
    return e;
}

// One step (a.pass == 0): the photons, then the leptons with the newborns;
// or a further launch for newborns left behind (a.pass > 0).  loop: the
// lepton pass sets the condition of the step graph's while node h.
template <class T>
qed_status launch_pass(qed_ctx *ctx, PassArgs &a, bool photons, cudaGraphConditionalHandle h, int loop) {
    qed_status e = QED_OK;
    if (a.pass == 0 && photons) {
#if !SFQ_GRID
        if (sizeof(T) == 4 && a.field_kind != QED_FIELD_STANDING_CP && a.field_zero != 0) {
            const int bp = resident_blocks(ctx, k_photon_pass2, 256);
            e = timed_launch(ctx, 1, [&] { k_photon_pass2<<<bp, 256, 0, ctx->stream>>>(a); });
        } else
#endif
        {
            const int bp = resident_blocks(ctx, k_photon_pass<T>, 256);
            e = timed_launch(ctx, 1, [&] { k_photon_pass<T><<<bp, 256, 0, ctx->stream>>>(a); });
        }
        if (e != QED_OK) return e;
        SFQ_LAUNCHED(ctx, 1);
    }
    if (a.mlp_w16)
        e = a.pass == 0 ? launch_leptons<T, true, true>(ctx, a, h, loop) : launch_leptons<T, false, true>(ctx, a, h, loop);
    else
        e = a.pass == 0 ? launch_leptons<T, true, false>(ctx, a, h, loop) : launch_leptons<T, false, false>(ctx, a, h, loop);
    if (e != QED_OK) return e;
    SFQ_CUDA(cudaGetLastError());
    return QED_OK;
}

// Blocks of the one-launch emission run for n leptons; 0: the steps are taken
// one by one.  A block keeps its 256 (FP64 128) leptons through all steps, so
// with more leptons than resident threads it runs all steps for one tile after
// another, drains its stack in every step of every tile, and has none of the
// pass's staged loads; the pass's launches then cost less than that.  One
// launch against a launch per step (graph), gain at 2 / 10 / 40 steps, uniform
// B (a wave is 77824 leptons in both precisions):
//   FP32  1 wave 1.20 / 1.84 / 2.71   2 waves 0.99 / 1.43 / 1.72   3 waves
//         0.99 / 1.18 / 1.34   4 waves 1.00 / 1.07 / 1.14   6 waves 0.88 /
//         0.87 / 0.89   13 waves 0.68 / 0.61 / 0.61 (2.4 times as slow at 4e6 leptons)
//   FP64  1 wave 1.13 / 1.52 / 1.70   2 waves 0.86 / 1.00 / 1.07   3 waves
//         0.72 / 0.82 / 0.85   13 waves 0.56 / 0.57 / 0.57
// and much the same in the other analytic fields; on the grid FP32 3 waves
// 0.98 / 1.00 / 1.00, 4 waves 0.84 / 0.89 / 0.92, FP64 2 waves 0.78 / 0.90 / 0.94.
template <class T>
int steps_blocks(const qed_ctx *ctx, int64_t n, int nsteps) {
    const int waves = (sizeof(T) == 4 ? 3 : 1) + (!SFQ_GRID && nsteps >= 16 ? 1 : 0);
    const int bl = resident_blocks(ctx, k_lepton_steps<T>, LB<T>);
    return n <= (int64_t)waves * bl * LB<T> ? bl : 0;
}

template <class T>
qed_status launch_steps(qed_ctx *ctx, PassArgs &a, int64_t step0, int nsteps, int blocks) {
    qed_status e = timed_launch(ctx, 0, [&] {
        k_lepton_steps<T><<<blocks, LB<T>, 0, ctx->stream>>>(a, (unsigned long long)step0, nsteps);
    });
    if (e != QED_OK) return e;
    SFQ_LAUNCHED(ctx, 1);
    SFQ_CUDA(cudaGetLastError());
    return QED_OK;
}

// the optical-depth method: one launch per species kind and step
template <class T>
qed_status launch_od(qed_ctx *ctx, PassArgs &a, bool photons) {
    cudaStream_t st = ctx->stream;
    const int bl = resident_blocks(ctx, k_lepton_od<T>, 256);
    qed_status e = timed_launch(ctx, 0, [&] { k_lepton_od<T><<<bl, 256, 0, st>>>(a); });
    if (e != QED_OK) return e;
    SFQ_LAUNCHED(ctx, 1);
    if (photons) {
        const int bp = resident_blocks(ctx, k_photon_od<T>, 256);
        e = timed_launch(ctx, 1, [&] { k_photon_od<T><<<bp, 256, 0, st>>>(a); });
        if (e != QED_OK) return e;
        SFQ_LAUNCHED(ctx, 1);
    }
    SFQ_CUDA(cudaGetLastError());
    return QED_OK;
}

}  // namespace SFQ_PASS_NS
}  // namespace sfq
