// K4 / K5: removal of dead particles and global leveling
// (arXiv:2409.17299 Sec. 4.2: the merge step is where filtering and thinning
// happen; Sec. 5.1: "global leveling" keeps the particle count bounded).
//
// Compaction is in place and deterministic: with A alive entries among
// [0, N), the r-th dead slot below A receives the r-th alive entry at or
// above A (ranks from block scans), so no entry is read after it is written.
//
// Leveling: the threshold w* solves sum_i min(1, w_i / w*) = cap (solved on
// the device, see k_level).  Particle i is kept with probability
// min(1, w_i / w*) from Philox(seed; id, step, 0xFFFFFFFF), and kept
// particles below w* get weight w*.
#include <math.h>
#include <string.h>

#include "sfqed_device.cuh"
#include "sfqed_internal.h"

namespace sfq {
namespace {

constexpr int CT = 256;            // threads per compaction block
constexpr int CITEMS = 4;          // items per thread
constexpr int CTILE = CT * CITEMS; // entries per block

template <class T> __device__ __forceinline__ bool alive_at(const void *w, unsigned long long i) {
    return ld<T>(w, i) > (T)0;
}

// exclusive scan of one value per thread over the block; returns the prefix,
// writes the block total
__device__ __forceinline__ unsigned block_scan(unsigned v, unsigned *sw, unsigned *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sw[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned t = lane < (int)(blockDim.x >> 5) ? sw[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sw[lane] = t;   // inclusive warp totals
    }
    __syncthreads();
    const unsigned before = (wid > 0 ? sw[wid - 1] : 0u) + x - v;
    *total = sw[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before;
}

template <class T>
__global__ void __launch_bounds__(CT) k_count_alive(const void *w, const DevCtl *ctl, int s,
                                                    unsigned long long *blk) {
    const unsigned long long n = ctl->count[s];
    const unsigned long long base = (unsigned long long)blockIdx.x * CTILE;
    unsigned c = 0;
    for (int r = 0; r < CITEMS; ++r) {
        const unsigned long long i = base + r * CT + threadIdx.x;
        if (i < n && alive_at<T>(w, i)) ++c;
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    __shared__ unsigned sw[32];
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0;
        for (int k = 0; k < CT / 32; ++k) t += sw[k];
        blk[blockIdx.x] = t;
    }
}

// single block: exclusive scan of the per-block counts, total -> alive[s]
__global__ void k_scan_blocks(unsigned long long *blk, long long nb, DevCtl *ctl, int s) {
    __shared__ unsigned long long sw[32];
    __shared__ unsigned long long carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (long long b0 = 0; b0 < nb; b0 += blockDim.x) {
        const long long i = b0 + threadIdx.x;
        const unsigned long long v = i < nb ? blk[i] : 0ull;
        unsigned long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sw[wid] = x;
        __syncthreads();
        if (wid == 0) {
            unsigned long long t = lane < (int)(blockDim.x >> 5) ? sw[lane] : 0ull;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            sw[lane] = t;
        }
        __syncthreads();
        const unsigned long long before = carry + (wid > 0 ? sw[wid - 1] : 0ull) + x - v;
        if (i < nb) blk[i] = before;
        __syncthreads();
        if (threadIdx.x == 0) carry += sw[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        ctl->alive[s] = carry;
        ctl->holes[s] = 0;
    }
}

// dead slots below A record their rank (= number of dead entries before them)
// and are counted (H, the number of holes)
template <class T>
__global__ void __launch_bounds__(CT) k_mark_holes(const void *w, DevCtl *ctl, int s,
                                                   const unsigned long long *blk, unsigned long long *slots) {
    __shared__ unsigned sw[32];
    const unsigned long long n = ctl->count[s], A = ctl->alive[s];
    const unsigned long long base = (unsigned long long)blockIdx.x * CTILE;
    unsigned long long run = blk[blockIdx.x];
    unsigned my_holes = 0;
    for (int r = 0; r < CITEMS; ++r) {
        const unsigned long long i = base + r * CT + threadIdx.x;
        const bool al = i < n && alive_at<T>(w, i);
        unsigned tot;
        const unsigned before = block_scan(al ? 1u : 0u, sw, &tot);
        if (i < A && !al) {
            slots[i - (run + before)] = i;     // rank < A <= n (slots holds n entries)
            ++my_holes;
        }
        run += tot;
    }
    for (int o = 16; o > 0; o >>= 1) my_holes += __shfl_down_sync(0xffffffffu, my_holes, o);
    if ((threadIdx.x & 31) == 0 && my_holes) atomicAdd(&ctl->holes[s], (unsigned long long)my_holes);
}

template <class T> __device__ __forceinline__ void move_entry(const SpeciesDev &S, unsigned long long d,
                                                              unsigned long long i) {
    st<T>(S.x, d, ld<T>(S.x, i)); st<T>(S.y, d, ld<T>(S.y, i)); st<T>(S.z, d, ld<T>(S.z, i));
    st<T>(S.px, d, ld<T>(S.px, i)); st<T>(S.py, d, ld<T>(S.py, i)); st<T>(S.pz, d, ld<T>(S.pz, i));
    st<T>(S.w, d, ld<T>(S.w, i));
    S.id[d] = S.id[i];
    S.nev[d] = S.nev[i];
    if (S.od) st<T>(S.od, d, ld<T>(S.od, i));
}

// alive entries at or above A move into the holes, in rank order: the mover
// rank is the number of alive entries in [A, i) = alive_before(i) - (A - H)
template <class T>
__global__ void __launch_bounds__(CT) k_fill_holes(SpeciesDev S, DevCtl *ctl, int s, const unsigned long long *blk,
                                                   const unsigned long long *slots) {
    __shared__ unsigned sw[32];
    const unsigned long long n = ctl->count[s], A = ctl->alive[s], H = ctl->holes[s];
    const unsigned long long alive_below_A = A - H;
    const unsigned long long base = (unsigned long long)blockIdx.x * CTILE;
    if (base + CTILE <= A) return;                 // whole tile below A: nothing moves
    unsigned long long run = blk[blockIdx.x];
    for (int r = 0; r < CITEMS; ++r) {
        const unsigned long long i = base + r * CT + threadIdx.x;
        const bool al = i < n && alive_at<T>(S.w, i);
        unsigned tot;
        const unsigned before = block_scan(al ? 1u : 0u, sw, &tot);
        if (al && i >= A) {
            const unsigned long long ab = run + before;     // alive entries before i
            const unsigned long long rank = ab - alive_below_A;
            if (ab >= alive_below_A && rank < H) {
                const unsigned long long d = slots[rank];
                if (d < A) move_entry<T>(S, d, i);
                else atomicExch(&ctl->bad_index, i + 1);
            } else {
                atomicExch(&ctl->bad_index, i + 1);
            }
        }
        run += tot;
    }
}

// Entries a tile pass covers: the count (at most the capacity), none once a
// step ran out of capacity or a device check failed (the state is then left
// as it is for the caller's replay).
__device__ __forceinline__ unsigned long long tile_count(const DevCtl *ctl, int s) {
    if (ctl->overflow || ctl->timeout || ctl->bad_index) return 0;
    const unsigned long long c = ctl->count[s], cp = ctl->capacity[s];
    return c < cp ? c : cp;
}

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
constexpr unsigned long long INF_BITS = 0x7ff0000000000000ull;    // +inf as double bits

// ---- leveling: device-resident piecewise-exact Newton iteration ----
// S(w) = sum_i min(1, w_i / w) = A(w) / w + C(w) with A = sum of weights below
// w and C = count at or above w.  On the piece of w containing the root,
// S = A/w + C, whose root is A / (cap - C): evaluating (A, C) at w and jumping
// to A / (cap - C) lands on the root once the piece is right, otherwise it
// moves toward it; a bisection bracket keeps every step inside [lo, hi].
// Block partial sums are reduced in a fixed order (deterministic result).
constexpr int LEVEL_ITERS = 40;

// smallest float >= a positive double (v < d <=> v < ceil_f(d) for floats v)
__host__ __device__ __forceinline__ float ceil_f(double d) {
#ifdef __CUDA_ARCH__
    return __double2float_ru(d);
#else
    float f = (float)d;
    if ((double)f < d) f = nextafterf(f, INFINITY);
    return f;
#endif
}

__host__ __device__ __forceinline__ double double_of_bits(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, sizeof d);
    return d;
#endif
}

// Warm start: the first pass evaluates at the species' previous threshold
// times the last growth of the threshold (in a cascade that grows steadily
// the next root lies close by), else at +inf.  The start changes only the
// path: the root of its own piece is the same from any start.
__device__ __forceinline__ LevelIter lev_start(double prev, double ratio) {
    LevelIter it;
    const double inf = __longlong_as_double(0x7ff0000000000000ll);
    const double w0 = prev > 0.0 && prev < inf ? (ratio > 0.0 ? prev * ratio : prev) : inf;
    it.lo = 0.0;
    it.hi = inf;
    it.w = w0;
    it.w_up = w0 < inf ? ceil_f(w0) : __int_as_float(0x7f800000);
    it.wstar = 0.0;
    it.wstar_up = it.wstar_f = it.wstar_inv_f = 0.f;
    it.done = 0;
    it.iters = 0;
    it.alive = 0;
    return it;
}

// error-free float-float accumulation (TwoSum), accurate to ~2^-48 relative
struct FF {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float b) {
        const float t = hi + b;
        const float bp = t - hi;
        const float e = (hi - (t - bp)) + (b - bp);
        hi = t;
        lo += e;
    }
};

// double-double accumulation (TwoSum) for the reduction of block partials
struct DD {
    double hi = 0.0, lo = 0.0;
    __device__ __forceinline__ void add(double b) {
        const double t = hi + b;
        const double bp = t - hi;
        lo += (hi - (t - bp)) + (b - bp);
        hi = t;
    }
};

__host__ __device__ __forceinline__ void lev_finish(LevelIter &it, double wstar) {
    it.done = 1;
    it.wstar = wstar;
    it.wstar_up = wstar > 0.0 ? ceil_f(wstar) : 0.f;
    it.wstar_f = (float)wstar;
    it.wstar_inv_f = wstar > 0.0 ? (float)(1.0 / wstar) : 0.f;
}

// Newton step from the sums at it.w: A (weights below w), C (count at or
// above w), N (alive count), M (largest weight, double bits).  PL and PH
// (double bits; PH = 0: not given) bound the piece of w: the largest weight
// below w and the smallest at or above it.  A Newton point c with
// PL < c <= PH lies on w's piece, where A and C are those just summed, so the
// next pass would return c itself and finish there: the iteration finishes at
// c now, with the same result and one pass fewer.
__host__ __device__ void lev_advance(LevelIter &it, double A, unsigned long long C, unsigned long long N,
                                     unsigned long long M, long long cap, unsigned long long PL = 0,
                                     unsigned long long PH = 0) {
    const double inf = double_of_bits(0x7ff0000000000000ull);
    const double w = it.w;
    if (it.iters == 0) {                           // first pass: at +inf or at a warm start w
        it.alive = N;
        if (N <= (unsigned long long)cap) { lev_finish(it, 0.0); return; }
        it.hi = double_of_bits(M) * (double)N / (double)cap;                    // S(hi) <= cap
        it.lo = 0.0;
        if (w < inf) {
            const double S = A / w + (double)C;
            if (S > (double)cap) it.lo = w;
            else if (w < it.hi) it.hi = w;
        }
    } else {
        const double S = A / w + (double)C;
        if (S > (double)cap) it.lo = w; else it.hi = w;
    }
    ++it.iters;
    double c = (double)cap > (double)C ? A / ((double)cap - (double)C) : inf;
    if (c == w) { lev_finish(it, w); return; }     // root of its own piece
    const bool newton = c > it.lo && c <= it.hi;
    if (!newton) c = 0.5 * (it.lo + it.hi);
    // stop at double resolution of the bracket (hi, evaluated, is the answer)
    if (!(c > it.lo && c <= it.hi) || (c == it.hi && it.hi == w) || it.iters >= LEVEL_ITERS) {
        lev_finish(it, it.hi);
        return;
    }
    if (newton && PH != 0 && c > double_of_bits(PL) && c <= double_of_bits(PH)) {
        lev_finish(it, c);
        return;
    }
    it.w = c;
    it.w_up = ceil_f(c);
}

constexpr int LEV_T = 256;

// This thread's share of the sums at w_at (w_up in FP32) over entries t0, t0 + stride, ...
template <class T>
__device__ __forceinline__ void lev_accumulate(const void *w, unsigned long long n, unsigned long long t0,
                                               unsigned long long stride, double w_at, float w_up, double &A,
                                               unsigned long long &C, unsigned long long &N, unsigned long long &M,
                                               unsigned long long &L, unsigned long long &H) {
    C = 0;
    N = 0;
    M = 0;
    L = 0;
    H = INF_BITS;
    if constexpr (sizeof(T) == 4) {
        // FP32 weights: exact float comparisons and float-float sums, no FP64 per element
        const float wc = w_up;
        FF acc;
        unsigned mb = 0, c = 0, nn = 0, lb = 0, hb = 0x7f800000u;    // positive floats order like their bits
        auto one = [&](float v) {
            if (v > 0.f) {
                ++nn;
                mb = max(mb, __float_as_uint(v));
                if (v < wc) {
                    acc.add(v);
                    lb = max(lb, __float_as_uint(v));
                } else {
                    ++c;
                    hb = min(hb, __float_as_uint(v));
                }
            }
        };
        const float *wf = reinterpret_cast<const float *>(w);
        unsigned long long i0 = 0;
        if ((reinterpret_cast<uintptr_t>(wf) & 15u) == 0) {
            const float4 *w4 = reinterpret_cast<const float4 *>(wf);
            const unsigned long long n4 = n / 4;
            unsigned long long j = t0;
            for (; j + 3 * stride < n4; j += 4 * stride) {      // four 16-byte loads in flight
                const float4 a = __ldg(w4 + j), b = __ldg(w4 + j + stride);
                const float4 c4 = __ldg(w4 + j + 2 * stride), d = __ldg(w4 + j + 3 * stride);
                one(a.x); one(a.y); one(a.z); one(a.w);
                one(b.x); one(b.y); one(b.z); one(b.w);
                one(c4.x); one(c4.y); one(c4.z); one(c4.w);
                one(d.x); one(d.y); one(d.z); one(d.w);
            }
            for (; j < n4; j += stride) {
                const float4 a = __ldg(w4 + j);
                one(a.x); one(a.y); one(a.z); one(a.w);
            }
            i0 = n4 * 4;
        }
        for (unsigned long long i = i0 + t0; i < n; i += stride) one(wf[i]);
        A = (double)acc.hi + (double)acc.lo;
        C = c;
        N = nn;
        M = nn ? dbits((double)__uint_as_float(mb)) : 0ull;
        L = lb ? dbits((double)__uint_as_float(lb)) : 0ull;
        H = hb < 0x7f800000u ? dbits((double)__uint_as_float(hb)) : INF_BITS;
    } else {
        const double wc = w_at;
        double comp = 0.0;           // Kahan
        A = 0.0;
        for (unsigned long long i = t0; i < n; i += stride) {
            const double v = (double)ld<T>(w, i);
            if (!(v > 0.0)) continue;
            ++N;
            M = max(M, dbits(v));
            if (v < wc) {
                const double y = v - comp;
                const double t = A + y;
                comp = (t - A) - y;
                A = t;
                L = max(L, dbits(v));
            } else {
                ++C;
                H = min(H, dbits(v));
            }
        }
    }
}

struct LevSums {
    double A;                               // sum of the weights below w
    unsigned long long C, N, M, L, H;       // at or above w; alive; largest; the bounds of w's piece (double bits)
};

// One pass over a species: this block's sums at w, written to its place of
// the block partials.
template <class T>
__device__ __forceinline__ void lev_block_sums(const void *w, unsigned long long n, double w_at, float w_up,
                                               LevelWork *lw, int s) {
    const unsigned long long t0 = (unsigned long long)blockIdx.x * LEV_T + threadIdx.x;
    const unsigned long long stride = (unsigned long long)gridDim.x * LEV_T;
    LevSums v;
    lev_accumulate<T>(w, n, t0, stride, w_at, w_up, v.A, v.C, v.N, v.M, v.L, v.H);
    __shared__ LevSums sw[LEV_T / 32];
    for (int o = 16; o > 0; o >>= 1) {
        v.A += __shfl_down_sync(0xffffffffu, v.A, o);
        v.C += __shfl_down_sync(0xffffffffu, v.C, o);
        v.N += __shfl_down_sync(0xffffffffu, v.N, o);
        v.M = max(v.M, __shfl_down_sync(0xffffffffu, v.M, o));
        v.L = max(v.L, __shfl_down_sync(0xffffffffu, v.L, o));
        v.H = min(v.H, __shfl_down_sync(0xffffffffu, v.H, o));
    }
    __syncthreads();                        // sw is read by the previous species' sums
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        LevSums t = sw[0];
        for (int k = 1; k < LEV_T / 32; ++k) {
            t.A += sw[k].A; t.C += sw[k].C; t.N += sw[k].N;
            t.M = max(t.M, sw[k].M); t.L = max(t.L, sw[k].L); t.H = min(t.H, sw[k].H);
        }
        const int b = s * LEVEL_MAX_BLOCKS + blockIdx.x;
        lw->partA[b] = t.A;
        lw->partC[b] = t.C;
        lw->partN[b] = t.N;
        lw->partM[b] = t.M;
        lw->partL[b] = t.L;
        lw->partH[b] = t.H;
    }
}

// The block partials of a species reduced by one warp in a fixed order
// (partials lane, lane + 32, ..., then a butterfly), so that the result does
// not depend on which block does it.
__device__ __forceinline__ LevSums lev_reduce(const LevelWork *lw, int s, int blocks) {
    const int base = s * LEVEL_MAX_BLOCKS;
    DD acc;
    unsigned long long c = 0, nn = 0, m = 0, pl = 0, ph = INF_BITS;
    for (int b = threadIdx.x & 31; b < blocks; b += 32) {
        acc.add(__ldcg(&lw->partA[base + b]));
        c += __ldcg(&lw->partC[base + b]);
        nn += __ldcg(&lw->partN[base + b]);
        m = max(m, __ldcg(&lw->partM[base + b]));
        pl = max(pl, __ldcg(&lw->partL[base + b]));
        ph = min(ph, __ldcg(&lw->partH[base + b]));
    }
    for (int o = 16; o > 0; o >>= 1) {
        DD x = acc;
        const double oh = __shfl_down_sync(0xffffffffu, acc.hi, o), ol = __shfl_down_sync(0xffffffffu, acc.lo, o);
        x.add(oh);
        x.lo += ol;
        acc = x;
        c += __shfl_down_sync(0xffffffffu, c, o);
        nn += __shfl_down_sync(0xffffffffu, nn, o);
        m = max(m, __shfl_down_sync(0xffffffffu, m, o));
        pl = max(pl, __shfl_down_sync(0xffffffffu, pl, o));
        ph = min(ph, __shfl_down_sync(0xffffffffu, ph, o));
    }
    return LevSums{acc.hi + acc.lo, c, nn, m, pl, ph};       // valid in lane 0
}

struct LevWeights {
    const void *w[3];       // the species' weights (null: not leveled in this launch)
};

// Leveling thresholds of all species in one cooperative launch: each species
// above the cap runs its iteration (lev_advance) over the same passes; in a
// pass every block sums its share of each species' weights, the last block
// to arrive reduces the partials and advances the iterations, and the others
// wait for it (bounded; a wait that runs out marks the step as timed out).
// Arrivals are counted in the control block, which every batch of steps and
// every merge call opens anew: a wait that ran out leaves arrivals behind, and
// no later leveling may count them.
//
// A pass over 1e7 weights takes 6 us from DRAM and less from L2, but as two
// launches of a graph's while loop per pass and species it took 19 to 25 us,
// and the standing-wave cascade takes about five passes for each of three
// species: 0.36 ms of a 1.9 ms step (1e7 per species), 0.07 ms here (three
// passes from the better start; a warp per species reduces the partials:
// 0.26 ms with a block-wide tree per species and the old start).  With the
// merged compaction launches: 40 steps of that cascade 88.2 -> 72.4 ms, 20
// steps on the grid (1e6 per species) 20.8 -> 13.3 ms, 20 steps at the start
// of a cascade 2.86 -> 2.00 ms, 40 steps at 5e7 photons 87.0 -> 83.9 ms.
constexpr unsigned LEV_POLLS = 1u << 24;      // unless cfg.level_polls gives another limit

template <class T>
__global__ void __launch_bounds__(LEV_T, 4) k_level(LevWeights lwt, DevCtl *ctl, LevelWork *lw, long long cap,
                                                    unsigned max_polls) {
    __shared__ int s_last, s_out;
    __shared__ double s_w[3];
    __shared__ float s_wup[3];
    __shared__ int s_done[3];
    const int t = threadIdx.x;
    const bool stop = ctl->overflow || ctl->timeout || ctl->bad_index;
    unsigned long long n[3];
    bool any = false;
    for (int s = 0; s < 3; ++s) {
        n[s] = min(ctl->count[s], ctl->capacity[s]);
        const bool on = lwt.w[s] && !stop && cap > 0 && n[s] > (unsigned long long)cap;
        if (!on) n[s] = 0;
        any = any || on;
        if (t == 0) {
            const LevelIter it = lev_start(lw->prev[s], lw->ratio[s]);
            s_w[s] = it.w;
            s_wup[s] = it.w_up;
            s_done[s] = !on;
            if (!on && blockIdx.x == 0) {
                LevelIter off = it;
                lev_finish(off, 0.0);
                lw->it[s] = off;
                lw->on[s] = 0;
            }
        }
    }
    if (!any) return;
    const unsigned long long round0 = *reinterpret_cast<volatile unsigned long long *>(&lw->round);
    __syncthreads();
    for (int pass = 0; pass <= LEVEL_ITERS; ++pass) {
        for (int s = 0; s < 3; ++s)
            if (!s_done[s]) lev_block_sums<T>(lwt.w[s], n[s], s_w[s], s_wup[s], lw, s);
        if (t == 0) {
            __threadfence();
            s_last = atomicAdd(&ctl->arrive, 1ull) == gridDim.x - 1;
            __threadfence();
        }
        __syncthreads();
        if (s_last) {
            const int s = t >> 5;                   // a warp per species
            if (s < 3 && !s_done[s]) {
                const LevSums v = lev_reduce(lw, s, (int)gridDim.x);
                if ((t & 31) == 0) {
                    LevelIter it;
                    if (pass == 0) it = lev_start(lw->prev[s], lw->ratio[s]);
                    else it = lw->it[s];
                    lev_advance(it, v.A, v.C, v.N, v.M, cap, v.L, v.H);
                    if (it.done && it.wstar > 0.0) {
                        const double r = it.wstar / lw->prev[s];
                        lw->ratio[s] = lw->prev[s] > 0.0 && r > 0.5 && r < 2.0 ? r : 1.0;
                        lw->prev[s] = it.wstar;
                    }
                    lw->it[s] = it;
                    lw->on[s] = 1;
                    __threadfence();
                }
            }
            __syncthreads();
            if (t == 0) {
                ctl->arrive = 0;
                __threadfence();
                atomicExch(&lw->round, round0 + pass + 1);
            }
        }
        if (t == 0) {
            unsigned polls = 0;
            s_out = 0;
            while (!s_last && *reinterpret_cast<volatile unsigned long long *>(&lw->round) != round0 + pass + 1) {
                if (++polls > max_polls) {
                    atomicExch(&ctl->timeout, 1ull);
                    s_out = 1;
                    break;
                }
                __nanosleep(40);
            }
            __threadfence();
            bool all = true;
            for (int s = 0; s < 3; ++s) {
                if (!s_done[s]) {
                    s_done[s] = __ldcg(&lw->it[s].done) != 0;
                    s_w[s] = __ldcg(&lw->it[s].w);
                    s_wup[s] = __ldcg(&lw->it[s].w_up);
                }
                all = all && s_done[s];
            }
            if (all) s_out = 1;
        }
        __syncthreads();
        if (s_out) break;
    }
}

// The sums of one species at w (a shard's part of a leveling over processes)
template <class T>
__global__ void __launch_bounds__(LEV_T) k_lev_eval(const void *w, unsigned long long n, double at, float up, int s,
                                                    LevelWork *lw) {
    __shared__ int s_last;
    lev_block_sums<T>(w, n, at, up, lw, s);
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&lw->arrive, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    if (threadIdx.x >= 32) return;
    const LevSums v = lev_reduce(lw, s, (int)gridDim.x);
    if (threadIdx.x == 0) {
        lw->sumA = v.A;
        lw->sumC = v.C;
        lw->sumN = v.N;
        lw->sumM = v.M;
        lw->arrive = 0;
    }
}

// ---- compaction by tiles (used after leveling and for converted photons) ----
// A tile of 4096 entries is one block of 256 threads; warp k owns entries
// [512 k, 512 k + 512) of the tile, 32 per round (coalesced).  Pass 1 lists
// the dead entries of each tile in index order (16-bit tile offsets) and
// counts the alive ones; a scan gives A (alive total) and H (dead entries
// below A); pass 2 lists the alive entries at or above A (the movers) by
// rank; pass 3 moves mover r into the r-th dead slot below A.  The passes
// cover all species of the merge step in one launch each (a species' step
// took seven launches of its own: 25 us of a 145 us step with few particles).
constexpr int LT = 256;
constexpr int LROUNDS = 16;
constexpr int LTILE = LT * LROUNDS;       // entries per tile (offsets fit 16 bits)
constexpr int LSPAN = 32 * LROUNDS;       // contiguous entries per warp

// Tiles holding entries of a species of n entries, and the tile grid: a
// kernel loops over tiles (grid stride), so its grid can be fixed by the
// species' capacity (a captured step graph) while the device count decides
// the work.
__device__ __forceinline__ long long tiles_of(unsigned long long n) { return (long long)((n + LTILE - 1) / LTILE); }

// What the passes work on: the species of `always`, and with `leveled` those
// whose leveling ran.
struct MergeArgs {
    SpeciesDev sp[3];
    DevCtl *ctl;
    LevelWork *lw;
    unsigned long long *blk[3];       // per tile: alive entries, then (pass 2 on) those before it
    unsigned short *dl[3];            // dead entries by tile
    unsigned long long *movers[3];
    long long nb[3];                  // tiles the buffers hold
    PhiloxKeys keys;
    unsigned step;                    // step index keying the draws, unless
    int step_from_ctl;                // it is the control block's current step
    int always, leveled;              // bits of species; leveled: bits of species that may have been
    int may_defer;
};

// entries of species s that the passes cover
__device__ __forceinline__ unsigned long long merge_count(const MergeArgs &m, int s) {
    const bool run = ((m.always >> s) & 1) || (((m.leveled >> s) & 1) && m.lw->on[s]);
    return run ? tile_count(m.ctl, s) : 0;
}

// Pass 1.  LEVEL: first keep particle i (0 < w_i < w*) with probability
// w_i / w*: the comparison u < w_i / w* is made in FP32 with a relative
// margin, and in FP64 (the oracle's test) only for draws within that margin
// of the boundary; kept particles get weight w*.
template <class T, bool LEVEL>
__global__ void __launch_bounds__(LT, 4) k_tile_dead(const __grid_constant__ MergeArgs m) {
    __shared__ unsigned wdead[LT / 32];
    DevCtl *ctl = m.ctl;
    const PhiloxKeys &keys = m.keys;
    // one species per row of blocks: its arrays and threshold are uniform
    const int s = 2 - (int)blockIdx.y;
    const unsigned long long n = merge_count(m, s);
    const long long nbe = tiles_of(n);
    const SpeciesDev S = m.sp[s];
    bool thin = false;
    double wstar = 0.0;
    float inv_f = 0.f, wup = 0.f, wnew = 0.f;
    if constexpr (LEVEL) {
        const LevelIter &it = m.lw->it[s];
        wstar = it.wstar;
        thin = ((m.leveled >> s) & 1) && it.done && wstar > 0.0;
        inv_f = it.wstar_inv_f;
        wup = it.wstar_up;
        wnew = it.wstar_f;
    }
    unsigned step = m.step;
    if (m.step_from_ctl) step = ctl->sv_step;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned removed = 0;
    // FP32 leveling: groups of four entries whose draws are computed together
    constexpr bool SPEC = LEVEL && sizeof(T) == 4;
    // entries per group of loads (with leveling four: eight FP64 weights and
    // ids and the next eight spill 88 bytes; level_apply at 1e7 weights 346 us against 334)
    constexpr int G = LEVEL ? 4 : 8;
    static_assert(LROUNDS % G == 0, "groups tile the rounds");
    for (long long tile = blockIdx.x; tile < nbe; tile += gridDim.x) {
        const unsigned long long base = (unsigned long long)tile * LTILE;
        const unsigned long long wbase = base + (unsigned long long)wid * LSPAN;
        unsigned mask[LROUNDS];
        unsigned cnt = 0;
        // weights and (leveling) ids of G entries issued together, and those of
        // the next G before this group's draws and stores.  The weights are
        // written by this kernel, so plain loads; the ids are not.
        T v[G], vn[G];
        unsigned long long idv[G], idn[G];
        auto load = [&](int c0, T (&vv)[G], unsigned long long (&ii)[G]) {
#pragma unroll
            for (int r = 0; r < G; ++r) {
                const unsigned long long i = wbase + (c0 + r) * 32 + lane;
                vv[r] = i < n ? ld<T>(S.w, i) : (T)0;
                ii[r] = (LEVEL && thin && i < n) ? __ldg(S.id + i) : 0ull;
            }
        };
        load(0, vn, idn);
#pragma unroll
        for (int c0 = 0; c0 < LROUNDS; c0 += G) {
#pragma unroll
            for (int r = 0; r < G; ++r) {
                v[r] = vn[r];
                idv[r] = idn[r];
            }
            if (c0 + G < LROUNDS) load(c0 + G, vn, idn);
            bool below[G];
#pragma unroll
            for (int r = 0; r < G; ++r) {
                if constexpr (sizeof(T) == 4) below[r] = LEVEL && thin && v[r] > (T)0 && (float)v[r] < wup;
                else below[r] = LEVEL && thin && v[r] > (T)0 && (double)v[r] < wstar;
            }
            // FP32 leveling: the G draws are computed together, outside the
            // per-entry branch, so their Philox rounds interleave (one draw
            // per branch ran the ten dependent rounds back to back); only the
            // entries below w* use theirs
            uint4 qv[G];
            if constexpr (SPEC) {
                if (thin) {
#pragma unroll
                    for (int r = 0; r < G; ++r) qv[r] = event_draw(keys, idv[r], step, 0xFFFFFFFFu);
                }
            }
#pragma unroll
            for (int r = 0; r < G; ++r) {
                const unsigned long long i = wbase + (c0 + r) * 32 + lane;
                bool dead = i < n && !(v[r] > (T)0);
                if (LEVEL && below[r]) {
                    const uint4 q = SPEC ? qv[r] : event_draw(keys, idv[r], step, 0xFFFFFFFFu);
                    const float uf = __uint2float_rn(q.x) * 0x1p-32f;     // u to within 2^-32 + FP32 rounding
                    const float pf = (float)v[r] * inv_f;
                    bool keep;
                    if (uf < pf * (1.0f - 1e-6f) - 0x1p-31f) keep = true;
                    else if (uf > pf * (1.0f + 1e-6f) + 0x1p-31f) keep = false;
                    else {
                        double u, vv;
                        Uniform<double>::draw(q.x, q.y, u, vv);
                        keep = u < (double)v[r] / wstar;
                    }
                    if (keep) {
                        if constexpr (sizeof(T) == 4) st<T>(S.w, i, wnew);
                        else st<T>(S.w, i, wstar);
                    } else {
                        st<T>(S.w, i, (T)0);
                        dead = true;
                        ++removed;
                    }
                }
                mask[c0 + r] = __ballot_sync(0xffffffffu, dead);
                cnt += __popc(mask[c0 + r]);
            }
        }
        if (lane == 0) wdead[wid] = cnt;
        __syncthreads();
        unsigned before = 0, total = 0;
#pragma unroll
        for (int k = 0; k < LT / 32; ++k) {
            const unsigned c = wdead[k];
            before += k < wid ? c : 0u;
            total += c;
        }
        unsigned short *tdl = m.dl[s] + base;
        const unsigned lt = (1u << lane) - 1u;
        unsigned run = before;
#pragma unroll
        for (int r = 0; r < LROUNDS; ++r) {
            if ((mask[r] >> lane) & 1u) tdl[run + __popc(mask[r] & lt)] = (unsigned short)(wid * LSPAN + r * 32 + lane);
            run += __popc(mask[r]);
        }
        if (threadIdx.x == 0) {
            const unsigned long long tn = n - base < (unsigned long long)LTILE ? n - base : (unsigned long long)LTILE;
            m.blk[s][tile] = tn - total;
        }
        __syncthreads();                       // wdead is rewritten by the next tile
    }
    if constexpr (LEVEL) {
        for (int o = 16; o > 0; o >>= 1) removed += __shfl_down_sync(0xffffffffu, removed, o);
        if (lane == 0 && removed) atomicAdd(&ctl->thinned, (unsigned long long)removed);
    }
}

// One block per species: exclusive scan of the counts of the tiles holding
// entries (blk[nbe] = A; each thread takes a run of consecutive tiles), then H
// from the alive entries of the tile that holds A.
// may_defer: while dead entries are at most DEFER_DEN-th of the species and
// the count leaves a fifth of the capacity free, the move is deferred (H = 0,
// the count stays): the dead entries (weight 0) are skipped by every pass
// until a later step compacts, with holes denser and fewer moves per step.
constexpr unsigned long long DEFER_DEN = 4;
constexpr int SCAN_T = 1024;

template <class T> __global__ void __launch_bounds__(SCAN_T) k_scan_tiles(const __grid_constant__ MergeArgs m) {
    __shared__ unsigned long long sw[SCAN_T / 32];
    const int s = blockIdx.x;
    DevCtl *ctl = m.ctl;
    const unsigned long long n = merge_count(m, s);
    if (n == 0) {
        if (threadIdx.x == 0) {                     // nothing moves, no entry counted
            ctl->alive[s] = min(ctl->count[s], ctl->capacity[s]);
            ctl->holes[s] = 0;
        }
        return;
    }
    const void *w = m.sp[s].w;
    unsigned long long *blk = m.blk[s];
    const long long nbe_all = tiles_of(n), nbe = nbe_all < m.nb[s] ? nbe_all : m.nb[s];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long per = (nbe + SCAN_T - 1) / SCAN_T;
    const long long i0 = min((long long)threadIdx.x * per, nbe), i1 = min(i0 + per, nbe);
    unsigned long long v = 0;
    for (long long i = i0; i < i1; ++i) v += blk[i];
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sw[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long t = sw[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sw[lane] = t;
    }
    __syncthreads();
    unsigned long long run = (wid > 0 ? sw[wid - 1] : 0ull) + x - v;
    for (long long i = i0; i < i1; ++i) {
        const unsigned long long c = blk[i];
        blk[i] = run;
        run += c;
    }
    const unsigned long long A = sw[SCAN_T / 32 - 1];
    const unsigned long long a = A / LTILE;
    unsigned long long below = A;                   // A on a tile boundary past the data: no holes
    __syncthreads();                                // blk and sw: written and read above
    if ((long long)a < nbe) {
        unsigned c = 0;
        for (unsigned long long i = a * LTILE + threadIdx.x; i < A; i += SCAN_T) c += alive_at<T>(w, i) ? 1u : 0u;
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if (lane == 0) sw[wid] = c;
        __syncthreads();
        unsigned long long tc = 0;
        for (int k = 0; k < SCAN_T / 32; ++k) tc += sw[k];
        below = blk[a] + tc;
    }
    if (threadIdx.x == 0) {
        blk[nbe] = A;
        if (m.may_defer && (n - A) * DEFER_DEN <= n && 5 * n <= 4 * ctl->capacity[s]) {
            ctl->alive[s] = n;                      // nothing moves; count unchanged
            ctl->holes[s] = 0;
            ctl->deferred[s] = n - A;
        } else {
            ctl->alive[s] = A;
            ctl->holes[s] = A - below;
            if (A - below) atomicAdd(&ctl->moved, A - below);
            ctl->deferred[s] = 0;
        }
    }
}

// pass 2: movers (alive entries at or above A) by rank, over the tiles that
// reach past A
template <class T> __global__ void __launch_bounds__(LT) k_tile_movers(const __grid_constant__ MergeArgs m) {
    __shared__ unsigned walive[LT / 32];
    DevCtl *ctl = m.ctl;
    for (int s = 0; s < 3; ++s) {
        const unsigned long long n = merge_count(m, s), A = ctl->alive[s], H = ctl->holes[s];
        if (n == 0 || H == 0) continue;
        const void *w = m.sp[s].w;
        const unsigned long long *blk = m.blk[s];
        const unsigned long long below_A = A - H;      // alive entries below A
        const long long nbe = tiles_of(n);
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        for (long long tile = (long long)(A / LTILE) + blockIdx.x; tile < nbe; tile += gridDim.x) {
            const unsigned long long base = (unsigned long long)tile * LTILE;
            const unsigned long long wbase = base + (unsigned long long)wid * LSPAN;
            unsigned amask[LROUNDS];
            unsigned cnt = 0;
#pragma unroll
            for (int r = 0; r < LROUNDS; ++r) {
                const unsigned long long i = wbase + r * 32 + lane;
                amask[r] = __ballot_sync(0xffffffffu, i < n && alive_at<T>(w, i));
                cnt += __popc(amask[r]);
            }
            if (lane == 0) walive[wid] = cnt;
            __syncthreads();
            unsigned before = 0;
            for (int k = 0; k < wid; ++k) before += walive[k];
            const unsigned lt = (1u << lane) - 1u;
            unsigned long long run = blk[tile] + before;   // alive entries before this warp's span
#pragma unroll
            for (int r = 0; r < LROUNDS; ++r) {
                const unsigned long long i = wbase + r * 32 + lane;
                if (((amask[r] >> lane) & 1u) && i >= A) {
                    const unsigned long long ab = run + __popc(amask[r] & lt);
                    const unsigned long long rank = ab - below_A;
                    if (ab >= below_A && rank < H) m.movers[s][rank] = i;
                    else atomicExch(&ctl->bad_index, i + 1);
                }
                run += __popc(amask[r]);
            }
            __syncthreads();                       // walive is rewritten by the next tile
        }
    }
}

// pass 3: the k-th dead entry of tile b has rank (dead entries before the
// tile) + k; dead entries below A receive the mover of their rank.  (One
// warp per tile with four moves in flight per lane was measured slower: the
// moves are bound by the scattered 32-byte sectors they write, not by the
// latency of their loads.)  The last block to finish takes over the counts.
template <class T> __global__ void __launch_bounds__(LT) k_tile_fill(const __grid_constant__ MergeArgs m) {
    __shared__ int s_last;
    DevCtl *ctl = m.ctl;
    unsigned long long n3[3];
    for (int s = 0; s < 3; ++s) {
        const unsigned long long n = merge_count(m, s), A = ctl->alive[s], H = ctl->holes[s];
        n3[s] = n;
        if (n == 0 || H == 0) continue;
        const SpeciesDev &S = m.sp[s];
        const unsigned long long *blk = m.blk[s];
        const long long nfill = tiles_of(A);
        for (long long tile = blockIdx.x; tile < nfill; tile += gridDim.x) {
            const unsigned long long base = (unsigned long long)tile * LTILE;
            const unsigned long long tn = n - base < (unsigned long long)LTILE ? n - base : (unsigned long long)LTILE;
            const unsigned long long alive_t = blk[tile + 1] - blk[tile];
            const unsigned dead_t = (unsigned)(tn - alive_t);
            const unsigned long long dead_before = base - blk[tile];
            const unsigned short *tdl = m.dl[s] + base;
            for (unsigned k = threadIdx.x; k < dead_t; k += LT) {
                const unsigned long long i = base + tdl[k];
                if (i >= A) break;                      // offsets ascend: the rest lie at or above A too
                const unsigned long long r = dead_before + k;
                if (r < H) {
                    const unsigned long long src = m.movers[s][r];
                    if (src >= A && src < n) move_entry<T>(S, i, src);
                    else atomicExch(&ctl->bad_index, i + 1);
                } else {
                    atomicExch(&ctl->bad_index, i + 1);
                }
            }
        }
    }
    // every block has read the counts above
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&ctl->arrive, 1ull) == gridDim.x - 1;
        __threadfence();
        if (s_last) {
            ctl->arrive = 0;
            for (int s = 0; s < 3; ++s)
                if (n3[s]) ctl->count[s] = ctl->end[s] = ctl->begin[s] = ctl->alive[s];
        }
    }
}

// Resident blocks of a tile kernel (its grid loops over tiles), at most one
// block per tile.
template <class K> static unsigned tile_grid(const qed_ctx *ctx, K kernel, long long nb) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, LT, 0) != cudaSuccess || per_sm < 1) per_sm = 1;
    const long long g = (long long)ctx->sm_count * per_sm;
    return (unsigned)(nb < g ? (nb > 0 ? nb : 1) : g);
}

// The work buffers of one merge over species of at most bound[s] entries:
// a word per tile and two more, and per entry 16 bits of dead list and half a
// mover index.  bound: an upper bound of the device's count (the host's count,
// or the capacity where only the device knows the count).
static int64_t merge_blk_words(const int64_t bound[3]) {
    int64_t n = 0;
    for (int s = 0; s < 3; ++s) n += (bound[s] + LTILE - 1) / LTILE + 2;
    return n;
}

// words of species s: the dead list, then the movers
static int64_t dead_words(int64_t bound) { return (bound + 3) / 4 + 1; }
static int64_t mover_words(int64_t bound) { return bound / 2 + 1; }
static int64_t merge_slot_words(const int64_t bound[3]) {
    int64_t n = 0;
    for (int s = 0; s < 3; ++s) n += dead_words(bound[s]) + mover_words(bound[s]);
    return n;
}

template <class T>
static qed_status merge_args(qed_ctx *ctx, const qed_particles *p, const int64_t bound[3], MergeArgs &m) {
    memset(&m, 0, sizeof m);
    if (ctx->blk_cap < merge_blk_words(bound) || ctx->slots_cap < merge_slot_words(bound)) return QED_ERR_STATE;
    unsigned long long *blk = ctx->blk, *slots = ctx->slots;
    for (int s = 0; s < 3; ++s) {
        const qed_species &S = p->s[s];
        m.sp[s] = SpeciesDev{S.x, S.y, S.z, S.px, S.py, S.pz, S.w, reinterpret_cast<unsigned long long *>(S.id),
                             S.nevents, nullptr, ctx->od[s]};
        m.nb[s] = (bound[s] + LTILE - 1) / LTILE;
        m.blk[s] = blk;
        blk += m.nb[s] + 2;
        m.dl[s] = reinterpret_cast<unsigned short *>(slots);
        slots += dead_words(bound[s]);
        m.movers[s] = slots;
        slots += mover_words(bound[s]);
    }
    m.ctl = ctx->ctl;
    m.lw = ctx->lev;
    m.keys = philox_keys(ctx->cfg.seed);
    return QED_OK;
}

// The four compaction passes over the species of m.always and, with
// m.leveled, those whose leveling ran (four launches for all of them).
template <class T, bool LEVEL> static qed_status compact_launch(qed_ctx *ctx, const MergeArgs &m) {
    long long nb_max = 0;
    for (int s = 0; s < 3; ++s)
        if ((((m.always | m.leveled) >> s) & 1) && m.nb[s] > nb_max) nb_max = m.nb[s];
    if (nb_max == 0) return QED_OK;
    cudaStream_t st = ctx->stream;
    k_tile_dead<T, LEVEL><<<dim3(tile_grid(ctx, k_tile_dead<T, LEVEL>, nb_max), 3), LT, 0, st>>>(m);
    k_scan_tiles<T><<<3, SCAN_T, 0, st>>>(m);
    k_tile_movers<T><<<tile_grid(ctx, k_tile_movers<T>, nb_max), LT, 0, st>>>(m);
    k_tile_fill<T><<<tile_grid(ctx, k_tile_fill<T>, nb_max), LT, 0, st>>>(m);
    SFQ_LAUNCHED(ctx, 4);
    SFQ_CUDA(cudaGetLastError());
    return QED_OK;
}

// Leveling thresholds of the species of `mask` (device: those whose count
// exceeds the cap), one cooperative launch.
template <class T> static qed_status level_launch(qed_ctx *ctx, const qed_particles *p, int mask) {
    LevWeights w{};
    for (int s = 0; s < 3; ++s) w.w[s] = ((mask >> s) & 1) && p->s[s].capacity > 0 ? p->s[s].w : nullptr;
    int per_sm = 0;
    SFQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_level<T>, LEV_T, 0));
    int blocks = ctx->sm_count * (per_sm < 4 ? (per_sm > 0 ? per_sm : 1) : 4);
    blocks = blocks > LEVEL_MAX_BLOCKS ? LEVEL_MAX_BLOCKS : blocks;
    long long cap = (long long)ctx->cfg.thin_cap;
    unsigned polls = ctx->cfg.level_polls > 0 ? (unsigned)ctx->cfg.level_polls : LEV_POLLS;
    void *args[] = {&w, &ctx->ctl, &ctx->lev, &cap, &polls};
    SFQ_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<void *>(k_level<T>), dim3((unsigned)blocks), dim3(LEV_T), args,
                                         0, ctx->stream));
    SFQ_LAUNCHED(ctx, 1);
    return QED_OK;
}

// A merge step: species of level_mask are leveled when their count exceeds
// the cap (decided on the device), dead entries are removed from those and
// from the species of `always`.  bound: an upper bound of each device count.
template <class T>
static qed_status merge_impl(qed_ctx *ctx, const qed_particles *p, const int64_t bound[3], int level_mask, int always,
                             int64_t step, bool step_from_ctl, bool may_defer) {
    MergeArgs m;
    for (int s = 0; s < 3; ++s)
        if (bound[s] <= 0) {
            level_mask &= ~(1 << s);
            always &= ~(1 << s);
        }
    if (!(level_mask | always)) return QED_OK;
    qed_status e = merge_args<T>(ctx, p, bound, m);
    if (e != QED_OK) return e;
    m.step = (unsigned)step;
    m.step_from_ctl = step_from_ctl ? 1 : 0;
    m.always = always;
    m.leveled = level_mask;
    m.may_defer = may_defer ? 1 : 0;
    if (!level_mask) return compact_launch<T, false>(ctx, m);
    e = level_launch<T>(ctx, p, level_mask);
    return e != QED_OK ? e : compact_launch<T, true>(ctx, m);
}

// ---- leveling over shards (one species split across processes) ----
// The threshold is a property of all shards together: each shard evaluates
// its sums at the current point (level_eval), the caller adds them over the
// shards (an all-reduce) and advances the iteration with the same step the
// device uses (sfq_level_advance), then each shard applies w* (level_apply).
template <class T>
qed_status level_eval_impl(qed_ctx *ctx, qed_species *sp, double w, double *A, int64_t *C, int64_t *N, double *M) {
    cudaStream_t st = ctx->stream;
    int blocks = ctx->sm_count * 4;
    blocks = blocks > LEVEL_MAX_BLOCKS ? LEVEL_MAX_BLOCKS : blocks;
    const unsigned long long n = (unsigned long long)sp->count;
    *A = *M = 0.0;
    *C = *N = 0;
    if (n == 0) return QED_OK;
    k_lev_eval<T><<<blocks, LEV_T, 0, st>>>(sp->w, n, w, ceil_f(w), 0, ctx->lev);
    SFQ_LAUNCHED(ctx, 1);
    SFQ_CUDA(cudaGetLastError());
    struct {
        double A;
        unsigned long long C, N, M;
    } h;
    SFQ_CUDA(cudaMemcpyAsync(&h, &ctx->lev->sumA, sizeof h, cudaMemcpyDeviceToHost, st));
    SFQ_CUDA(cudaStreamSynchronize(st));
    *A = h.A;
    *C = (int64_t)h.C;
    *N = (int64_t)h.N;
    *M = double_of_bits(h.M);
    return QED_OK;
}

}  // namespace
}  // namespace sfq

using namespace sfq;

// The captured step holds addresses inside these buffers: it goes when one of
// them does, and the next batch of steps captures anew.
qed_status sfq_ensure_work(qed_ctx *ctx, int64_t n_blocks, int64_t n_slots) {
    if (ctx->blk_cap < n_blocks || ctx->slots_cap < n_slots) sfq_step_graph_free(ctx);
    if (ctx->blk_cap < n_blocks) {
        if (ctx->blk) SFQ_CUDA(cudaFreeAsync(ctx->blk, ctx->stream));
        ctx->blk = nullptr;
        ctx->blk_cap = 0;
        if (cudaMallocAsync(&ctx->blk, sizeof(unsigned long long) * (size_t)n_blocks, ctx->stream) != cudaSuccess)
            return QED_ERR_NOMEM;
        ctx->blk_cap = n_blocks;
    }
    if (ctx->slots_cap < n_slots) {
        if (ctx->slots) SFQ_CUDA(cudaFreeAsync(ctx->slots, ctx->stream));
        ctx->slots = nullptr;
        ctx->slots_cap = 0;
        if (cudaMallocAsync(&ctx->slots, sizeof(unsigned long long) * (size_t)n_slots, ctx->stream) != cudaSuccess)
            return QED_ERR_NOMEM;
        ctx->slots_cap = n_slots;
    }
    return QED_OK;
}

qed_status sfq_ensure_merge(qed_ctx *ctx, const int64_t bound[3]) {
    return sfq_ensure_work(ctx, merge_blk_words(bound), merge_slot_words(bound));
}

unsigned *sfq_entry_words(const qed_ctx *ctx, const int64_t bound[3], int s) {
    int64_t at = dead_words(bound[s]);                  // the movers of species s: half a 64-bit word per entry
    for (int k = 0; k < s; ++k) at += dead_words(bound[k]) + mover_words(bound[k]);
    return reinterpret_cast<unsigned *>(ctx->slots + at);
}

qed_status sfq_merge(qed_ctx *ctx, const qed_particles *p, const int64_t bound[3], int level_mask, int always,
                     int64_t step, bool step_from_ctl, bool may_defer) {
    if (ctx->cfg.precision == QED_FP32)
        return merge_impl<float>(ctx, p, bound, level_mask, always, step, step_from_ctl, may_defer);
    return merge_impl<double>(ctx, p, bound, level_mask, always, step, step_from_ctl, may_defer);
}

qed_status sfq_level_eval(qed_ctx *ctx, qed_species *sp, double w, double *A, int64_t *C, int64_t *N, double *M) {
    if (ctx->cfg.precision == QED_FP32) return level_eval_impl<float>(ctx, sp, w, A, C, N, M);
    return level_eval_impl<double>(ctx, sp, w, A, C, N, M);
}

qed_status sfq_level_apply_species(qed_ctx *ctx, const qed_particles *p, int s, double wstar, int64_t step) {
    LevelIter h{};
    lev_finish(h, wstar > 0.0 ? wstar : 0.0);
    SFQ_CUDA(cudaMemcpyAsync(&ctx->lev->it[s], &h, sizeof h, cudaMemcpyHostToDevice, ctx->stream));
    const int64_t bound[3] = {p->s[0].count, p->s[1].count, p->s[2].count};
    if (bound[s] <= 0) return QED_OK;
    qed_status e = sfq_ensure_merge(ctx, bound);
    if (e != QED_OK) return e;
    MergeArgs m;
    const bool f32 = ctx->cfg.precision == QED_FP32;
    e = f32 ? merge_args<float>(ctx, p, bound, m) : merge_args<double>(ctx, p, bound, m);
    if (e != QED_OK) return e;
    m.step = (unsigned)step;
    m.always = m.leveled = 1 << s;             // w* is given: no threshold to find
    return f32 ? compact_launch<float, true>(ctx, m) : compact_launch<double, true>(ctx, m);
}

void sfq_level_advance(double *lo, double *hi, double *w, double *wstar, int64_t *iters, int64_t *done,
                       int64_t *alive, double A, int64_t C, int64_t N, double M, int64_t cap) {
    LevelIter it{};
    it.lo = *lo;
    it.hi = *hi;
    it.w = *w;
    it.wstar = *wstar;
    it.iters = (unsigned long long)*iters;
    it.done = (unsigned long long)*done;
    it.alive = (unsigned long long)*alive;
    unsigned long long mb;
    memcpy(&mb, &M, sizeof mb);
    lev_advance(it, A, (unsigned long long)C, (unsigned long long)N, mb, (long long)cap);
    *lo = it.lo;
    *hi = it.hi;
    *w = it.w;
    *wstar = it.wstar;
    *iters = (int64_t)it.iters;
    *done = (int64_t)it.done;
    *alive = (int64_t)it.alive;
}

// ---------------------------------------------------------------------------
// Compaction that allocates nothing.  Some callers cannot call cudaMalloc:
// their device memory is owned entirely by another allocator (a host code's
// memory pool), or they cannot accept the device-wide synchronisation that
// cudaMalloc / cudaFree may cause inside their time loop.  This variant keeps
// its scratch (control words, per-block counts, hole ranks) in one
// file-scope device array of fixed size, which every GPU that loads the
// library holds until the process exits.
// ---------------------------------------------------------------------------
namespace sfq {
namespace {
constexpr long long NA_MAX_ENTRIES = 1ll << 20;                       // largest species count accepted
constexpr long long NA_CTL_WORDS = ((long long)sizeof(DevCtl) + 255) / 256 * 32;
constexpr long long NA_BLK_WORDS = (NA_MAX_ENTRIES / CTILE + 2 + 31) / 32 * 32;
constexpr long long NA_WORDS = NA_CTL_WORDS + NA_BLK_WORDS + NA_MAX_ENTRIES;

__global__ void k_noalloc_begin(DevCtl *ctl, unsigned long long count) {
    // the array keeps the previous call's contents: reset what must start at zero
    ctl->count[0] = count;
    ctl->capacity[0] = count;
    ctl->alive[0] = 0;
    ctl->holes[0] = 0;
    ctl->bad_index = 0;
}
}  // namespace
}  // namespace sfq

static __device__ __align__(256) unsigned long long g_noalloc_scratch[sfq::NA_WORDS];

namespace {
constexpr int NA_MAX_DEVICES = 64;
unsigned long long *g_noalloc_addr[NA_MAX_DEVICES];   // device address of the array, per device
}

template <class T>
static qed_status noalloc_compact(qed_species *sp, void *od, cudaStream_t st, unsigned long long *base) {
    using namespace sfq;
    DevCtl *ctl = reinterpret_cast<DevCtl *>(base);
    unsigned long long *blk = base + NA_CTL_WORDS;
    unsigned long long *slots = blk + NA_BLK_WORDS;
    const long long n = sp->count;
    const long long nb = (n + CTILE - 1) / CTILE;
    SpeciesDev S{sp->x, sp->y, sp->z, sp->px, sp->py, sp->pz, sp->w,
                 reinterpret_cast<unsigned long long *>(sp->id), sp->nevents, nullptr, od};
    k_noalloc_begin<<<1, 1, 0, st>>>(ctl, (unsigned long long)n);
    k_count_alive<T><<<(unsigned)nb, CT, 0, st>>>(sp->w, ctl, 0, blk);
    k_scan_blocks<<<1, 1024, 0, st>>>(blk, nb, ctl, 0);
    k_mark_holes<T><<<(unsigned)nb, CT, 0, st>>>(sp->w, ctl, 0, blk, slots);
    k_fill_holes<T><<<(unsigned)nb, CT, 0, st>>>(S, ctl, 0, blk, slots);
    SFQ_CUDA(cudaGetLastError());
    unsigned long long res[2];   // alive, bad index
    SFQ_CUDA(cudaMemcpyAsync(&res[0], &ctl->alive[0], sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    SFQ_CUDA(cudaMemcpyAsync(&res[1], &ctl->bad_index, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    SFQ_CUDA(cudaStreamSynchronize(st));
    if (res[1]) return QED_ERR_STATE;
    sp->count = (int64_t)res[0];
    return QED_OK;
}

extern "C" qed_status qed_compact_species_noalloc(qed_species *sp, void *od_dev, int precision, void *cuda_stream) {
    using namespace sfq;
    if (!sp || (precision != QED_FP64 && precision != QED_FP32)) return QED_ERR_INVALID;
    // the optical-depth array moves with the particles; element alignment as in qed_set_optical_depth
    if (od_dev && (reinterpret_cast<uintptr_t>(od_dev) % (precision == QED_FP32 ? 4u : 8u))) return QED_ERR_INVALID;
    if (sp->count < 0 || sp->count > sp->capacity) return QED_ERR_INVALID;
    if (sp->count > NA_MAX_ENTRIES) return QED_ERR_INVALID;
    if (sp->count == 0) return QED_OK;
    const void *ptrs[] = {sp->x, sp->y, sp->z, sp->px, sp->py, sp->pz, sp->w, sp->id, sp->nevents};
    for (const void *q : ptrs)
        if (!q || (reinterpret_cast<uintptr_t>(q) & 15u)) return QED_ERR_INVALID;
    int dev = 0;
    SFQ_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= NA_MAX_DEVICES) return QED_ERR_INVALID;
    if (!g_noalloc_addr[dev]) {
        // once per device, with that device current: the host-side name of the
        // array is not a device address, so ask the runtime for it
        void *p = nullptr;
        SFQ_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        g_noalloc_addr[dev] = static_cast<unsigned long long *>(p);
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (precision == QED_FP32) return noalloc_compact<float>(sp, od_dev, st, g_noalloc_addr[dev]);
    return noalloc_compact<double>(sp, od_dev, st, g_noalloc_addr[dev]);
}
