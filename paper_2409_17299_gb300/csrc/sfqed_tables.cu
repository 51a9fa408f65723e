// K1: build the rate approximant and the inverse-CDF tables on the device.
//
// arXiv:2409.17299 Sec. 3: event rates come from polynomial approximations of
// precomputed rates and photon / pair energies from precomputed tables of the
// inverse cumulative probability over (chi, energy).  The underlying
// probabilities are the quasi-classical (LCFA) ones:
//   emission  dW/dd ~ ((1-d) + 1/(1-d)) K_{2/3}(y) - int_y^inf K_{1/3},  y = 2d/(3 chi (1-d))
//   pair      dW/dd ~ (d/(1-d) + (1-d)/d) K_{2/3}(y) + int_y^inf K_{1/3},  y = 2/(3 chi d (1-d))
// Both are integrated on the whole line in z (emission y = e^z; pair
// d = 1/(1+e^-z)) with composite 16-point Gauss-Legendre panels.
//
// Two builders.  FP32 contexts read the tables rounded to float: their
// nodes come from Chebyshev interpolants of the Bessel functions
// (sfqed_tables32.cu, 1e-15 from the sums here, 1.6 ms).  FP64 contexts get
// the sums below, rounded as they have always been, because trajectories in
// strong standing waves amplify a last-bit change of the tables (1e-15 to
// 1e-2 in 500 steps of the paper's test problem).
//
// What bounds the FP64 build: FP64 arithmetic, K_{2/3} and the integral of
// K_{1/3} in the root solves of the 44,126 table nodes (up to 100 iterations
// of 17 points each).  One block per table row, which also recomputed the
// emission panels' Bessel values for every chi and cosh t and e^{-y cosh t}
// for each of the two functions, took 432 ms per context; 94 ms now: panels
// and nodes are spread over the whole chip, the emission panels' values (they
// depend on y alone) are computed once, and the two trapezoid sums share
// their exponentials and read cosh t from a table where the step is 0.1.
// Products and sums that the compiler may or may not fuse are written out.
#include <math.h>

#include "sfqed_device.cuh"
#include "sfqed_internal.h"
#include "sfqed_tables.cuh"

namespace sfq {
namespace {

// Trapezoid points t_j = 0.1 j: cosh t, cosh(2 t / 3), cosh(t / 3)
constexpr int NTRIG = 64;
struct Trig {
    double ch[NTRIG], c23[NTRIG], c13[NTRIG];
};

// what the quadrature keeps between its kernels
struct TableWork {
    Trig trig;
    double gamma[4];                  // Gamma(1/3), Gamma(5/3), Gamma(2/3), Gamma(4/3)
    double chi[ROWS];
    struct { double y, k23, k13; } em[EZ_NP * GLN];      // the emission panels' nodes, whatever chi
    double mass[ROWS * EZ_NP];        // panel integrals per row
    double below[(EM_NCHI + PAIR_NCHI) * (EZ_NP + 1)], above[(EM_NCHI + PAIR_NCHI) * (EZ_NP + 1)];
    double fnode[NCOEF];              // rate form at the Chebyshev nodes
};

// what the kernels keep in shared memory
struct TableShared {
    Trig trig;
    double gamma[4];
};

__device__ __forceinline__ void load_shared(TableShared &s, const TableWork *W) {
    for (int i = threadIdx.x; i < NTRIG; i += blockDim.x) {
        s.trig.ch[i] = W->trig.ch[i];
        s.trig.c23[i] = W->trig.c23[i];
        s.trig.c13[i] = W->trig.c13[i];
    }
    if (threadIdx.x < 4) s.gamma[threadIdx.x] = W->gamma[threadIdx.x];
    __syncthreads();
}

// Modified Bessel function of the second kind and int_y^inf K_{1/3}.
//   y < 1 : ascending series, K_nu = pi/(2 sin(nu pi)) (I_{-nu} - I_nu)
//   y >= 1: trapezoid rule on K_nu(y) = int_0^inf e^{-y cosh t} cosh(nu t) dt
//           (and the same with 1/cosh t for the integral of K_{1/3})
// tg: Gamma(mu + 1)
__device__ __forceinline__ double series_I(double mu, double tg, double y, bool integrated) {
    const double h = 0.5 * y, h2 = h * h;
    double term = pow(h, mu) / tg;
    double s = integrated ? term * y / (mu + 1.0) : term;
    for (int k = 1; k < 40; ++k) {
        term *= h2 / (k * (k + mu));
        const double add = integrated ? term * y / (2.0 * k + mu + 1.0) : term;
        s += add;
        if (fabs(add) < 1e-18 * fabs(s)) break;
    }
    return s;
}

// K_{2/3}(y) and int_y^inf K_{1/3}
__device__ __noinline__ double2 bessel(const TableShared &S, double y) {
    double k23, k13;
    if (y < 1.0) {
        const double nu = 2.0 / 3.0;
        k23 = PI / (2.0 * sin(nu * PI)) * (series_I(-nu, S.gamma[0], y, false) - series_I(nu, S.gamma[1], y, false));
        const double c = PI / sqrt(3.0);   // int_0^inf K_{1/3} = pi/sqrt3 = pi/(2 sin(pi/3))
        k13 = c * (1.0 - series_I(-1.0 / 3.0, S.gamma[2], y, true) + series_I(1.0 / 3.0, S.gamma[3], y, true));
    } else if (y > 740.0) {
        k23 = 0.0;
        k13 = 0.0;
    } else {
        // both trapezoid sums over the same points; each stops at its own end
        const double h = fmin(0.1, 0.4 * rsqrt(y));
        const bool tab = h == 0.1;
        double s23 = 0.5 * exp(-y), s13 = s23;
        bool d23 = false, d13 = false;
        for (int j = 1; j < 20000 && !(d23 && d13); ++j) {
            double ch, a23, a13;
            if (tab && j < NTRIG) {
                ch = S.trig.ch[j]; a23 = S.trig.c23[j]; a13 = S.trig.c13[j];
            } else {
                const double t = j * h;
                ch = cosh(t); a23 = cosh((2.0 / 3.0) * t); a13 = cosh((1.0 / 3.0) * t);
            }
            const double yc = __dmul_rn(y, ch), e = exp(-yc);
            if (!d23) {
                const double f = __dmul_rn(e, a23);
                s23 = __dadd_rn(s23, f);
                d23 = yc > 1.0 && f <= __dmul_rn(1e-18, s23);
            }
            if (!d13) {
                const double f = __dmul_rn(e, a13) / ch;
                s13 = __dadd_rn(s13, f);
                d13 = yc > 1.0 && f <= __dmul_rn(1e-18, s13);
            }
        }
        k23 = __dmul_rn(h, s23);
        k13 = __dmul_rn(h, s13);
    }
    return make_double2(k23, k13);
}

// emission integrand in z = ln y (bracket times d delta / dz)
__device__ __forceinline__ double g_emission_at(double y, double k23, double k13, double chi) {
    const double a = 3.0 * chi * y;
    const double om = 2.0 / (2.0 + a);                   // 1 - delta
    const double jac = y * 6.0 * chi / ((2.0 + a) * (2.0 + a));
    return __dsub_rn(__dmul_rn(om + 1.0 / om, k23), k13) * jac;
}

__device__ __forceinline__ double g_emission(const TableShared &S, double z, double chi) {
    const double y = exp(z);
    const double2 k = bessel(S, y);
    return g_emission_at(y, k.x, k.y, chi);
}

// pair integrand in z, delta = 1/(1+e^-z)
__device__ __forceinline__ double g_pairs(const TableShared &S, double z, double chi) {
    const double d = 1.0 / (1.0 + exp(-z));
    const double om = 1.0 / (1.0 + exp(z));
    const double jac = d * om;
    const double y = 2.0 / (3.0 * chi * jac);
    const double2 k = bessel(S, y);
    return __dadd_rn(__dmul_rn(d / om + om / d, k.x), k.y) * jac;
}

__device__ __forceinline__ double gl_panel(const TableShared &S, bool pair, double chi, double a, double b) {
    const double m = 0.5 * (a + b), hw = 0.5 * (b - a);
    double s = 0.0;
    for (int i = 0; i < GLN; ++i) {
        const double z = m + hw * GLX[i];
        s += GLW[i] * (pair ? g_pairs(S, z, chi) : g_emission(S, z, chi));
    }
    return s * hw;
}

__device__ double block_sum(double v, double *red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    __syncthreads();
    return s;
}

// the constants of the sums and the rows' chi (one thread each)
constexpr int TT = 128;
__global__ void k_table_constants(TableWork *W) {
    const int i = blockIdx.x * TT + threadIdx.x;
    if (i < NTRIG) {
        const double t = i * 0.1;
        W->trig.ch[i] = cosh(t);
        W->trig.c23[i] = cosh((2.0 / 3.0) * t);
        W->trig.c13[i] = cosh((1.0 / 3.0) * t);
    } else if (i < NTRIG + 4) {
        const double mu = i == NTRIG ? -2.0 / 3.0 : i == NTRIG + 1 ? 2.0 / 3.0 : i == NTRIG + 2 ? -1.0 / 3.0 : 1.0 / 3.0;
        W->gamma[i - NTRIG] = tgamma(mu + 1.0);
    }
    if (i < ROWS) W->chi[i] = row_chi(i);
}

// Bessel values at the emission panels' Gauss nodes: one thread per node
__global__ void __launch_bounds__(TT) k_emission_nodes(TableWork *W) {
    __shared__ TableShared S;
    load_shared(S, W);
    const int i = blockIdx.x * TT + threadIdx.x;
    if (i >= EZ_NP * GLN) return;
    const int p = i / GLN;
    const double a = EZ_LO + p * EZ_W, b = EZ_LO + (p + 1) * EZ_W;
    const double m = 0.5 * (a + b), hw = 0.5 * (b - a);
    const double y = exp(m + hw * GLX[i % GLN]);
    const double2 k = bessel(S, y);
    W->em[i] = {y, k.x, k.y};
}

// panel integrals: one thread per (row, panel)
__global__ void __launch_bounds__(TT) k_panel_masses(TableWork *W) {
    __shared__ TableShared S;
    load_shared(S, W);
    const int r = blockIdx.y, p = blockIdx.x * TT + threadIdx.x;
    const bool pair = row_is_pair(r);
    if (p >= (pair ? PZ_NP : EZ_NP)) return;
    const double chi = W->chi[r];
    double v;
    if (pair) {
        v = gl_panel(S, true, chi, PZ_LO + p * PZ_W, PZ_LO + (p + 1) * PZ_W);
    } else {
        const double a = EZ_LO + p * EZ_W, b = EZ_LO + (p + 1) * EZ_W, hw = 0.5 * (b - a);
        double s = 0.0;
        for (int i = 0; i < GLN; ++i) {
            const auto n = W->em[p * GLN + i];
            s += GLW[i] * g_emission_at(n.y, n.k23, n.k13, chi);
        }
        v = s * hw;
    }
    W->mass[(size_t)r * EZ_NP + p] = v;
}

// Per row: the cumulative integrals from both ends (table rows; the two
// running sums by two warps), or the total rate at the Chebyshev nodes
// (emission decades 0..5 on log10 chi in [-3, 3] store F/chi; pair decades
// 6..10 on [-2, 3] store ln F + 8/(3 chi)).
__global__ void __launch_bounds__(TT) k_row_sums(TableWork *W) {
    __shared__ TableShared S;
    __shared__ double m[EZ_NP];
    __shared__ double red[32];
    load_shared(S, W);
    const int r = blockIdx.x;
    const bool pair = row_is_pair(r);
    const int np = pair ? PZ_NP : EZ_NP;
    for (int p = threadIdx.x; p < np; p += TT) m[p] = W->mass[(size_t)r * EZ_NP + p];
    __syncthreads();
    const double chi = W->chi[r];
    if (r < ROW_EM_RATE) {
        double *below = W->below + (size_t)r * (EZ_NP + 1), *above = W->above + (size_t)r * (EZ_NP + 1);
        if (threadIdx.x == 0) {
            double s = pair ? 0.0 : 3.0 * g_emission(S, EZ_LO, chi);
            below[0] = s;
            for (int p = 0; p < np; ++p) below[p + 1] = s = s + m[p];
        } else if (threadIdx.x == 32) {
            double s = 0.0;
            above[np] = s;
            for (int p = np - 1; p >= 0; --p) above[p] = s = s + m[p];
        }
    } else {
        double acc = 0.0;
        for (int p = threadIdx.x; p < np; p += TT) acc += m[p];
        const double tot = block_sum(acc, red);
        if (threadIdx.x == 0) {
            if (!pair) {
                const double F = (tot + 3.0 * g_emission(S, EZ_LO, chi)) / (sqrt(3.0) * PI);
                W->fnode[r - ROW_EM_RATE] = F / chi;
            } else {
                const double F = 2.0 * tot / (sqrt(3.0) * PI);
                W->fnode[r - ROW_EM_RATE] = log(F) + 8.0 / (3.0 * chi);
            }
        }
    }
}

// Chebyshev coefficients from the node values (discrete cosine transform).
__global__ void k_cheb_coef(const double *fnode, double *coef64) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NCOEF) return;
    const int dec = i / CHEB_N, j = i % CHEB_N;
    double s = 0.0;
    for (int k = 0; k < CHEB_N; ++k) s += fnode[dec * CHEB_N + k] * cos(PI * j * (k + 0.5) / CHEB_N);
    coef64[i] = 2.0 * s / CHEB_N;
}

// FP32 cubic pieces: piece i of a decade interpolates the FP64 Chebyshev form
// at t = 0, 1/3, 2/3, 1 (so neighbouring pieces meet), written as monomial
// coefficients in t from the forward differences.  Interpolation error below
// 1e-8 of the function; the FP32 evaluation rounds at ~3e-7.
__global__ void k_rate_segments(const double *coef64, float *seg) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= EM_NSEG + PAIR_NSEG) return;
    const bool pair = i >= EM_NSEG;
    const int k = pair ? i - EM_NSEG : i;
    const int dec = k / RSEG, r = k % RSEG;
    const double *c = coef64 + (pair ? EM_NDEC * CHEB_N : 0) + dec * CHEB_N;
    double f[4];
    for (int q = 0; q < 4; ++q) {
        const double x = 2.0 * ((r + q / 3.0) / RSEG) - 1.0;    // Chebyshev variable of the decade
        double b1 = 0.0, b2 = 0.0;
        for (int j = CHEB_N - 1; j >= 1; --j) {
            const double b0 = c[j] + 2.0 * x * b1 - b2;
            b2 = b1;
            b1 = b0;
        }
        f[q] = 0.5 * c[0] + x * b1 - b2;
    }
    const double d1 = f[1] - f[0], d2 = f[2] - 2.0 * f[1] + f[0], d3 = f[3] - 3.0 * f[2] + 3.0 * f[1] - f[0];
    // p(t) = f0 + d1 tau + d2 tau (tau - 1)/2 + d3 tau (tau - 1)(tau - 2)/6, tau = 3 t
    seg[4 * i + 0] = (float)f[0];
    seg[4 * i + 1] = (float)(3.0 * (d1 - d2 / 2.0 + d3 / 3.0));
    seg[4 * i + 2] = (float)(9.0 * (d2 / 2.0 - d3 / 2.0));
    seg[4 * i + 3] = (float)(27.0 * (d3 / 6.0));
}

// Newton's method inside one panel [za, zb] for int_za^z g = target
// (from_top: int_z^zb g = target), bracketed by bisection.  whole: the
// panel's integral.  SL lanes share a node: each evaluates every SL-th Gauss
// point of the partial integral, which every lane then sums in the points'
// order, so a node's chain of integrand evaluations is 16 / SL + 1 per
// iteration instead of 17 (a few nodes take tens of iterations, and one lane
// per node left the chip waiting for them: 132 ms against 95 ms).
constexpr int SL = 8;
__device__ __forceinline__ double solve_panel(const TableShared &S, bool pair, double chi, double za, double zb,
                                              double whole, double target, bool from_top) {
    const int lane = threadIdx.x & 31, part = lane % SL;
    const unsigned group = (SL == 32 ? 0xffffffffu : (1u << SL) - 1u) << (lane - part);
    double lo = za, hi = zb;
    const double f = whole > 0.0 ? fmin(fmax(target / whole, 0.0), 1.0) : 0.5;
    double z = from_top ? __fma_rn(-f, zb - za, zb) : __fma_rn(f, zb - za, za);
    for (int it = 0; it < 100; ++it) {
        const double a = from_top ? z : za, b = from_top ? zb : z;
        const double m = 0.5 * (a + b), hw = 0.5 * (b - a);
        double g[GLN / SL], s = 0.0;
        for (int i = 0; i < GLN / SL; ++i) {
            const double x = m + hw * GLX[i * SL + part];
            g[i] = pair ? g_pairs(S, x, chi) : g_emission(S, x, chi);
        }
#pragma unroll
        for (int i = 0; i < GLN; ++i) s = __fma_rn(GLW[i], __shfl_sync(group, g[i / SL], i % SL, SL), s);
        const double gz = pair ? g_pairs(S, z, chi) : g_emission(S, z, chi);
        const double r = __fma_rn(s, hw, -target), d = from_top ? -gz : gz;
        const bool z_high = from_top ? (r < 0.0) : (r > 0.0);
        if (z_high) hi = z; else lo = z;
        double zn = d != 0.0 ? z - r / d : 0.5 * (lo + hi);
        if (!(zn > lo && zn < hi)) zn = 0.5 * (lo + hi);
        const double step = fabs(zn - z);
        z = zn;
        if (step <= 1e-15 * (1.0 + fabs(z)) || hi - lo <= 1e-15 * (1.0 + fabs(z))) break;
    }
    return z;
}

// Table nodes, SL lanes each: rows 0..120 emission (ln y), 121..221 pair (ln delta).
constexpr int ST = 64;
__global__ void __launch_bounds__(ST) k_icdf_nodes(const TableWork *W, double *em64, double *pair64) {
    __shared__ TableShared S;
    load_shared(S, W);
    const bool pair = blockIdx.y >= EM_NCHI;
    const int row = pair ? blockIdx.y - EM_NCHI : blockIdx.y;
    const int np = pair ? PZ_NP : EZ_NP;
    const double zlo = pair ? PZ_LO : EZ_LO, wp = pair ? PZ_W : EZ_W;
    const double chi = W->chi[blockIdx.y];
    const double *mass = W->mass + (size_t)blockIdx.y * EZ_NP;
    const double *below = W->below + (size_t)blockIdx.y * (EZ_NP + 1), *above = W->above + (size_t)blockIdx.y * (EZ_NP + 1);
    const double tail = below[0];
    const double total = pair ? 2.0 * below[np] : below[np];
    const int ns = pair ? PAIR_NS : EM_NS;
    const int j = (blockIdx.x * ST + threadIdx.x) / SL;
    if (j >= ns) return;                            // all lanes of a node alike
    const double s = pair ? -16.0 + 16.0 * j / (PAIR_NS - 1) : -16.0 + 32.0 * j / (EM_NS - 1);
    const double u = 1.0 / (1.0 + exp(-s)), v = 1.0 / (1.0 + exp(s));
    const bool top = !(pair || u <= 0.5);
    double target = (top ? v : u) * total, z;
    if (!top && target <= tail) {
        z = zlo + 3.0 * log(target / tail);
    } else {
        int a = 0, b = np - 1;
        while (a < b) {
            if (!top) {                             // first panel with below[p+1] >= target
                const int m = (a + b) >> 1;
                if (below[m + 1] < target) a = m + 1; else b = m;
            } else {                                // last panel with above[p] >= target
                const int m = (a + b + 1) >> 1;
                if (above[m] >= target) a = m; else b = m - 1;
            }
        }
        target = top ? __dsub_rn(target, above[a + 1]) : __dsub_rn(target, below[a]);
        z = solve_panel(S, pair, chi, zlo + a * wp, zlo + (a + 1) * wp, mass[a], target, top);
    }
    if (threadIdx.x % SL) return;
    if (pair) pair64[(size_t)row * PAIR_NS + j] = -log1p(exp(-z));
    else em64[(size_t)row * EM_NS + j] = z;
}

__global__ void k_to_f32(const double *a, float *b, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}

}  // namespace
}  // namespace sfq

qed_status sfq_build_tables(qed_ctx *ctx) {
    using namespace sfq;
    cudaStream_t st = ctx->stream;
    const bool fp32 = ctx->cfg.precision == QED_FP32;
    void *work = nullptr;
    SFQ_CUDA(cudaMallocAsync(&work, fp32 ? sfq_tables32_bytes() : sizeof(TableWork), st));
    const double *fnode;
    if (fp32) {
        fnode = sfq_tables32(work, ctx->icdf_em64, ctx->icdf_pair64, st);
    } else {
        TableWork *W = static_cast<TableWork *>(work);
        fnode = W->fnode;
        k_table_constants<<<(ROWS + TT - 1) / TT, TT, 0, st>>>(W);
        k_emission_nodes<<<(EZ_NP * GLN + TT - 1) / TT, TT, 0, st>>>(W);
        k_panel_masses<<<dim3((EZ_NP + TT - 1) / TT, ROWS), TT, 0, st>>>(W);
        k_row_sums<<<ROWS, TT, 0, st>>>(W);
        k_icdf_nodes<<<dim3((EM_NS * SL + ST - 1) / ST, EM_NCHI + PAIR_NCHI), ST, 0, st>>>(W, ctx->icdf_em64,
                                                                                           ctx->icdf_pair64);
    }
    k_cheb_coef<<<1, 128, 0, st>>>(fnode, ctx->coef64);
    k_rate_segments<<<1, 256, 0, st>>>(ctx->coef64, ctx->coef32);
    k_to_f32<<<(EM_NCHI * EM_NS + 255) / 256, 256, 0, st>>>(ctx->icdf_em64, ctx->icdf_em32, EM_NCHI * EM_NS);
    k_to_f32<<<(PAIR_NCHI * PAIR_NS + 255) / 256, 256, 0, st>>>(ctx->icdf_pair64, ctx->icdf_pair32,
                                                                PAIR_NCHI * PAIR_NS);
    SFQ_CUDA(cudaGetLastError());
    SFQ_CUDA(cudaFreeAsync(work, st));
    SFQ_CUDA(cudaStreamSynchronize(st));
    return QED_OK;
}
