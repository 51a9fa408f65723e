// The tables of FP32 contexts (sfqed_tables.cu says what they hold): the same
// quadrature as in FP64 contexts, with the Bessel functions taken from
// Chebyshev interpolants in ln y.  Their values are within a few ulp of the
// direct sums, and the FP32 tables are these rounded to float.
//
// What bounds it: FP64 arithmetic, about 4e6 integrand evaluations, most of
// them in the root solves.  The Bessel functions are evaluated from their
// definitions only at 472 x 12 points; every kernel spreads its independent
// pieces (panels, nodes) over the whole chip.  1.6 ms of kernels per context
// on one GB300, against 432 ms for the direct sums with one block per row.
#include <math.h>

#include "sfqed_internal.h"
#include "sfqed_tables.cuh"

namespace sfq {
namespace {

// Modified Bessel function of the second kind and int_y^inf K_{1/3}.
//   y < 1 : ascending series, K_nu = pi/(2 sin(nu pi)) (I_{-nu} - I_nu)
//   y >= 1: trapezoid rule on K_nu(y) = int_0^inf e^{-y cosh t} cosh(nu t) dt
//           (and the same with 1/cosh t for the integral of K_{1/3})
__device__ double series_I(double mu, double y, bool integrated) {
    const double h = 0.5 * y, h2 = h * h;
    double term = pow(h, mu) / tgamma(mu + 1.0);
    double s = integrated ? term * y / (mu + 1.0) : term;
    for (int k = 1; k < 40; ++k) {
        term *= h2 / (k * (k + mu));
        const double add = integrated ? term * y / (2.0 * k + mu + 1.0) : term;
        s += add;
        if (fabs(add) < 1e-18 * fabs(s)) break;
    }
    return s;
}

// y < 1
__device__ double bessel_k23_small(double y) {
    const double nu = 2.0 / 3.0;
    return PI / (2.0 * sin(nu * PI)) * (series_I(-nu, y, false) - series_I(nu, y, false));
}

__device__ double int_k13_small(double y) {
    const double c = PI / sqrt(3.0);   // int_0^inf K_{1/3} = pi/sqrt3 = pi/(2 sin(pi/3))
    return c * (1.0 - series_I(-1.0 / 3.0, y, true) + series_I(1.0 / 3.0, y, true));
}

// e^y K_{2/3}(y) and e^y int_y^inf K_{1/3} for y >= 1 by the lanes of a warp:
// the trapezoid terms j = lane, lane + 32, ... with cosh t - 1 = 2 sinh^2(t/2)
__device__ void trap_scaled(double y, double &k23, double &k13) {
    const double h = fmin(0.1, 0.4 * rsqrt(y));
    double s23 = 0.0, s13 = 0.0;
    for (int j0 = 0; j0 < 320; j0 += 32) {
        const int j = j0 + (int)(threadIdx.x & 31);
        const double t = j * h, sh = sinh(0.5 * t), c1 = 2.0 * sh * sh;
        const double f = (j == 0 ? 0.5 : 1.0) * exp(-y * c1);
        s23 += f * cosh((2.0 / 3.0) * t);
        s13 += f * cosh((1.0 / 3.0) * t) / (1.0 + c1);
        // the last lane's term is the smallest of this round, and the next
        // rounds' terms fall faster than geometrically
        if (__shfl_sync(0xffffffffu, f * cosh((2.0 / 3.0) * t), 31) < 1e-20) break;
    }
    for (int o = 16; o > 0; o >>= 1) {
        s23 += __shfl_xor_sync(0xffffffffu, s23, o);
        s13 += __shfl_xor_sync(0xffffffffu, s13, o);
    }
    k23 = h * s23;
    k13 = h * s13;
}

// ---- Bessel interpolants ----
// On each emission panel (width 0.25 in z = ln y) e^y K_{2/3}(y) and
// e^y int_y^inf K_{1/3} are interpolated at BC Chebyshev points.  Both are
// entire in z and grow slowly in the strip |Im z| < 2, so the interpolation
// error on a half width of 1/8 is about 4 * 32^-12 of the value, below FP64
// rounding; the exponential is applied at the point itself.
constexpr int BC = 12;

// coefficient table: bc[2 * (panel * BC + k)] (K_{2/3}), + 1 (the integral)
__device__ __forceinline__ void bessel_at(const double *bc, int panel, double x, double y, double &k23, double &k13) {
    const double2 *c = reinterpret_cast<const double2 *>(bc) + panel * BC;
    const double x2 = x + x;
    double a1 = 0.0, a2 = 0.0, b1 = 0.0, b2 = 0.0;
#pragma unroll
    for (int k = BC - 1; k >= 1; --k) {
        const double2 v = __ldg(c + k);
        const double a0 = fma(x2, a1, v.x - a2), b0 = fma(x2, b1, v.y - b2);
        a2 = a1; a1 = a0;
        b2 = b1; b1 = b0;
    }
    const double2 v = __ldg(c);
    const double ey = exp(-y);
    k23 = fma(x, a1, v.x - a2) * ey;
    k13 = fma(x, b1, v.y - b2) * ey;
}

// at any y with its logarithm (0 beyond the panels, where e^-y underflows;
// the smallest y asked for is that of the first emission panel)
__device__ __forceinline__ void bessel_any(const double *bc, double lny, double y, double &k23, double &k13) {
    if (y > 740.0) {
        k23 = 0.0;
        k13 = 0.0;
        return;
    }
    const double u = (lny - EZ_LO) * (1.0 / EZ_W);
    int p = (int)u;
    p = p < 0 ? 0 : (p > EZ_NP - 1 ? EZ_NP - 1 : p);
    bessel_at(bc, p, 2.0 * (u - p) - 1.0, y, k23, k13);
}

// emission integrand (bracket times d delta / dz) from y and the functions there
__device__ __forceinline__ double em_integrand(double chi, double y, double k23, double k13) {
    const double a = 3.0 * chi * y;
    const double inv = 1.0 / (2.0 + a);                  // 1 - delta = 2 inv
    const double jac = 6.0 * chi * y * (inv * inv);
    return ((2.0 * inv + 0.5 * (2.0 + a)) * k23 - k13) * jac;
}

// pair integrand: s = e^z + e^-z, 1 / (delta (1 - delta)) = 2 + s
__device__ __forceinline__ double pair_integrand(const double *bc, double c, double lnc, double s, double lns2) {
    const double y = c * (2.0 + s);                      // c = 2 / (3 chi)
    double k23, k13;
    bessel_any(bc, lnc + lns2, y, k23, k13);
    return (s * k23 + k13) / (2.0 + s);
}

__device__ __forceinline__ double em_density(const double *bc, double chi, int panel, double z) {
    const double za = EZ_LO + panel * EZ_W, y = exp(z);
    if (y > 740.0) return 0.0;
    double k23, k13;
    bessel_at(bc, panel, (2.0 / EZ_W) * (z - za) - 1.0, y, k23, k13);
    return em_integrand(chi, y, k23, k13);
}

__device__ __forceinline__ double pair_density(const double *bc, double c, double lnc, double z) {
    const double s = exp(z) + exp(-z);
    return pair_integrand(bc, c, lnc, s, log(2.0 + s));
}

// what the quadrature needs at the Gauss nodes of every panel, whatever chi
struct BesselWork {
    double bc[2 * EZ_NP * BC];        // interpolant coefficients
    struct { double y, k23, k13, w; } em[EZ_NP * GLN];   // w: weight x half width
    struct { double s, ln, w; } pr[PZ_NP * GLN];         // s = e^z + e^-z, ln = ln(2 + s)
    double chi[ROWS];
    double mass[ROWS * EZ_NP];        // panel integrals per row
    double below[(EM_NCHI + PAIR_NCHI) * (EZ_NP + 1)], above[(EM_NCHI + PAIR_NCHI) * (EZ_NP + 1)];
    double fnode[NCOEF];              // rate form at the Chebyshev nodes
};

// Panel b of the interpolants: the BC node values (a warp per node where the
// trapezoid sum runs, y >= 1; a thread per node where the ascending series
// does), their Chebyshev coefficients, and the values at the panel's Gauss
// nodes.
constexpr int BT = 32 * BC;
__global__ void __launch_bounds__(BT) k_bessel_panels(BesselWork *W) {
    __shared__ double f23[BC], f13[BC], cs[BC][BC];
    const int b = blockIdx.x, t = threadIdx.x;
    const double za = EZ_LO + b * EZ_W;
    const bool series = za + EZ_W <= 0.0;
    const int node = series ? t : t >> 5;
    if (node < BC) {
        const double z = za + 0.5 * EZ_W * (1.0 + cospi((node + 0.5) / BC));
        const double y = exp(z);
        double k23, k13;
        if (series) {
            const double e = exp(y);
            k23 = bessel_k23_small(y) * e;
            k13 = int_k13_small(y) * e;
        } else {
            trap_scaled(y, k23, k13);
        }
        f23[node] = k23;
        f13[node] = k13;
    }
    if (t < BC * BC) cs[t / BC][t % BC] = cospi((t / BC) * ((t % BC) + 0.5) / BC);
    __syncthreads();
    if (t < 2 * BC) {
        const int k = t >> 1;
        const double *f = t & 1 ? f13 : f23;
        double s = 0.0;
        for (int j = 0; j < BC; ++j) s += f[j] * cs[k][j];
        W->bc[2 * (b * BC + k) + (t & 1)] = (k == 0 ? 1.0 : 2.0) / BC * s;
    }
    __syncthreads();                                     // the block reads its own coefficients
    __threadfence_block();
    if (t < GLN) {
        const double x = GLX[t], y = exp(za + 0.5 * EZ_W * (1.0 + x));
        // plain loads: the coefficients were written by this launch
        double a1 = 0.0, a2 = 0.0, c1 = 0.0, c2 = 0.0;
        const double2 *c = reinterpret_cast<const double2 *>(W->bc) + b * BC;
        for (int k = BC - 1; k >= 1; --k) {
            const double a0 = fma(2.0 * x, a1, c[k].x - a2), c0 = fma(2.0 * x, c1, c[k].y - c2);
            a2 = a1; a1 = a0;
            c2 = c1; c1 = c0;
        }
        const double ey = y > 740.0 ? 0.0 : exp(-y);
        W->em[b * GLN + t] = {y, fma(x, a1, c[0].x - a2) * ey, fma(x, c1, c[0].y - c2) * ey, GLW[t] * 0.5 * EZ_W};
    } else if (t >= 32 && t < 32 + GLN && b < PZ_NP) {
        const int i = t - 32;
        const double z = PZ_LO + b * PZ_W + 0.5 * PZ_W * (1.0 + GLX[i]);
        const double s = exp(z) + exp(-z);
        W->pr[b * GLN + i] = {s, log(2.0 + s), GLW[i] * 0.5 * PZ_W};
    } else if (t == 64 && b < ROWS) {
        W->chi[b] = row_chi(b);
    }
}

// Panel integrals: one thread per (row, panel).
constexpr int MT = 128;
__global__ void __launch_bounds__(MT) k_panel_masses(BesselWork *W) {
    const int r = blockIdx.y, p = blockIdx.x * MT + threadIdx.x;
    const bool pair = row_is_pair(r);
    if (p >= (pair ? PZ_NP : EZ_NP)) return;
    const double chi = W->chi[r];
    double s = 0.0;
    if (!pair) {
        for (int i = 0; i < GLN; ++i) {
            const auto n = W->em[p * GLN + i];
            s += n.w * em_integrand(chi, n.y, n.k23, n.k13);
        }
    } else {
        const double c = 2.0 / (3.0 * chi), lnc = log(c);
        for (int i = 0; i < GLN; ++i) {
            const auto n = W->pr[p * GLN + i];
            s += n.w * pair_integrand(W->bc, c, lnc, n.s, n.ln);
        }
    }
    W->mass[(size_t)r * EZ_NP + p] = s;
}

// Per row: the cumulative integrals from both ends (table rows) or the rate
// form at the Chebyshev node (emission decades store F/chi, pair decades
// ln F + 8/(3 chi)).  The two running sums are two lanes of different warps.
__global__ void __launch_bounds__(64) k_row_sums(BesselWork *W) {
    __shared__ double m[EZ_NP];
    const int r = blockIdx.x;
    const bool pair = row_is_pair(r);
    const int np = pair ? PZ_NP : EZ_NP;
    for (int p = threadIdx.x; p < np; p += 64) m[p] = W->mass[(size_t)r * EZ_NP + p];
    __syncthreads();
    const double chi = W->chi[r];
    const double tail = pair ? 0.0 : 3.0 * em_density(W->bc, chi, 0, EZ_LO);
    if (r < ROW_EM_RATE) {
        double *below = W->below + (size_t)r * (EZ_NP + 1), *above = W->above + (size_t)r * (EZ_NP + 1);
        if (threadIdx.x == 0) {
            double s = tail;
            below[0] = s;
            for (int p = 0; p < np; ++p) below[p + 1] = s += m[p];
        } else if (threadIdx.x == 32) {
            double s = 0.0;
            above[np] = s;
            for (int p = np - 1; p >= 0; --p) above[p] = s += m[p];
        }
    } else if (threadIdx.x == 0) {
        double s = 0.0;
        for (int p = 0; p < np; ++p) s += m[p];
        const double F = (pair ? 2.0 * s : s + tail) / (sqrt(3.0) * PI);
        W->fnode[r - ROW_EM_RATE] = pair ? log(F) + 8.0 / (3.0 * chi) : F / chi;
    }
}

// Table nodes: rows 0..120 emission (ln y), 121..221 pair (ln delta); one
// thread per node, Newton's method on the cumulative integral inside the
// node's panel, bracketed by bisection.  The integral is taken from the
// nearer end of the distribution, so that both tails keep their relative
// accuracy.  Newton's error after a step s is about s^2 times half the
// density's logarithmic slope (at most ~20 per unit z here), so a step below
// 1e-9 leaves 1e-17 and no confirming evaluation is needed.
constexpr int ST = 64;
__global__ void __launch_bounds__(ST) k_solve_nodes(const BesselWork *W, double *em64, double *pair64) {
    const int row = blockIdx.y, j = blockIdx.x * ST + threadIdx.x;
    const bool pair = row >= ROW_PAIR;
    const int ns = pair ? PAIR_NS : EM_NS, np = pair ? PZ_NP : EZ_NP;
    if (j >= ns) return;
    const double zlo = pair ? PZ_LO : EZ_LO, wp = pair ? PZ_W : EZ_W;
    const double *below = W->below + (size_t)row * (EZ_NP + 1), *above = W->above + (size_t)row * (EZ_NP + 1);
    const double chi = W->chi[row], c = 2.0 / (3.0 * chi), lnc = pair ? log(c) : 0.0;
    const double s = pair ? -16.0 + 16.0 * j / (PAIR_NS - 1) : -16.0 + 32.0 * j / (EM_NS - 1);
    const double u = 1.0 / (1.0 + exp(-s)), v = 1.0 / (1.0 + exp(s));
    const double tail = below[0];                       // 0 for pairs
    const double total = pair ? 2.0 * below[np] : below[np];
    const bool low = pair || u <= 0.5;
    double target = (low ? u : v) * total;
    double z;
    if (low && target <= tail) {
        z = zlo + 3.0 * log(target / tail);
    } else {
        int a = 0, b = np - 1;
        while (a < b) {
            if (low) {                                  // first panel with below[p + 1] >= target
                const int m = (a + b) >> 1;
                if (below[m + 1] < target) a = m + 1; else b = m;
            } else {                                    // last panel with above[p] >= target
                const int m = (a + b + 1) >> 1;
                if (above[m] >= target) a = m; else b = m - 1;
            }
        }
        const double za = zlo + a * wp, zb = zlo + (a + 1) * wp;
        target -= low ? below[a] : above[a + 1];
        const double whole = W->mass[(size_t)row * EZ_NP + a];
        const double f = whole > 0.0 ? fmin(fmax(target / whole, 0.0), 1.0) : 0.5;
        z = low ? za + f * (zb - za) : zb - f * (zb - za);
        double lo = za, hi = zb;
        for (int it = 0; it < 100; ++it) {
            const double e0 = low ? za : z, hw = 0.5 * (low ? z - za : zb - z);
            double r = 0.0;
            for (int i = 0; i < GLN; ++i) {
                const double x = e0 + hw * (1.0 + GLX[i]);
                r += GLW[i] * (pair ? pair_density(W->bc, c, lnc, x) : em_density(W->bc, chi, a, x));
            }
            r = r * hw - target;
            if (!low) r = -r;                           // increasing in z from either end
            const double d = pair ? pair_density(W->bc, c, lnc, z) : em_density(W->bc, chi, a, z);
            if (r > 0.0) hi = z; else lo = z;
            double zn = d != 0.0 ? z - r / d : 0.5 * (lo + hi);
            const bool newton = zn >= lo && zn <= hi;
            if (!newton) zn = 0.5 * (lo + hi);
            const double step = fabs(zn - z);
            z = zn;
            if ((newton && step <= 1e-9) || hi - lo <= 1e-15 * (1.0 + fabs(z))) break;
        }
    }
    if (pair) pair64[(size_t)(row - ROW_PAIR) * PAIR_NS + j] = -log1p(exp(-z));
    else em64[(size_t)row * EM_NS + j] = z;
}

}  // namespace
}  // namespace sfq

size_t sfq_tables32_bytes() { return sizeof(sfq::BesselWork); }

const double *sfq_tables32(void *work, double *em64, double *pair64, cudaStream_t st) {
    using namespace sfq;
    BesselWork *W = static_cast<BesselWork *>(work);
    k_bessel_panels<<<EZ_NP, BT, 0, st>>>(W);
    k_panel_masses<<<dim3((EZ_NP + MT - 1) / MT, ROWS), MT, 0, st>>>(W);
    k_row_sums<<<ROWS, 64, 0, st>>>(W);
    k_solve_nodes<<<dim3((EM_NS + ST - 1) / ST, EM_NCHI + PAIR_NCHI), ST, 0, st>>>(W, em64, pair64);
    return W->fnode;
}
