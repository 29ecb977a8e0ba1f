// K1: per-sample tables of the regularized Brinkmanlet kernel functions (FP64 build).
//
// For each sample (alpha, delta) this builds, on the device,
//   g1(r) = B''(r),  g2(r) = (r B''(r) - B'(r))/r^3     (Sec. 2.1, Eq. BrV)
// with (Lap - alpha^2) B = G and Lap G = phi_delta (Eq. eqnblob).  With
//   M0(r) = int_0^r phi s ds = (1 - delta^3/R^3)/(2 pi)            (closed form)
//   A1(r) = int_0^r (I0(alpha s) - 1) phi s ds
//   C(r)  = int_r^inf K0(alpha s) phi s ds
// and x = alpha r, the solution of the radial problem by variation of parameters
// (Green's function -K0(alpha |x|)/(2 pi), averaged over circles) gives
//   g1 = [1/x^2 - W] M0 - W A1 - (I0 + I2) C / 2,             W = (K0 + K2)/2
//   g2 = [(2/x^2 - K2) M0 - K2 A1 - I2 C] / r^2
// where the bracketed differences are evaluated from their power series for x <= 2.
// alpha = 0 is the regularized Stokeslet in closed form (Cortez 2001).
//
// Numerics (all FP64).  The table's nodes lie at fixed u = 1 + sigma^2, sigma = r/delta, and so
// do the Gauss-Legendre points of the integrals between consecutive nodes: sigma, ln sigma,
// M0, the quadrature weights times phi s ds and the like are the same for every sample and are
// made once per device (build_universal); a sample enters through beta = alpha delta alone,
// x = beta sigma.  Each interval takes as many points as its distance from the integrands'
// singularities (s = 0 and s = +-i delta) asks for 1e-16.  Bessel I: power series for x <= 8,
// beyond that, and for K beyond x = 2, polynomials in 1/x fitted on the host at Chebyshev nodes
// to sqrt(x) e^-x I and sqrt(x) e^x K (I from its power series and Hankel's expansion, K from
// the trapezoid rule on K_nu(x) e^x = int_0^inf exp(-x (cosh t - 1)) cosh(nu t) dt); K for
// x <= 2 from its ascending series (A&S 9.6.11/9.6.13).
//
// What bounds it: the FP64 pipe (two FMAs a clock and SM: a warp instruction takes 16 clocks).
// Every integral by the trapezoid rule and a power series with FP64 tests, point by point, took
// 20.6 ms for 1024 FP64 samples of N = 128 and 3.1 ms for a lone one; the fixed points and the
// polynomials take 0.9 and 0.05 ms.  FP32 handles, whose arithmetic is fixed (below): 8.1 to
// 2.3 ms for 1024 samples, 1.7 to 0.2 ms for 40, by taking both integrals of an interval at
// the same points, the polynomial for K0 beyond x = 2, tests on the high words alone, and no
// FP64 table beside the FP32 one.
//
// Output per sample: FP64 handles the FP64 table, FP32 handles quadratic coefficients in the
// mantissa F in [1, 2) of u (64 panels per octave).
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "table_eval.cuh"

namespace {

constexpr double PI = 3.14159265358979323846;
constexpr double EGAMMA = 0.57721566490153286061;
constexpr int GL_N = 16;
// FP32 handles: the FP64 node values feed an FP32 table only, and ~1e-9 is enough: 6 nodes a panel
constexpr int LITE_NODES = 6;
__constant__ double c_gl_x[GL_N];   // 16-point Gauss-Legendre on [-1, 1]
__constant__ double c_gl_w[GL_N];
__constant__ double c_gl12_x[12];   // 12 points, for the tail
__constant__ double c_gl12_w[12];
// FP64 table: coefficients of a panel from the 10 node values of its build panel
constexpr int F64_SPLIT = F64_FINE / F64_SUB, F64_COEF = 8;
__constant__ double c_fit64[F64_SPLIT][F64_COEF][F64_NODES];
// FP32 handles: 8 points, the 6 nodes' places and transform, the quadratic's 3 nodes
__constant__ double c_gl8_x[8], c_gl8_w[8];
__constant__ double c_cheb_t6[LITE_NODES], c_dct6[LITE_NODES][LITE_NODES];
__constant__ double c_node3[3], c_dct3[3][3];
constexpr int F32_SPLIT = F32_SUB / F64_SUB;  // FP32 panels per FP64 panel
constexpr int NSER = 160;
__constant__ double c_inv_k[NSER];      // 1/k (index 0 unused)
__constant__ double c_inv_kk[2][NSER];  // 1/((k+1)(k+1+nu)) for nu = 0, 2
constexpr int HARM = 64;
__constant__ double c_harm[HARM];       // H_k, summed in order

// Bessel coefficients (host-made): series in y = x^2/4, and polynomials in z = 1/x, each in its
// range's variable t in [-1, 1]
constexpr int SER = 25, SER_K = 13;
__constant__ double c_i0[SER], c_i2[SER];       // 1/(k!)^2, 1/(k! (k+2)!)
__constant__ double c_k0t[SER_K], c_t2[SER_K];  // H_k/(k!)^2, (H_k + H_{k+2})/(2 k! (k+2)!)
constexpr int DEG_K = 16, DEG_I1 = 18, DEG_I2 = 12;
constexpr double K_SPLIT = 6.0, I_SERIES = 8.0, I_SPLIT = 20.0;
__constant__ double c_k0[2][DEG_K + 1], c_k1[2][DEG_K + 1];   // x in (2, 6], (6, inf)
__constant__ double c_i0p[DEG_I1 + 1], c_i2p[DEG_I1 + 1];     // x in (8, 20]
__constant__ double c_i0q[DEG_I2 + 1], c_i2q[DEG_I2 + 1];     // x in (20, inf)

// FP64 handles: the sample-independent tables
struct __align__(16) NodeRec {
    double sig, lns, rsq, inv2, m0, pad;  // sigma, ln sigma, sigma^-1/2, sigma^-2, M0 (delta = 1)
};
struct __align__(16) QuadRec {
    double sig, lns, rsq, w;  // a Gauss-Legendre point: w = weight * phi * sigma
};
constexpr int QUAD_MIN = 5;  // points of an interval at least
constexpr int QUAD_CAP = 6 * NODES_MAX;
__device__ NodeRec g_node[NODES_MAX];
__device__ QuadRec g_quad[QUAD_CAP];
__device__ int g_quad_at[NODES_MAX + 1];  // interval q: [at[q], at[q + 1])
// beta times an interval's width beyond which its fixed points do not resolve e^(-beta s) (5
// points: (beta w)^10 4e-13 relative); such intervals, far out where x > 40, are split anew
constexpr double WIDTH_MAX = 0.7;

template <int N>
__device__ __forceinline__ double horner(const double *c, double t) {
    double s = c[N - 1];
#pragma unroll
    for (int k = N - 2; k >= 0; --k) s = fma(s, t, c[k]);
    return s;
}

// t in [-1, 1] of z = 1/x in [1/hi, 1/lo]
__host__ __device__ constexpr double z_scale(double lo, double inv_hi) { return 2.0 / (1.0 / lo - inv_hi); }
__host__ __device__ constexpr double z_shift(double lo, double inv_hi) { return -(1.0 / lo + inv_hi) / (1.0 / lo - inv_hi); }

// polynomials of K_nu e^x sqrt(x) at z = 1/x, x > 2
__device__ __forceinline__ double k_poly(const double (*c)[DEG_K + 1], bool far, double z) {
    return far ? horner<DEG_K + 1>(c[1], fma(z, z_scale(K_SPLIT, 0.0), z_shift(K_SPLIT, 0.0)))
               : horner<DEG_K + 1>(c[0], fma(z, z_scale(2.0, 1.0 / K_SPLIT), z_shift(2.0, 1.0 / K_SPLIT)));
}

// I_nu e^-x sqrt(x) at z = 1/x, x > 8
__device__ __forceinline__ double i_poly(const double *p, const double *q, bool far, double z) {
    return far ? horner<DEG_I2 + 1>(q, fma(z, z_scale(I_SPLIT, 0.0), z_shift(I_SPLIT, 0.0)))
               : horner<DEG_I1 + 1>(p, fma(z, z_scale(I_SERIES, 1.0 / I_SPLIT), z_shift(I_SERIES, 1.0 / I_SPLIT)));
}

// K0(x), and I0(x) - 1 without cancellation when want_i.  lx = ln(x/2) + gamma and rs = x^(-1/2)
// come with the point.
__device__ __forceinline__ void bessel_k0_i0m1(double x, double lx, double rs, bool want_i, double &k0, double &i0m1) {
    const double y = 0.25 * x * x;
    if (x <= 2.0) {
        // the series' lengths by size of y <= 1 (terms below 1e-18)
        double im, tail;
        if (y <= 0.0625) {
            im = y * horner<7>(c_i0 + 1, y);
            tail = y * horner<7>(c_k0t + 1, y);
        } else {
            im = y * horner<SER_K - 1>(c_i0 + 1, y);
            tail = y * horner<SER_K - 1>(c_k0t + 1, y);
        }
        i0m1 = im;
        k0 = fma(-lx, 1.0 + im, tail);  // K0 = -lx I0 + sum H_k y^k/(k!)^2
        return;
    }
    const double z = rs * rs;
    k0 = exp(-x) * rs * k_poly(c_k0, x > K_SPLIT, z);
    if (want_i)
        i0m1 = x <= I_SERIES ? y * horner<SER - 1>(c_i0 + 1, y)
                             : exp(x) * rs * i_poly(c_i0p, c_i0q, x > I_SPLIT, z) - 1.0;
}

// ---------------------------------------------------------------------------------
// integrands and panel integrals
// ---------------------------------------------------------------------------------
// int_a^b f(s) ds (delta = 1), f = (I0(beta s) - 1) phi s and K0(beta s) phi s, split so that no
// piece is wider than 0.5/beta or half the distance scale max(a, 1/4): the intervals whose
// fixed points would not do
__device__ __noinline__ void split_integral(double a, double b, double beta, double &ia, double &ic) {
    const double w = b - a;
    int n = (int)ceil(fmax(beta * w / 0.5, w / (0.5 * fmax(a, 0.25))));
    n = n < 1 ? 1 : n > 4096 ? 4096 : n;
    const double hw = 0.5 * w / n, lb = log(0.5 * beta) + EGAMMA;
    ia = ic = 0.0;
    for (int p = 0; p < n; ++p) {
        const double c = a + (2 * p + 1) * hw;
        for (int g = 0; g < GL_N; ++g) {
            const double s = c + hw * c_gl_x[g], R2 = s * s + 1.0;
            const double wt = hw * c_gl_w[g] * 3.0 * s / (2.0 * PI * R2 * R2 * sqrt(R2));
            const double x = beta * s;
            double k0, im = 0.0;
            bessel_k0_i0m1(x, lb + log(s), rsqrt(x), true, k0, im);
            ia = fma(wt, im, ia);
            ic = fma(wt, k0, ic);
        }
    }
}

// ---------------------------------------------------------------------------------
// FP32 handles.  Their tables are FP64 node values rounded to FP32 quadratics, and a run in
// FP32 follows every rounding of them, so the arithmetic that a node value depends on to its last
// bits (the recurrences, their order, the 8-point integrals) is fixed here, apart from that of the
// FP64 handles above.  K0 inside the integral C enters a node value scaled by (delta/r)^3: beyond
// x = 2 (in the tail: six units of x into it, and from the start where the weight is below 4e-6)
// the polynomial above takes the place of the trapezoid rule, whose last bits no node value shows
// there (bit-equal tables at 8000 samples of the sperm model, where the weight is largest).
// ---------------------------------------------------------------------------------
// term < 2^-e s for positive numbers from their high words alone: the series' tests, without
// FP64 instructions (a term more or less lies below the sums' last bit)
__device__ __forceinline__ bool below(double term, double s, int e) {
    return __double2hiint(term) + (e << 20) < __double2hiint(s);
}

// I_nu(x), nu in {0, 2}: power series for x <= 30, Hankel asymptotic expansion beyond.
__device__ double series_i(int nu, double x) {
    if (x <= 30.0) {
        double y = 0.25 * x * x;
        double term = nu == 0 ? 1.0 : 0.5;  // 1/nu!
        const double *inv = c_inv_kk[nu == 0 ? 0 : 1];
        double s = 0.0;
        for (int k = 0; k < NSER; ++k) {
            s += term;
            term *= y * inv[k];
            if (below(term, s, 60)) break;
        }
        return s * (nu == 0 ? 1.0 : y);  // (x/2)^2 = y for nu = 2
    }
    double mu = 4.0 * nu * nu;
    double s = 1.0, term = 1.0, inv8x = 0.125 / x;
    for (int k = 1; k < 60; ++k) {
        double a = (mu - (2.0 * k - 1.0) * (2.0 * k - 1.0)) * c_inv_k[k] * inv8x;
        double nt = -term * a;
        if (fabs(nt) > fabs(term)) break;
        term = nt;
        s += term;
        if (fabs(term) < 1e-18 * fabs(s)) break;
    }
    return exp(x) / sqrt(2.0 * PI * x) * s;
}

// I0(x) - 1 without cancellation
__device__ __forceinline__ double series_i0m1(double x) {
    if (x > 1.0) return series_i(0, x) - 1.0;
    double y = 0.25 * x * x, term = y, s = 0.0;
    for (int k = 1; k < 60; ++k) {
        s += term;
        term *= y * c_inv_kk[0][k];  // 1/((k+1)^2)
        if (below(term, s, 60)) break;
    }
    return s;
}

// K0(x) for x <= 2 = -(ln(x/2) + gamma) I0(x) + sum_{k>=1} H_k y^k/(k!)^2, y = x^2/4 (one pass)
__device__ __forceinline__ double series_k0(double x) {
    double y = 0.25 * x * x, term = 1.0, i0 = 1.0, tail = 0.0;
    for (int k = 1; k < 60; ++k) {
        term *= y * c_inv_kk[0][k - 1];
        i0 += term;
        tail += c_harm[k] * term;
        if (below(term, i0, 63)) break;
    }
    return -(log(0.5 * x) + EGAMMA) * i0 + tail;
}

// K0(x) for x > 2 by the trapezoid rule on K0(x) e^x = int_0^inf exp(-x (cosh t - 1)) dt
__device__ __noinline__ double trapezoid_k0(double x) {
    double d = acos(1.0 - 1.0 / x);
    double h = d / 6.5;
    double s0 = 0.5;
    const double eh = exp(h), emh = 1.0 / eh;
    double ep = 1.0, em = 1.0;  // e^{m h}, e^{-m h}
    for (int m = 1; m < 4000; ++m) {
        ep *= eh;
        em *= emh;
        double c = 0.5 * (ep + em);  // cosh(m h)
        double e = exp(-x * (c - 1.0));
        s0 += e;
        if (below(e, s0, 63)) break;
    }
    return h * s0 * exp(-x);
}

struct BesselSet {
    double i0, i2, k0, k2, t2k2, ix2w;  // t2k2 = 2/x^2 - K2, ix2w = 1/x^2 - (K0+K2)/2
};

// K0(x) e^x and K1(x) e^x for x > 2 by the trapezoid rule on the integral representation
__device__ void trapezoid_k01(double x, double *k0e, double *k1e) {
    double d = acos(1.0 - 1.0 / x);
    double h = d / 6.5;
    double s0 = 0.5, s1 = 0.5;
    const double eh = exp(h), emh = 1.0 / eh;
    double ep = 1.0, em = 1.0;  // e^{m h}, e^{-m h}
    for (int m = 1; m < 4000; ++m) {
        ep *= eh;
        em *= emh;
        double c = 0.5 * (ep + em);  // cosh(m h)
        double e = exp(-x * (c - 1.0));
        s0 += e;
        s1 += e * c;
        if (below(e, s0, 63)) break;
    }
    *k0e = h * s0;
    *k1e = h * s1;
}

__device__ BesselSet bessel_set(double x) {
    BesselSet b;
    b.i0 = series_i(0, x);
    b.i2 = series_i(2, x);
    if (x <= 2.0) {
        double y = 0.25 * x * x;
        double lx = log(0.5 * x) + EGAMMA;
        // K0 = -lx I0 + sum_{k>=1} H_k y^k/(k!)^2
        double term = 1.0, tail = 0.0;
        for (int k = 1; k < 60; ++k) {
            term *= y * c_inv_kk[0][k - 1];  // 1/k^2
            tail += c_harm[k] * term;
            if (below(term, 1.0, 63)) break;
        }
        b.k0 = -lx * b.i0 + tail;
        // 2/x^2 - K2 = 1/2 + y sum_k [lx - (H_k + H_{k+2})/2] y^k/(k!(k+2)!)
        double s = 0.0;
        term = 0.5;
        double hk0 = 0.0, hk2 = 1.5;  // H_0, H_2
        for (int k = 0; k < 60; ++k) {
            s += (lx - 0.5 * (hk0 + hk2)) * term;
            term *= y * c_inv_kk[1][k];  // 1/((k+1)(k+3))
            hk0 += c_inv_k[k + 1];
            hk2 += c_inv_k[k + 3];
            if (below(term, 1.0, 66)) break;
        }
        b.t2k2 = 0.5 + y * s;
        b.k2 = 2.0 / (x * x) - b.t2k2;
        b.ix2w = 0.5 * b.t2k2 - 0.5 * b.k0;
    } else {
        double k0e, k1e;
        trapezoid_k01(x, &k0e, &k1e);
        double ex = exp(-x);
        b.k0 = k0e * ex;
        double k1 = k1e * ex;
        b.k2 = b.k0 + 2.0 * k1 / x;
        b.t2k2 = 2.0 / (x * x) - b.k2;
        b.ix2w = 1.0 / (x * x) - 0.5 * (b.k0 + b.k2);
    }
    return b;
}

__device__ __forceinline__ double blob(double s, double delta) {
    double R2 = s * s + delta * delta;
    return 3.0 * delta * delta * delta / (2.0 * PI * R2 * R2 * sqrt(R2));
}

__device__ double m0_closed(double r, double delta) {
    double R = sqrt(r * r + delta * delta);
    return (r * r / (R + delta)) * (R * R + R * delta + delta * delta) / (R * R * R) / (2.0 * PI);
}

__device__ __forceinline__ double node6_u(int m) {
    // node m -> (octave, panel, ascending Chebyshev index)
    int panel = m / LITE_NODES, ii = m % LITE_NODES;
    int e = panel >> F64_SUB_LOG2, j = panel & (F64_SUB - 1);
    double f = 0.5 * (c_cheb_t6[ii] + 1.0);
    return ldexp(1.0 + (j + f) / F64_SUB, e);
}

// int_a^b of (I0(alpha s) - 1) phi s and of K0(alpha s) phi s, 8 points a piece, split so that no
// piece is wider than 0.5/alpha or half the distance scale max(a, delta/4)
__device__ void panel_integrals8(double a, double b, double alpha, double delta, bool want_k, double &ia, double &ic) {
    double w = b - a;
    int n = (int)ceil(fmax(alpha * w / 0.5, w / (0.5 * fmax(a, 0.25 * delta))));
    if (n < 1) n = 1;
    if (n > 4096) n = 4096;
    double hw = 0.5 * w / n, ta = 0.0, tc = 0.0;
    for (int p = 0; p < n; ++p) {
        double c = a + (2 * p + 1) * hw, aa = 0.0, ac = 0.0;
        for (int g = 0; g < 8; ++g) {
            double s = c + hw * c_gl8_x[g], x = alpha * s, bl = blob(s, delta);
            double f = series_i0m1(x) * bl * s;
            aa += c_gl8_w[g] * f;
            if (want_k) {
                double k0, im;
                if (x <= 2.0)
                    k0 = series_k0(x);
                else
                    bessel_k0_i0m1(x, 0.0, rsqrt(x), false, k0, im);
                f = k0 * bl * s;
                ac += c_gl8_w[g] * f;
            }
        }
        ta += aa * hw;
        tc += ac * hw;
    }
    ia = ta;
    ic = tc;
}

__device__ void stokes_g(double r, double delta, double *g1, double *g2) {
    double R = sqrt(r * r + delta * delta);
    *g1 = (log(R + delta) - delta * (R + 2.0 * delta) / (R * (R + delta))) / (4.0 * PI);
    *g2 = (R + 2.0 * delta) / (4.0 * PI * R * (R + delta) * (R + delta));
}

// ---------------------------------------------------------------------------------
// per-sample parameters from theta
// ---------------------------------------------------------------------------------
__global__ void prepare_kernel(int B, const double *__restrict__ theta, const int *__restrict__ n_pts,
                               swimmer_config cfg, SampleParams *__restrict__ sp, int *__restrict__ order) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    SampleParams p;
    p.n = n_pts ? n_pts[b] : default_flagellum_points(cfg);
    p.nh = cfg.n_head;
    const int np = n_params(cfg);
    p.alpha = theta[np * b + 0];
    p.kc = pow(10.0, theta[np * b + 1]);
    p.amp = theta[np * b + 2];
    p.sig = np == 4 ? theta[np * b + 3] : 1.0;
    p.length = cfg.ds_fixed > 0.0 ? (p.n - 1) * cfg.ds_fixed : cfg.length;
    p.status = SWIMMER_OK;
    if (p.n < 3 || (cfg.n_swimmers == 2 ? 2 : 1) * (p.n + p.nh) > cfg.n_max) {
        p.n = 3;
        p.status = SWIMMER_BAD_SAMPLE;
    }
    p.ds = p.length / (p.n - 1);
    p.delta = cfg.delta_over_ds * p.ds;
    double rho = R_MAX_OVER_L * sample_reach(cfg, p.n, p.ds) / p.delta;  // r_max/delta, as handle_octaves()
    int n_oct = (int)floor(log2(1.0 + rho * rho)) + 1;
    if (n_oct > N_OCT_MAX) {
        n_oct = N_OCT_MAX;
        p.status = SWIMMER_BAD_SAMPLE;
    }
    p.n_oct = n_oct;
    if (!(p.sig > 0.0) || !isfinite(p.sig)) p.status = SWIMMER_BAD_SAMPLE;
    if (!(p.alpha >= 0.0) || p.alpha * R_MAX_OVER_L * sample_reach(cfg, p.n, p.ds) > X_MAX || !isfinite(p.kc) ||
        !isfinite(p.amp) || !(p.kc > 0.0))
        p.status = SWIMMER_BAD_SAMPLE;
    sp[b] = p;
    order[b] = b;
}

// Longest-first processing order for the persistent work queue (the classic LPT rule):
// batches of uneven size by n, largest first (a run costs n^2 per step); batches of one size
// by ascending bending stiffness K_C, whose growth lowers forward Euler's stability limit, so
// that the runs likely to stop early (DIVERGED) come last and the queue, which deals runs to
// the SMs in turn, spreads them over the SMs.  Counting sort in one CTA (log10 K_C in 1024
// buckets over [-5, 5]); samples with a bad status go last (they do no work).
constexpr int SORT_THREADS = 1024;
__device__ __forceinline__ int order_key(const SampleParams &p, bool by_kc) {
    if (p.status != SWIMMER_OK) return N_PTS_MAX + 1;
    if (by_kc) return min(max((int)floor((log10(p.kc) + 5.0) * 102.4), 0), N_PTS_MAX);
    return N_PTS_MAX + 1 - min(max(p.n, 0), N_PTS_MAX);
}
__global__ void __launch_bounds__(SORT_THREADS) order_kernel(int B, const SampleParams *__restrict__ sp,
                                                           int *__restrict__ order, int by_kc) {
    __shared__ int cnt[N_PTS_MAX + 2];
    __shared__ int start[N_PTS_MAX + 2];
    const int tid = threadIdx.x;
    for (int i = tid; i < N_PTS_MAX + 2; i += SORT_THREADS) cnt[i] = 0;
    __syncthreads();
    for (int b = tid; b < B; b += SORT_THREADS) atomicAdd(&cnt[order_key(sp[b], by_kc)], 1);
    __syncthreads();
    if (tid == 0) {
        int acc = 0;
        for (int k = 0; k < N_PTS_MAX + 2; ++k) {
            start[k] = acc;
            acc += cnt[k];
        }
    }
    __syncthreads();
    for (int b = tid; b < B; b += SORT_THREADS) order[atomicAdd(&start[order_key(sp[b], by_kc)], 1)] = b;
}

// ---------------------------------------------------------------------------------
// K1a: one thread per node: the integrals over the interval that ends at the node and the
// Bessel factors at the node, for all samples; the last row of CTAs takes the integral of
// K0 phi s beyond the last node
// ---------------------------------------------------------------------------------
constexpr int K1_THREADS = 256;
constexpr int K1A_THREADS = 128;
// tail pieces beyond sigma_last: each sqrt(2) - 1 of its start wide, at most 4/beta, until 60/beta
// beyond or s^-3 has fallen by 1e-18; 12 points a piece
constexpr int TAIL_PIECES = 60, TAIL_POINTS = 12;
// FP32 handles: at most 64 pieces of up to 5 parts (a piece is at most 2/alpha wide, a part
// 0.5/alpha; 5 by rounding), 8 points a part.  The last of 64 pieces runs to the end whatever
// its width: with as many its share is below 1e-18 of the first's.
constexpr int TAIL8_MAX = 64, TAIL8_SUB = 5, TAIL8_POINTS = TAIL8_MAX * TAIL8_SUB * 8;

__device__ __forceinline__ int node_count(const SampleParams &p, int NP, int max_oct) {
    return min(p.n_oct, max_oct) * F64_SUB * NP;
}

// scratch row of a sample: K1_ROWS values per node, then the tail
enum { K1_IA, K1_IC, K1_E1, K1_WA, K1_WC, K1_E2, K1_VA, K1_VC };
enum { K1_I0 = 2, K1_I2, K1_K0, K1_K2, K1_T2K2, K1_IX2W };  // FP32 handles

__global__ void __launch_bounds__(K1A_THREADS)
table_nodes_kernel(const SampleParams *__restrict__ sp, double *__restrict__ scratch, int lite, int max_oct) {
    __shared__ double s_edge[TAIL8_MAX + 1], s_red[K1A_THREADS / 32];
    __shared__ int s_pieces, s_at[TAIL8_MAX + 1];
    static_assert(TAIL_PIECES <= TAIL8_MAX && TAIL8_MAX <= K1A_THREADS, "tail pieces");
    const SampleParams p = sp[blockIdx.x];
    if (p.status != SWIMMER_OK || !(p.alpha > 0.0)) return;
    const int NP = lite ? LITE_NODES : F64_NODES;
    const int M = node_count(p, NP, max_oct);
    const double beta = p.alpha * p.delta;
    double *out = scratch + (size_t)blockIdx.x * K1_SCRATCH;
    if (lite && blockIdx.y == gridDim.y - 1) {
        // the tail: pieces whose widths double from the last node up to 2/alpha, then stay; a
        // thread per point, then a thread per piece sums its points in order
        __shared__ double s_f[TAIL8_POINTS];
        if (threadIdx.x == 0) {
            const double r_last = p.delta * sqrt(node6_u(M - 1) - 1.0);
            const double end = fmin(r_last + 60.0 / p.alpha, 1e6 * p.delta);
            double s = r_last;
            int k = 0, at = 0;
            while (k < TAIL8_MAX && s < end) {
                const double w = fmin(fmax(s, 0.25 * p.delta), 2.0 / p.alpha);
                const double e = (k == TAIL8_MAX - 1) ? end : fmin(s + w, end);
                s_edge[k] = s;
                const double we = e - s;
                int n = (int)ceil(fmax(p.alpha * we / 0.5, we / (0.5 * fmax(s, 0.25 * p.delta))));
                s_at[k] = at;
                at += n < 1 ? 1 : n > TAIL8_SUB ? TAIL8_SUB : n;
                s = e;
                s_edge[++k] = s;
            }
            s_at[k] = at;
            s_pieces = k;
        }
        __syncthreads();
        const int K = s_pieces;
        const double dr = p.delta / s_edge[0];
        const double x_exact = dr * dr * dr > 4e-6 ? p.alpha * s_edge[0] + 6.0 : 2.0;
        for (int i = threadIdx.x; i < 8 * s_at[K]; i += K1A_THREADS) {
            int k = 0;
            while (s_at[k + 1] <= i / 8) ++k;
            const int n = s_at[k + 1] - s_at[k], q = i / 8 - s_at[k];
            const double hw = 0.5 * (s_edge[k + 1] - s_edge[k]) / n, c = s_edge[k] + (2 * q + 1) * hw;
            const double s = c + hw * c_gl8_x[i % 8], x = p.alpha * s;
            double k0, im;
            if (x <= 2.0)
                k0 = series_k0(x);
            else if (x <= x_exact)
                k0 = trapezoid_k0(x);
            else
                bessel_k0_i0m1(x, 0.0, rsqrt(x), false, k0, im);
            s_f[i] = k0 * blob(s, p.delta) * s;
        }
        __syncthreads();
        double tot = 0.0;
        if (threadIdx.x < K) {
            const int k = threadIdx.x, n = s_at[k + 1] - s_at[k];
            const double hw = 0.5 * (s_edge[k + 1] - s_edge[k]) / n;
            for (int q = 0; q < n; ++q) {
                double acc = 0.0;
                for (int g = 0; g < 8; ++g) acc += c_gl8_w[g] * s_f[8 * (s_at[k] + q) + g];
                tot += acc * hw;
            }
        }
        __syncthreads();
        if (threadIdx.x < K) s_f[threadIdx.x] = tot;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = K - 1; k >= 0; --k) t += s_f[k];  // far (small) pieces first
            out[K1_ROWS * (size_t)NODES_MAX] = t;
        }
        return;
    }
    if (blockIdx.y == gridDim.y - 1) {  // the tail
        const double s0 = g_node[M - 1].sig;
        if (threadIdx.x == 0) {
            double s = s0;
            const double wmax = 4.0 / beta, end = s0 + 60.0 / beta, last = fmin(1e6, 1e6 * s0);
            int k = 0;
            s_edge[0] = s;
            while (k < TAIL_PIECES && s < end && s < last) {
                s = fmin(s + fmin(0.41421356237309515 * s, wmax), end);
                s_edge[++k] = s;
            }
            s_pieces = k;
        }
        __syncthreads();
        const double lb = log(0.5 * beta) + EGAMMA;
        double sum = 0.0;
        for (int i = threadIdx.x; i < s_pieces * TAIL_POINTS; i += K1A_THREADS) {
            const int k = i / TAIL_POINTS, g = i % TAIL_POINTS;
            const double a = s_edge[k], hw = 0.5 * (s_edge[k + 1] - a);
            const double s = a + hw + hw * c_gl12_x[g], q = rsqrt(fma(s, s, 1.0)), q2 = q * q, x = beta * s;
            double k0, im;
            bessel_k0_i0m1(x, lb + log(s), rsqrt(x), false, k0, im);
            sum = fma(hw * c_gl12_w[g] * (3.0 / (2.0 * PI)) * s * q2 * q2 * q, k0, sum);
        }
        for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < K1A_THREADS / 32; ++k) t += s_red[k];
            out[K1_ROWS * (size_t)NODES_MAX] = t;
        }
        return;
    }
    const int q = blockIdx.y * K1A_THREADS + threadIdx.x;
    if (q >= M) return;
    // ---- the interval [sigma_{q-1}, sigma_q] (from 0 for the first node, where only A1's counts)
    double ia = 0.0, ic = 0.0;
    if (lite) {
        const double r = p.delta * sqrt(node6_u(q) - 1.0), rprev = q ? p.delta * sqrt(node6_u(q - 1) - 1.0) : 0.0;
        panel_integrals8(rprev, r, p.alpha, p.delta, q > 0, ia, ic);
        const BesselSet bs = bessel_set(p.alpha * r);
        out[K1_IA * (size_t)NODES_MAX + q] = ia;
        out[K1_IC * (size_t)NODES_MAX + q] = ic;
        out[K1_I0 * (size_t)NODES_MAX + q] = bs.i0;
        out[K1_I2 * (size_t)NODES_MAX + q] = bs.i2;
        out[K1_K0 * (size_t)NODES_MAX + q] = bs.k0;
        out[K1_K2 * (size_t)NODES_MAX + q] = bs.k2;
        out[K1_T2K2 * (size_t)NODES_MAX + q] = bs.t2k2;
        out[K1_IX2W * (size_t)NODES_MAX + q] = bs.ix2w;
        return;
    }
    const double lb = log(0.5 * beta) + EGAMMA, rsb = rsqrt(beta);
    const NodeRec nd = g_node[q];
    const double sprev = q ? g_node[q - 1].sig : 0.0;
    if (beta * (nd.sig - sprev) > WIDTH_MAX) {
        split_integral(sprev, nd.sig, beta, ia, ic);
    } else {
        const int e = g_quad_at[q + 1];
        for (int i = g_quad_at[q]; i < e; ++i) {
            const QuadRec c = g_quad[i];
            double k0, im = 0.0;
            bessel_k0_i0m1(beta * c.sig, lb + c.lns, rsb * c.rsq, true, k0, im);
            ia = fma(c.w, im, ia);
            ic = fma(c.w, k0, ic);
        }
    }
    out[K1_IA * (size_t)NODES_MAX + q] = ia;
    out[K1_IC * (size_t)NODES_MAX + q] = ic;
    // ---- the node: g1 = E1 - WA A1 - WC C, delta^2 g2 = E2 - VA A1 - VC C
    const double x = beta * nd.sig, rs = rsb * nd.rsq, z = rs * rs;
    double i0, i2, k0, k2, t2k2, ix2w;  // t2k2 = 2/x^2 - K2, ix2w = 1/x^2 - (K0 + K2)/2
    const double y = 0.25 * x * x;
    if (x <= I_SERIES) {
        if (x <= 2.0) {
            i0 = horner<SER_K>(c_i0, y);
            i2 = horner<SER_K>(c_i2, y);
        } else {
            i0 = horner<SER>(c_i0, y);
            i2 = horner<SER>(c_i2, y);
        }
    } else {
        const double ex = exp(x) * rs;
        i0 = ex * i_poly(c_i0p, c_i0q, x > I_SPLIT, z);
        i2 = ex * i_poly(c_i2p, c_i2q, x > I_SPLIT, z);
    }
    if (x <= 2.0) {
        const double lx = log(0.5 * x) + EGAMMA;  // (the sum lb + ln sigma would round twice more)
        k0 = fma(-lx, i0, y * horner<SER_K - 1>(c_k0t + 1, y));
        // 2/x^2 - K2 = 1/2 + y sum_k [lx - (H_k + H_{k+2})/2] y^k/(k! (k+2)!)
        t2k2 = fma(y, fma(lx, i2, -horner<SER_K>(c_t2, y)), 0.5);
        k2 = 0.5 / y - t2k2;
        ix2w = 0.5 * (t2k2 - k0);
        i2 *= y;
    } else {
        const double ex = exp(-x) * rs;
        const bool far = x > K_SPLIT;
        k0 = ex * k_poly(c_k0, far, z);
        k2 = fma(2.0 * z, ex * k_poly(c_k1, far, z), k0);
        t2k2 = fma(2.0 * z, z, -k2);
        ix2w = fma(z, z, -0.5 * (k0 + k2));
        if (x <= I_SERIES) i2 *= y;
    }
    out[K1_E1 * (size_t)NODES_MAX + q] = ix2w * nd.m0;
    out[K1_WA * (size_t)NODES_MAX + q] = 0.5 * (k0 + k2);
    out[K1_WC * (size_t)NODES_MAX + q] = 0.5 * (i0 + i2);
    out[K1_E2 * (size_t)NODES_MAX + q] = t2k2 * nd.m0 * nd.inv2;
    out[K1_VA * (size_t)NODES_MAX + q] = k2 * nd.inv2;
    out[K1_VC * (size_t)NODES_MAX + q] = i2 * nd.inv2;
}

// ---------------------------------------------------------------------------------
// K1b: per sample: prefix/suffix sums, node values, the table's fit.  A lone sample's fit is
// split over gridDim.y CTAs, each of which repeats the (short) sums and fits its part.
// ---------------------------------------------------------------------------------
template <bool LITE>
__global__ void __launch_bounds__(K1_THREADS)
table_build_kernel(SampleParams *__restrict__ sp, const double *__restrict__ scratch, float4 *__restrict__ tab64,
                   float4 *__restrict__ tab32, int max_oct) {
    extern __shared__ double sm[];
    __shared__ double s_part[2][K1_THREADS / 32];
    const int b = blockIdx.x;
    SampleParams p = sp[b];
    if (p.n_oct > max_oct) {  // never beyond the shared-memory node arrays
        p.n_oct = max_oct;
        __syncthreads();
        if (threadIdx.x == 0) sp[b].n_oct = max_oct;  // (every CTA of the sample writes the same)
    }
    constexpr int NP = LITE ? LITE_NODES : F64_NODES;  // nodes per FP64 panel
    const int M = p.n_oct * F64_SUB * NP;
    double *g1s = sm, *g2s = sm + M;  // [M] node values
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float4 *t64 = tab64 + (size_t)b * TAB64_STRIDE;
    float4 *t32 = tab32 + (size_t)b * TAB32_STRIDE;
    const int at = blockIdx.y * K1_THREADS + tid, step = gridDim.y * K1_THREADS;

    if (p.status != SWIMMER_OK) {
        // keep the table finite so that a stray read cannot produce garbage
        if (!LITE)
            for (int i = at; i < TAB64_STRIDE; i += step) t64[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        else
            for (int i = at; i < TAB32_STRIDE; i += step) t32[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const double *row = scratch + (size_t)b * K1_SCRATCH;
    const double tail = row[K1_ROWS * (size_t)NODES_MAX];

    if (!(p.alpha > 0.0)) {
        for (int m = tid; m < M; m += blockDim.x) {
            double g1, g2;
            stokes_g(LITE ? p.delta * sqrt(node6_u(m) - 1.0) : p.delta * g_node[m].sig, p.delta, &g1, &g2);
            g1s[m] = g1;
            g2s[m] = LITE ? g2 : g2 * p.delta * p.delta;
        }
    } else if (LITE) {
        // A1 (prefix) and C (suffix) by warp 0: lanes own contiguous chunks (the order of these
        // sums is part of what keeps the FP32 tables bit for bit the same)
        double *nodeA = g1s, *nodeC = g2s;
        for (int m = tid; m < M; m += K1_THREADS) {
            nodeA[m] = row[K1_IA * (size_t)NODES_MAX + m];
            nodeC[m] = m + 1 < M ? row[K1_IC * (size_t)NODES_MAX + m + 1] : tail;
        }
        __syncthreads();
        if (tid < 32) {
            int chunk = (M + 31) / 32;
            int lo = tid * chunk, hi = min(M, lo + chunk);
            double sa = 0.0, sc = 0.0;
            for (int m = lo; m < hi; ++m) sa += nodeA[m];
            for (int m = lo; m < hi; ++m) sc += nodeC[m];
            // exclusive scans of the chunk totals (A: from the left, C: from the right)
            double pa = sa, pc = sc;
            for (int o = 1; o < 32; o <<= 1) {
                double va = __shfl_up_sync(0xffffffffu, pa, o);
                double vc = __shfl_down_sync(0xffffffffu, pc, o);
                if (tid >= o) pa += va;
                if (tid + o < 32) pc += vc;
            }
            double offa = pa - sa, offc = pc - sc;
            double run = offa;
            for (int m = lo; m < hi; ++m) {
                run += nodeA[m];
                nodeA[m] = run;
            }
            run = offc;
            for (int m = hi - 1; m >= lo; --m) {
                run += nodeC[m];
                nodeC[m] = run;
            }
        }
        __syncthreads();
        for (int m = tid; m < M; m += K1_THREADS) {
            double r = p.delta * sqrt(node6_u(m) - 1.0);
            BesselSet bs;
            bs.i0 = row[K1_I0 * (size_t)NODES_MAX + m];
            bs.i2 = row[K1_I2 * (size_t)NODES_MAX + m];
            bs.k0 = row[K1_K0 * (size_t)NODES_MAX + m];
            bs.k2 = row[K1_K2 * (size_t)NODES_MAX + m];
            bs.t2k2 = row[K1_T2K2 * (size_t)NODES_MAX + m];
            bs.ix2w = row[K1_IX2W * (size_t)NODES_MAX + m];
            double M0 = m0_closed(r, p.delta), A = nodeA[m], C = nodeC[m];
            double w = 0.5 * (bs.k0 + bs.k2);
            double g1 = bs.ix2w * M0 - w * A - 0.5 * (bs.i0 + bs.i2) * C;
            double g2 = (bs.t2k2 * M0 - bs.k2 * A - bs.i2 * C) / (r * r);
            g1s[m] = g1;
            g2s[m] = g2;
        }
    } else {
        // A1 at node m: sum of the intervals up to it; C: the tail and the intervals beyond it.
        // Thread t owns the nodes [t chunk, (t + 1) chunk).
        const int chunk = (M + K1_THREADS - 1) / K1_THREADS;
        const int lo = min(M, tid * chunk), hi = min(M, lo + chunk);
        double sa = 0.0, sc = 0.0;
        for (int m = lo; m < hi; ++m) sa += row[K1_IA * (size_t)NODES_MAX + m];
        for (int m = hi - 1; m >= lo; --m) sc += m + 1 < M ? row[K1_IC * (size_t)NODES_MAX + m + 1] : tail;
        double pa = sa, pc = sc;  // inclusive scans within the warp (A from the left, C from the right)
        for (int o = 1; o < 32; o <<= 1) {
            const double va = __shfl_up_sync(0xffffffffu, pa, o), vc = __shfl_down_sync(0xffffffffu, pc, o);
            if (lane >= o) pa += va;
            if (lane + o < 32) pc += vc;
        }
        if (lane == 31) s_part[0][warp] = pa;
        if (lane == 0) s_part[1][warp] = pc;
        // what lies before (A) and beyond (C) the chunk: the neighbours' inclusive sums, not a
        // difference (C falls steeply, and inclusive minus own would cancel)
        const double before = __shfl_up_sync(0xffffffffu, pa, 1), beyond = __shfl_down_sync(0xffffffffu, pc, 1);
        __syncthreads();
        double A = 0.0, C = 0.0;
        for (int k = 0; k < warp; ++k) A += s_part[0][k];
        for (int k = K1_THREADS / 32 - 1; k > warp; --k) C += s_part[1][k];
        if (lane > 0) A += before;
        if (lane < 31) C += beyond;
        for (int m = lo; m < hi; ++m) {
            A += row[K1_IA * (size_t)NODES_MAX + m];
            g1s[m] = A;
        }
        for (int m = hi - 1; m >= lo; --m) {
            C += m + 1 < M ? row[K1_IC * (size_t)NODES_MAX + m + 1] : tail;
            const double a = g1s[m];
            g1s[m] = row[K1_E1 * (size_t)NODES_MAX + m] - row[K1_WA * (size_t)NODES_MAX + m] * a -
                     row[K1_WC * (size_t)NODES_MAX + m] * C;
            g2s[m] = row[K1_E2 * (size_t)NODES_MAX + m] - row[K1_VA * (size_t)NODES_MAX + m] * a -
                     row[K1_VC * (size_t)NODES_MAX + m] * C;
        }
    }
    __syncthreads();

    if (!LITE) {
        // the panels' records (table_eval.cuh), four panels to a build panel
        const int np = p.n_oct * F64_SUB;
        for (int q = at; q < p.n_oct * F64_FINE; q += step) {  // (a warp shares its rows of c_fit64)
            const int panel = q % np, part = q / np;
            float4 *rec = t64 + F64_REC * (panel * F64_SPLIT + part);
            const double *ga = g1s + panel * F64_NODES, *gb = g2s + panel * F64_NODES;
            // the fit of the differences from a middle node: they are exact, and the rounding of
            // the higher coefficients' sums of alternating terms stays in proportion to them
            const double ma = ga[F64_NODES / 2], mb = gb[F64_NODES / 2];
            double ca[F64_COEF], cb[F64_COEF];
#pragma unroll
            for (int k = 0; k < F64_COEF; ++k) {
                double x = 0.0, y = 0.0;
                for (int i = 0; i < F64_NODES; ++i) {
                    const double w = c_fit64[part][k][i];
                    x = fma(w, ga[i] - ma, x);
                    y = fma(w, gb[i] - mb, y);
                }
                ca[k] = x;
                cb[k] = y;
            }
            *(double2 *)rec = make_double2(ma + ca[0], mb + cb[0]);
#pragma unroll
            for (int k = 1; k <= 5; ++k) {
                const float ha = (float)ca[k], hb = (float)cb[k];
                rec[k] = make_float4(ha, hb, (float)(ca[k] - (double)ha), (float)(cb[k] - (double)hb));
            }
            rec[6] = make_float4((float)ca[6], (float)cb[6], (float)ca[7], (float)cb[7]);
        }
        return;
    }
    // Chebyshev coefficients of the 6 node values, in place (each thread its panels)
    const int np = p.n_oct * F64_SUB;
    for (int q = tid; q < 2 * np; q += K1_THREADS) {
        double *g = (q < np ? g1s : g2s) + (q % np) * LITE_NODES, c[LITE_NODES];
        for (int k = 0; k < LITE_NODES; ++k) {
            double s = 0.0;
            for (int ii = 0; ii < LITE_NODES; ++ii) s += g[ii] * c_dct6[k][ii];
            c[k] = s;
        }
        for (int k = 0; k < LITE_NODES; ++k) g[k] = c[k];
    }
    __syncthreads();
    // FP32 quadratic per eighth of an FP64 panel from its series (Chebyshev fit at 3 nodes, then
    // monomial coefficients in G = 1 + f / F32_SUB, f in [0, 1) across the panel); the FP32 table
    // holds -g1 (the sign the pair sum's mobility -g1 I + h e e^T takes) and h = delta^2 g2, for
    // separations measured in units of delta
    float2 *t32b = (float2 *)(t32 + F32_PANELS_MAX);
    for (int q = at; q < p.n_oct * F32_SUB; q += step) {
        const int panel = q / F32_SPLIT, jj = q % F32_SPLIT;
        double cf[2][3];
        for (int fn = 0; fn < 2; ++fn) {
            const double *c = (fn == 0 ? g1s : g2s) + panel * LITE_NODES;
            double vals[3];
            for (int i = 0; i < 3; ++i) {
                double f32 = 0.5 * (c_node3[i] + 1.0);  // node of the FP32 panel
                double f64 = (jj + f32) / F32_SPLIT;
                double t = 2.0 * f64 - 1.0;
                double b1 = 0.0, b2 = 0.0;
                for (int k = LITE_NODES - 1; k >= 1; --k) {
                    double b0 = 2.0 * t * b1 - b2 + c[k];
                    b2 = b1;
                    b1 = b0;
                }
                vals[i] = t * b1 - b2 + c[0];
            }
            double a[3];
            for (int k = 0; k < 3; ++k) a[k] = vals[0] * c_dct3[k][0] + vals[1] * c_dct3[k][1] + vals[2] * c_dct3[k][2];
            // p(t) = a0 + a1 t + a2 (2 t^2 - 1), t = 2 f - 1: p = m0 + m1 f + m2 f^2.  The kernel
            // reads G = 1 + f / S (S = F32_SUB) straight from the low mantissa bits of u, so
            // p = c0 + c1 G + c2 G^2 with f = S (G - 1)
            const double m0 = a[0] - a[1] + a[2], m1 = 2.0 * a[1] - 8.0 * a[2], m2 = 8.0 * a[2];  // in f
            const double S = F32_SUB, sc = fn == 1 ? p.delta * p.delta : -1.0;  // -g1; delta^2 g2
            cf[fn][0] = sc * (m0 - S * m1 + S * S * m2);
            cf[fn][1] = sc * (S * m1 - 2.0 * S * S * m2);
            cf[fn][2] = sc * (S * S * m2);
        }
        t32[q] = make_float4((float)cf[0][0], (float)cf[0][1], (float)cf[0][2], (float)cf[1][0]);
        t32b[q] = make_float2((float)cf[1][1], (float)cf[1][2]);
    }
}

__global__ void set_sample_kernel(SampleParams *sp, double alpha, double delta, double r_max) {
    SampleParams p;
    p.alpha = alpha;
    p.kc = 1.0;
    p.amp = 0.0;
    p.length = r_max / R_MAX_OVER_L;
    p.n = 3;
    p.nh = 0;
    p.sig = 1.0;
    p.ds = p.length / 2;
    p.delta = delta;
    double rho = r_max / delta;
    int n_oct = (int)floor(log2(1.0 + rho * rho)) + 1;
    p.status = SWIMMER_OK;
    if (n_oct > N_OCT_MAX || !(alpha >= 0.0) || alpha * r_max > X_MAX) p.status = SWIMMER_BAD_SAMPLE;
    p.n_oct = min(n_oct, N_OCT_MAX);
    sp[0] = p;
}

// ---------------------------------------------------------------------------------
// kernel-function evaluation through the tables (testing entry point)
// ---------------------------------------------------------------------------------
__global__ void kernel_eval_kernel(int m, const double *__restrict__ r, double *__restrict__ g1,
                                   double *__restrict__ g2, const SampleParams *__restrict__ sp,
                                   const float4 *__restrict__ tab64, const float4 *__restrict__ tab32,
                                   int precision) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const SampleParams p = sp[0];
    double rr = r[i];
    if (precision == SWIMMER_FP64) {
        double u = 1.0 + rr * rr / (p.delta * p.delta);
        if (!(u >= 1.0) || !(u < ldexp(1.0, p.n_oct))) {
            g1[i] = g2[i] = nan("");
            return;
        }
        double h;
        kern_f64(tab64, p.n_oct * F64_FINE - 1, u, g1[i], h);
        g2[i] = h / (p.delta * p.delta);
    } else {
        float inv_d2 = (float)(1.0 / (p.delta * p.delta));
        float r2 = (float)(rr * rr);
        float u = fmaf(r2, inv_d2, 1.0f);
        unsigned bits = __float_as_uint(u);
        unsigned panel = (bits >> (23 - F32_SUB_LOG2)) - (127u << F32_SUB_LOG2);
        if (!(u >= 1.0f) || panel >= (unsigned)(p.n_oct * F32_SUB)) {
            g1[i] = g2[i] = nan("");
            return;
        }
        float G = __uint_as_float(0x3f800000u | (bits & ((1u << (23 - F32_SUB_LOG2)) - 1u)));
        float4 a = tab32[panel];
        float2 c = ((const float2 *)(tab32 + F32_PANELS_MAX))[panel];
        g1[i] = -fmaf(G, fmaf(G, a.z, a.y), a.x);           // the table holds -g1
        g2[i] = fmaf(G, fmaf(G, c.y, c.x), a.w) * inv_d2;  // and delta^2 g2
    }
}

}  // namespace

// Gauss-Legendre nodes/weights on [-1, 1] by Newton's method on P_n (host).
static void gauss_legendre(int n, double *x, double *w) {
    for (int i = 0; i < n; ++i) {
        double z = cos(PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            double dz = p1 / dp;
            z -= dz;
            if (fabs(dz) < 1e-16) break;
        }
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= n; ++k) {
            double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = n * (z * p1 - p0) / (z * z - 1.0);
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// ---- host Bessel functions at the fit's nodes
// K_0 e^x sqrt(x) and K_1 e^x sqrt(x), x >= 2: the trapezoid rule on the integral representation,
// whose error decays like exp(-2 pi d/h) for the strip half-width d = acos(1 - 1/x)
static void host_k_scaled(double x, double *k0, double *k1) {
    const double d = acos(1.0 - 1.0 / x), h = d / 6.5;
    double s0 = 0.5, s1 = 0.5;
    for (int m = 1; m < 4000; ++m) {
        const double sh = sinh(0.5 * m * h), c1 = 2.0 * sh * sh;  // cosh(m h) - 1
        const double e = exp(-x * c1);
        s0 += e;
        s1 += e * (1.0 + c1);
        if (e < 1e-19 * s0) break;
    }
    *k0 = h * s0 * sqrt(x);
    *k1 = h * s1 * sqrt(x);
}
// I_nu e^-x sqrt(x), nu = 0 or 2, x >= 8: power series to x = 30, Hankel's expansion beyond
static double host_i_scaled(int nu, double x) {
    if (x <= 30.0) {
        const double y = 0.25 * x * x;
        double term = nu == 0 ? 1.0 : 0.5 * y, s = 0.0;
        for (int k = 0; k < 200; ++k) {
            s += term;
            term *= y / ((k + 1.0) * (k + 1.0 + nu));
            if (term < 1e-18 * s) break;
        }
        return s * exp(-x) * sqrt(x);
    }
    const double mu = 4.0 * nu * nu;
    double s = 1.0, term = 1.0;
    for (int k = 1; k < 60; ++k) {
        const double t = -term * (mu - (2.0 * k - 1.0) * (2.0 * k - 1.0)) / (8.0 * k * x);
        if (fabs(t) > fabs(term)) break;
        term = t;
        s += term;
        if (fabs(term) < 1e-18 * fabs(s)) break;
    }
    return s / sqrt(2.0 * PI);
}

// Chebyshev coefficients in [-1, 1] to powers (in place, n of them)
template <class T>
static void cheb_to_powers(T *c, int n) {
    std::vector<T> out(n, 0.0), t0(n, 0.0), t1(n, 0.0), t2(n, 0.0);
    t0[0] = 1.0;
    if (n > 1) t1[1] = 1.0;
    for (int k = 0; k < n; ++k) {
        const std::vector<T> &tk = k == 0 ? t0 : t1;
        for (int i = 0; i < n; ++i) out[i] += c[k] * tk[i];
        if (k >= 1) {
            for (int i = 0; i < n; ++i) t2[i] = (i ? 2.0 * t1[i - 1] : 0.0) - t0[i];
            t0 = t1;
            t1 = t2;
        }
    }
    std::copy(out.begin(), out.end(), c);
}
// The fit of a function on [-1, 1] in powers of t: its polynomial through n Chebyshev nodes as a Chebyshev
// series cut to degree deg (so that what is cut is small).  node [n]; weight [deg + 1][n] takes the values there
// to the coefficients.  In extended precision: rounding of these sums would show in the leading coefficient's
// last places.
void fit_matrix(int n, int deg, long double *node, long double *weight) {
    const long double pi = acosl(-1.0L);
    for (int i = 0; i < n; ++i) {
        node[i] = cosl(pi * (i + 0.5L) / n);
        std::vector<long double> c(deg + 1);
        for (int k = 0; k <= deg; ++k) c[k] = cosl(pi * k * (i + 0.5L) / n) * (k == 0 ? 1.0L : 2.0L) / n;
        cheb_to_powers(c.data(), deg + 1);
        for (int k = 0; k <= deg; ++k) weight[k * n + i] = c[k];
    }
}

// powers of t = z_scale z + z_shift of f(1/z) on x in [lo, 1/inv_hi], degree deg
template <class F>
static void fit_inverse(double lo, double inv_hi, int deg, F f, double *c) {
    const int n = deg + 1;
    std::vector<double> v(n);
    for (int i = 0; i < n; ++i) v[i] = f(z_scale(lo, inv_hi) / (cos(PI * (i + 0.5) / n) - z_shift(lo, inv_hi)));
    for (int k = 0; k < n; ++k) {
        double s = 0.0;
        for (int i = 0; i < n; ++i) s += v[i] * cos(PI * k * (i + 0.5) / n);
        c[k] = s * (k == 0 ? 1.0 : 2.0) / n;
    }
    cheb_to_powers(c, n);
}

// the sample-independent nodes and quadrature points
static void build_universal(std::vector<NodeRec> &node, std::vector<QuadRec> &quad, std::vector<int> &at) {
    const int np = F64_NODES, M = F64_PANELS_MAX * np;
    std::vector<double> gx[GL_N + 1], gw[GL_N + 1];
    for (int n = QUAD_MIN; n <= GL_N; ++n) {
        gx[n].resize(n);
        gw[n].resize(n);
        gauss_legendre(n, gx[n].data(), gw[n].data());
    }
    double prev = 0.0;
    at.assign(1, 0);
    for (int m = 0; m < M; ++m) {
        const int panel = m / np, i = np - 1 - m % np;  // ascending nodes
        const double f = 0.5 * (cos(PI * (i + 0.5) / np) + 1.0);
        const int e = panel >> F64_SUB_LOG2, j = panel & (F64_SUB - 1);
        // u - 1 without cancellation in the first octave
        const double um1 = e == 0 ? (j + f) / F64_SUB : ldexp(1.0 + (j + f) / F64_SUB, e) - 1.0;
        NodeRec r;
        r.sig = sqrt(um1);
        r.lns = 0.5 * log(um1);
        r.rsq = 1.0 / sqrt(r.sig);
        r.inv2 = 1.0 / um1;
        const double R = sqrt(1.0 + um1);
        r.m0 = (um1 / (R + 1.0)) * (R * R + R + 1.0) / (R * R * R) / (2.0 * PI);
        r.pad = 0.0;
        node.push_back(r);
        // the interval's points: enough for 1e-16 in the Bernstein ellipse that reaches s = 0
        // (ln s; not for the first, which starts there and carries I0 - 1 alone) and s = +-i
        const double c = 0.5 * (r.sig + prev), hw = 0.5 * (r.sig - prev);
        double rho = 1e30;
        if (m > 0) rho = c / hw + sqrt(c / hw * (c / hw) - 1.0);
        // |z + sqrt(z^2 - 1)| at z = (c + i)/hw by the ellipse's semi-axes sum
        const double d1 = hypot(c / hw + 1.0, 1.0 / hw), d2 = hypot(c / hw - 1.0, 1.0 / hw), a = 0.5 * (d1 + d2);
        rho = std::min(rho, a + sqrt(a * a - 1.0));
        const int n = std::min(GL_N, std::max(QUAD_MIN, (int)ceil(37.0 / (2.0 * log(rho))) + 1));
        for (int g = n - 1; g >= 0; --g) {  // ascending points
            QuadRec q;
            q.sig = c + hw * gx[n][g];
            q.lns = log(q.sig);
            q.rsq = 1.0 / sqrt(q.sig);
            const double R2 = q.sig * q.sig + 1.0;
            q.w = hw * gw[n][g] * 3.0 * q.sig / (2.0 * PI * R2 * R2 * sqrt(R2));
            quad.push_back(q);
        }
        at.push_back((int)quad.size());
        prev = r.sig;
    }
}

// constant and sample-independent tables for the table builder (host; device memory is per
// device, so once per device)
int gl_init() {
    static bool done[256] = {};
    static std::mutex mutex;
    std::lock_guard<std::mutex> lock(mutex);
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) {
        set_error("device ordinal %d out of range", dev);
        return SWIMMER_E_ARG;
    }
    if (done[dev]) return 0;
    double x[GL_N], w[GL_N];
    gauss_legendre(GL_N, x, w);
    CUDA_TRY(cudaMemcpyToSymbol(c_gl_x, x, sizeof(x)));
    CUDA_TRY(cudaMemcpyToSymbol(c_gl_w, w, sizeof(w)));
    gauss_legendre(12, x, w);
    CUDA_TRY(cudaMemcpyToSymbol(c_gl12_x, x, sizeof(double) * 12));
    CUDA_TRY(cudaMemcpyToSymbol(c_gl12_w, w, sizeof(double) * 12));
    // Bessel series
    double i0[SER], i2[SER], k0t[SER_K], t2[SER_K], harmonic[SER_K + 2] = {0.0};
    for (int k = 1; k < SER_K + 2; ++k) harmonic[k] = harmonic[k - 1] + 1.0 / k;
    i0[0] = 1.0;
    i2[0] = 0.5;
    for (int k = 1; k < SER; ++k) {
        i0[k] = i0[k - 1] / ((double)k * k);
        i2[k] = i2[k - 1] / ((double)k * (k + 2.0));
    }
    for (int k = 0; k < SER_K; ++k) {
        k0t[k] = harmonic[k] * i0[k];
        t2[k] = 0.5 * (harmonic[k] + harmonic[k + 2]) * i2[k];
    }
    CUDA_TRY(cudaMemcpyToSymbol(c_i0, i0, sizeof(i0)));
    CUDA_TRY(cudaMemcpyToSymbol(c_i2, i2, sizeof(i2)));
    CUDA_TRY(cudaMemcpyToSymbol(c_k0t, k0t, sizeof(k0t)));
    CUDA_TRY(cudaMemcpyToSymbol(c_t2, t2, sizeof(t2)));
    // Bessel fits in 1/x
    double pk[2][2][DEG_K + 1], pi1[2][DEG_I1 + 1], pi2[2][DEG_I2 + 1];
    for (int nu = 0; nu < 2; ++nu) {
        auto k = [nu](double v) {
            double a, b;
            host_k_scaled(v, &a, &b);
            return nu == 0 ? a : b;
        };
        fit_inverse(2.0, 1.0 / K_SPLIT, DEG_K, k, pk[nu][0]);
        fit_inverse(K_SPLIT, 0.0, DEG_K, k, pk[nu][1]);
        auto i = [nu](double v) { return host_i_scaled(2 * nu, v); };
        fit_inverse(I_SERIES, 1.0 / I_SPLIT, DEG_I1, i, pi1[nu]);
        fit_inverse(I_SPLIT, 0.0, DEG_I2, i, pi2[nu]);
    }
    CUDA_TRY(cudaMemcpyToSymbol(c_k0, pk[0], sizeof(pk[0])));
    CUDA_TRY(cudaMemcpyToSymbol(c_k1, pk[1], sizeof(pk[1])));
    CUDA_TRY(cudaMemcpyToSymbol(c_i0p, pi1[0], sizeof(pi1[0])));
    CUDA_TRY(cudaMemcpyToSymbol(c_i2p, pi1[1], sizeof(pi1[1])));
    CUDA_TRY(cudaMemcpyToSymbol(c_i0q, pi2[0], sizeof(pi2[0])));
    CUDA_TRY(cudaMemcpyToSymbol(c_i2q, pi2[1], sizeof(pi2[1])));
    // FP64 table fits: the degree-9 polynomial through the 10 nodes, on a quarter of its panel,
    // t = (tau + 2 part - 3) / 4, as a Chebyshev series in tau cut to degree 7 (what is cut is below
    // 1e-17), in powers of tau
    std::vector<double> fit(F64_SPLIT * F64_COEF * F64_NODES);
    for (int part = 0; part < F64_SPLIT; ++part)
        for (int ii = 0; ii < F64_NODES; ++ii) {
            const int i = F64_NODES - 1 - ii;  // ascending node ii is Chebyshev index i
            double v[F64_NODES], c[F64_NODES];
            for (int j = 0; j < F64_NODES; ++j) {
                const double t = 0.25 * (cos(PI * (j + 0.5) / F64_NODES) + 2.0 * part - 3.0);
                v[j] = 1.0 / F64_NODES;
                for (int k = 1; k < F64_NODES; ++k)
                    v[j] += (2.0 / F64_NODES) * cos(PI * k * (i + 0.5) / F64_NODES) * cos(k * acos(t));
            }
            for (int k = 0; k < F64_NODES; ++k) {
                c[k] = 0.0;
                for (int j = 0; j < F64_NODES; ++j)
                    c[k] += (k ? 2.0 : 1.0) / F64_NODES * v[j] * cos(PI * k * (j + 0.5) / F64_NODES);
            }
            cheb_to_powers(c, F64_COEF);
            for (int k = 0; k < F64_COEF; ++k) fit[(part * F64_COEF + k) * F64_NODES + ii] = c[k];
        }
    CUDA_TRY(cudaMemcpyToSymbol(c_fit64, fit.data(), sizeof(double) * fit.size()));
    // FP32 handles
    double ik[NSER], ikk[2][NSER], hk[HARM];
    for (int k = 0; k < NSER; ++k) {
        ik[k] = k ? 1.0 / k : 0.0;
        ikk[0][k] = 1.0 / ((k + 1.0) * (k + 1.0));
        ikk[1][k] = 1.0 / ((k + 1.0) * (k + 3.0));
    }
    hk[0] = 0.0;
    for (int k = 1; k < HARM; ++k) hk[k] = hk[k - 1] + ik[k];
    CUDA_TRY(cudaMemcpyToSymbol(c_inv_k, ik, sizeof(ik)));
    CUDA_TRY(cudaMemcpyToSymbol(c_inv_kk, ikk, sizeof(ikk)));
    CUDA_TRY(cudaMemcpyToSymbol(c_harm, hk, sizeof(hk)));
    gauss_legendre(8, x, w);
    CUDA_TRY(cudaMemcpyToSymbol(c_gl8_x, x, sizeof(double) * 8));
    CUDA_TRY(cudaMemcpyToSymbol(c_gl8_w, w, sizeof(double) * 8));
    double ct6[LITE_NODES], dct6[LITE_NODES][LITE_NODES];
    for (int ii = 0; ii < LITE_NODES; ++ii) {
        int i = LITE_NODES - 1 - ii;
        ct6[ii] = cos(PI * (i + 0.5) / LITE_NODES);
        for (int k = 0; k < LITE_NODES; ++k)
            dct6[k][ii] = (2.0 / LITE_NODES) * cos(PI * k * (i + 0.5) / LITE_NODES) * (k == 0 ? 0.5 : 1.0);
    }
    CUDA_TRY(cudaMemcpyToSymbol(c_cheb_t6, ct6, sizeof(ct6)));
    CUDA_TRY(cudaMemcpyToSymbol(c_dct6, dct6, sizeof(dct6)));
    double n3[3], d3[3][3];
    for (int i = 0; i < 3; ++i) {
        n3[i] = cos(PI * (i + 0.5) / 3.0);
        for (int k = 0; k < 3; ++k) d3[k][i] = (2.0 / 3.0) * cos(PI * k * (i + 0.5) / 3.0) * (k == 0 ? 0.5 : 1.0);
    }
    CUDA_TRY(cudaMemcpyToSymbol(c_node3, n3, sizeof(n3)));
    CUDA_TRY(cudaMemcpyToSymbol(c_dct3, d3, sizeof(d3)));
    // FP64 handles: nodes and quadrature points
    std::vector<NodeRec> node;
    std::vector<QuadRec> quad;
    std::vector<int> at;
    build_universal(node, quad, at);
    if (quad.size() > QUAD_CAP) {
        set_error("the table build's quadrature needs %zu points", quad.size());
        return SWIMMER_E_ARG;
    }
    CUDA_TRY(cudaMemcpyToSymbol(g_node, node.data(), sizeof(NodeRec) * node.size()));
    CUDA_TRY(cudaMemcpyToSymbol(g_quad, quad.data(), sizeof(QuadRec) * quad.size()));
    CUDA_TRY(cudaMemcpyToSymbol(g_quad_at, at.data(), sizeof(int) * at.size()));
    done[dev] = true;
    return 0;
}

int handle_octaves(const swimmer_handle *h) {
    // the sample with the most flagellum points and, for two swimmers, the smallest ds
    const int nfm = default_flagellum_points(h->cfg);
    const double ds = h->cfg.ds_fixed > 0.0 ? h->cfg.ds_fixed : h->cfg.length / (nfm - 1);
    double rho = R_MAX_OVER_L * sample_reach(h->cfg, nfm, ds) / (h->cfg.delta_over_ds * ds);
    int n_oct = (int)floor(log2(1.0 + rho * rho)) + 1;
    return n_oct > N_OCT_MAX ? N_OCT_MAX : n_oct;
}

int launch_prepare(swimmer_handle *h, int B, const double *theta, const int *n_pts, cudaStream_t s) {
    prepare_kernel<<<(B + 127) / 128, 128, 0, s>>>(B, theta, n_pts, h->cfg, h->sp, h->order);
    CUDA_TRY(cudaGetLastError());
    prof_count(h, 1);
    {  // longest first: by n for uneven sizes, else by K_C
        order_kernel<<<1, SORT_THREADS, 0, s>>>(B, h->sp, h->order, n_pts ? 0 : 1);
        CUDA_TRY(cudaGetLastError());
        prof_count(h, 1);
    }
    return 0;
}

// the two table kernels on B samples whose scratch rows start at `scratch`
static int table_kernels(int B, SampleParams *sp, double *scratch, float4 *tab64, float4 *tab32, bool lite, int oct,
                         int sms, cudaStream_t s) {
    const int M = oct * F64_SUB * (lite ? LITE_NODES : F64_NODES);
    const dim3 ga(B, (M + K1A_THREADS - 1) / K1A_THREADS + 1);
    table_nodes_kernel<<<ga, K1A_THREADS, 0, s>>>(sp, scratch, lite ? 1 : 0, oct);
    CUDA_TRY(cudaGetLastError());
    // the fit of few samples over several CTAs each (at most one per octave)
    const dim3 gb(B, std::max(1, std::min(oct, sms / B)));
    const size_t smem = 2 * (size_t)M * sizeof(double);
    if (lite)
        table_build_kernel<true><<<gb, K1_THREADS, smem, s>>>(sp, scratch, tab64, tab32, oct);
    else
        table_build_kernel<false><<<gb, K1_THREADS, smem, s>>>(sp, scratch, tab64, tab32, oct);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_table_build(swimmer_handle *h, int B, int need64, cudaStream_t s) {
    // node arrays for the handle's octaves (kernel_eval may need the full range)
    // need64: 0 = FP32 table, 1 = FP64 table, 2/3 = FP64 / FP32 table over the full range
    const int oct = need64 >= 2 ? N_OCT_MAX : handle_octaves(h);
    const bool lite = need64 == 0 || need64 == 3;
    for (int b = 0; b < B; b += K1_SLICE) {  // the scratch holds K1_SLICE samples
        int rc = table_kernels(std::min(K1_SLICE, B - b), h->sp + b, h->k1_scratch, h->tab64 + (size_t)b * TAB64_STRIDE,
                               h->tab32 + (size_t)b * TAB32_STRIDE, lite, oct, h->num_sms, s);
        if (rc) return rc;
        prof_count(h, 2);
    }
    return 0;
}

int launch_set_sample(swimmer_handle *h, double alpha, double delta, double r_max, cudaStream_t s) {
    set_sample_kernel<<<1, 1, 0, s>>>(h->sp, alpha, delta, r_max);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_kernel_eval(swimmer_handle *h, int m, const double *r, double *g1, double *g2,
                       int precision, cudaStream_t s) {
    kernel_eval_kernel<<<(m + 127) / 128, 128, 0, s>>>(m, r, g1, g2, h->sp, h->tab64, h->tab32, precision);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

// ---------------------------------------------------------------------------------
// Allocation-free kernel-function evaluation
// ---------------------------------------------------------------------------------
// Some callers may not allocate device memory at all: services that fix their device-memory
// budget at start-up and must not grow it per request.  For them the
// table build of one sample (the kernels above that use scratch memory) runs on scratch
// that lives in file-scope device arrays: every GPU that loads this library holds these
// ~0.25 MB until the process exits, and every call on a device shares them (as handles do the
// ~0.5 MB of universal nodes and quadrature points).
namespace {
__device__ __align__(256) double g_noalloc_scratch[K1_SCRATCH];
__device__ __align__(256) float4 g_noalloc_tab64[TAB64_STRIDE];
__device__ __align__(256) float4 g_noalloc_tab32[TAB32_STRIDE];
__device__ __align__(256) SampleParams g_noalloc_sp[1];

struct NoallocPtrs {
    double *scratch;
    float4 *tab64, *tab32;
    SampleParams *sp;
    bool ready;
};
NoallocPtrs g_noalloc[256];
std::mutex g_noalloc_mutex;

// once per device, with that device current: the device addresses of the arrays (their names
// are host-side stand-ins in host code), constant tables and kernel attributes
int noalloc_setup(int dev, NoallocPtrs *out) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoallocPtrs &p = g_noalloc[dev];
    if (!p.ready) {
        int rc = gl_init();
        if (rc) return rc;
        CUDA_TRY(cudaGetSymbolAddress((void **)&p.scratch, g_noalloc_scratch));
        CUDA_TRY(cudaGetSymbolAddress((void **)&p.tab64, g_noalloc_tab64));
        CUDA_TRY(cudaGetSymbolAddress((void **)&p.tab32, g_noalloc_tab32));
        CUDA_TRY(cudaGetSymbolAddress((void **)&p.sp, g_noalloc_sp));
        // load every kernel of the call now: with lazy module loading a kernel first launched
        // later (kernel_eval_kernel after calls with m = 0) would load its code then
        cudaFuncAttributes fa;
        CUDA_TRY(cudaFuncGetAttributes(&fa, set_sample_kernel));
        CUDA_TRY(cudaFuncGetAttributes(&fa, table_nodes_kernel));
        CUDA_TRY(cudaFuncGetAttributes(&fa, table_build_kernel<false>));
        CUDA_TRY(cudaFuncGetAttributes(&fa, table_build_kernel<true>));
        CUDA_TRY(cudaFuncGetAttributes(&fa, kernel_eval_kernel));
        p.ready = true;
    }
    *out = p;
    return 0;
}
}  // namespace

extern "C" int swimmer_kernel_eval_noalloc(double alpha, double delta, double r_max, int m, const double *r,
                                           double *g1, double *g2, int precision, void *stream) {
    ARG_CHECK(m >= 0, "m must be >= 0");
    ARG_CHECK(m == 0 || (r && g1 && g2), "r, g1, g2 must be device pointers");
    ARG_CHECK(alpha >= 0.0 && delta > 0.0 && r_max > 0.0, "need alpha >= 0, delta > 0, r_max > 0");
    ARG_CHECK(r_max / delta < 4000.0, "r_max/delta = %g beyond the maximum 4000 of the static tables",
              r_max / delta);
    ARG_CHECK(alpha * r_max <= X_MAX, "alpha * r_max beyond %g", X_MAX);
    ARG_CHECK(precision == SWIMMER_FP64 || precision == SWIMMER_FP32C, "precision must be 0 or 1");
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    ARG_CHECK(dev >= 0 && dev < 256, "device ordinal %d out of range", dev);
    NoallocPtrs p;
    int rc = noalloc_setup(dev, &p);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const bool lite = precision != SWIMMER_FP64;  // as FP32 handles build their table
    set_sample_kernel<<<1, 1, 0, s>>>(p.sp, alpha, delta, r_max);
    CUDA_TRY(cudaGetLastError());
    rc = table_kernels(1, p.sp, p.scratch, p.tab64, p.tab32, lite, N_OCT_MAX, N_OCT_MAX, s);
    if (rc) return rc;
    if (m > 0) {
        kernel_eval_kernel<<<(m + 127) / 128, 128, 0, s>>>(m, r, g1, g2, p.sp, p.tab64, p.tab32, precision);
        CUDA_TRY(cudaGetLastError());
    }
    return 0;
}
