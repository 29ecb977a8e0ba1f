// Flow and pressure at target points (Eqs. BrP, BrV with targets x other than the
// swimmer's points): v(x) = (1/mu) sum_j [-F_j g1(r) + (F_j . d) d g2(r)] and
// p(x) = sum_j F_j . grad G_delta = sum_j (F_j . d) G_delta'(r)/r, d = x - X_j, with
// G_delta'(r)/r = (R^2 + R delta + delta^2) / (2 pi R^3 (R + delta)), R = sqrt(r^2 + delta^2)
// (the blob's moment over r^2, finite at r = 0).  FP64.
//
// Bound by the FP64 pipe (16 clocks a warp instruction).  One thread per target; the sample's
// table, the pressure kernel's (delta^2 G_delta'/r is a function of u = 1 + r^2/delta^2 alone, made
// once per device in the same form) and the sources sit in shared memory, so a pair takes 16 FP64
// instructions: separation and u 5, the three kernel functions one each, the sums 8.  With the
// Clenshaw recurrences, square root and division in FP64 and the table read from L1 it took 75
// (512 x 512 targets and 74 points: 2.8 ms a call, of it 2.75 here; now 0.65 ms a call).
// Against extended precision (30 points) the pressure is 3.6e-17 of its terms' sizes off in the mean square and the
// velocity 8.2e-17, where the closed form and the recurrences in FP64 were 4.4e-17 and 15e-17; with the
// pressure's table fitted in FP64 it had been 17e-17.
// CTAs are persistent: one or two per SM load the tables once and walk the targets.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "table_eval.cuh"

int launch_set_sample(swimmer_handle *h, double alpha, double delta, double r_max, cudaStream_t s);
int launch_table_build(swimmer_handle *h, int B, int need64, cudaStream_t s);
void fit_matrix(int n, int deg, long double *node, long double *weight);

namespace {

constexpr int FLOW_THREADS = 256;
constexpr int FLOW_SOURCES = 512;  // sources in shared memory at a time
constexpr int PRES_REC = 4;        // float4 per panel of the pressure kernel's table
constexpr int PRES_PANELS = N_OCT_MAX * F64_FINE;
__device__ float4 g_pressure[PRES_PANELS * PRES_REC];

// delta^2 G_delta'(r)/r as a function of u: with q = u^(-1/2), q^2 (1 + q^2/(1 + q)) / (2 pi); on the
// host, for the table's fit, in extended precision
__device__ __noinline__ double pressure_of_u(double u) {
    const double q = 1.0 / sqrt(u);
    return q * q * (1.0 + q * q / (1.0 + q)) / (2.0 * 3.14159265358979323846);
}
long double pressure_to_fit(long double u) {
    const long double q = 1.0L / sqrtl(u);
    return q * q * (1.0L + q * q / (1.0L + q)) / (2.0L * acosl(-1.0L));
}

__global__ void __launch_bounds__(FLOW_THREADS) flow_kernel(int n, const double *__restrict__ state,
                                                            const float4 *__restrict__ tab64,
                                                            const SampleParams *__restrict__ sp, double mu, int G,
                                                            const double *__restrict__ grid, int oct,
                                                            double *__restrict__ vel, double *__restrict__ pres) {
    extern __shared__ __align__(16) float4 sm[];
    const SampleParams p = sp[0];
    if (p.status != SWIMMER_OK) {
        for (int g = blockIdx.x * FLOW_THREADS + threadIdx.x; g < G; g += gridDim.x * FLOW_THREADS) {
            if (vel) vel[2 * g] = vel[2 * g + 1] = nan("");
            if (pres) pres[g] = nan("");
        }
        return;
    }
    const int panels = min(p.n_oct, oct) * F64_FINE;  // (oct: what the shared memory holds)
    float4 *src = sm, *tab = src + 2 * FLOW_SOURCES, *ptab = tab + panels * F64_REC;
    for (int i = threadIdx.x; i < panels * F64_REC; i += FLOW_THREADS) tab[i] = tab64[i];
    if (pres)
        for (int i = threadIdx.x; i < panels * PRES_REC; i += FLOW_THREADS) ptab[i] = g_pressure[i];
    const double inv_d2 = 1.0 / (p.delta * p.delta), inv_mu = 1.0 / mu;
    // high word of u at the tables' end (an FP64 comparison would cost a pair a sixteenth)
    const unsigned u_end = 0x3ff00000u + ((unsigned)panels << (20 - F64_FINE_LOG2));
    const bool one_load = n <= FLOW_SOURCES;
    // every thread of the CTA takes the same number of turns (the barriers below)
    for (int g0 = blockIdx.x * FLOW_THREADS; g0 < G; g0 += gridDim.x * FLOW_THREADS) {
        const int g = g0 + threadIdx.x;
        const double x = g < G ? grid[2 * (size_t)g] : 0.0, y = g < G ? grid[2 * (size_t)g + 1] : 0.0;
        double ax = 0.0, ay = 0.0, vx = 0.0, vy = 0.0, pr = 0.0;  // sums of F g1, of (F . d) d h, of pressure
        for (int j0 = 0; j0 < n; j0 += FLOW_SOURCES) {
            const int m = min(FLOW_SOURCES, n - j0);
            if (!one_load || g0 == blockIdx.x * FLOW_THREADS) {
                __syncthreads();  // the previous sources are read
                double *d = (double *)src;
                for (int i = threadIdx.x; i < 4 * m; i += FLOW_THREADS) d[i] = state[4 * (size_t)j0 + i];
                __syncthreads();
            }
            if (g >= G) continue;
            for (int j = 0; j < m; ++j) {
                const double2 X = *(const double2 *)(src + 2 * j), F = *(const double2 *)(src + 2 * j + 1);
                const double dx = x - X.x, dy = y - X.y;
                const double u = fma(fma(dx, dx, dy * dy), inv_d2, 1.0);
                float th, tl;
                const int pan = panel_f64(u, panels - 1, th, tl);
                const double fd = fma(F.x, dx, F.y * dy);
                if (vel) {
                    const float4 *rec = tab + F64_REC * pan;
                    const double2 c0 = *(const double2 *)rec;
                    float2 qh, ql;
                    poly_f64(rec, th, tl, qh, ql);
                    const double g1 = c0.x + join(qh.x, ql.x), w = fd * (c0.y + join(qh.y, ql.y));
                    ax = fma(F.x, g1, ax);
                    ay = fma(F.y, g1, ay);
                    vx = fma(w, dx, vx);
                    vy = fma(w, dy, vy);
                }
                // (the pressure holds at any distance: beyond the octaves of r_max by its closed form)
                if (pres)
                    pr = fma(fd, (unsigned)__double2hiint(u) < u_end ? poly1_f64(ptab + PRES_REC * pan, th, tl)
                                                                     : pressure_of_u(u), pr);
            }
        }
        if (g < G) {
            if (vel) {
                vel[2 * (size_t)g] = fma(vx, inv_d2, -ax) * inv_mu;
                vel[2 * (size_t)g + 1] = fma(vy, inv_d2, -ay) * inv_mu;
            }
            if (pres) pres[g] = pr * inv_d2;
        }
    }
}

}  // namespace

// the pressure kernel's table, once per device
int pressure_init() {
    static bool done[256] = {};
    static std::mutex mutex;
    std::lock_guard<std::mutex> lock(mutex);
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    ARG_CHECK(dev >= 0 && dev < 256, "device ordinal %d out of range", dev);
    if (done[dev]) return 0;
    std::vector<float4> all(PRES_PANELS * PRES_REC);
    constexpr int NODES = 10, COEFS = 8;
    long double node[NODES], weight[COEFS][NODES];
    fit_matrix(NODES, COEFS - 1, node, weight[0]);
    for (int q = 0; q < PRES_PANELS; ++q) {
        const double oct = ldexp(1.0, q / F64_FINE), w = oct / F64_FINE, lo = oct + (q % F64_FINE) * w;
        long double c[COEFS] = {};
        for (int i = 0; i < NODES; ++i) {
            const long double v = pressure_to_fit(lo + 0.5L * w * (node[i] + 1.0L));
            for (int k = 0; k < COEFS; ++k) c[k] += weight[k][i] * v;
        }
        float h[6], l[6];
        for (int k = 1; k <= 5; ++k) {
            h[k] = (float)c[k];
            l[k] = (float)(c[k] - (long double)h[k]);
        }
        float4 *rec = &all[q * PRES_REC];
        const double c0 = (double)c[0];
        memcpy(rec, &c0, sizeof(double));
        rec[0].z = h[1];
        rec[0].w = l[1];
        rec[1] = make_float4(h[5], l[5], h[4], l[4]);
        rec[2] = make_float4(h[3], l[3], h[2], l[2]);
        rec[3] = make_float4((float)c[6], (float)c[7], 0.f, 0.f);
    }
    CUDA_TRY(cudaMemcpyToSymbol(g_pressure, all.data(), sizeof(float4) * all.size()));
    CUDA_TRY(cudaFuncSetAttribute(flow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(sizeof(float4) * (2 * FLOW_SOURCES + PRES_PANELS * (F64_REC + PRES_REC)))));
    done[dev] = true;
    return 0;
}

extern "C" int swimmer_flow_field(swimmer_handle *h, double alpha, double delta, double r_max, int n,
                                  const double *state, int G, const double *grid, double *vel, double *pres,
                                  void *stream) {
    ARG_CHECK(h != nullptr, "handle is NULL");
    ARG_CHECK(alpha >= 0.0 && delta > 0.0 && r_max > 0.0, "need alpha >= 0, delta > 0, r_max > 0");
    ARG_CHECK(n >= 1 && G >= 0, "need n >= 1 points and G >= 0 targets");
    ARG_CHECK(state != nullptr && (G == 0 || grid != nullptr), "NULL device pointer");
    ARG_CHECK(vel != nullptr || pres != nullptr, "no output requested");
    if (G == 0) return 0;
    cudaStream_t s = (cudaStream_t)stream;
    int rc = launch_set_sample(h, alpha, delta, r_max, s);
    if (!rc) rc = launch_table_build(h, 1, 2, s);  // full-range FP64 table in sample slot 0
    if (rc) return rc;
    // the table covers the octaves of r_max (as launch_set_sample counts them)
    const double rho = r_max / delta;
    const int oct = std::max(1, std::min(N_OCT_MAX, (int)std::min(64.0, floor(log2(1.0 + rho * rho)) + 1.0)));
    const size_t smem = sizeof(float4) * (2 * FLOW_SOURCES + (size_t)oct * F64_FINE * (F64_REC + PRES_REC));
    const int ctas = (G + FLOW_THREADS - 1) / FLOW_THREADS, per_sm = smem + 1024 <= (size_t)h->max_smem / 2 ? 2 : 1;
    flow_kernel<<<std::min(ctas, per_sm * h->num_sms), FLOW_THREADS, smem, s>>>(n, state, h->tab64, h->sp, h->cfg.mu, G,
                                                                               grid, oct, vel, pres);
    CUDA_TRY(cudaGetLastError());
    prof_count(h, 1);
    return 0;
}
