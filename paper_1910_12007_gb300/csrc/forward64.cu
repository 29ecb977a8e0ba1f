// K2 in FP64: fused forward model + log-likelihood, one run per CTA or, when the batch leaves SMs
// idle, per cluster of CTAs (the model, the phases and the outputs are those of forward.cu).
//
// Bound by the FP64 pipe: GB300 issues a warp's FP64 instruction every 16 clocks of an SM, 64 times
// slower than FP32.  So
//   - the pair sum reads positions in units of delta (u = 1 + |e|^2 takes two FMAs), and the kernel functions
//     come from table_eval.cuh with one FP64 addition each: 13 FP64 instructions per ordered pair
//     (separation 2, u 2, kernel functions 2, F . e and its product 3, the sums 4) where two
//     Clenshaw recurrences took 54;
//   - the threads that share a target leave their partial sums in shared memory and one thread adds
//     them and updates the point: as warp shuffles, additions and the update cost their 16 clocks in
//     every warp, for two or four useful lanes each;
//   - a run's positions themselves are in the caller's units, and what rounding takes from one goes into
//     its next displacement.  In units of delta their last place was up to 1.5 times coarser and the errors
//     of all steps added up: against extended precision (400 steps, N = 64) positions were 1.4e-16 to
//     2.9e-16 off in the mean square, now below 0.72e-16, and the forces at the end 1.7 to 6 times as far as
//     now.  It costs a lone run 1 % of its time (N = 64, 2000 steps 13.9 -> 14.05 ms), a batch 0.3 %;
//   - (cos, sin)(omega t) is made for 32 steps at a time, a lane each, and the preferred curvature
//     is P_k cos + Q_k sin; springs and curvature take one reciprocal square root each.
// Of a run that has a CTA to itself every unordered pair is evaluated once, in the blocks and units of
// forward.cu (19 FP64 instructions: the symmetric mobility 5, two sums 4 each): 1024 runs of N = 128 85.6 ->
// 65.5 ms.
// Where the padding to blocks would cost more than that saves, where the warps' arrays do not fit
// and in a cluster, target i meets source i + d mod n at step d (the lanes of a warp share d: on a
// smooth filament they read the same table panel).  A lone run is spread over a cluster of up to 16 SMs: a CTA owns
// n / C points; forces and new positions go to every CTA's shared memory (double-buffered
// positions, two cluster barriers a step).
// Measured (whole calls): a lone run of N = 64, 2000 steps 53.1 -> 14.05 ms (26.5 -> 7.0 us a step) on a
// cluster of 16; 1024 runs of N = 128, 200 steps 109 -> 65 ms (99 as a kernel of its own, 86 with 13
// FP64 instructions a pair, 65 with the symmetric sum); 152 pairs of sperm models (148 points), 400
// steps 44 -> 31.6 ms.
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "forward_args.cuh"
#include "table_eval.cuh"

namespace {

constexpr double PI = 3.14159265358979323846;
constexpr int MAX_CLUSTER = 16;
constexpr int CLUSTER_THREADS = 256;  // threads of a CTA of a cluster (more when it owns more points)
constexpr int CLUSTER_POINTS = 4;     // points of a CTA of a cluster at least

// a Hookean spring E = K (l/l0 - 1)^2 l0: 1/l0^2, and 2 K / l0
struct Rest {
    double inv_l02, k2;
};

// t with force on i = t (X_j - X_i), and the strain l/l0 - 1 from l^2/l0^2 - 1, without cancellation
__device__ __forceinline__ double spring(double2 xi, double2 xj, const Rest &r, double &ex, double &ey, double &strain) {
    ex = xj.x - xi.x;
    ey = xj.y - xi.y;
    const double s2 = fma(fma(ex, ex, ey * ey), r.inv_l02, -1.0), one = 1.0 + s2;
    const double rs = rsqrt(one);  // l0/l
    strain = s2 / fma(one, rs, 1.0);
    return r.k2 * strain * rs;
}

// a value at the same place of every CTA of the cluster (its own among them: no branch in the loop).  One
// thread sends them, a step's barrier waits for it: a lone run of N = 64 takes 14.20 ms with the loop unrolled by
// 2, 14.05 by 4, 13.90 by 8, and 30 runs of N = 100 on clusters of 4 4.89, 4.89 and 4.93
__device__ __forceinline__ void put_all(double2 *p, double2 v, int C) {
    if (C == 1) {
        *p = v;
        return;
    }
    const unsigned at = smem_addr(p);
#pragma unroll 4
    for (int r = 0; r < C; ++r)
        asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(remote(at, r)), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void put_all(double2 *p, double2 v, double2 *q, double2 w, int C) {
    if (C == 1) {
        *p = v;
        *q = w;
        return;
    }
    const unsigned at = smem_addr(p), off = smem_addr(q) - at;
#pragma unroll 4
    for (int r = 0; r < C; ++r) {
        const unsigned to = remote(at, r);
        asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(to), "d"(v.x), "d"(v.y) : "memory");
        asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(to + off), "d"(w.x), "d"(w.y) : "memory");
    }
}
__device__ __forceinline__ void put_all(int *p, int v, int C) {
    if (C == 1) {
        *p = v;
        return;
    }
    for (int r = 0; r < C; ++r)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote(smem_addr(p), r)), "r"(v) : "memory");
}

// shared memory before the table (the pair sum's partial velocities lie over the stencils' terms, which the
// force phase has read by then)
__host__ __device__ inline size_t state_bytes(int n_max, int threads, int pair_warps) {
    const size_t np = (n_max + 31) & ~31;
    size_t part = pair_warps * np;
    if (part < (size_t)threads) part = threads;
    if (part < 3 * np) part = 3 * np;
    const size_t b = sizeof(double2) * (5 * np + part);
    return (b + 127) & ~size_t(127);
}

// mean of the points from k0 on as seen from ref (one warp, fixed order); all lanes get it
__device__ __forceinline__ double2 centre(const double2 *P, double2 ref, int k0, int count, int lane) {
    double x = 0.0, y = 0.0;
    for (int m = lane; m < count; m += 32) {
        x += P[k0 + m].x - ref.x;
        y += P[k0 + m].y - ref.y;
    }
    for (int o = 16; o >= 1; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    return make_double2(x / count, y / count);
}

// One unit of the symmetric pair sum (a warp, 16 steps): lane l holds target I*32 + l and at step d =
// d0 .. d0 + 15 meets source J*32 + (l + d) mod 32; the pair's term is the symmetric mobility M = h e e^T
// - g1 I applied to both forces, and the source's sum moves down one lane per step with its source.
// A diagonal block (I = J) runs d = 1 .. 16, at 16 with half the lanes (the units of forward.cu).
template <bool DIAG>
__device__ __forceinline__ void pair_unit64(const double2 *__restrict__ X, const double2 *__restrict__ frc,
                                            const float4 *__restrict__ tab, int pmax, int lane, int I, int Jb, int d0,
                                            double2 *__restrict__ mypart) {
    const double2 xi = X[32 * I + lane], fi = frc[32 * I + lane];
    double vx = 0.0, vy = 0.0, ax = 0.0, ay = 0.0;
#pragma unroll 2
    for (int s = 0; s < 16; ++s) {
        const int j = 32 * Jb + ((lane + d0 + s) & 31);
        const double2 xj = X[j], f = frc[j];
        const double ex = xi.x - xj.x, ey = xi.y - xj.y;
        double g1, h;
        kern_f64(tab, pmax, fma(ex, ex, fma(ey, ey, 1.0)), g1, h);
        if (DIAG && s == 15 && lane >= 16) g1 = h = 0.0;
        const double hx = h * ex, hy = h * ey;
        const double m11 = fma(hx, ex, -g1), m12 = hx * ey, m22 = fma(hy, ey, -g1);
        vx = fma(m11, f.x, fma(m12, f.y, vx));
        vy = fma(m12, f.x, fma(m22, f.y, vy));
        ax = fma(m11, fi.x, fma(m12, fi.y, ax));
        ay = fma(m12, fi.x, fma(m22, fi.y, ay));
        ax = __shfl_sync(0xffffffffu, ax, (lane + 1) & 31);
        ay = __shfl_sync(0xffffffffu, ay, (lane + 1) & 31);
    }
    // lane l holds the sum of source (l + d0 + 16) mod 32: to its own lane
    const int from = (lane - d0 - 16) & 31;
    ax = __shfl_sync(0xffffffffu, ax, from);
    ay = __shfl_sync(0xffffffffu, ay, from);
    double2 pv = mypart[32 * I + lane];
    pv.x += vx;
    pv.y += vy;
    if (DIAG) {
        pv.x += ax;
        pv.y += ay;
    }
    mypart[32 * I + lane] = pv;
    if (!DIAG) {
        double2 pa = mypart[32 * Jb + lane];
        pa.x += ax;
        pa.y += ay;
        mypart[32 * Jb + lane] = pa;
    }
}

// whether a run of n points is worth the symmetric sum: 19 FP64 instructions per unordered pair of
// the points padded to blocks of 32, against 26 of the points
__host__ __device__ inline bool symmetric_pays(int n) {
    const int np = (n + 31) & ~31;
    return 19 * np * np < 26 * n * n;
}

// MODEL 0: the flagellum; 1: the full sperm model (head points and neck); 2: two sperm models
// coupled by the fluid.  MAXT 1024, for runs above 512 points, is held to 64 registers and spills (360 to 560
// bytes of loads a thread): 100 runs take, us a step, N = 600 2000, N = 768 3120, N = 1024 7400, a fifth to a
// quarter of what the Clenshaw kernel took (10500, 16700, 29100).  C CTAs (a cluster when C > 1) share a run.
template <int MODEL, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) forward64_kernel(FwdArgs a, int C, int pw) {
    constexpr bool HEAD = MODEL >= 1, TWO = MODEL == 2;
    extern __shared__ __align__(128) unsigned char smraw[];
    const int n_max = a.n_max, T = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    const int np = (n_max + 31) & ~31;     // points in blocks of 32
    double2 *P = (double2 *)smraw;         // [np] positions relative to (L/2, 0)
    double2 *pos = P + np;                 // [2][np] the same in units of delta, for the pair sum
    double2 *frc = pos + 2 * np;           // [np] point forces
    double2 *pq = frc + np;                // [np] preferred-curvature coefficients
    double2 *tv = pq + np;                 // [np] tension of segment (k, next)
    double2 *b0 = tv + np, *b4 = b0 + np;  // [np] bending of centre k on its neighbours
    double2 *part = tv;                    // partial velocities: [T], or [pw][np] of the symmetric sum's warps
    const float4 *tab = (const float4 *)(smraw + state_bytes(n_max, T, pw));
    __shared__ int s_work, s_bad[2];
    __shared__ Rest s_rest[6];  // flagellum segment, head membrane, diametral, neck A, neck B, neck gap
    // stencils of the flagellum [0] and the head [1]: 1/(2 h), 1/h^2, 2 K h; then 1/H_r and 2 K_NA
    __shared__ double s_st[2][3], s_ihr, s_kang;
    // at the previous observation: the first head point and the head's centre as seen from there (a velocity
    // is the difference of the large parts, which is exact, and of the small ones)
    __shared__ double2 s_first, s_centre;
    __shared__ double2 s_rot[32];  // (cos, sin)(omega t) of 32 steps
    unsigned rank_ = 0;
    if (C > 1) asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_));
    const int rank = (int)rank_;
    // every CTA of the cluster has started: only then may the others write to its shared memory
    if (C > 1) run_sync(C);

    for (;;) {
        if (rank == 0 && tid == 0) put_all(&s_work, atomicAdd(a.queue, 1), C);
        run_sync(C);
        const int w = s_work;
        if (w >= a.B) break;
        const int b = a.order[w];
        const SampleParams p = a.sp[b];
        const int nf = p.n, nh = HEAD ? p.nh : 0, h2 = nh >> 1;
        const int nsw = nf + nh;            // points per swimmer: flagellum, then head
        const int n = TWO ? 2 * nsw : nsw;  // all points of the sample
        const long long n_obs = a.steps / a.obs_every;
        if (p.status != SWIMMER_OK) {
            if (rank == 0) {
                if (tid == 0) {
                    a.status[b] = p.status;
                    if (a.loglik) a.loglik[b] = -INFINITY;
                    if (a.speed) a.speed[b] = nan("");
                    if (a.speculative) a.run_work[b] = 0;
                }
                if (a.head_traj)
                    for (long long o = tid; o < 2 * n_obs; o += T) a.head_traj[(size_t)b * 2 * n_obs + o] = nan("");
                if (a.final_state)
                    for (int k = tid; k < 4 * n_max; k += T) a.final_state[(size_t)b * n_max * 4 + k] = nan("");
            }
            run_sync(C);
            continue;
        }
        // ---- set-up: the table, the straight filament (and head circle), constants
        const int npan = min(a.tab_panels, p.n_oct * F64_FINE);
        {
            const float4 *g = a.tab64 + (size_t)b * TAB64_STRIDE;
            for (int i = tid; i < npan * F64_REC; i += T) ((float4 *)tab)[i] = g[i];
        }
        const double ds = p.ds, L = p.length, delta = p.delta, inv_d = 1.0 / p.delta;
        const double xref = 0.5 * L;
        const double hr = a.hr_over_ds * ds, gap = a.gap_over_ds * ds;
        const double dth = nh ? 2.0 * PI / nh : 0.0, dsh = hr * dth;
        for (int k = tid; k < n; k += T) {
            const int sw = TWO && k >= nsw;  // second swimmer: displaced by d along y
            const int kl = k - sw * nsw;
            double x0, y0 = 0.0;
            if (kl < nf) {
                x0 = kl * ds - xref;
            } else {
                double sn, cs;
                sincos((kl - nf) * dth, &sn, &cs);
                x0 = L + gap + hr + hr * cs - xref;
                y0 = hr * sn;
            }
            if (sw) y0 += a.swim_d;
            P[k] = make_double2(x0, y0);
            pos[k] = make_double2(x0 * inv_d, y0 * inv_d);
            if (kl < nf) {
                // the preferred curvature (Appendix: y^ = a (1 - s/L) sin(eta s - omega t),
                // zeta^ = d^2 y^/ds^2) as P_k cos(omega t) + Q_k sin(omega t)
                const double sk = kl * ds;
                double sn, cs;
                sincos(a.eta * sk, &sn, &cs);
                const double c1 = 2.0 * a.eta / L, c2 = (1.0 - sk / L) * a.eta * a.eta;
                pq[k] = make_double2(-p.amp * (c1 * cs + c2 * sn), -p.amp * (c1 * sn - c2 * cs));
            }
        }
        // force-free sources ds apart beyond the last point fill the last block (symmetric sum)
        const int nbk = (n + 31) >> 5;
        for (int k = n + tid; k < 32 * nbk; k += T) {
            const double end = nh ? L + gap + 2.0 * hr : L;
            pos[k] = pos[np + k] = make_double2((end - xref + (k - n + 1) * ds) * inv_d, TWO ? a.swim_d * inv_d : 0.0);
            frc[k] = make_double2(0.0, 0.0);
        }
        const bool sym = pw > 0 && symmetric_pays(n);
        const unsigned *units = a.units + UNIT_HDR + a.units[nbk - 1];  // the one-target list of nbk blocks
        if (tid == 0) {
            const double c1 = hr * (1.0 - cos(dth)), s1 = hr * sin(dth);
            const double l0[6] = {ds, 2.0 * hr * sin(0.5 * dth), 2.0 * hr, hypot(gap + c1, s1), hypot(ds + gap + c1, s1),
                                  gap};
            const double kk[6] = {a.kt, a.k_head_tens, a.k_head_tens, a.k_neck_tens, a.k_neck_tens, a.k_neck_tens};
            for (int q = 0; q < 6; ++q) {
                const double lq = l0[q] > 0.0 ? l0[q] : 1.0;  // unused without a head
                s_rest[q].inv_l02 = 1.0 / (lq * lq);
                s_rest[q].k2 = 2.0 * kk[q] / lq;
            }
            for (int q = 0; q < (nh ? 2 : 1); ++q) {
                const double h = q ? dsh : ds;
                s_st[q][0] = 0.5 / h;
                s_st[q][1] = 1.0 / (h * h);
                s_st[q][2] = 2.0 * (q ? a.k_head_c : p.kc) * h;
            }
            s_ihr = nh ? 1.0 / hr : 0.0;
            s_kang = 2.0 * a.k_neck_ang;
            s_bad[0] = s_bad[1] = 0;
        }
        // the CTA's own points, and the threads of the pair sum: thread -> (own point, split)
        const int k_lo = (int)((long long)n * rank / C), m = (int)((long long)n * (rank + 1) / C) - k_lo;
        // (m <= T by the launch's choice; a short sample can leave a CTA of a cluster no point)
        const int S = m > 0 ? T / m : 0, pt = m > 0 ? tid % m : 0, split = m > 0 ? tid / m : 0;
        // lanes that add a point's partial sums: eight for a few points, else one
        const int G = m < 32 && 8 * m <= T ? 8 : 1;
        const int my = G == 8 ? tid >> 3 : tid;  // own point that this thread updates (if < m)
        const double dt_mu = a.dt / a.mu;
        const double self_g1 = [&] {
            __syncthreads();
            double g1, h;
            kern_f64(tab, npan - 1, 1.0, g1, h);
            return g1;
        }();
        // the thread that keeps the log-likelihood: thread 0 of the first CTA for observations that
        // a warp makes, else the one that updates the proximal flagellum point nf - 1
        const bool vobs = vel_obs(a, nh);
        const bool head_thread = vobs ? rank == 0 && tid == 0
                                      : my == nf - 1 - k_lo && my < m && (G == 1 || (tid & 7) == 0);
        double2 rest = make_double2(0.0, 0.0);  // what rounding took from the position that this thread updates
        double J = 0.0;
        int status = SWIMMER_OK;
        long long steps_done = a.steps;
        if (vobs && rank == 0 && tid < 32) {  // head centre at the previous observation
            const double2 c = centre(P, P[nf], nf, nh, lane);
            if (tid == 0) {
                s_first = P[nf];
                s_centre = c;
            }
        }
        run_sync(C);

        // with a final state requested, one more pass of the force phases at t = steps dt
        const long long last = a.steps + (a.final_state ? 1 : 0);
        const int obs_every = (int)min(a.obs_every, (long long)INT_MAX);  // > steps: no observation
        int obs_left = obs_every, obs_idx = 0;
        for (int step = 0; step < (int)last; ++step) {
            const double2 *X = pos + (step & 1) * np;
            const bool obs_step = --obs_left == 0;
            int bad = 0;
            if ((step & 31) == 0) {  // (the last reads of s_rot lie before a barrier)
                if (tid >= T - 32) {
                    double sn, cs;
                    sincos(a.omega * ((double)(step + lane) * a.dt), &sn, &cs);
                    s_rot[lane] = make_double2(cs, sn);
                }
                __syncthreads();
            }
            // ---- A+B: tension and curvature stencils of the own points and of the neighbours whose
            //      stencils act on them: the points before the first and after the last, and a head
            //      ring's other end
            for (int q = tid; q < m + 2 + (HEAD ? 4 : 0); q += T) {
                int k = k_lo + q;
                if (q >= m) {
                    const int e = q - m;
                    if (e < 2) {
                        k = e == 0 ? k_lo - 1 : k_lo + m;
                    } else {  // ring of swimmer (e - 2) / 2: its last point when its first is own, and the reverse
                        const int first = ((e - 2) >> 1) * nsw + nf, end = first + nh - 1;
                        if (first >= n) continue;
                        const int own = (e & 1) ? end : first;
                        if (own < k_lo || own >= k_lo + m) continue;
                        k = (e & 1) ? first : end;
                    }
                    if (k < 0 || k >= n || (k >= k_lo && k < k_lo + m)) continue;
                }
                const int base = (TWO && k >= nsw) ? nsw : 0;  // the point's swimmer
                const int kl = k - base;
                const bool hd = HEAD && kl >= nf;
                const int mh = kl - nf;
                const int next = hd ? base + nf + (mh + 1 == nh ? 0 : mh + 1) : (kl + 1 < nf ? k + 1 : -1);
                const int prev = hd ? base + nf + (mh == 0 ? nh - 1 : mh - 1) : k - 1;
                const bool center = hd || (kl >= 1 && kl + 1 < nf);
                const double2 xk = P[k];
                double epx = 0.0, epy = 0.0;
                if (next >= 0) {
                    double strain;
                    const double t = spring(xk, P[next], s_rest[hd ? 1 : 0], epx, epy, strain);
                    if (!(fabs(strain) <= STRETCH_MAX)) bad = 1;
                    tv[k] = make_double2(t * epx, t * epy);
                }
                if (center) {
                    const double *st = s_st[hd ? 1 : 0];
                    const double emx = xk.x - P[prev].x, emy = xk.y - P[prev].y;
                    const double A = (emx + epx) * st[0], Bv = (emy + epy) * st[0];
                    const double Cc = (epx - emx) * st[1], D = (epy - emy) * st[1];
                    const double rs = rsqrt(fma(A, A, Bv * Bv)), r2 = rs * rs, S15 = r2 * rs;
                    const double cross = fma(A, D, -Bv * Cc), zeta = cross * S15;
                    double zhat = s_ihr;  // preferred head curvature 1/H_r
                    if (!hd) {
                        const double2 c = pq[k], rot = s_rot[step & 31];
                        zhat = fma(c.x, rot.x, c.y * rot.y);
                    }
                    const double ck = st[2] * (zeta - zhat), p1 = ck * st[0], p2 = ck * st[1] * S15;
                    const double s25 = 3.0 * zeta * r2;
                    const double Px = fma(D, S15, -A * s25) * p1, Py = -fma(Cc, S15, Bv * s25) * p1;
                    const double Qx = -Bv * p2, Qy = A * p2;
                    b0[k] = make_double2(Qx - Px, Qy - Py);
                    b4[k] = make_double2(Qx + Px, Qy + Py);
                }
            }
            __syncthreads();
            // ---- C: point forces, gathered per point (no atomics): segment tensions, the bending
            //      stencils of the centres k-1, k, k+1, and for the head model the diametral and neck
            //      springs and the neck angle (Appendix)
            for (int q = tid; q < m; q += T) {
                const int k = k_lo + q;
                const int base = (TWO && k >= nsw) ? nsw : 0;
                const int kl = k - base;
                const bool hd = HEAD && kl >= nf;
                const int mh = kl - nf;
                const int next = hd ? base + nf + (mh + 1 == nh ? 0 : mh + 1) : (kl + 1 < nf ? k + 1 : -1);
                const int prev = hd ? base + nf + (mh == 0 ? nh - 1 : mh - 1) : (kl >= 1 ? k - 1 : -1);
                double fx = 0.0, fy = 0.0;
                if (next >= 0) {
                    fx += tv[k].x;
                    fy += tv[k].y;
                }
                if (prev >= 0) {
                    fx -= tv[prev].x;
                    fy -= tv[prev].y;
                }
                if (hd || kl >= 2) {  // centre prev acts on k as its next neighbour
                    fx -= b4[prev].x;
                    fy -= b4[prev].y;
                }
                if (hd || (kl >= 1 && kl + 1 < nf)) {
                    fx += b0[k].x + b4[k].x;
                    fy += b0[k].y + b4[k].y;
                }
                if (hd || kl + 2 < nf) {  // centre next acts on k as its previous neighbour
                    fx -= b0[next].x;
                    fy -= b0[next].y;
                }
                if (HEAD && nh > 0) {
                    // springs (k, j): force on k = t e, e = X_j - X_k; up to three per point
                    for (int g = 0; g < 3; ++g) {
                        int j = -1, kind = 0;  // kind: 0 diametral, 1 neck A, 2 neck B, 3 neck gap
                        if (hd) {
                            if (g == 0) {
                                j = nf + (mh + h2 >= nh ? mh + h2 - nh : mh + h2);
                            } else if (mh == h2 - 1 || mh == h2 + 1) {
                                j = g == 1 ? nf - 1 : nf - 2;
                                kind = g;
                            } else if (mh == h2 && g == 1) {
                                j = nf - 1;
                                kind = 3;
                            }
                        } else if (kl == nf - 1) {
                            j = nf + h2 - 1 + g;
                            kind = g == 1 ? 3 : 1;
                        } else if (kl == nf - 2 && g < 2) {
                            j = nf + h2 - 1 + 2 * g;
                            kind = 2;
                        }
                        if (j < 0) continue;
                        double ex, ey, strain;
                        const double t = spring(P[k], P[j + base], s_rest[2 + kind], ex, ey, strain);
                        fx += t * ex;
                        fy += t * ey;
                        if (!(fabs(strain) <= STRETCH_MAX)) bad = 1;
                    }
                    // neck angle E = K (z1 . z2)^2, z1 = H(pi) - X_{nf-1}, z2 = H(pi+dth) - H(pi-dth)
                    const int ihp = base + nf + h2, iplus = ihp + 1, iminus = ihp - 1, iend = base + nf - 1;
                    if (k == ihp || k == iplus || k == iminus || k == iend) {
                        const double z1x = P[ihp].x - P[iend].x, z1y = P[ihp].y - P[iend].y;
                        const double z2x = P[iplus].x - P[iminus].x, z2y = P[iplus].y - P[iminus].y;
                        const double ww = s_kang * (z1x * z2x + z1y * z2y);
                        if (k == ihp) {
                            fx -= ww * z2x;
                            fy -= ww * z2y;
                        } else if (k == iend) {
                            fx += ww * z2x;
                            fy += ww * z2y;
                        } else if (k == iplus) {
                            fx -= ww * z1x;
                            fy -= ww * z1y;
                        } else {
                            fx += ww * z1x;
                            fy += ww * z1y;
                        }
                    }
                }
                put_all(frc + k, make_double2(fx, fy), C);
            }
            run_sync(C);
            if (step == a.steps) {  // final state: positions and the forces there
                for (int q = tid; q < m; q += T) {
                    const int k = k_lo + q;
                    double *o = a.final_state + ((size_t)b * n_max + k) * 4;
                    o[0] = P[k].x + xref;
                    o[1] = P[k].y;
                    o[2] = frc[k].x;
                    o[3] = frc[k].y;
                }
                break;
            }
            // ---- D: pair sum of the own points, e = d / delta, h = delta^2 g2:
            //      v_i = (1/mu) sum_j [-F_j g1 + (F_j . e) e h]
            double vx = 0.0, vy = 0.0;
            if (sym) {
                // every unordered pair once; warp w takes units w, w + pw, ... and adds them into its
                // own array, the arrays are added in order
                const int warp = tid >> 5;
                if (warp < pw) {
                    double2 *mypart = part + warp * np;
                    for (int k = lane; k < 32 * nbk; k += 32) mypart[k] = make_double2(0.0, 0.0);
                    for (int un = warp; un < nbk * nbk; un += pw) {
                        const unsigned pk = units[un];
                        const int I = pk & 31, Jb = (pk >> 5) & 31, code = (pk >> 25) & 3;
                        if (I == Jb)
                            pair_unit64<true>(X, frc, tab, npan - 1, lane, I, Jb, 1, mypart);
                        else
                            pair_unit64<false>(X, frc, tab, npan - 1, lane, I, Jb, code << 4, mypart);
                    }
                }
                __syncthreads();
                if (my < m && (G == 1 || (tid & 7) == 0)) {
                    const double2 f = frc[my];
                    vx = -f.x * self_g1;
                    vy = -f.y * self_g1;
                    for (int w = 0; w < pw; ++w) {
                        const double2 v = part[w * np + my];
                        vx += v.x;
                        vy += v.y;
                    }
                }
            } else if (split < S) {
                const int i = k_lo + pt;
                const double2 xi = X[i];
                if (split == 0) {
                    const double2 f = frc[i];
                    vx = -f.x * self_g1;
                    vy = -f.y * self_g1;
                }
                // offsets 1 .. n - 1, split over the S threads of the point
                int j = i + 1 + split;
                if (j >= n) j -= n;
                for (int d = 1 + split; d < n; d += S) {
                    const double2 xj = X[j], f = frc[j];
                    j += S;
                    if (j >= n) j -= n;
                    const double ex = xi.x - xj.x, ey = xi.y - xj.y;
                    const double u = fma(ex, ex, fma(ey, ey, 1.0));
                    double g1, h;
                    kern_f64(tab, npan - 1, u, g1, h);
                    const double wv = fma(f.x, ex, f.y * ey) * h;
                    vx = fma(wv, ex, fma(-f.x, g1, vx));
                    vy = fma(wv, ey, fma(-f.y, g1, vy));
                }
            }
            if (!sym && S > 1) {
                if (split < S) part[split * m + pt] = make_double2(vx, vy);
                __syncthreads();
                vx = vy = 0.0;
                if (G == 1) {
                    if (tid < m)
                        for (int s = 0; s < S; ++s) {
                            const double2 v = part[s * m + tid];
                            vx += v.x;
                            vy += v.y;
                        }
                } else if (tid < ((8 * m + 31) & ~31)) {
                    if (my < m)
                        for (int s = tid & 7; s < S; s += 8) {
                            const double2 v = part[s * m + my];
                            vx += v.x;
                            vy += v.y;
                        }
                    for (int o = 4; o >= 1; o >>= 1) {
                        vx += __shfl_xor_sync(0xffffffffu, vx, o);
                        vy += __shfl_xor_sync(0xffffffffu, vy, o);
                    }
                }
            }
            // ---- E: Euler step into the other position buffer, divergence, observations
            if (my < m && (G == 1 || (tid & 7) == 0)) {
                const int k = k_lo + my;
                // the displacement with what the last sum left over
                const double2 was = P[k];
                const double2 moved = make_double2(fma(vx, dt_mu, rest.x), fma(vy, dt_mu, rest.y));
                if (!isfinite(moved.x) || !isfinite(moved.y) || fmax(fabs(moved.x), fabs(moved.y)) > ds) bad = 1;
                const double2 xn = make_double2(was.x + moved.x, was.y + moved.y);
                put_all(pos + ((step + 1) & 1) * np + k, make_double2(xn.x * inv_d, xn.y * inv_d), P + k, xn, C);
                rest = make_double2(moved.x - (xn.x - was.x), moved.y - (xn.y - was.y));
                // the head point's observation: squared residual into J, trajectory row
                if (obs_step && !vobs && k == nf - 1) {
                    const double hxo = xn.x + xref, hyo = xn.y;
                    const long long o = obs_idx;
                    if (a.obs) {
                        const double rx = a.obs[2 * o] - hxo, ry = (a.obs[2 * o + 1] - hyo) / a.sigma_ratio;
                        J = fma(rx, rx, fma(ry, ry, J));
                    }
                    if (a.head_traj) {
                        a.head_traj[((size_t)b * n_obs + o) * 2] = hxo;
                        a.head_traj[((size_t)b * n_obs + o) * 2 + 1] = hyo;
                    }
                }
            }
            // (two flags in turn: a CTA ahead in the next step must not be read here)
            if (bad) put_all(&s_bad[step & 1], 1, C);
            run_sync(C);
            if (s_bad[step & 1]) {
                status = SWIMMER_DIVERGED;
                steps_done = step + 1;
                break;
            }
            if (vobs && obs_step && rank == 0 && tid < 32) {
                double ox, oy;
                if (TWO && a.obs_kind == SWIMMER_OBS_PAIR_DISTANCES) {
                    // distances between the tail tips and between the head centres (Sec. 4.2)
                    const double2 f0 = P[nf], f1 = P[nsw + nf];
                    const double2 c0 = centre(P, f0, nf, nh, lane), c1 = centre(P, f1, nsw + nf, nh, lane);
                    const double cx = (f1.x - f0.x) + (c1.x - c0.x), cy = (f1.y - f0.y) + (c1.y - c0.y);
                    const double tx = P[nsw].x - P[0].x, ty = P[nsw].y - P[0].y;
                    ox = sqrt(tx * tx + ty * ty);
                    oy = sqrt(cx * cx + cy * cy);
                } else {
                    // head-centre velocity over the observation interval (Sec. 4.1)
                    const double2 f = P[nf], c = centre(P, f, nf, nh, lane);
                    const double inv = 1.0 / ((double)a.obs_every * a.dt);
                    ox = ((f.x - s_first.x) + (c.x - s_centre.x)) * inv;
                    oy = ((f.y - s_first.y) + (c.y - s_centre.y)) * inv;
                    __syncwarp();
                    if (tid == 0) {
                        s_first = f;
                        s_centre = c;
                    }
                }
                if (tid == 0) {
                    const long long o = obs_idx;
                    if (a.obs) {
                        const double rx = a.obs[2 * o] - ox, ry = (a.obs[2 * o + 1] - oy) / a.sigma_ratio;
                        J = fma(rx, rx, fma(ry, ry, J));
                    }
                    if (a.head_traj) {
                        a.head_traj[((size_t)b * n_obs + o) * 2] = ox;
                        a.head_traj[((size_t)b * n_obs + o) * 2 + 1] = oy;
                    }
                }
            }
            if (obs_step) {
                obs_left = obs_every;
                ++obs_idx;
            }
        }
        // ---- outputs
        if (a.final_state && rank == 0) {  // rows past the sample's points, or of a run that stopped: NaN
            const int k0 = status == SWIMMER_OK ? n : 0;
            for (int k = k0 + tid; k < n_max; k += T)
                for (int c = 0; c < 4; ++c) a.final_state[((size_t)b * n_max + k) * 4 + c] = nan("");
        }
        if (a.speed && rank == 0 && tid < 32) {
            // mean speed: x-displacement of the flagellum's centroid (which starts at 0 in the stored
            // coordinates) or, with a head, of the head centre (the first swimmer's, with two), over
            // the run's duration; one warp sums in a fixed order
            const int k0 = nh > 0 ? nf : 0;
            const double2 ref = nh > 0 ? P[k0] : make_double2(0.0, 0.0), c = centre(P, ref, k0, nsw - k0, lane);
            if (tid == 0) {
                const double c0 = nh > 0 ? L + (a.gap_over_ds + a.hr_over_ds) * ds - xref : 0.0;
                a.speed[b] = status == SWIMMER_OK ? ((ref.x - c0) + c.x) / (a.steps * a.dt) : nan("");
            }
        }
        if (rank == 0 && tid == 0) {
            const unsigned long long wk = (unsigned long long)n * (unsigned long long)n * (unsigned long long)steps_done;
            atomicAdd(a.work, wk);
            if (a.speculative)
                a.run_work[b] = wk;
            else
                atomicAdd(a.work + 1, wk);
        }
        if (head_thread) {
            a.status[b] = status;
            if (a.loglik) {
                // Sigma = diag(sigma^2, (sigma_ratio sigma)^2) per observation (Sec. 3.1; two noise
                // levels, Sec. 4.2): residuals of the second component are divided by sigma_ratio in J
                const double sg = a.sigma * p.sig, s2 = sg * sg;  // the sample's noise level
                a.loglik[b] = status == SWIMMER_OK
                                  ? -(double)n_obs * (log(2.0 * PI * s2) + log(a.sigma_ratio)) - 0.5 * J / s2
                                  : -INFINITY;
            }
            if (status != SWIMMER_OK && a.head_traj) {
                // observations after the divergence were never taken
                for (long long o = steps_done / a.obs_every; o < n_obs; ++o) {
                    a.head_traj[((size_t)b * n_obs + o) * 2] = nan("");
                    a.head_traj[((size_t)b * n_obs + o) * 2 + 1] = nan("");
                }
            }
        }
        run_sync(C);
    }
}

typedef void (*Kernel64)(FwdArgs, int, int);

Kernel64 kernel_for(const swimmer_config &c, int threads) {
    const int model = c.n_swimmers == 2 ? 2 : c.n_head > 0 ? 1 : 0;
    if (threads <= 512)
        return model == 2 ? forward64_kernel<2, 512> : model == 1 ? forward64_kernel<1, 512> : forward64_kernel<0, 512>;
    return model == 2 ? forward64_kernel<2, 1024> : model == 1 ? forward64_kernel<1, 1024> : forward64_kernel<0, 1024>;
}

}  // namespace

size_t forward64_smem(int n_max, int panels, int threads, int pair_warps) {
    return state_bytes(n_max, threads, pair_warps) + sizeof(float4) * F64_REC * (size_t)panels;
}

// Warps of the symmetric pair sum in a launch with one run per CTA: at most one per unit, and 16, 8 or 4
// as their arrays fit; 0 where it does not pay for the largest sample, or, above 512 points, where a run is
// alone on its SM, if fewer than 8 fit (100 runs, us a step: N = 768 8 warps 3120, every ordered pair in 32
// 4530; N = 1024 4 warps 8010, 7400).
int forward64_pair_warps(const swimmer_handle *h, int threads) {
    const int n = h->cfg.n_max, nb = (n + 31) / 32, least = std::min(n > 512 ? 8 : 4, nb * nb);
    if (!symmetric_pays(n)) return 0;
    for (int w = std::min(16, std::min(threads / 32, nb * nb)); w >= least; w >>= 1)
        if (forward64_smem(n, handle_octaves(h) * F64_FINE, threads, w) + 2048 <= (size_t)h->max_smem) return w;
    return 0;
}

// CTAs per SM of a launch with one run per CTA (0: does not fit)
int forward64_resident(const swimmer_handle *h, int threads) {
    const size_t smem = forward64_smem(h->cfg.n_max, handle_octaves(h) * F64_FINE, threads, forward64_pair_warps(h, threads));
    Kernel64 kern = kernel_for(h->cfg, threads);
    int per_sm = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess) {
        cudaGetLastError();  // clear the error state a failed query leaves
        per_sm = 0;
    }
    return per_sm;
}

// One run per CTA, or per cluster of C CTAs when clusters of that size for every run of the batch
// fit the device at once and a CTA is left CLUSTER_POINTS points: a step's pair sum is what a run
// waits for (13 of 16 us at N = 64 on one SM), and it shrinks with the SMs that share it; with fewer
// points a CTA the stencils of the neighbours and the barriers would outweigh it.  Speculative launches
// (the pre-fetch rounds of a stage, whose rows outnumber the SMs) stay with one.
int launch_forward64(swimmer_handle *h, const FwdArgs &a, int threads, int max_runs, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cfg.attrs = attr;
    for (int C = a.speculative || 2 * a.B > h->num_sms ? 1 : MAX_CLUSTER; C > 1; C >>= 1) {
        if (a.n_max < C * CLUSTER_POINTS || C * a.B > h->num_sms) continue;
        int T = CLUSTER_THREADS;
        while (T < (a.n_max + C - 1) / C + 1) T <<= 1;  // a thread per own point
        const size_t smem = forward64_smem(a.n_max, a.tab_panels, T, 0);
        if (T > 1024 || smem + 2048 > (size_t)h->max_smem) continue;
        Kernel64 kern = kernel_for(h->cfg, T);
        CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        if (C > 8) CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.numAttrs = 1;
        cfg.gridDim = dim3(a.B * C);
        cfg.blockDim = dim3(T);
        cfg.dynamicSmemBytes = smem;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) != cudaSuccess) {
            cudaGetLastError();  // a size that the device does not offer
            continue;
        }
        if (fit < a.B) continue;
        CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, a, C, 0));
        return 0;
    }
    const int per = forward64_resident(h, threads), pw = forward64_pair_warps(h, threads);
    const size_t smem = forward64_smem(a.n_max, a.tab_panels, threads, pw);
    if (per < 1) {
        set_error("forward kernel does not fit on an SM (threads %d, smem %zu)", threads, smem);
        return SWIMMER_E_CUDA;
    }
    // CTAs per SM: no more than the launch has runs per SM (see launch_forward)
    const int runs = max_runs > 0 && max_runs < a.B ? max_runs : a.B;
    const int per_sm = std::min(per, std::max(1, (runs + h->num_sms - 1) / h->num_sms));
    kernel_for(h->cfg, threads)<<<std::min(per_sm * h->num_sms, a.B), threads, smem, s>>>(a, 1, pw);
    CUDA_TRY(cudaGetLastError());
    return 0;
}
