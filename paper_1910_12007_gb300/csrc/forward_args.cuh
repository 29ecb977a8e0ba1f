// Arguments of the forward kernels (forward.cu: FP32, forward64.cu: FP64).
#pragma once

#include "common.cuh"

struct FwdArgs {
    int B;
    const SampleParams *sp;
    const int *order;
    int *queue;
    const float4 *tab64;
    const float4 *tab32;
    float2 *pq;  // FP32 kernel: [B][n_max] preferred-curvature coefficients (P_k, Q_k) per run
    double mu, dt, kt, eta, omega;
    double hr_over_ds, gap_over_ds, k_head_tens, k_head_c, k_neck_tens, k_neck_ang;  // head model
    int obs_kind;
    double swim_d;        // two swimmers: initial separation along y
    double sigma_ratio;   // noise of the second observed component / the first
    long long steps, obs_every;
    const double *obs;
    double sigma;
    double *loglik;
    double *head_traj;
    double *speed;
    double *final_state;  // optional [B][n_max][4]: (x, y, Fx, Fy) at the end of the run
    int *status;
    unsigned long long *work;      // [0] executed, [1] useful pair evaluations
    unsigned long long *run_work;  // per-run pair evaluations (speculative launches)
    int speculative;               // 1: the caller decides later which runs were useful
    int n_max;
    int threads;
    int tab_panels;  // panels of the shared-memory table region (handle's octaves x panels/octave)
    const unsigned *units;  // FP32 pair-unit lists (offsets header, then the lists)
    int mode;               // FP32 pair units: 0 one-, 1 two-, 2 four-target
    int list_threads;       // FP32: the pair sum is split into as many lists as this many threads have warps
    int cluster;            // FP32: CTAs per run
};

// observations computed by warp 0 after a step (head-centre velocities, two-swimmer
// distances) rather than by the thread that updates the proximal point
static __device__ __forceinline__ bool vel_obs(const FwdArgs &a, int nh) {
    return (a.obs_kind == SWIMMER_OBS_HEAD_VELOCITY || a.obs_kind == SWIMMER_OBS_PAIR_DISTANCES) && nh > 0;
}

// A run on a cluster of C CTAs: an address of this CTA's shared memory as that of the CTA of a rank, and
// the barrier
static __device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
static __device__ __forceinline__ unsigned remote(unsigned addr, unsigned rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// barrier over the run's CTAs (every thread of every CTA reaches the same ones: all branches
// around them depend on values that the CTAs share)
static __device__ __forceinline__ void run_sync(int C) {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}

// forward64.cu: dynamic shared memory of an FP64 launch and the launch itself (threads per CTA
// as chosen by forward_threads)
size_t forward64_smem(int n_max, int panels, int threads, int pair_warps);
int forward64_pair_warps(const swimmer_handle *h, int threads);
int forward64_resident(const swimmer_handle *h, int threads);
int launch_forward64(swimmer_handle *h, const FwdArgs &a, int threads, int max_runs, cudaStream_t s);
