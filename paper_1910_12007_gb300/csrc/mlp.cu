// K5/K6: the learned surrogate, an MLP 5 -> 256 -> 256 -> 256 -> 80 with GELU hidden
// activations (not in the paper).  Weights are kept as an FP32 master copy and rounded to
// BF16 when they enter a product; every product accumulates in FP32.
//
// What bounds it: latency.  A step on 2048 samples is 1.9 GFLOP, a microsecond of tensor pipe; as
// one GEMM launch per product (21 launches, operands staged from FP32 with a division of their
// index per element, 64 x 64 tiles that left most SMs idle) it took 312 us with Adam.  Now
//   - one kernel takes a tile of 16 or 32 rows through the whole network and back down to the first
//     layer (mlp_kernel): activations stay in shared memory as BF16, pre-activations as FP32, and
//     the weights come from L2 as ready-made MMA fragments (pack_kernel), 16 bytes a lane, a batch
//     of loads ahead of the batch in use;
//   - the weight gradients (reductions over the batch) are one launch over all layers' 64 x 64
//     tiles and up to SPLIT_MAX slices of the batch, BF16 operands by cp.async;
//   - one launch adds the slices and the tiles' bias and first-layer sums in a fixed order (no
//     atomics: gradients are deterministic).
// Measured: backward and Adam on 2048 samples 312 -> 43 us (35 us of it on the GPU: packing 3, the
// network 15, gradients 5, reduction 3, Adam 3 and gaps), the log-likelihood of 4096 samples 97 ->
// 19 us.  The network kernel waits for its weights (two batches of L2 loads a layer) and for erff and
// expf, in about equal parts; the tensor pipe idles, and tcgen05's larger tiles would leave fewer
// SMs with work.
//
// The products are warp-level m16n8k16 BF16 MMAs along k in order, so that a row's outputs do not
// depend on the tile it falls in (nor on the kernel's earlier form): an output that moved by an ulp
// could round the other way to BF16 on entering the next layer.  The first layer (5 inputs, which
// stay FP32) is an FP32 product with BF16 weights.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "table_eval.cuh"

namespace {

constexpr int IN = SWIMMER_MLP_IN, HID = SWIMMER_MLP_HIDDEN, OUT = SWIMMER_MLP_OUT;
constexpr int NLAYER = 4;
__host__ __device__ constexpr int fan_in(int l) { return l == 0 ? IN : HID; }
__host__ __device__ constexpr int fan_out(int l) { return l == NLAYER - 1 ? OUT : HID; }
__host__ __device__ constexpr int w_off(int l) {
    return l == 0 ? 0 : w_off(l - 1) + fan_in(l - 1) * fan_out(l - 1) + fan_out(l - 1);
}
__host__ __device__ constexpr int b_off(int l) { return w_off(l) + fan_in(l) * fan_out(l); }
static_assert(b_off(NLAYER - 1) + OUT == SWIMMER_MLP_NPARAM, "parameter layout");

constexpr float INV_SQRT2 = 0.70710678118654752f;
constexpr float INV_SQRT2PI = 0.39894228040143268f;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * INV_SQRT2)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * INV_SQRT2)) + z * expf(-0.5f * z * z) * INV_SQRT2PI;
}
__device__ __forceinline__ float bf16r(float w) { return __bfloat162float(__float2bfloat16_rn(w)); }
__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
    const unsigned a = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
    const unsigned b = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
    return a | (b << 16);
}
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], const __nv_bfloat16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], const __nv_bfloat16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// ---------------------------------------------------------------------------------
// weights as MMA B fragments: per (n8 tile j, k32 block kb) one uint4 a lane, the two registers
// of its first k16 step, then of its second
// ---------------------------------------------------------------------------------
// matrices: forward products of layers 1, 2, 3 (B(k, n) = W[n][k]), input gradients of layers 3,
// 2, 1 (B(k, n) = W[k][n]; layer 3's k = 80 is padded with zeros to 96)
constexpr int KB = HID / 32, KB3 = (OUT + 31) / 32;
constexpr int NT = HID / 8, NT3 = OUT / 8;
__host__ __device__ constexpr int frag_at(int q) {  // in uint4
    return q == 0 ? 0 : frag_at(q - 1) + 32 * (q - 1 == 2 ? NT3 * KB : q - 1 == 3 ? NT * KB3 : NT * KB);
}
constexpr int FRAG_FORWARD = frag_at(3), FRAG_ALL = frag_at(6);

__global__ void pack_kernel(int count, const float *__restrict__ P, uint4 *__restrict__ frag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    int q = 0;
    while (q < 5 && i >= frag_at(q + 1)) ++q;
    const int r = (i - frag_at(q)) >> 5, lane = i & 31, gid = lane >> 2, tig = lane & 3;
    const int kbs = q == 3 ? KB3 : KB, j = r / kbs, kb = r % kbs, n = 8 * j + gid;
    const int l = q < 3 ? q + 1 : 6 - q;
    const float *W = P + w_off(l);
    unsigned v[4];
    for (int h = 0; h < 4; ++h) {
        const int k = 32 * kb + 16 * (h >> 1) + 8 * (h & 1) + 2 * tig;
        float a, b;
        if (q < 3) {
            a = W[(size_t)n * HID + k];
            b = W[(size_t)n * HID + k + 1];
        } else {
            a = k < fan_out(l) ? W[(size_t)k * HID + n] : 0.f;
            b = k + 1 < fan_out(l) ? W[(size_t)(k + 1) * HID + n] : 0.f;
        }
        v[h] = pack_bf16(a, b);
    }
    frag[i] = make_uint4(v[0], v[1], v[2], v[3]);
}

// ---------------------------------------------------------------------------------
// a tile of MT rows through the network
// ---------------------------------------------------------------------------------
constexpr int THREADS = 256, WARPS = THREADS / 32;
constexpr int LDA = HID + 8;  // BF16 row stride (rows 16 bytes apart modulo 128: ldmatrix conflict-free)
constexpr int LDZ = HID + 2;  // FP32 row stride
constexpr int BATCH = 4;      // k32 blocks of weights loaded at a time

// per tile of rows: sums of d loss / d pre-activation (biases) and of the first layer's products
constexpr int SUM_B3 = 0, SUM_B2 = SUM_B3 + OUT, SUM_B1 = SUM_B2 + HID, SUM_0 = SUM_B1 + HID;  // then [6][HID]
constexpr int SUMS = SUM_0 + (IN + 1) * HID;

struct Surr {  // the surrogate's inputs and likelihood
    int np, stride;
    long long n_obs;
    const double *theta, *norm, *obs;
    double lo[3], hi[3];  // of theta; the other two inputs are the same for every sample:
    float x3, x4;
    double sigma, log_term;  // log_term: -n_obs log(2 pi sigma^2) of the launch's noise level
    double *ll;
};

struct NetArgs {
    int n;
    const float *P, *x, *t;  // t: targets (training)
    float *y;                // outputs, or nullptr
    const uint4 *frag;
    __nv_bfloat16 *H[3], *dZ[3];  // training: activations and output gradients of layers 1 .. 3, [n][256] ([n][80])
    float *sums, *loss;           // training: [tiles][SUMS], [tiles]
    Surr s;
};

template <int NTW, int KBS>
struct Weights {  // a warp's fragments of one layer: its n8 tiles w, w + step, ...
    const uint4 *p;
    int step;  // between a warp's tiles
    uint4 v[2][BATCH][NTW];
    __device__ __forceinline__ void load(int slot, int kb0, int tiles) {
#pragma unroll
        for (int b = 0; b < BATCH; ++b)
#pragma unroll
            for (int j = 0; j < NTW; ++j)
                if (kb0 + b < KBS && j < tiles) v[slot][b][j] = p[(size_t)(j * step * KBS + kb0 + b) * 32];
    }
};

// acc += A (MT x 32 KBS, BF16 in shared memory) times the warp's tiles
template <int MT, int NTW, int KBS>
__device__ __forceinline__ void product(const __nv_bfloat16 *A, Weights<NTW, KBS> &w, int tiles, float (&acc)[MT / 16][NTW][4]) {
    const int lane = threadIdx.x & 31;
    const __nv_bfloat16 *base = A + (lane & 15) * LDA + (lane >> 4) * 8;
#pragma unroll
    for (int kb0 = 0; kb0 < KBS; kb0 += BATCH) {
        const int slot = (kb0 / BATCH) & 1;
        if (kb0 + BATCH < KBS) w.load(slot ^ 1, kb0 + BATCH, tiles);
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            if (kb0 + b >= KBS) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unsigned a[MT / 16][4];
#pragma unroll
                for (int i = 0; i < MT / 16; ++i) ldsm4(a[i], base + 16 * i * LDA + 32 * (kb0 + b) + 16 * h);
#pragma unroll
                for (int j = 0; j < NTW; ++j) {
                    if (j >= tiles) break;
                    const uint4 &f = w.v[slot][b][j];
#pragma unroll
                    for (int i = 0; i < MT / 16; ++i) mma_bf16_16816(acc[i][j], a[i], h ? f.z : f.x, h ? f.w : f.y);
                }
            }
        }
    }
}

template <int MT>
constexpr size_t net_smem(bool train) {
    return sizeof(__nv_bfloat16) * 2 * MT * LDA + sizeof(float) * (MT * 8 + MT * OUT) +
           (train ? sizeof(float) * 3 * MT * LDZ : 0);
}

template <int MT, bool TRAIN, bool SURR>
__global__ void __launch_bounds__(THREADS, 1) mlp_kernel(NetArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    __nv_bfloat16 *Abuf[2] = {(__nv_bfloat16 *)sm, (__nv_bfloat16 *)sm + MT * LDA};
    float *xs = (float *)(Abuf[1] + MT * LDA);  // [MT][8] inputs
    float *ys = xs + MT * 8;                    // [MT][80] outputs, then their gradients
    float *Z = ys + MT * OUT;                   // training: [3][MT][LDZ] pre-activations, then their gradients
    __shared__ float s_red[WARPS];
    __shared__ double res_c[SURR ? OUT : 1], res_s[SURR ? OUT : 1];  // residual = res_c - res_s y
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const int r0 = blockIdx.x * MT, rows = min(MT, a.n - r0);

    // the first batch of layer 1's weights is under way while the inputs and layer 0 are made
    Weights<4, KB> w;
    w.p = a.frag + (size_t)(4 * warp) * KB * 32 + lane;
    w.step = 1;
    w.load(0, 0, 4);
    // ---- inputs
    for (int e = tid; e < MT * IN; e += THREADS) {
        const int r = e / IN, k = e % IN;
        float v = 0.f;
        if (r < rows) {
            if (SURR) {
                const Surr &s = a.s;
                if (k >= 3) {
                    v = k == 3 ? s.x3 : s.x4;
                } else {
                    const double span = s.hi[k] - s.lo[k];
                    v = span > 0.0 ? (float)(2.0 * (s.theta[(size_t)s.np * (r0 + r) + k] - s.lo[k]) / span - 1.0) : 0.f;
                }
            } else {
                v = a.x[(size_t)(r0 + r) * IN + k];
            }
        }
        xs[r * 8 + k] = v;
    }
    if (SURR && tid < OUT) {
        const long long row = (long long)(tid >> 1) * a.s.stride + a.s.stride - 1;
        res_c[tid] = a.s.obs[2 * row + (tid & 1)] - a.s.norm[tid];
        res_s[tid] = a.s.norm[OUT + tid];
    }
    __syncthreads();
    // ---- layer 0: a thread per output, FP32
    {
        float w0[IN];
        for (int k = 0; k < IN; ++k) w0[k] = bf16r(a.P[w_off(0) + tid * IN + k]);
        const float bias = a.P[b_off(0) + tid];
        for (int r = 0; r < MT; ++r) {
            float v = 0.f;
            for (int k = 0; k < IN; ++k) v = fmaf(xs[r * 8 + k], w0[k], v);
            v += bias;
            if (TRAIN) Z[r * LDZ + tid] = v;
            const __nv_bfloat16 h = __float2bfloat16_rn(gelu(v));
            Abuf[0][r * LDA + tid] = h;
            if (TRAIN && r < rows) a.H[0][(size_t)(r0 + r) * HID + tid] = h;
        }
    }
    __syncthreads();
    // ---- layers 1, 2: a warp owns 32 outputs
#pragma unroll 1
    for (int l = 1; l <= 2; ++l) {
        float acc[MT / 16][4][4] = {};
        product<MT, 4, KB>(Abuf[(l - 1) & 1], w, 4, acc);
        if (l == 1) {
            w.p = a.frag + frag_at(1) + (size_t)(4 * warp) * KB * 32 + lane;
            w.load(0, 0, 4);
        }
        const float *bias = a.P + (l == 1 ? b_off(1) : b_off(2));
#pragma unroll
        for (int i = 0; i < MT / 16; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 32 * warp + 8 * j + 2 * tig;
                const float b0 = bias[c], b1 = bias[c + 1];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 16 * i + 8 * h + gid;
                    const float v0 = acc[i][j][2 * h] + b0, v1 = acc[i][j][2 * h + 1] + b1;
                    if (TRAIN) *(float2 *)(Z + (l * MT + r) * LDZ + c) = make_float2(v0, v1);
                    const unsigned hv = pack_bf16(gelu(v0), gelu(v1));
                    *(unsigned *)(Abuf[l & 1] + r * LDA + c) = hv;
                    if (TRAIN && r < rows) *(unsigned *)(a.H[l] + (size_t)(r0 + r) * HID + c) = hv;
                }
            }
        __syncthreads();
    }
    // ---- layer 3: n8 tiles warp and warp + 8 of 10
    Weights<4, KB3> w3;  // the input gradient's first batch (its only one)
    if (TRAIN) {
        w3.p = a.frag + frag_at(3) + (size_t)(4 * warp) * KB3 * 32 + lane;
        w3.step = 1;
        w3.load(0, 0, 4);
    }
    {
        Weights<2, KB> wo;
        const int tiles = warp + WARPS < NT3 ? 2 : 1;
        wo.p = a.frag + frag_at(2) + (size_t)warp * KB * 32 + lane;
        wo.step = WARPS;
        wo.load(0, 0, tiles);
        float acc[MT / 16][2][4] = {};
        product<MT, 2, KB>(Abuf[0], wo, tiles, acc);
        const float *bias = a.P + b_off(3);
#pragma unroll
        for (int i = 0; i < MT / 16; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (j >= tiles) break;
                const int c = 8 * (warp + j * WARPS) + 2 * tig;
#pragma unroll
                for (int q = 0; q < 4; ++q) ys[(16 * i + (q >> 1) * 8 + gid) * OUT + c + (q & 1)] = acc[i][j][q] + bias[c + (q & 1)];
            }
    }
    __syncthreads();
    if (SURR) {
        // Gaussian log-likelihood over the 40 subsampled observation rows, 8 lanes a sample: FP64,
        // two instructions an output (the pipe takes 16 clocks each), floats widened by integers
        const Surr &s = a.s;
        for (int r = tid >> 3; r < MT; r += THREADS / 8) {
            double J = 0.0;
            for (int c = tid & 7; c < OUT; c += 8) {
                const float y = ys[r * OUT + c];
                // (widen takes finite numbers only)
                const double res = fma(-res_s[c], isfinite(y) ? widen(y) : (double)y, res_c[c]);
                J = fma(res, res, J);
            }
            for (int o = 4; o >= 1; o >>= 1) J += __shfl_xor_sync(0xffffffffu, J, o);
            if ((tid & 7) == 0 && r < rows) {
                const int b = r0 + r;
                J *= 0.5 * (double)s.n_obs / (double)(OUT / 2);
                double sg = s.sigma, term = s.log_term;
                if (s.np == 4) {  // the sample's noise level: theta[3] times sigma
                    sg *= s.theta[(size_t)s.np * b + 3];
                    term = -(double)s.n_obs * log(2.0 * 3.14159265358979323846 * (sg * sg));
                }
                s.ll[b] = isnan(s.theta[(size_t)s.np * b]) || !(sg > 0.0) ? -INFINITY : term - J / (sg * sg);
            }
        }
        return;
    }
    if (a.y)
        for (int e = tid; e < rows * OUT; e += THREADS) a.y[(size_t)r0 * OUT + e] = ys[e];
    if (!TRAIN) return;
    // ---- loss and its gradient: dY = 2 (Y - T)/(n 80), FP32 in ys, BF16 as the next operand
    {
        const float sc = 2.0f / ((float)a.n * (float)OUT);
        float part = 0.f;
        __nv_bfloat16 *A = Abuf[1];
        for (int e = tid; e < MT * 96; e += THREADS) {
            const int r = e / 96, c = e % 96;
            float g = 0.f;
            if (r < rows && c < OUT) {
                const float d = ys[r * OUT + c] - a.t[(size_t)(r0 + r) * OUT + c];
                part = fmaf(d, d, part);
                g = sc * d;
            }
            const __nv_bfloat16 gb = __float2bfloat16_rn(g);
            A[r * LDA + c] = gb;
            if (c < OUT) {
                ys[r * OUT + c] = g;
                if (r < rows) a.dZ[2][(size_t)(r0 + r) * OUT + c] = gb;
            }
        }
        for (int o = 16; o >= 1; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) s_red[warp] = part;
    }
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        for (int k = 0; k < WARPS; ++k) s += s_red[k];
        a.loss[blockIdx.x] = s;
    }
    float *sums = a.sums + (size_t)blockIdx.x * SUMS;
    if (tid < OUT) {
        float s = 0.f;
        for (int r = 0; r < MT; ++r) s += ys[r * OUT + tid];
        sums[SUM_B3 + tid] = s;
    }
    // ---- input gradients: dZ_{l-1} = (dZ_l W_l) gelu'(Z_{l-1}), l = 3, 2, 1
#pragma unroll 1
    for (int l = 3; l >= 1; --l) {
        float acc[MT / 16][4][4] = {};
        if (l == 3) {
            w.p = a.frag + frag_at(4) + (size_t)(4 * warp) * KB * 32 + lane;
            w.load(0, 0, 4);
            product<MT, 4, KB3>(Abuf[1], w3, 4, acc);
        } else {
            product<MT, 4, KB>(Abuf[l == 2 ? 0 : 1], w, 4, acc);
            if (l == 2) {
                w.p = a.frag + frag_at(5) + (size_t)(4 * warp) * KB * 32 + lane;
                w.load(0, 0, 4);
            }
        }
        float *Zl = Z + (l - 1) * MT * LDZ;
        __nv_bfloat16 *An = Abuf[l == 3 ? 0 : 1];
#pragma unroll
        for (int i = 0; i < MT / 16; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 32 * warp + 8 * j + 2 * tig;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 16 * i + 8 * h + gid;
                    float2 *z = (float2 *)(Zl + r * LDZ + c);
                    const float2 zz = *z;
                    const float g0 = acc[i][j][2 * h] * gelu_grad(zz.x), g1 = acc[i][j][2 * h + 1] * gelu_grad(zz.y);
                    *z = make_float2(g0, g1);
                    if (l > 1) {
                        const unsigned gv = pack_bf16(g0, g1);
                        *(unsigned *)(An + r * LDA + c) = gv;
                        if (r < rows) *(unsigned *)(a.dZ[l - 2] + (size_t)(r0 + r) * HID + c) = gv;
                    }
                }
            }
        __syncthreads();
        // column sums (rows past the batch hold zeros); for the first layer also its weights'
        float s[IN + 1] = {};
        for (int r = 0; r < MT; ++r) {
            const float g = Zl[r * LDZ + tid];
            s[0] += g;
            if (l == 1)
                for (int k = 0; k < IN; ++k) s[k + 1] = fmaf(g, xs[r * 8 + k], s[k + 1]);
        }
        if (l > 1) {
            sums[(l == 3 ? SUM_B2 : SUM_B1) + tid] = s[0];
        } else {
            for (int k = 0; k <= IN; ++k) sums[SUM_0 + k * HID + tid] = s[k];
        }
    }
}

// ---------------------------------------------------------------------------------
// weight gradients: dW_l[o][i] = sum_s dZ_l[s][o] H_{l-1}[s][i] over a slice of the batch, one 64 x 64
// tile a CTA of four warps (2 x 2, each 32 x 32), 64 samples at a time, three stages of cp.async
// ---------------------------------------------------------------------------------
constexpr int GT = 64, GK = 64, GLD = GT + 8, STAGES = 3;
constexpr int TILES_H = (HID / GT) * (HID / GT), TILES_3 = ((OUT + GT - 1) / GT) * (HID / GT);
constexpr int GRAD_TILES = 2 * TILES_H + TILES_3;
constexpr int GRAD_W = 2 * HID * HID + OUT * HID;  // weights of layers 1, 2, 3
constexpr int SPLIT_MAX = 6;                       // slices of the batch at most

struct GradArgs {
    int n, rows;  // samples, samples per slice (a multiple of GK)
    const __nv_bfloat16 *H[3], *dZ[3];
    float *part;  // [slices][GRAD_W]
};

__device__ __forceinline__ void cp16(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(ok ? 16 : 0));
}

__global__ void __launch_bounds__(128) grad_kernel(GradArgs a) {
    extern __shared__ __align__(16) __nv_bfloat16 gs[];  // [STAGES][2][GK][GLD]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int tile = blockIdx.x;
    const int l = tile < TILES_H ? 0 : tile < 2 * TILES_H ? 1 : 2;
    tile -= l * TILES_H;
    const int o0 = (tile / (HID / GT)) * GT, i0 = (tile % (HID / GT)) * GT, fo = l == 2 ? OUT : HID;
    const int s0 = blockIdx.y * a.rows, s1 = min(a.n, s0 + a.rows);
    const __nv_bfloat16 *G = a.dZ[l], *H = a.H[l];
    auto stage = [&](int st, int k0) {
        __nv_bfloat16 *sg = gs + st * 2 * GK * GLD, *sh = sg + GK * GLD;
        for (int e = tid; e < GK * GT / 8; e += 128) {
            const int r = e / (GT / 8), c = 8 * (e % (GT / 8)), s = k0 + r;
            const bool in = s < s1, og = in && o0 + c < fo;
            cp16(sg + r * GLD + c, G + (og ? (size_t)s * fo + o0 + c : 0), og);
            cp16(sh + r * GLD + c, H + (in ? (size_t)s * HID + i0 + c : 0), in);
        }
        asm volatile("cp.async.commit_group;");
    };
    const int steps = (s1 - s0 + GK - 1) / GK;
    for (int st = 0; st < STAGES - 1; ++st)
        if (st < steps) stage(st, s0 + st * GK);
        else asm volatile("cp.async.commit_group;");
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int q = lane >> 3, r8 = lane & 7;
    float acc[2][4][4] = {};
    for (int it = 0; it < steps; ++it) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2));
        __syncthreads();
        const __nv_bfloat16 *sg = gs + (it % STAGES) * 2 * GK * GLD, *sh = sg + GK * GLD;
        if (it + STAGES - 1 < steps) stage((it + STAGES - 1) % STAGES, s0 + (it + STAGES - 1) * GK);
        else asm volatile("cp.async.commit_group;");
#pragma unroll
        for (int k = 0; k < GK; k += 16) {
            unsigned af[2][4], bf[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) ldsm4t(af[i], sg + (k + (q >> 1) * 8 + r8) * GLD + wm + 16 * i + (q & 1) * 8);
#pragma unroll
            for (int j = 0; j < 2; ++j) ldsm4t(bf[j], sh + (k + (q & 1) * 8 + r8) * GLD + wn + 16 * j + (q >> 1) * 8);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16_16816(acc[i][j], af[i], bf[j >> 1][2 * (j & 1)], bf[j >> 1][2 * (j & 1) + 1]);
        }
    }
    float *out = a.part + (size_t)blockIdx.y * GRAD_W + (size_t)l * HID * HID;
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int o = o0 + wm + 16 * i + 8 * h + gid, c = i0 + wn + 8 * j + 2 * tig;
                if (o < fo) *(float2 *)(out + (size_t)o * HID + c) = make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
            }
}

// slices added in order into the weight gradients; the tiles' sums (eight partial sums of every
// eighth tile, then those in order) into bias and first-layer gradients and the loss
constexpr int RED_W = (GRAD_W / 4 + 255) / 256, RED_S = (SUMS + 1 + 31) / 32;
__global__ void __launch_bounds__(256) grad_reduce_kernel(int n, int slices, const float *__restrict__ part, int tiles,
                                                          const float *__restrict__ sums, const float *__restrict__ loss,
                                                          float *__restrict__ grad, float *__restrict__ loss_out) {
    __shared__ float red[8][33];
    const int tid = threadIdx.x;
    if (blockIdx.x < RED_W) {
        const int i = 4 * (blockIdx.x * 256 + tid);
        if (i >= GRAD_W) return;
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int z = 0; z < slices; ++z) {
            const float4 v = *(const float4 *)(part + (size_t)z * GRAD_W + i);
            t.x += v.x;
            t.y += v.y;
            t.z += v.z;
            t.w += v.w;
        }
        const int l = i < HID * HID ? 1 : i < 2 * HID * HID ? 2 : 3;
        float *g = grad + (l == 1 ? w_off(1) : l == 2 ? w_off(2) : w_off(3)) + (i - (l - 1) * HID * HID);
        g[0] = t.x;
        g[1] = t.y;
        g[2] = t.z;
        g[3] = t.w;
        return;
    }
    const int c = (blockIdx.x - RED_W) * 32 + (tid & 31), part8 = tid >> 5;
    float s = 0.f;
    if (c < SUMS)
        for (int k = part8; k < tiles; k += 8) s += sums[(size_t)k * SUMS + c];
    else if (c == SUMS)
        for (int k = part8; k < tiles; k += 8) s += loss[k];
    red[part8][tid & 31] = s;
    __syncthreads();
    if (part8 != 0 || c > SUMS) return;
    float t = 0.f;
    for (int k = 0; k < 8; ++k) t += red[k][tid];
    if (c == SUMS) {
        loss_out[0] = t / ((float)n * (float)OUT);
    } else if (c < SUM_B2) {
        grad[b_off(3) + c] = t;
    } else if (c < SUM_B1) {
        grad[b_off(2) + c - SUM_B2] = t;
    } else if (c < SUM_0) {
        grad[b_off(1) + c - SUM_B1] = t;
    } else {
        const int k = (c - SUM_0) / HID, o = (c - SUM_0) % HID;
        grad[k == 0 ? b_off(0) + o : w_off(0) + o * IN + k - 1] = t;
    }
}

__global__ void adam_kernel(int n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float gi = g[i];
    float mi = b1 * m[i] + (1.f - b1) * gi;
    float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// workspace for n samples, 16-byte aligned parts: the packed weights, then for training the
// activations and output gradients in BF16, the tiles' sums and losses, the slices' partial gradients
struct Ws {
    uint4 *frag;
    __nv_bfloat16 *H[3], *dZ[3];
    float *sums, *loss, *part;
};
constexpr int MT_MIN = 16;
int grad_slices(int n) { return std::min(SPLIT_MAX, (n + GK - 1) / GK); }
size_t align16(size_t b) { return (b + 15) & ~size_t(15); }
Ws carve(void *base, int n, size_t *used = nullptr) {
    unsigned char *p = (unsigned char *)align16((size_t)base);
    auto take = [&](size_t bytes) {
        unsigned char *q = p;
        p += align16(bytes);
        return q;
    };
    Ws w;
    w.frag = (uint4 *)take(sizeof(uint4) * FRAG_ALL);
    for (int l = 0; l < 3; ++l) {
        w.H[l] = (__nv_bfloat16 *)take(2 * (size_t)n * HID);
        w.dZ[l] = (__nv_bfloat16 *)take(2 * (size_t)n * (l == 2 ? OUT : HID));
    }
    const size_t tiles = ((size_t)n + MT_MIN - 1) / MT_MIN;
    w.sums = (float *)take(sizeof(float) * tiles * SUMS);
    w.loss = (float *)take(sizeof(float) * tiles);
    w.part = (float *)take(sizeof(float) * (size_t)grad_slices(n) * GRAD_W);
    if (used) *used = (size_t)(p - (unsigned char *)base);
    return w;
}

int pack(cudaStream_t s, const float *P, uint4 *frag, bool train) {
    const int count = train ? FRAG_ALL : FRAG_FORWARD;
    pack_kernel<<<(count + 255) / 256, 256, 0, s>>>(count, P, frag);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

template <int MT, bool TRAIN, bool SURR>
int launch_net(cudaStream_t s, const NetArgs &a) {
    constexpr size_t smem = net_smem<MT>(TRAIN);
    CUDA_TRY(cudaFuncSetAttribute(mlp_kernel<MT, TRAIN, SURR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    mlp_kernel<MT, TRAIN, SURR><<<(a.n + MT - 1) / MT, THREADS, smem, s>>>(a);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

// rows per tile: 16 while those tiles leave no SM with two (a tile's latency, not its work, is what
// a small batch waits for), else 32 (half the weight traffic per row)
int tile_rows(int n, int sms) { return n <= 16 * sms ? 16 : 32; }

int sm_count(int *sms) {
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
    return 0;
}

}  // namespace

extern "C" size_t mlp_workspace_bytes(int n) {
    size_t used = 0;
    carve(nullptr, n, &used);
    return used + 16;  // the caller's buffer may start anywhere
}

extern "C" int mlp_forward(int n, const float *params, const float *x, float *y, float *workspace, void *stream) {
    ARG_CHECK(n >= 1, "n must be >= 1");
    ARG_CHECK(params && x && y && workspace, "NULL device pointer");
    cudaStream_t s = (cudaStream_t)stream;
    int sms = 0, rc = sm_count(&sms);
    if (rc) return rc;
    NetArgs a = {};
    a.n = n;
    a.P = params;
    a.x = x;
    a.y = y;
    a.frag = carve(workspace, n).frag;
    rc = pack(s, params, carve(workspace, n).frag, false);
    if (rc) return rc;
    return tile_rows(n, sms) == 16 ? launch_net<16, false, false>(s, a) : launch_net<32, false, false>(s, a);
}

extern "C" int mlp_backward(int n, const float *params, const float *x, const float *t, float *grad,
                            float *loss_out, float *workspace, void *stream) {
    ARG_CHECK(n >= 1, "n must be >= 1");
    ARG_CHECK(params && x && t && grad && loss_out && workspace, "NULL device pointer");
    cudaStream_t s = (cudaStream_t)stream;
    int sms = 0, rc = sm_count(&sms);
    if (rc) return rc;
    const Ws w = carve(workspace, n);
    rc = pack(s, params, w.frag, true);
    if (rc) return rc;
    NetArgs a = {};
    a.n = n;
    a.P = params;
    a.x = x;
    a.t = t;
    a.frag = w.frag;
    GradArgs g = {};
    for (int l = 0; l < 3; ++l) {
        a.H[l] = w.H[l];
        a.dZ[l] = w.dZ[l];
        g.H[l] = w.H[l];
        g.dZ[l] = w.dZ[l];
    }
    a.sums = w.sums;
    a.loss = w.loss;
    const int mt = tile_rows(n, sms);
    rc = mt == 16 ? launch_net<16, true, false>(s, a) : launch_net<32, true, false>(s, a);
    if (rc) return rc;
    g.n = n;
    g.rows = ((n + grad_slices(n) - 1) / grad_slices(n) + GK - 1) / GK * GK;
    g.part = w.part;
    const int slices = (n + g.rows - 1) / g.rows;
    constexpr size_t smem = sizeof(__nv_bfloat16) * STAGES * 2 * GK * GLD;
    CUDA_TRY(cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    grad_kernel<<<dim3(GRAD_TILES, slices), 128, smem, s>>>(g);
    CUDA_TRY(cudaGetLastError());
    grad_reduce_kernel<<<RED_W + RED_S, 256, 0, s>>>(n, slices, w.part, (n + mt - 1) / mt, w.sums, w.loss, grad, loss_out);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

extern "C" int mlp_adam(float *params, const float *grad, float *m, float *v, int step, float lr, void *stream) {
    ARG_CHECK(params && grad && m && v, "NULL device pointer");
    ARG_CHECK(step >= 1, "step counts from 1");
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    adam_kernel<<<(SWIMMER_MLP_NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(SWIMMER_MLP_NPARAM, params, grad, m,
                                                                                   v, lr, b1, b2, eps, c1, c2);
    CUDA_TRY(cudaGetLastError());
    return 0;
}

// ---------------------------------------------------------------------------------
// surrogate log-likelihood for delayed acceptance: one launch, inputs from theta, the network with
// the weights packed by swimmer_surrogate_set, the likelihood
// ---------------------------------------------------------------------------------
int run_surrogate_loglik(swimmer_handle *h, int B, const double *theta, const double *obs, double sigma,
                         double *loglik, cudaStream_t s) {
    NetArgs a = {};
    a.n = B;
    a.P = h->surr_params;
    a.frag = h->surr_frag;
    a.s.np = n_params(h->cfg);
    a.s.theta = theta;
    const double *lo = h->surr_in_lo, *hi = h->surr_in_hi, fixed[2] = {h->surr_log10_kt, h->surr_omega};
    for (int k = 0; k < IN; ++k) {
        if (k < 3) {
            a.s.lo[k] = lo[k];
            a.s.hi[k] = hi[k];
        } else {
            const double span = hi[k] - lo[k];
            (k == 3 ? a.s.x3 : a.s.x4) = span > 0.0 ? (float)(2.0 * (fixed[k - 3] - lo[k]) / span - 1.0) : 0.f;
        }
    }
    a.s.norm = h->surr_norm;
    a.s.obs = obs;
    a.s.stride = h->surr_obs_stride;
    a.s.n_obs = h->cfg.steps / h->cfg.obs_every;
    a.s.sigma = sigma;
    a.s.log_term = -(double)a.s.n_obs * log(2.0 * 3.14159265358979323846 * (sigma * sigma));
    a.s.ll = loglik;
    return tile_rows(B, h->num_sms) == 16 ? launch_net<16, false, true>(s, a) : launch_net<32, false, true>(s, a);
}

extern "C" int swimmer_surrogate_set(swimmer_handle *h, const float *params, const double *in_lo, const double *in_hi,
                                     const double *out_mean, const double *out_std, int obs_stride, double log10_kt,
                                     double omega) {
    ARG_CHECK(h != nullptr, "handle is NULL");
    ARG_CHECK(params && in_lo && in_hi && out_mean && out_std, "NULL pointer");
    ARG_CHECK(obs_stride >= 1, "obs_stride must be >= 1");
    ARG_CHECK((long long)(OUT / 2) * obs_stride <= h->cfg.steps / h->cfg.obs_every,
              "surrogate outputs beyond the observation record");
    if (!h->surr_frag) CUDA_TRY(cudaMalloc((void **)&h->surr_frag, sizeof(uint4) * FRAG_FORWARD));
    for (int k = 0; k < 5; ++k) {
        h->surr_in_lo[k] = in_lo[k];
        h->surr_in_hi[k] = in_hi[k];
    }
    CUDA_TRY(cudaMemcpy(h->surr_params, params, sizeof(float) * SWIMMER_MLP_NPARAM, cudaMemcpyDeviceToDevice));
    CUDA_TRY(cudaMemcpy(h->surr_norm, out_mean, sizeof(double) * OUT, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(h->surr_norm + OUT, out_std, sizeof(double) * OUT, cudaMemcpyHostToDevice));
    // the weights as the likelihood kernel reads them; as synchronous as the copies around it
    int rc = pack(0, h->surr_params, h->surr_frag, false);
    if (rc) return rc;
    CUDA_TRY(cudaStreamSynchronize(0));
    const int trusted = 1;  // a surrogate set anew may screen until the plain model judges it
    CUDA_TRY(cudaMemcpy(h->surr_trust, &trusted, sizeof(int), cudaMemcpyHostToDevice));
    h->surr_obs_stride = obs_stride;
    h->surr_log10_kt = log10_kt;
    h->surr_omega = omega;
    h->surr_ready = 1;
    return 0;
}

extern "C" int surrogate_loglik_batch(swimmer_handle *h, int B, const double *theta, const double *obs, double sigma,
                                      double *loglik, void *stream) {
    ARG_CHECK(h != nullptr, "handle is NULL");
    ARG_CHECK(h->surr_ready, "surrogate not set (swimmer_surrogate_set)");
    ARG_CHECK(B >= 1 && B <= h->cfg.b_max, "B outside [1, b_max]");
    ARG_CHECK(theta && obs && loglik, "NULL device pointer");
    ARG_CHECK(sigma > 0.0, "sigma must be > 0");
    return run_surrogate_loglik(h, B, theta, obs, sigma, loglik, (cudaStream_t)stream);
}
