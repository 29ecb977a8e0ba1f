// FP64 evaluation of a sample's kernel-function table (g1 = B'' and h = delta^2 g2,
// g2 = (r B'' - B')/r^3, Eq. BrV) with almost no FP64 instruction.  GB300 issues an FP64 instruction of a warp every 16
// clocks of an SM and an FP32 one every quarter clock, so a degree-9 Clenshaw recurrence for two
// functions (36 FP64 FMAs) is what a pair evaluation used to wait for.
//
// Panels: 32 per octave of u = 1 + r^2/delta^2, indexed by the double's exponent and top 5
// mantissa bits; t in [-1, 1) across a panel is the remaining 47 bits, split exactly into two
// floats th + tl by integer operations.  On so short a panel g = c0 + q, q = t (c1 + t (c2 + ...))
// of degree 7, where q is at most 2^-5 of g's size nearby and each further term another 2^-5.5: c0 is a double,
// c1 .. c5 are pairs of floats evaluated with error-free products and sums (48 bits, so q carries
// less than an ulp of that size; where g1 crosses zero its error is one of its size nearby, as a series
// in FP64 has it), c6 and c7 floats.  Both functions run in the two halves of the packed FP32
// instructions.  The pair becomes a double by integer operations (join), so FP64 is left with one
// addition per function.  1024 FP64 runs of N = 128, 200 steps: 321 -> 109 ms (two additions), and
// 98 -> 86 ms by the join.  Against 22-digit references (alpha 0.3 to 30) g1 is 2.1e-16 rms off, g2
// 5.0e-16; as Chebyshev series in FP64 they were 6.0e-16 and 8.4e-16.
//
// Record of a panel (F64_REC float4): {c0 of g1, c0 of h} as doubles; for k = 1 .. 5 the high
// parts of c_k of g1 and h, then the low parts; c6 of g1, h, c7 of g1, h.
#pragma once

#include "common.cuh"

// a float as a double by integer operations (the conversion instruction runs at the FP64 rate);
// zero and denormals come out below 1e-38, which no sum here shows
static __device__ __forceinline__ double widen(float v) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// h + l as a double by integer operations, for |l| at most half of h's last place (a normalized
// pair): l in units of the last place of h's double is a whole number of 28 bits (rounded: half
// of that place), added to the bits.  Where h is a power of two (the sum could leave its binade) or
// so small that the unit is no float, the sum is FP64's.
static __device__ __forceinline__ double join(float h, float l) {
    const unsigned b = __float_as_uint(h), e = (b >> 23) & 0xffu;
    if ((b & 0x7fffffu) == 0u || e < 60u) return widen(h) + widen(l);
    const int n = __float2int_rn(l * __uint_as_float((306u - e) << 23));  // l 2^(52 - (e - 127))
    const int s = (int)b >> 31, d = (n ^ s) - s;                         // towards h's sign
    const unsigned hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u);
    return __longlong_as_double(((long long)hi << 32 | (long long)(b << 29)) + (long long)d);
}

static __device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// panel of u (clamped to pmax) and its local coordinate th + tl
static __device__ __forceinline__ int panel_f64(double u, int pmax, float &th, float &tl) {
    const unsigned hi = (unsigned)__double2hiint(u), lo = (unsigned)__double2loint(u);
    const int p = (int)min((hi - 0x3ff00000u) >> (20 - F64_FINE_LOG2), (unsigned)pmax);
    // the 47 bits below the panel's: the top 23, rounded, and the signed rest
    const unsigned top = (((hi & ((1u << (20 - F64_FINE_LOG2)) - 1u)) << 8) | (lo >> 24)) + ((lo >> 23) & 1u);
    th = fmaf(__uint_as_float(0x3f800000u + top), 2.f, -3.f);
    tl = (float)((int)(lo << 8) >> 8) * 0x1p-46f;
    return p;
}

// q of a record's two functions as normalized pairs of floats qh + ql
static __device__ __forceinline__ void poly_f64(const float4 *__restrict__ rec, float th, float tl, float2 &qh,
                                                float2 &ql) {
    const float2 t = make_float2(th, th), l = make_float2(tl, tl);
    const float4 c67 = rec[6];
    float2 ph = __ffma2_rn(make_float2(c67.z, c67.w), t, make_float2(c67.x, c67.y)), pl = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 5; k >= 1; --k) {
        const float4 c = rec[k];
        const float2 ch = make_float2(c.x, c.y), cl = make_float2(c.z, c.w);
        const float2 prod = __fmul2_rn(ph, t);
        float2 err = __ffma2_rn(ph, t, make_float2(-prod.x, -prod.y));
        err = __ffma2_rn(ph, l, err);
        if (k < 5) err = __ffma2_rn(pl, t, err);
        // TwoSum of ch and prod
        const float2 s = __fadd2_rn(ch, prod), b = sub2(s, ch);
        const float2 e = __fadd2_rn(sub2(ch, sub2(s, b)), sub2(prod, b));
        pl = __fadd2_rn(__fadd2_rn(e, err), cl);
        ph = s;
    }
    const float2 prod = __fmul2_rn(ph, t);
    float2 err = __ffma2_rn(ph, t, make_float2(-prod.x, -prod.y));
    err = __ffma2_rn(ph, l, err);
    err = __ffma2_rn(pl, t, err);
    // normalized: |l| is at most half of a nonzero |t|, so err of prod
    qh = __fadd2_rn(prod, err);
    ql = sub2(err, sub2(qh, prod));
}

// one function in the same form: record {c0 as a double, c1}, {c5, c4}, {c3, c2} (high and low
// part each), {c6, c7, 0, 0}
static __device__ __forceinline__ double poly1_f64(const float4 *__restrict__ rec, float th, float tl) {
    const double c0 = *(const double *)rec;
    const float2 c1 = *((const float2 *)rec + 1), c67 = *(const float2 *)(rec + 3);
    const float4 c54 = rec[1], c32 = rec[2];
    const float hi[6] = {0.f, c1.x, c32.z, c32.x, c54.z, c54.x}, lo[6] = {0.f, c1.y, c32.w, c32.y, c54.w, c54.y};
    float ph = fmaf(c67.y, th, c67.x), pl = 0.f;
#pragma unroll
    for (int k = 5; k >= 1; --k) {
        const float prod = __fmul_rn(ph, th);
        float err = fmaf(ph, th, -prod);
        err = fmaf(ph, tl, err);
        err = fmaf(pl, th, err);
        const float s = __fadd_rn(hi[k], prod), b = __fsub_rn(s, hi[k]);
        const float e = __fadd_rn(__fsub_rn(hi[k], __fsub_rn(s, b)), __fsub_rn(prod, b));
        pl = __fadd_rn(__fadd_rn(e, err), lo[k]);
        ph = s;
    }
    const float prod = __fmul_rn(ph, th);
    float err = fmaf(ph, th, -prod);
    err = fmaf(ph, tl, err);
    err = fmaf(pl, th, err);
    const float qh = __fadd_rn(prod, err);
    return c0 + join(qh, __fsub_rn(err, __fsub_rn(qh, prod)));
}

static __device__ __forceinline__ void kern_f64(const float4 *__restrict__ tab, int pmax, double u, double &g1,
                                                double &h) {
    float th, tl;
    const float4 *rec = tab + F64_REC * panel_f64(u, pmax, th, tl);
    const double2 c0 = *(const double2 *)rec;
    float2 qh, ql;
    poly_f64(rec, th, tl, qh, ql);
    g1 = c0.x + join(qh.x, ql.x);
    h = c0.y + join(qh.y, ql.y);
}
