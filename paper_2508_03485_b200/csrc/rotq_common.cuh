// Pieces shared by the rotate + quantize kernels: the per-token parameters of Eq. 1 and the saturating packers.
#pragma once
#include "lrq_internal.cuh"
#include "f32x2.cuh"

namespace lrq_rq {

// Per-token quantization parameters from the token's extremes of the un-normalised transform.
// s_u is the step in the un-normalised domain; the reported scale is s_u * nrm.
struct TokenQ { float inv; float negz; };

__device__ __forceinline__ uint32_t pack_u8x4(int q0, int q1, int q2, int q3) {
    uint32_t t, d;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(t) : "r"(q3), "r"(q2), "r"(0));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(q1), "r"(q0), "r"(t));
    return d;
}

__device__ __forceinline__ uint32_t pack_u4x8(const int* q) {
    uint32_t t = 0;
#pragma unroll
    for (int i = 3; i >= 0; --i)
        asm("cvt.pack.sat.u4.s32.b32 %0, %1, %2, %3;" : "=r"(t) : "r"(q[2 * i + 1]), "r"(q[2 * i]), "r"(t));
    return t;
}

// The contraction's operand: codes less the token's centre c, the code that stands for zero (-z, or the nearest code when zero is
// outside the token's range), and z + c in the place of the zero-point, 0 for every token whose range holds zero.  So what
// the tensor cores sum is y / s, which has no part that the zero-point term would have to cancel.  Centred at the middle of the
// range instead, a token that lies to one side of zero lost what the sum of 2^(b-1) T rounds off: K = 4608, 2-bit weights, inputs of 4
// +- 0.1 behind a Hadamard rotation 4.1e-4 of the outputs' norm (uncentred on the CUDA cores 1.7e-5; so 3.2e-6), and a
// token of zeros did not give zeros.
template <int A_BITS>
struct Centre {
    lrq_f2::f32x2 back;           // from the rounding constant to the operand
    uint32_t lo, hi;              // the operand's ends, as pairs of bf16
    int c;
    __device__ __forceinline__ explicit Centre(float negz) {       // negz = -z, rounded to fp32
        constexpr float QMAX = (float)((1 << A_BITS) - 1);
        const float f = fminf(fmaxf(negz, 0.f), QMAX);
        back = lrq_f2::pack2(-12582912.f - f, -12582912.f - f);
        lo = __float_as_uint(-f) >> 16; lo |= lo << 16;            // whole numbers up to 256 are bf16 numbers
        hi = __float_as_uint(QMAX - f) >> 16; hi |= hi << 16;
        c = (int)f;
    }
};
// Two codes as the operand: clamp(rint(x), 0, 2^b - 1) - c, x = y / s - z.  Adding 1.5 * 2^23 rounds to an integer, ties to even,
// as cvt.rni does; every integer up to 256 is exactly a bf16 number, so the clamp can run on the packed result.
template <int A_BITS>
__device__ __forceinline__ uint32_t centred_bf16x2(lrq_f2::f32x2 x, const Centre<A_BITS>& ctr) {
    const lrq_f2::f32x2 MAGIC = lrq_f2::pack2(12582912.f, 12582912.f);
    float a, b;
    lrq_f2::unpack2(lrq_f2::add2(lrq_f2::add2(x, MAGIC), ctr.back), a, b);
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    asm("max.bf16x2 %0, %0, %1;" : "+r"(d) : "r"(ctr.lo));
    asm("min.bf16x2 %0, %0, %1;" : "+r"(d) : "r"(ctr.hi));
    return d;
}

// The same parameters for the fast kernel, where every warp works them out: one fp64 reciprocal refined
// from the fp32 approximation (two Newton steps, relative error below 1e-14) instead of fp64 divisions.
__device__ __forceinline__ TokenQ token_params_fast(float mn, float mx, int a_bits, int mode, double nrm,
                                                    float* scale_out, int32_t* zp_out) {
    const bool asym = mode == LRQ_ACT_ASYM;
    const double qsteps = asym ? (double)((1 << a_bits) - 1) : (double)((1 << (a_bits - 1)) - 1);
    // (mn > mx: a token without a number in it, whose range is empty in either mode)
    const double range = asym ? (double)mx - (double)mn : mn <= mx ? (double)fmaxf(fabsf(mn), fabsf(mx)) : 0.0;
    const float r0 = __frcp_rn((float)range);
    double s, inv;
    if (range > 0.0 && r0 > 0.f && r0 < 3.0e38f) {
        double r = (double)r0;
        r = fma(r, fma(-range, r, 1.0), r);
        r = fma(r, fma(-range, r, 1.0), r);
        inv = qsteps * r;
        s = range * (1.0 / qsteps);
    } else if (range > 0.0) {      // outside fp32's reciprocal range: plain division
        s = range / qsteps;
        inv = 1.0 / s;
    } else {                       // empty range: unit step in the normalised domain
        s = 1.0 / nrm;
        inv = nrm;
    }
    const double z = asym ? rint((double)mn * inv) : -(double)(1 << (a_bits - 1));
    *scale_out = (float)(s * nrm);
    *zp_out = (int32_t)z;
    TokenQ t;
    t.inv = (float)inv;
    t.negz = (float)(-z);
    return t;
}

// Step and zero-point of a token (Eq. 1) from its extremes, in fp32 with error-free corrections, for the common
// case; the fp64 routine takes over when the token's range is degenerate or when min/s comes within 2e-3 of a
// rounding boundary, so that the zero-point is always the one exact arithmetic gives.  The reciprocal step is
// refined from the hardware approximation against the exact range (max - min as an unevaluated sum hi + lo), which
// leaves it within an ulp of the correctly rounded value: the same accuracy as rounding the fp64 result.
// scale_mul = nrm / qsteps rounded to fp32.
template <int A_BITS>
__device__ __forceinline__ TokenQ token_params_f32(float mn, float mx, int mode, float scale_mul, double nrm,
                                                   float* scale_out, int32_t* zp_out) {
    const bool asym = mode == LRQ_ACT_ASYM;
    const float qs = asym ? (float)((1 << A_BITS) - 1) : (float)((1 << (A_BITS - 1)) - 1);
    float hi, lo;
    if (asym) {
        hi = mx - mn;                                          // TwoSum(mx, -mn): hi + lo is the exact range
        const float bv = hi - mx;
        lo = (mx - (hi - bv)) + (-mn - bv);
    } else {
        hi = fmaxf(fabsf(mn), fabsf(mx)); lo = 0.f;
    }
    if (hi > 1e-30f && hi < 1e30f) {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(hi));
        float inv = qs * r;
        float e = fmaf(-hi, inv, qs);
        e = fmaf(-lo, inv, e);
        inv = fmaf(e, r, inv);
        const float p = mn * inv, zr = rintf(p);
        if (!asym || fabsf(fabsf(p - zr) - 0.5f) > 2e-3f) {
            const float z = asym ? zr : -(float)(1 << (A_BITS - 1));
            *scale_out = hi * scale_mul;
            *zp_out = (int32_t)z;
            TokenQ t;
            t.inv = inv; t.negz = -z;
            return t;
        }
    }
    return token_params_fast(mn, mx, A_BITS, mode, nrm, scale_out, zp_out);
}

// Smoothing multipliers (Sec. 5.1) in shared memory, laid out so that threads which own runs of 4 * PER consecutive channels
// read them without conflicts: float4 i of thread j at i * tpt + j.  Read from global memory as they lie, a warp's 128-bit
// loads touched 32 lines each, once per token (32768 x 4608, B = 128: 227 us against 106 without multipliers, 139 now).
template <int PER>
__device__ __forceinline__ void stage_prescale(float4* ps, const float* __restrict__ prescale, int K, int tpt) {
    for (int q = threadIdx.x; q < (K >> 2); q += blockDim.x)
        ps[(q % PER) * tpt + q / PER] = __ldg(reinterpret_cast<const float4*>(prescale) + q);
}
template <int PER>
__device__ __forceinline__ void apply_prescale(lrq_f2::f32x2* P, const float4* ps, int j, int tpt) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const float4 f = ps[i * tpt + j];
        P[2 * i] = lrq_f2::mul2(P[2 * i], lrq_f2::pack2(f.x, f.y));
        P[2 * i + 1] = lrq_f2::mul2(P[2 * i + 1], lrq_f2::pack2(f.z, f.w));
    }
}

}  // namespace lrq_rq
