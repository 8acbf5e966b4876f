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

// Two codes as the contraction's bf16 operand: clamp(rint(x), 0, 2^b - 1) - C with C = 2^(b-1) (Eq. 1 before centring;
// x = y / s - z).  Adding 1.5 * 2^23 rounds to an integer, ties to even, as cvt.rni does; every integer up to 256 is
// exactly a bf16 number, so the clamp can run on the packed result.
template <int A_BITS>
__device__ __forceinline__ uint32_t centred_bf16x2(lrq_f2::f32x2 x) {
    constexpr float C = A_BITS == 8 ? 128.f : 8.f;
    const lrq_f2::f32x2 MAGIC = lrq_f2::pack2(12582912.f, 12582912.f), BACK = lrq_f2::pack2(-12582912.f - C, -12582912.f - C);
    float a, b;
    lrq_f2::unpack2(lrq_f2::add2(lrq_f2::add2(x, MAGIC), BACK), a, b);
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    asm("max.bf16x2 %0, %0, %1;" : "+r"(d) : "r"(A_BITS == 8 ? 0xC300C300u : 0xC100C100u));      // -128 / -8
    asm("min.bf16x2 %0, %0, %1;" : "+r"(d) : "r"(A_BITS == 8 ? 0x42FE42FEu : 0x40E040E0u));      // 127 / 7
    return d;
}

// The same parameters for the fast kernel, where every warp works them out: one fp64 reciprocal refined
// from the fp32 approximation (two Newton steps, relative error below 1e-14) instead of fp64 divisions.
__device__ __forceinline__ TokenQ token_params_fast(float mn, float mx, int a_bits, int mode, double nrm,
                                                    float* scale_out, int32_t* zp_out) {
    const bool asym = mode == LRQ_ACT_ASYM;
    const double qsteps = asym ? (double)((1 << a_bits) - 1) : (double)((1 << (a_bits - 1)) - 1);
    const double range = asym ? (double)mx - (double)mn : (double)fmaxf(fabsf(mn), fabsf(mx));
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
