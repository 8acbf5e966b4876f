// Twin-log weight quantization with search-based clipping (Sec. 4.1, Eqs. 4-9).
//
// Offline step.  One CTA of two warps per output row walks the row's groups.  The search of Eq. 6 is a
// comparison of sums of squared errors, and near-ties between two clipping factors do occur (two factors that
// give the same codes and differ only in the lowest level): which one wins then depends on how the fp64 sum
// was rounded.  The sum is therefore taken exactly as its definition reads - over the side's elements in
// increasing k, one add after another, products and sums rounded separately - and the parallelism is across
// candidates instead of across elements: warp 0 scores the positive side, warp 1 the negative side, each lane
// one clipping factor of the caller's grid, all lanes walking over the same elements.  Every decision (codes,
// chosen factor) is the one fp64 arithmetic with explicitly rounded operations gives.
//
// What bounds it is the number of instructions per element and factor, so nothing but the three operations of the sum
// itself is left in fp64 there:
//   * the code is rint(l/s) - z in fp32, from log2f, two elements per instruction; an element within the fp32 error of a rounding boundary
//     (|x - rint x| > 1/2 - E, E worked out from the candidate's range) takes the fp64 expression, a division, instead;
//   * levels have 8-bit significands, so the upper word of the double is the level: 32-bit look-ups;
//   * a side's elements are compacted into shared memory CHUNK source elements at a time and read as broadcasts.
// 4608 x 1152, 4 bits, 31 factors a side: 545 us with fp64 codes and elements handed round by shuffles, 164 now;
// 4608 x 1536, 3 bits, groups of 128: 1086 and 380.
#include "lrq_internal.cuh"
#include "f32x2.cuh"
#include <climits>

namespace {

constexpr int kMaxGrid = 64;
constexpr int kThreads = 64;
constexpr int kChunk = 256;                        // source elements compacted at a time
struct ClipGrid { double a[kMaxGrid]; double b[kMaxGrid]; int na, nb; };

__device__ __forceinline__ double level_value(double e, int I) {
    // Eqs. 8-9: 2^e ~ II * 2^(f-I) with f = floor(e), II = rint(2^(e-f) * 2^I)
    const double f = floor(e);
    const double II = rint(exp2(__dsub_rn(e, f)) * (double)(1 << I));      // the factor is a power of two: exact
    const int x = (int)f - I;
    if (x >= -1000 && x <= 1000) return II * __hiloint2double((1023 + x) << 20, 0);   // a product with a power of two: exact
    return ldexp(II, x);
}

// code of Eq. 5 on one side: clamp(rint(l / s) - z, 0, nq), l = log2 of the magnitude
__device__ __forceinline__ int side_code(double l, double s, double z, int nq) {
    return (int)fmin(fmax(__dsub_rn(rint(__ddiv_rn(l, s)), z), 0.0), (double)nq);
}

__device__ __forceinline__ double shfl_double(double v, int src) {
    return __hiloint2double(__shfl_sync(0xffffffffu, __double2hiint(v), src), __shfl_sync(0xffffffffu, __double2loint(v), src));
}

// The upper word of a level's double (its 8 significant bits fit there), from fp32: exp2f is within 2 ulp, so II is what the
// fp64 expression gives unless 2^(e-f) * 2^I comes within 2e-4 of a rounding boundary, which takes that expression.
__device__ __forceinline__ int level_word(double e, int I) {
    const double f = floor(e);
    const float x = exp2f((float)__dsub_rn(e, f)) * (float)(1 << I), r = rintf(x);
    const int fi = (int)f;
    if (fabsf(x - r) < 0.4998f && fi > -900 && fi < 900) return (int)(__float_as_uint(r) >> 3) + 0x38000000 + (fi - I) * (1 << 20);
    return __double2hiint(level_value(e, I));
}

// The same from fp32: x = l32 * inv + negz is within E of the exact l/s - z, with E = 2^-20 (max|l| / s + nq + 2): log2f is
// within an ulp of l (2^-23 of |l/s|), the reciprocal of the rounded step within 2^-22, the fused multiply-add rounds once
// (2^-24), all taken more than twice over.  `thr` = 1/2 - E; a candidate whose E is too large (E >= 1/2) always takes the fp64
// expression, and so does one whose z is not an fp32 integer, since then |l/s| is above 2^23.  The side's smallest element
// has the code rint(smin / s) - z = 0 and no element a lower one, so only the upper clamp of Eq. 5 is left to do.
constexpr float kMagic = 12582912.f;                // 1.5 * 2^23: adding it rounds to an integer, ties to even
struct FastCode { float inv, negz, thr, top; };
__device__ __forceinline__ FastCode fast_code(double s, double z, float lmax, int nq) {     // lmax >= |l| of every element
    FastCode f;
    f.inv = 1.0f / (float)s;
    f.negz = (float)-z;
    const float e = 9.5367431640625e-7f * (lmax * f.inv + (float)nq + 2.0f);
    f.thr = e < 0.5f && f.inv > 0.f ? (0.5f - e) * 0.999999f : -1.f;
    f.top = kMagic + (float)nq;
    return f;
}
// The code in the low bits of the returned float; `exact` is false for a NaN or an out-of-range x as well.
__device__ __forceinline__ float fast_round(float l32, const FastCode& f, bool& exact) {
    const float x = fmaf(l32, f.inv, f.negz), r = x + kMagic;
    exact = fabsf(x - (r - kMagic)) <= f.thr;
    return fminf(r, f.top);
}

using namespace lrq_f2;

struct Side { double s, z, factor; };

__global__ void __launch_bounds__(kThreads, 16)
tlq_quantize_kernel(const float* __restrict__ W, int N, int K, int G, int bits, int I, ClipGrid grid, int pack3,
                    uint8_t* __restrict__ codes, float* __restrict__ levels, double* __restrict__ meta,
                    float* __restrict__ wsum) {
    __shared__ int cand_lev[2][9][32];             // level table of each lane's candidate, per side (upper word of the double)
    // a side's elements of one chunk, in increasing k: magnitude and its log2
    __shared__ __align__(16) double mag[2][kChunk];
    __shared__ __align__(16) float lg[2][kChunk];
    __shared__ FastCode best_fc[2];
    __shared__ float ext[2][2][2];                 // [warp][side][max, min] of |w|
    __shared__ int ext_cnt[2][2];
    __shared__ Side best[2];
    __shared__ double T[16];
    __shared__ double red[2];

    const int n = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = 1 << (bits - 1), nlev = 1 << bits, ngrp = K / G;
    double row_sum = 0.0;                          // meaningful in thread 0
    lrq_pdl_trigger();
    lrq_pdl_wait();                                // the weights may be the previous kernel's output

    for (int g = 0; g < ngrp; ++g) {
        const float* w = W + (size_t)n * K + (size_t)g * G;
        // ---- extremes of |w| per side (order does not matter for max / min, and log2 is monotone on fp32 numbers)
        float amax[2] = {0.f, 0.f}, amin[2] = {INFINITY, INFINITY};
        int cnt[2] = {0, 0};
        for (int k = tid; k < G; k += kThreads) {
            const float v = w[k];
            if (v != 0.f) {
                const int sd = v < 0.f;
                const float av = fabsf(v);
                if (sd) { amax[1] = fmaxf(amax[1], av); amin[1] = fminf(amin[1], av); cnt[1]++; }
                else { amax[0] = fmaxf(amax[0], av); amin[0] = fminf(amin[0], av); cnt[0]++; }
            }
        }
#pragma unroll
        for (int sd = 0; sd < 2; ++sd) {
            // magnitudes: the bit patterns are ordered as the numbers
            const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(amax[sd])), mn = __reduce_min_sync(0xffffffffu, __float_as_uint(amin[sd]));
            const int c = __reduce_add_sync(0xffffffffu, cnt[sd]);
            if (lane == 0) { ext[warp][sd][0] = __uint_as_float(mx); ext[warp][sd][1] = __uint_as_float(mn); ext_cnt[warp][sd] = c; }
        }
        __syncthreads();
        // ---- search of the clipping factor: warp `sd` owns side sd, lane c the c-th factor of that side's grid
        const int sd = warp;
        const int nq = sd ? half : half - 1;       // highest code of the side = denominator of Eq. 6
        const float vmax = fmaxf(ext[0][sd][0], ext[1][sd][0]), vmin = fminf(ext[0][sd][1], ext[1][sd][1]);
        const int scnt = ext_cnt[0][sd] + ext_cnt[1][sd];
        const double smax = scnt ? log2((double)vmax) : -INFINITY, smin = scnt ? log2((double)vmin) : INFINITY;
        const float l_abs = scnt ? fmaxf(fabsf((float)smin), fabsf((float)smax)) * 1.000001f : 0.f;
        const int ng = sd ? grid.nb : grid.na;
        double best_err = INFINITY, best_s = 1.0, best_z = 0.0, best_f = 1.0;
        bool found = false;
        for (int c0 = 0; c0 < ng; c0 += 32) {
            const int c = c0 + lane;
            bool ok = false;
            double s = 1.0, z = 0.0, fac = 1.0;
            if (c < ng && scnt > 0 && nq > 0) {
                fac = sd ? grid.b[c] : grid.a[c];
                const double top = __dmul_rn(fac, smax), bot = smin;
                if (top > bot) {
                    s = __ddiv_rn(__dsub_rn(top, bot), (double)nq);
                    z = rint(__ddiv_rn(bot, s));
                    ok = true;
                }
            }
            __syncwarp();
            for (int q = 0; q <= nq; ++q)
                cand_lev[sd][q][lane] = ok ? level_word(__dmul_rn(s, __dadd_rn((double)q, z)), I) : 0;
            FastCode fc = fast_code(s, z, l_abs, nq);
            if (!ok) { fc.inv = 0.f; fc.negz = 0.f; fc.thr = 1.f; }                 // scored, but never looked at
            const uint32_t lev0 = (uint32_t)__cvta_generic_to_shared(&cand_lev[sd][0][lane]) - (__float_as_uint(kMagic) << 7);
            __syncwarp();
            // the side's elements in increasing k, one chunk at a time
            double err = 0.0;
            for (int k0 = 0; k0 < G; k0 += kChunk) {
                int n_el = 0;
#pragma unroll
                for (int u = 0; u < kChunk / 32; ++u) {
                    if (k0 + 32 * u >= G) break;
                    const int k = k0 + 32 * u + lane;
                    const float v = k < G ? w[k] : 0.f;
                    const bool mine = sd ? (v < 0.f) : (v > 0.f);
                    const unsigned m = __ballot_sync(0xffffffffu, mine);
                    if (mine) {
                        const int at = n_el + __popc(m & ((1u << lane) - 1u));
                        mag[sd][at] = (double)fabsf(v);
                        lg[sd][at] = log2f(fabsf(v));
                    }
                    n_el += __popc(m);
                }
                __syncwarp();
                auto level = [&](float r) {
                    int hi;
                    asm("ld.shared.b32 %0, [%1];" : "=r"(hi) : "r"(lev0 + (__float_as_uint(r) << 7)));
                    return __hiloint2double(hi, 0);
                };
                auto careful = [&](int j) {                     // one element, whatever its distance from a boundary
                    const double a = mag[sd][j];
                    bool exact;
                    float r = fast_round(lg[sd][j], fc, exact);
                    if (!exact) r = kMagic + (float)side_code(log2(a), s, z, nq);
                    const double d = __dsub_rn(a, level(r));
                    err = __dadd_rn(err, __dmul_rn(d, d));
                };
                constexpr int U = 8;
                const f32x2 INV = pack2(fc.inv, fc.inv), NEGZ = pack2(fc.negz, fc.negz), MAGIC = pack2(kMagic, kMagic);
                int j = 0;
                for (; j + U <= n_el; j += U) {
                    // two elements per instruction; the eight distances from an integer are looked at together
                    float r[U], off = 0.f;
#pragma unroll
                    for (int u = 0; u < U; u += 4) {
                        const float4 l4 = *reinterpret_cast<const float4*>(&lg[sd][j + u]);
#pragma unroll
                        for (int h = 0; h < 4; h += 2) {
                            const f32x2 x = fma2(h ? pack2(l4.z, l4.w) : pack2(l4.x, l4.y), INV, NEGZ), m = add2(x, MAGIC);
                            float d0, d1;
                            unpack2(sub2(x, sub2(m, MAGIC)), d0, d1);
                            off = max3(off, fabsf(d0), fabsf(d1));
                            unpack2(m, r[u + h], r[u + h + 1]);
                        }
                    }
                    if (off <= fc.thr) {
                        double d[U];
#pragma unroll
                        for (int u = 0; u < U; u += 2) {
                            const double2 a = *reinterpret_cast<const double2*>(&mag[sd][j + u]);
                            d[u] = __dsub_rn(a.x, level(fminf(r[u], fc.top)));
                            d[u + 1] = __dsub_rn(a.y, level(fminf(r[u + 1], fc.top)));
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) err = __dadd_rn(err, __dmul_rn(d[u], d[u]));
                    } else {
#pragma unroll 1
                        for (int u = 0; u < U; ++u) careful(j + u);
                    }
                }
#pragma unroll 1
                for (; j < n_el; ++j) careful(j);
                __syncwarp();
            }
            // first minimum in grid order: the smallest error, the lowest index among equals
            double e = ok ? err : INFINITY;
            int idx = ok ? c : INT_MAX;
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                const double e2 = shfl_double(e, lane ^ o);
                const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
                if (e2 < e || (e2 == e && i2 < idx)) { e = e2; idx = i2; }
            }
            if (idx != INT_MAX && e < best_err) {  // a later pass replaces the best only when strictly smaller
                const int src = idx - c0;
                best_err = e;
                best_s = shfl_double(s, src); best_z = shfl_double(z, src); best_f = shfl_double(fac, src);
                if (lane == src) best_fc[sd] = fc;
                found = true;
            }
        }
        if (!found) {                               // no usable range: unit step anchored at the smallest element
            best_s = 1.0; best_z = scnt ? rint(smin) : 0.0; best_f = 1.0;
            if (lane == 0) best_fc[sd] = fast_code(best_s, best_z, l_abs, nq);
        }
        if (lane == 0) { best[sd].s = best_s; best[sd].z = best_z; best[sd].factor = best_f; }
        __syncthreads();
        // ---- final level table of the group: entry u = c + half
        const int pcnt = ext_cnt[0][0] + ext_cnt[1][0], ncnt = ext_cnt[0][1] + ext_cnt[1][1];
        if (tid < nlev) {
            const int cc = tid - half;
            double v;
            if (cc > 0) v = pcnt ? level_value(__dmul_rn(best[0].s, __dadd_rn((double)cc, best[0].z)), I) : 0.0;
            else if (cc < 0) v = ncnt ? -level_value(__dmul_rn(best[1].s, __dadd_rn((double)(-cc), best[1].z)), I) : 0.0;
            else v = pcnt ? level_value(__dmul_rn(best[0].s, best[0].z), I) : 0.0;
            T[tid] = v;
            levels[((size_t)n * ngrp + g) * nlev + tid] = (float)v;
        }
        if (tid == 0 && meta) {
            double* mt = meta + ((size_t)n * ngrp + g) * 6;
            mt[0] = best[0].s; mt[1] = best[0].z; mt[2] = best[1].s; mt[3] = best[1].z;
            mt[4] = best[0].factor; mt[5] = best[1].factor;
        }
        __syncthreads();
        // ---- codes, eight to a 32-bit word ( of nibbles, or three bytes of packed 3-bit codes)
        double part = 0.0;
        const FastCode fcs[2] = {best_fc[0], best_fc[1]};
        // four lanes share eight codes, two elements each: the groups of 128 that grouped tables have keep every lane busy
        for (int j0 = 0; j0 < G / 2; j0 += kThreads) {
            const int j = j0 + tid;                  // pair of elements
            uint32_t word = 0;
            if (j < G / 2) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float v = w[2 * j + e];
                    int cc = 0;
                    if (v != 0.f) {
                        const bool neg = v < 0.f;
                        FastCode f;
                        f.inv = neg ? fcs[1].inv : fcs[0].inv; f.negz = neg ? fcs[1].negz : fcs[0].negz;
                        f.thr = neg ? fcs[1].thr : fcs[0].thr; f.top = neg ? fcs[1].top : fcs[0].top;
                        bool exact;
                        const float r = fast_round(log2f(fabsf(v)), f, exact);
                        const int q = exact ? (int)(__float_as_uint(r) - __float_as_uint(kMagic))
                                            : side_code(log2((double)fabsf(v)), best[neg].s, best[neg].z, neg ? half : half - 1);
                        cc = neg ? -q : q;
                    }
                    const int u = cc + half;
                    part += T[u];
                    word |= (uint32_t)u << ((pack3 ? 3 : 4) * (2 * (tid & 3) + e));
                }
            }
            word |= __shfl_xor_sync(0xffffffffu, word, 1);
            word |= __shfl_xor_sync(0xffffffffu, word, 2);
            if ((tid & 3) == 0 && j < G / 2) {
                if (pack3) {
                    uint8_t* dst = codes + ((size_t)n * K + (size_t)g * G) / 8 * 3 + (size_t)3 * (j >> 2);
                    dst[0] = (uint8_t)word; dst[1] = (uint8_t)(word >> 8); dst[2] = (uint8_t)(word >> 16);
                } else {
                    *reinterpret_cast<uint32_t*>(codes + ((size_t)n * K + (size_t)g * G) / 2 + (size_t)4 * (j >> 2)) = word;
                }
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) part += shfl_double(part, lane ^ o);
        if (lane == 0) red[warp] = part;
        __syncthreads();
        if (tid == 0) row_sum += red[0] + red[1];
        __syncthreads();
    }
    if (tid == 0) wsum[n] = (float)row_sum;
}

}  // namespace

extern "C" lrq_status lrq_tlq_quantize_weights(const float* W_rot, int N, int K, const lrq_tlq_params* p,
                                               uint8_t* codes, float* levels, double* meta, float* wsum,
                                               void* workspace, size_t workspace_bytes, void* cuda_stream) {
    (void)workspace; (void)workspace_bytes;
    if (!W_rot || !p || !codes || !levels || !wsum || N <= 0 || K <= 0) return LRQ_ERR_INVALID_ARG;
    if (!p->alpha || !p->beta) return LRQ_ERR_INVALID_ARG;
    if (!lrq_aligned(W_rot, 16) || !lrq_aligned(codes, 4) || !lrq_aligned(levels, 4)) return LRQ_ERR_INVALID_ARG;
    const int G = p->group_size > 0 ? p->group_size : K;
    if (p->w_bits < 2 || p->w_bits > 4) return LRQ_ERR_UNSUPPORTED;
    if (p->integerize_I < 1 || p->integerize_I > 7) return LRQ_ERR_UNSUPPORTED;
    if (p->n_alpha < 1 || p->n_alpha > kMaxGrid || p->n_beta < 1 || p->n_beta > kMaxGrid) return LRQ_ERR_UNSUPPORTED;
    if (K % G || G % 8 || (K & 1)) return LRQ_ERR_UNSUPPORTED;
    if (p->code_layout != LRQ_CODES_NIBBLE && p->code_layout != LRQ_CODES_PACKED3) return LRQ_ERR_INVALID_ARG;
    if (p->code_layout == LRQ_CODES_PACKED3 && p->w_bits != 3) return LRQ_ERR_UNSUPPORTED;
    ClipGrid grid;
    grid.na = p->n_alpha; grid.nb = p->n_beta;
    for (int i = 0; i < kMaxGrid; ++i) {
        grid.a[i] = i < grid.na ? p->alpha[i] : 0.0;
        grid.b[i] = i < grid.nb ? p->beta[i] : 0.0;
    }
    LRQ_CUDA_TRY(lrq_launch_pdl(tlq_quantize_kernel, dim3(N), dim3(kThreads), 0, (cudaStream_t)cuda_stream, W_rot, N, K, G, p->w_bits,
                                p->integerize_I, grid, p->code_layout == LRQ_CODES_PACKED3 ? 1 : 0, codes, levels, meta, wsum));
    return LRQ_OK;
}
