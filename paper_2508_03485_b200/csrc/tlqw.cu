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
// What bounds it is the number of instructions per element and factor:
//   * every factor's error is first summed in fp32, in any order.  That sum's relative error
//     is bounded (a few hundred roundings), so a factor further than twice the bound from the smallest cannot win; only
//     when more than one factor is that close is the sum above taken in fp64, for about one row in fifty;
//   * the code is rint(l/s) - z in fp32, from log2f; an element within the fp32 error of a rounding boundary
//     (|x - rint x| > 1/2 - E, E worked out from the candidate's range) takes the fp64 expression, a division, instead;
//   * levels have 8-bit significands: fp32 numbers, and the upper word of the double is the level;
//   * a side's elements are compacted into shared memory kChunk source elements at a time and read as broadcasts.
// 4608 x 1152, 4 bits, 31 factors a side: 545 us with the fp64 expression for every element and factor, 157 now;
// 4608 x 1536, 3 bits, groups of 128: 1086 and 315.
#include "lrq_internal.cuh"
#include <climits>
#include <type_traits>

namespace {

constexpr int kMaxGrid = 64;
constexpr int kThreads = 64;
constexpr int kChunk = 256;                        // source elements compacted at a time
struct ClipGrid { double a[kMaxGrid]; double b[kMaxGrid]; int na, nb; };

// (out of line, as the next one: both are rarely reached and long, and this kernel has to stay in the instruction cache)
__device__ __noinline__ double level_value(double e, int I) {
    // Eqs. 8-9: 2^e ~ II * 2^(f-I) with f = floor(e), II = rint(2^(e-f) * 2^I)
    const double f = floor(e);
    const double II = rint(exp2(__dsub_rn(e, f)) * (double)(1 << I));      // the factor is a power of two: exact
    const int x = (int)f - I;
    if (x >= -1000 && x <= 1000) return II * __hiloint2double((1023 + x) << 20, 0);   // a product with a power of two: exact
    return ldexp(II, x);
}

// code of Eq. 5 on one side: clamp(rint(l / s) - z, 0, nq), l = log2(a)
__device__ __noinline__ int side_code(float a, double s, double z, int nq) {
    return (int)fmin(fmax(__dsub_rn(rint(__ddiv_rn(log2((double)a), s)), z), 0.0), (double)nq);
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

struct Side { double s, z, factor; };

__global__ void __launch_bounds__(kThreads, 16)
tlq_quantize_kernel(const float* __restrict__ W, int N, int K, int G, int bits, int I, ClipGrid grid, int pack3,
                    uint8_t* __restrict__ codes, float* __restrict__ levels, double* __restrict__ meta,
                    float* __restrict__ wsum) {
    __shared__ int cand_lev[2][9][32];             // level table of each lane's candidate, per side (upper word of the double)
    __shared__ float cand_f32[2][9][32];           // the same in fp32
    // a side's elements of one chunk, in increasing k: magnitude and its log2
    __shared__ __align__(16) float mag[2][kChunk];
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
        // both logarithms in one evaluation: even lanes take the maximum's, odd lanes the minimum's
        const double lx = log2((double)((lane & 1) ? vmin : vmax));
        const double smax = scnt ? shfl_double(lx, 0) : -INFINITY, smin = scnt ? shfl_double(lx, 1) : INFINITY;
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
            for (int q = 0; q <= nq; ++q) {
                const int hi = ok ? level_word(__dmul_rn(s, __dadd_rn((double)q, z)), I) : 0;
                cand_lev[sd][q][lane] = hi;
                cand_f32[sd][q][lane] = (float)__hiloint2double(hi, 0);
            }
            FastCode fc = fast_code(s, z, l_abs, nq);
            if (!ok) { fc.inv = 0.f; fc.negz = 0.f; fc.thr = 1.f; }                 // scored, but never looked at
            const uint32_t magic_off = __float_as_uint(kMagic) << 7;
            const uint32_t lev0 = (uint32_t)__cvta_generic_to_shared(&cand_lev[sd][0][lane]) - magic_off;
            const uint32_t f32_0 = (uint32_t)__cvta_generic_to_shared(&cand_f32[sd][0][lane]) - magic_off;
            __syncwarp();
            // the side's elements among w[k0 .. k0 + kChunk), in increasing k, into the warp's list; returns how many
            auto fill = [&](int k0) {
                int n_el = 0;
                __syncwarp();
#pragma unroll
                for (int u = 0; u < kChunk / 32; ++u) {
                    if (k0 + 32 * u >= G) break;
                    const int k = k0 + 32 * u + lane;
                    const float v = k < G ? w[k] : 0.f;
                    const bool mine = sd ? (v < 0.f) : (v > 0.f);
                    const unsigned m = __ballot_sync(0xffffffffu, mine);
                    if (mine) {
                        const int at = n_el + __popc(m & ((1u << lane) - 1u));
                        mag[sd][at] = fabsf(v);
                        lg[sd][at] = log2f(fabsf(v));
                    }
                    n_el += __popc(m);
                }
                __syncwarp();
                return n_el;
            };
            auto code_of = [&](int j) {                         // one element, whatever its distance from a boundary
                bool exact;
                const float r = fast_round(lg[sd][j], fc, exact);
                return exact ? r : kMagic + (float)side_code(mag[sd][j], s, z, nq);
            };
            // ---- every factor's error in fp32 (terms within 3 u of the exact ones, eight partial sums of at most
            // scnt / 8 + chunk remainders terms), which leaves the factors within twice its bound of the smallest
            float part[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            float rest = 0.f;
            auto term = [&](int j, float r) {
                float L;
                asm("ld.shared.f32 %0, [%1];" : "=f"(L) : "r"(f32_0 + (__float_as_uint(r) << 7)));
                const float d = mag[sd][j] - L;
                rest = fmaf(d, d, rest);
            };
            auto group = [&](int j, auto U_) {
                constexpr int U = decltype(U_)::value;
                float r[U], off = 0.f;               // the distances from an integer are looked at together
#pragma unroll
                for (int u = 0; u < U; u += 4) {
                    const float4 l4 = *reinterpret_cast<const float4*>(&lg[sd][j + u]);
                    const float l[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const float x = fmaf(l[h], fc.inv, fc.negz);
                        r[u + h] = x + kMagic;
                        off = fmaxf(off, fabsf(x - (r[u + h] - kMagic)));
                    }
                }
                if (off <= fc.thr) {
#pragma unroll
                    for (int u = 0; u < U; u += 4) {
                        const float4 a4 = *reinterpret_cast<const float4*>(&mag[sd][j + u]);
                        const float a[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            float L;
                            asm("ld.shared.f32 %0, [%1];" : "=f"(L) : "r"(f32_0 + (__float_as_uint(fminf(r[u + h], fc.top)) << 7)));
                            const float d = a[h] - L;
                            part[u + h] = fmaf(d, d, part[u + h]);
                        }
                    }
                } else {
#pragma unroll 1
                    for (int u = 0; u < U; ++u) term(j + u, code_of(j + u));
                }
            };
            for (int k0 = 0; k0 < G; k0 += kChunk) {
                const int n_el = fill(k0);
                int j = 0;
                for (; j + 8 <= n_el; j += 8) group(j, std::integral_constant<int, 8>());
                if (j + 4 <= n_el) { group(j, std::integral_constant<int, 4>()); j += 4; }
#pragma unroll 1
                for (; j < n_el; ++j) term(j, code_of(j));
            }
            float e32;
            {
                e32 = (((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]))) + rest;
            }
            // errors are not negative, so their bit patterns are ordered as the numbers; NaN sorts above them all
            const float emin = __uint_as_float(__reduce_min_sync(0xffffffffu, ok ? __float_as_uint(e32) : 0x7fffffffu));
            const float eps = (float)(scnt / 8 + 3 * (G / kChunk + 1) + 64) * 2.4e-7f;      // 4 u per term of the longest sum
            const unsigned close = __ballot_sync(0xffffffffu, ok && e32 <= emin * (1.f + eps));
            const bool safe = ng <= 32 && emin > 1e-27f && emin < 1e30f && eps < 0.5f && vmax < 1e18f;
            if (safe && (close & (close - 1)) == 0) {
                // one factor is left: the smallest error, whatever the rounding
                const int src = __ffs(close) - 1;
                best_s = shfl_double(s, src); best_z = shfl_double(z, src); best_f = shfl_double(fac, src);
                if (lane == src) best_fc[sd] = fc;
                found = true;
                continue;
            }
            // ---- a near-tie (or sums out of fp32's range): the sum as it is defined
            double err = 0.0;
            for (int k0 = 0; k0 < G; k0 += kChunk) {
                const int n_el = fill(k0);
auto level = [&](float r) {
                    int hi;
                    asm("ld.shared.b32 %0, [%1];" : "=r"(hi) : "r"(lev0 + (__float_as_uint(r) << 7)));
                    return __hiloint2double(hi, 0);
                };
                int j = 0;
                for (; j + 4 <= n_el; j += 4) {
                    // four look-ups in flight: one element after the other, a row that lands here would be the last to finish
                    bool all = true;
                    float r[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) { bool exact; r[u] = fast_round(lg[sd][j + u], fc, exact); all &= exact; }
                    if (!all) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) r[u] = code_of(j + u);
                    }
                    double d[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) d[u] = __dsub_rn((double)mag[sd][j + u], level(r[u]));
#pragma unroll
                    for (int u = 0; u < 4; ++u) err = __dadd_rn(err, __dmul_rn(d[u], d[u]));
                }
#pragma unroll 1
                for (; j < n_el; ++j) { const double d = __dsub_rn((double)mag[sd][j], level(code_of(j))); err = __dadd_rn(err, __dmul_rn(d, d)); }
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
            const int sdc = cc < 0, q = sdc ? -cc : cc;
            v = (sdc ? ncnt : pcnt) ? __hiloint2double(level_word(__dmul_rn(best[sdc].s, __dadd_rn((double)q, best[sdc].z)), I), 0) : 0.0;
            if (sdc) v = -v;
            T[tid] = v;
            levels[((size_t)n * ngrp + g) * nlev + tid] = (float)v;
        }
        if (tid == 0 && meta) {
            double* mt = meta + ((size_t)n * ngrp + g) * 6;
            mt[0] = best[0].s; mt[1] = best[0].z; mt[2] = best[1].s; mt[3] = best[1].z;
            mt[4] = best[0].factor; mt[5] = best[1].factor;
        }
        __syncthreads();
        // ---- codes, eight to a 32-bit word (of nibbles, or three bytes of packed 3-bit codes)
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
                                            : side_code(fabsf(v), best[neg].s, best[neg].z, neg ? half : half - 1);
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
