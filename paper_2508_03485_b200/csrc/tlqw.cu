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
// What bounds it is the number of instructions.  Groups of more than 128 elements are not visited for every factor:
//   * a side's magnitudes are laid out in shared memory in ascending bins (of their bit patterns, so by a fraction of an
//     octave), with fp64 sums over every four of them.  A factor's codes change at nq magnitudes, so its error is a sum of
//     nq + 1 terms in the count and the sum of the elements above each, which takes a look at one bin per threshold;
//   * that error is off by fp64 roundings whose size is bounded, so a factor further than the bound from the smallest cannot
//     win; only when more than one factor is that close is the sum above taken, element by element.
// For shorter groups the bins cost as much as they save, and every factor's error is first summed in fp32, in any order: its
// relative error is bounded too (a few hundred roundings), and the rest is the same.  Common to both:
//   * a code is rint(l/s) - z in fp32; an element within the fp32 error of a rounding boundary (|x - rint x| > 1/2 - E, E
//     worked out from the candidate's range) takes the fp64 expression, a division, instead;
//   * levels have 8-bit significands: fp32 numbers, and the upper word of the double is the level.
// 31 factors a side, 4 bits: 4608 x 1152 545 us with the fp64 expression for every element and factor, 169 with fp32 sums over
// every element, 80 with bins; 2048 x 6144 485 and 122; 512 x 12288 685 and 96.  4608 x 1536 in groups of 128: 315 with fp32
// sums, 398 with bins; of 256 (4608 x 2048): 326 and 304.  These sums take two elements per instruction where there is one for it
// (four of the eleven an element): 3 bits, groups of 128, 303 -> 293.
#include "lrq_internal.cuh"
#include "f32x2.cuh"
#include <climits>
#include <type_traits>

namespace {

constexpr int kMaxGrid = 64;
constexpr int kChunk = 256;                        // source elements compacted at a time for the element-by-element sum
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

// log2 of a normal number to 2^-22 of max(1, |result|); minus infinity for a subnormal one, which fast_round does not call exact
__device__ __forceinline__ float log2_approx(float a) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// The same from fp32: x = l32 * inv + negz is within E of the exact l/s - z, with E = 2^-20 (max(1, |l|) / s + nq + 2): the
// logarithm is within 2^-22 of max(1, |l|), the reciprocal of the rounded step within 2^-22, the fused multiply-add rounds once
// (2^-24), all taken twice over.  `thr` = 1/2 - E; a candidate whose E is too large (E >= 1/2) always takes the fp64
// expression, and so does one whose z is not an fp32 integer, since then |l/s| is above 2^23.  The side's smallest element
// has the code rint(smin / s) - z = 0 and no element a lower one, so only the upper clamp of Eq. 5 is left to do.
constexpr float kMagic = 12582912.f;                // 1.5 * 2^23: adding it rounds to an integer, ties to even
struct __align__(16) FastCode { float inv, negz, thr, top; };
__device__ __forceinline__ FastCode fast_code(double s, double z, float lmax, int nq) {     // lmax >= max(1, |l|) of every element
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

// Bins of a side: bit patterns of its magnitudes above the smallest's, shifted so that the largest's falls below NB.
struct Bins { uint32_t base; int shift; };
template <int NB>
__device__ __forceinline__ Bins make_bins(float vmin, float vmax) {
    const uint32_t range = __float_as_uint(vmax) - __float_as_uint(vmin);
    const int top = 32 - __clz(range);
    return {__float_as_uint(vmin), max(0, top - (31 - __clz(NB)))};
}
__device__ __forceinline__ int bin_of(float a, const Bins& b) { return (int)((__float_as_uint(a) - b.base) >> b.shift); }

// Barrier over the warps of one side.
template <int WPS>
__device__ __forceinline__ void side_sync(int sd) {
    if (WPS == 1) __syncwarp();
    else if (sd) asm volatile("bar.sync 2, %0;" ::"n"(32 * WPS) : "memory");
    else asm volatile("bar.sync 1, %0;" ::"n"(32 * WPS) : "memory");
}

constexpr size_t binned_smem(int NB, int G) { return (size_t)2 * NB * 4 + (size_t)(G + 8) * 4 + (size_t)(G / 4 + 8) * 8; }

// WPS warps a side and NB bins (none: fp32 sums): one warp up to 256 elements, most of their work is per factor, not per
// element; two with 512 bins up to 2048 (4608 x 1152: 80 us; with one warp 106, with four 119); four with 1024 bins above,
// where a row's lists leave room for fewer CTAs (2048 x 6144: 122 us, with two warps 177).  `binned` is 0 when the lists do not
// fit in shared memory.
template <int WPS, int NB>
__global__ void __launch_bounds__(64 * WPS, 16 / WPS)
tlq_quantize_kernel(const float* __restrict__ W, int N, int K, int G, int bits, int I, ClipGrid grid, int pack3, int binned,
                    uint8_t* __restrict__ codes, float* __restrict__ levels, double* __restrict__ meta,
                    float* __restrict__ wsum) {
    constexpr int kThreads = 64 * WPS, kWarps = 2 * WPS;
    extern __shared__ __align__(16) unsigned char dyn[];       // both sides' bins, sums over fours, magnitudes
    __shared__ double epart[2][WPS][32], bpart[2][WPS][32];
    __shared__ int warp_count[2][WPS];
    __shared__ int cand_lev[2][9][32];             // level table of each lane's candidate, per side (upper word of the double)
    __shared__ float cand_f32[NB == 0 ? 2 : 1][NB == 0 ? 9 : 1][32];     // the same in fp32
    // a side's elements of one chunk, in increasing k: magnitude and its log2
    __shared__ __align__(16) float mag[2][kChunk];
    __shared__ __align__(16) float lg[2][kChunk];
    __shared__ FastCode best_fc[2];
    __shared__ unsigned ext[kWarps][2][2];         // [warp][side][max, ~min] of |w|, as bit patterns
    __shared__ int ext_cnt[kWarps][2];
    __shared__ Side best[2];
    __shared__ double T[16];
    __shared__ double red[kWarps];

    const int n = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = 1 << (bits - 1), nlev = 1 << bits, ngrp = K / G;
    // sum of each thread's codes; for the short groups in shared memory, since a register would be live across every search
    double kept = 0.0, *row_sum = &epart[0][0][0] + tid;
    if (NB == 0) *row_sum = 0.0;
    lrq_pdl_trigger();
    lrq_pdl_wait();                                // the weights may be the previous kernel's output

    for (int g = 0; g < ngrp; ++g) {
        const float* w = W + (size_t)n * K + (size_t)g * G;
        int* bins = reinterpret_cast<int*>(dyn);
        if (NB > 0 && binned)
            for (int i = tid; i < 2 * NB / 4; i += kThreads) reinterpret_cast<int4*>(bins)[i] = make_int4(0, 0, 0, 0);
        // ---- extremes of |w| per side (order does not matter for max / min, and log2 is monotone on fp32 numbers)
        auto pair_of = [&](int j) { return *reinterpret_cast<const float2*>(w + 2 * j); };
        {
            float amax[2] = {0.f, 0.f}, amin[2] = {INFINITY, INFINITY};
            int cnt[2] = {0, 0};
            for (int j = tid; j < G / 2; j += kThreads) {
                const float2 v2 = pair_of(j);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float v = e ? v2.y : v2.x, av = fabsf(v);
                    const bool neg = v < 0.f, pos = !neg && v != 0.f;
                    amax[0] = fmaxf(amax[0], neg ? 0.f : av); amax[1] = fmaxf(amax[1], neg ? av : 0.f);
                    amin[0] = fminf(amin[0], pos ? av : INFINITY); amin[1] = fminf(amin[1], neg ? av : INFINITY);
                    cnt[0] += pos; cnt[1] += neg;
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // magnitudes: the bit patterns are ordered as the numbers
                const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(amax[h])), mn = __reduce_min_sync(0xffffffffu, __float_as_uint(amin[h]));
                const int c = __reduce_add_sync(0xffffffffu, cnt[h]);
                if (lane == 0) { ext[warp][h][0] = mx; ext[warp][h][1] = ~mn; ext_cnt[warp][h] = c; }
            }
        }
        __syncthreads();
        unsigned top[2] = {0, 0}, low[2] = {0, 0};
        int cnts[2] = {0, 0};
#pragma unroll
        for (int i = 0; i < kWarps; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) { top[h] = max(top[h], ext[i][h][0]); low[h] = max(low[h], ext[i][h][1]); cnts[h] += ext_cnt[i][h]; }
        const float vmaxs[2] = {__uint_as_float(top[0]), __uint_as_float(top[1])};
        const float vmins[2] = {__uint_as_float(~low[0]), __uint_as_float(~low[1])};
        const int sd = warp / WPS, sw = warp % WPS;          // the warp's side and its place there; a lane is a factor
        const int nq = sd ? half : half - 1;       // highest code of the side = denominator of Eq. 6
        const float vmax = vmaxs[sd], vmin = vmins[sd];
        const int scnt = cnts[sd];
        int* side_bins = bins + sd * NB;
        double* side_sums = reinterpret_cast<double*>(dyn + 2 * NB * 4) + (sd ? (cnts[0] + 3) / 4 + 1 : 0);
        float* all_mags = reinterpret_cast<float*>(dyn + 2 * NB * 4 + (size_t)(G / 4 + 8) * 8);
        float* side_mags = all_mags + (sd ? (cnts[0] + 3) / 4 * 4 : 0);
        [[maybe_unused]] const Bins bn[2] = {make_bins<NB>(vmins[0], vmaxs[0]), make_bins<NB>(vmins[1], vmaxs[1])};
        double total = 0.0;
        if constexpr (NB > 0) if (binned) {
            // an element's bin, of both sides' 2 NB
            auto slot = [&](float v) {
                const bool neg = v < 0.f;
                return (neg ? NB : 0) + (int)(((__float_as_uint(v) & 0x7fffffffu) - (neg ? bn[1].base : bn[0].base)) >> (neg ? bn[1].shift : bn[0].shift));
            };
            for (int j = tid; j < G / 2; j += kThreads) {
                const float2 v = pair_of(j);
                if (fabsf(v.x) > 0.f) atomicAdd(&bins[slot(v.x)], 1);
                if (fabsf(v.y) > 0.f) atomicAdd(&bins[slot(v.y)], 1);
            }
            __syncthreads();
            // counts to starts, a run of bins per thread
            constexpr int RUN = NB / (32 * WPS);
            static_assert(RUN % 4 == 0, "");
            int4* run = reinterpret_cast<int4*>(side_bins + (sw * 32 + lane) * RUN);
            int c = 0;
#pragma unroll
            for (int i = 0; i < RUN / 4; ++i) { const int4 v = run[i]; c += v.x + v.y + v.z + v.w; }
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
            if (WPS > 1) {
                if (lane == 31) warp_count[sd][sw] = incl;
                side_sync<WPS>(sd);
            }
            int at = incl - c;
            for (int i = 0; i < sw; ++i) at += warp_count[sd][i];
#pragma unroll
            for (int i = 0; i < RUN / 4; ++i) {
                const int4 v = run[i];
                run[i] = make_int4(at, at + v.x, at + v.x + v.y, at + v.x + v.y + v.z);
                at += v.x + v.y + v.z + v.w;
            }
            __syncthreads();
            const int neg_at = (cnts[0] + 3) / 4 * 4;
            if (sw == 0 && lane < 3 && scnt + lane < (scnt + 3) / 4 * 4) side_mags[scnt + lane] = 0.f;       // the last four
            for (int j = tid; j < G / 2; j += kThreads) {    // afterwards a bin's entry is its end, the next one's start
                const float2 v = pair_of(j);
                if (fabsf(v.x) > 0.f) all_mags[atomicAdd(&bins[slot(v.x)], 1) + (v.x < 0.f ? neg_at : 0)] = fabsf(v.x);
                if (fabsf(v.y) > 0.f) all_mags[atomicAdd(&bins[slot(v.y)], 1) + (v.y < 0.f ? neg_at : 0)] = fabsf(v.y);
            }
            __syncthreads();
            if (sw == 0) {                                   // side_sums[i] = sum of the first 4 i magnitudes
                const int fours = (scnt + 3) / 4, each = (fours + 31) / 32;
                auto four = [&](int i) {
                    const float4 v = *reinterpret_cast<const float4*>(side_mags + 4 * i);
                    return ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w);
                };
                const int i0 = min(lane * each, fours), i1 = min(i0 + each, fours);
                double sum = 0.0;
                for (int i = i0; i < i1; ++i) sum += four(i);
                double run_sum = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const double v = __hiloint2double(__shfl_up_sync(0xffffffffu, __double2hiint(run_sum), o), __shfl_up_sync(0xffffffffu, __double2loint(run_sum), o));
                    if (lane >= o) run_sum += v;
                }
                double at_sum = run_sum - sum;               // any consistent value does: within the roundings allowed for
                for (int i = i0; i < i1; ++i) { side_sums[i] = at_sum; at_sum += four(i); }
                if (i0 < i1 && i1 == fours) side_sums[fours] = at_sum;
            }
            side_sync<WPS>(sd);
            total = scnt ? side_sums[(scnt + 3) / 4] : 0.0;
        }
        // ---- search of the clipping factor: lane c takes the c-th factor of the side's grid
        // both logarithms in one evaluation: even lanes take the maximum's, odd lanes the minimum's
        const double lx = log2((double)((lane & 1) ? vmin : vmax));
        const double smax = scnt ? shfl_double(lx, 0) : -INFINITY, smin = scnt ? shfl_double(lx, 1) : INFINITY;
        const float l_abs = scnt ? fmaxf(fmaxf(fabsf((float)smin), fabsf((float)smax)), 1.f) * 1.000001f : 1.f;
        const int ng = sd ? grid.nb : grid.na;
        // the thresholds below are relative to 2^-20: not for magnitudes all alike, nor for subnormal ones; a NaN is
        // counted and not binned
        const bool quick = NB > 0 && binned && ng <= 32 && side_bins[NB ? NB - 1 : 0] == scnt && vmin > 1e-37f && vmax < 1e37f && vmax > vmin * 1.001f;
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
            if constexpr (NB > 0) if (quick) {
                // error less the sum of the squares: sum over codes of n_q L_q^2 - 2 L_q S_q, by parts over the thresholds
                const int per = (nq + WPS - 1) / WPS, q0 = sw * per + 1, q1 = min(q0 + per, nq + 1);
                double e = 0.0, low = 0.0;
                auto level = [&](int q) { return ok ? __hiloint2double(level_word(__dmul_rn(s, __dadd_rn((double)q, z)), I), 0) : 0.0; };
                if (q0 < q1 || sw == 0) low = level(q0 - 1);
                if (sw == 0) e = low * fma((double)scnt, low, -2.0 * total);
#pragma unroll 1
                for (int q = q0; q < q1; ++q) {
                    const double L = level(q);
                    // magnitudes of code q and above start at 2^(s (z + q - 1/2)), here to 2^-21 of it
                    const double edge = s * (z + ((double)q - 0.5)), fl = floor(edge);
                    const int fi = (int)fmin(fmax(fl, -126.0), 127.0);
                    const float a0 = exp2f((float)(edge - fl)) * __int_as_float((fi + 127) << 23);
                    const float lo = a0 * 0.99999905f, hi = a0 * 1.00000095f;
                    int cnt = 0;
                    double sum = 0.0;
                    if (ok && lo <= vmax && edge < 127.0) {
                        const int kl = lo <= vmin ? 0 : bin_of(lo, bn[sd]), kh = hi <= vmin ? 0 : min(bin_of(hi, bn[sd]), NB - 1);
                        // fours that touch the edge's bins: what lies before them is smaller, what lies behind is larger
                        const int fours = (side_bins[kh] + 3) >> 2;
                        int maybe = 0;
                        for (int i = kl ? side_bins[kl - 1] >> 2 : 0; i < fours; ++i) {
                            const float4 v = *reinterpret_cast<const float4*>(side_mags + 4 * i);
                            const float a[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                maybe += a[h] >= lo;
                                if (a[h] >= hi) { ++cnt; sum += (double)a[h]; }
                            }
                        }
                        if (maybe != cnt)
                            for (int j = kl ? side_bins[kl - 1] & ~3 : 0; j < min(4 * fours, scnt); ++j) {
                                const float a = side_mags[j];
                                if (a >= lo && a < hi && side_code(a, s, z, nq) >= q) { ++cnt; sum += (double)a; }
                            }
                        cnt += scnt - min(4 * fours, scnt);
                        sum += total - side_sums[fours];
                    }
                    e += (L - low) * fma((double)cnt, L + low, -2.0 * sum);
                    low = L;
                }
                // roundings of the sums here and of the sum that defines the error: n of each, half an ulp, twice over
                epart[sd][sw][lane] = e;
                bpart[sd][sw][lane] = ((double)(scnt + 64)) * 4.5e-16 * ((double)scnt * ((double)vmax * (double)vmax + low * low) + 2.0 * low * total);
                side_sync<WPS>(sd);
                if (sw) continue;
#pragma unroll
                for (int i = 1; i < WPS; ++i) e += epart[sd][i][lane];
                double b = bpart[sd][0][lane];
#pragma unroll
                for (int i = 1; i < WPS; ++i) b = fmax(b, bpart[sd][i][lane]);
                // twice the largest bound, and the smallest error from the lanes that share its upper word
                const float bound = __uint_as_float(__reduce_max_sync(0xffffffffu, ok ? __float_as_uint((float)b * 2.001f) : 0u));
                const int key = ok ? lrq_ordered_int(__int_as_float(__double2hiint(e))) : INT_MAX, kmin = __reduce_min_sync(0xffffffffu, key);
                double emin = INFINITY;
                for (unsigned m = __ballot_sync(0xffffffffu, key == kmin); m; m &= m - 1) emin = fmin(emin, shfl_double(e, __ffs(m) - 1));
                const unsigned close = __ballot_sync(0xffffffffu, ok && !(e > emin + (double)bound));
                const bool fine = bound > 1e-30f && bound < 1e30f;         // below, fp32 does not hold it (0 would rule out every tie)
                if (fine && (close & (close - 1)) == 0) {
                    // one factor is left (or none is usable): the smallest error, whatever the rounding
                    if (close) {
                        const int src = __ffs(close) - 1;
                        best_s = shfl_double(s, src); best_z = shfl_double(z, src); best_f = shfl_double(fac, src);
                        found = true;
                    }
                    continue;
                }
            }
            if (sw) continue;
            __syncwarp();
            for (int q = 0; q <= nq; ++q) {
                const int hi = ok ? level_word(__dmul_rn(s, __dadd_rn((double)q, z)), I) : 0;
                cand_lev[sd][q][lane] = hi;
                if constexpr (NB == 0) cand_f32[sd][q][lane] = (float)__hiloint2double(hi, 0);
            }
            FastCode fc = fast_code(s, z, l_abs, nq);
            if (!ok) { fc.inv = 0.f; fc.negz = 0.f; fc.thr = 1.f; }                 // scored, but never looked at
            const uint32_t magic_off = __float_as_uint(kMagic) << 7;
            const uint32_t lev0 = (uint32_t)__cvta_generic_to_shared(&cand_lev[sd][0][lane]) - magic_off;
            [[maybe_unused]] const uint32_t f32_0 = (uint32_t)__cvta_generic_to_shared(&cand_f32[NB == 0 ? sd : 0][0][lane]) - magic_off;
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
                        lg[sd][at] = log2f(fabsf(v));          // finite for every element, subnormal ones too: `group` looks no further
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
            if constexpr (NB == 0) {
                // ---- every factor's error in fp32 (terms within 3 u of the exact ones, eight partial sums of at most
                // scnt / 8 + chunk remainders terms), which leaves the factors within twice its bound of the smallest
                using namespace lrq_f2;
                f32x2 part[4] = {0ull, 0ull, 0ull, 0ull};    // pairs: one instruction for two elements
                const f32x2 INV = pack2(fc.inv, fc.inv), NEGZ = pack2(fc.negz, fc.negz), MAGIC2 = pack2(kMagic, kMagic);
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
                        const f32x2 l[2] = {pack2(l4.x, l4.y), pack2(l4.z, l4.w)};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const f32x2 x = fma2(l[h], INV, NEGZ), rr = add2(x, MAGIC2);
                            float d0, d1;
                            unpack2(sub2(x, sub2(rr, MAGIC2)), d0, d1);
                            unpack2(rr, r[u + 2 * h], r[u + 2 * h + 1]);
                            off = max3(off, fabsf(d0), fabsf(d1));
                        }
                    }
                    if (off <= fc.thr) {
#pragma unroll
                        for (int u = 0; u < U; u += 4) {
                            const float4 a4 = *reinterpret_cast<const float4*>(&mag[sd][j + u]);
                            const f32x2 a[2] = {pack2(a4.x, a4.y), pack2(a4.z, a4.w)};
                            float L[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h)
                                asm("ld.shared.f32 %0, [%1];" : "=f"(L[h]) : "r"(f32_0 + (__float_as_uint(fminf(r[u + h], fc.top)) << 7)));
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const f32x2 d = sub2(a[h], pack2(L[2 * h], L[2 * h + 1]));
                                part[u / 2 + h] = fma2(d, d, part[u / 2 + h]);
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
                float ps[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) unpack2(part[i], ps[2 * i], ps[2 * i + 1]);
                const float e32 = (((ps[0] + ps[1]) + (ps[2] + ps[3])) + ((ps[4] + ps[5]) + (ps[6] + ps[7]))) + rest;
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
            }
            // ---- a near-tie (or a side the screen does not serve): the sum as it is defined, by one warp
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
        }
        if (sw == 0) {
            if (NB > 0 || !found) {                 // else the factor's lane has left it
                const FastCode f = fast_code(best_s, best_z, l_abs, nq);
                if (lane == 0) best_fc[sd] = f;
            }
            if (lane == 0) { best[sd].s = best_s; best[sd].z = best_z; best[sd].factor = best_f; }
        }
        __syncthreads();
        // ---- final level table of the group: entry u = c + half
        if (tid < nlev) {
            const int cc = tid - half;
            double v;
            const int sdc = cc < 0, q = sdc ? -cc : cc;
            v = cnts[sdc] ? __hiloint2double(level_word(__dmul_rn(best[sdc].s, __dadd_rn((double)q, best[sdc].z)), I), 0) : 0.0;
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
        // four lanes share eight codes, two elements each: the groups of 128 that grouped tables have keep every lane busy
        double part = 0.0;
        for (int j0 = 0; j0 < G / 2; j0 += kThreads) {
            const int j = j0 + tid;                  // pair of elements
            uint32_t word = 0;
            if (j < G / 2) {
                const float2 v2 = pair_of(j);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float v = e ? v2.y : v2.x;
                    int cc = 0;
                    if (v != 0.f) {
                        const bool neg = v < 0.f;
                        const FastCode f = best_fc[neg];
                        bool exact;
                        const float r = fast_round(log2_approx(fabsf(v)), f, exact);
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
        if (NB == 0) *row_sum += part; else kept += part;
        __syncthreads();                            // the tables are rewritten by the next group
    }
    double sum = NB == 0 ? *row_sum : kept;
#pragma unroll
    for (int o = 16; o; o >>= 1) sum += shfl_double(sum, lane ^ o);
    if (lane == 0) red[warp] = sum;
    __syncthreads();
    if (tid == 0) {
        for (int i = 1; i < kWarps; ++i) sum += red[i];
        wsum[n] = (float)sum;
    }
}

template <int WPS, int NB>
lrq_status launch(const float* W, int N, int K, int G, const lrq_tlq_params* p, const ClipGrid& grid, int pack3, uint8_t* codes, float* levels,
                  double* meta, float* wsum, cudaStream_t st) {
    constexpr size_t MAX_SMEM = 200 * 1024;
    const bool binned = NB > 0 && binned_smem(NB, G) <= MAX_SMEM;
    const size_t smem = binned ? binned_smem(NB, G) : 0;
    // the same limit whatever the length: with its own size here, a call could launch under the limit of another host thread's
    if (smem > 32 * 1024)
        LRQ_CUDA_TRY(cudaFuncSetAttribute(tlq_quantize_kernel<WPS, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MAX_SMEM));
    LRQ_CUDA_TRY(lrq_launch_pdl(tlq_quantize_kernel<WPS, NB>, dim3(N), dim3(64 * WPS), smem, st, W, N, K, G, p->w_bits, p->integerize_I, grid,
                                pack3, binned ? 1 : 0, codes, levels, meta, wsum));
    return LRQ_OK;
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
    const int pack3 = p->code_layout == LRQ_CODES_PACKED3 ? 1 : 0;
    return G <= 128 ? launch<1, 0>(W_rot, N, K, G, p, grid, pack3, codes, levels, meta, wsum, (cudaStream_t)cuda_stream)
         : G <= 256 ? launch<1, 128>(W_rot, N, K, G, p, grid, pack3, codes, levels, meta, wsum, (cudaStream_t)cuda_stream)
         : G <= 2048 ? launch<2, 512>(W_rot, N, K, G, p, grid, pack3, codes, levels, meta, wsum, (cudaStream_t)cuda_stream)
                    : launch<4, 1024>(W_rot, N, K, G, p, grid, pack3, codes, levels, meta, wsum, (cudaStream_t)cuda_stream);
}
