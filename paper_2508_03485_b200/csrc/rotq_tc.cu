// Rotation + per-token activation quantization (Sec. 4.2 Eq. 12, first case; Sec. 3.1 Eq. 1) for long batches and Hadamard blocks of
// 128 channels: the first four stages of the transform are products on the tensor cores.
//
//   y = x . blockdiag(H_128),  H_128 = H_8 (x) H_16
//
// What bounds the CUDA-core kernel (rotq_blk.cu) are its 11.3 instructions an element and the chain of a step; here a thread finds the sums
// of H_16 in TMEM, adds the last three stages and folds the extremes, and when the token's parameters are known reads the results again
// and codes them: 8.9, issue slots 58 % busy.
//   * Inputs are bf16 numbers and H_16 is +-1: a sum is one MMA of exact products, which rounds (toward zero) only when inputs more than
//     twelve octaves apart meet.  All else is the arithmetic of rotq_blk.cu, so that a token's results differ from those in a short batch
//     by such a rounding at most.  The seven stages as eight chained MMAs, each rounding toward zero, were 2 us faster (32768 x 4608
//     codes) and up to 2.7 times as far from the exact sums (inputs over 16 octaves: steps 13.1e-8 off, rms, 4.8e-8 by butterflies and here).
//   * One persistent CTA per SM.  A warp brings steps of T whole tokens (up to 128 blocks of 128 channels) to a ring of stages by
//     TMA, one issues a step's eight MMAs, four groups of four warps take the steps in turn, each with an accumulator of 128
//     columns, so that one group's barriers and reductions lie under the others' arithmetic and a stage is free as soon
//     as its MMAs are done.
//   * The tokens' blocks are the accumulator's lanes, the channels of a block its columns, so that the last stages are between a
//     thread's registers and a thread codes 128 consecutive channels.
// Loops over 32 columns are kept rolled: with 128 values a thread in registers between the passes and everything unrolled (8 warps of
// 200 registers) the warps waited for instructions; 64 at a time, or two turns of 32 unrolled, gave nothing (86 -> 90, 86).
// 32768 x 4608, 8-bit codes: 106 us before (rotq_blk.cu), 83.6 here (5.4 TB/s, 0.83 of the copy rate).
// Blocks of 2048 and 4096 channels are not taken: their remaining stages need the channels of a block along the accumulator's lanes, so
// that all seven first ones had to be chained MMAs.  That was 1.1 to 1.4 times as fast as rotq_big_kernel, but its sums were 1.4 times as far
// from the exact ones, a token's codes changed with the length of its batch, and sums that overflowed in the later stages left NaN
// in the contraction's operand.
#include "lrq_internal.cuh"
#include "f32x2.cuh"
#include "rotq_common.cuh"
#include "tlq_decode.cuh"
#include "tc_ptx.cuh"
#include "tma_host.cuh"
#include <mutex>

namespace {
using namespace lrq_f2;
using namespace lrq_rq;
using namespace lrq_tc;

constexpr int GROUPS = 4, GROUP_WARPS = 4;                   // groups of four warps, one per quadrant of the TMEM lanes
constexpr int TMA_WARP = GROUPS * GROUP_WARPS, MMA_WARP = TMA_WARP + 1, NUM_THREADS = (TMA_WARP + 2) * 32;
constexpr int COLS = 128, BUFS = GROUPS;                     // columns of an accumulator; accumulators, one per group
constexpr int MIN_BLOCKS = 6, MAX_TOK = COLS / MIN_BLOCKS;   // blocks of a token at least, tokens of a step at most
constexpr int H_BYTES = 16 * 128;                            // H_16: 16 rows of a 128-byte swizzled operand, of which 32 bytes are used
constexpr uint32_t HALF_BYTES = 128 * 128, STAGE_BYTES = 2 * HALF_BYTES;     // 64 channels of 128 blocks; both halves
constexpr int STAGES = 6;

struct __align__(16) Ctl {
    uint64_t full[STAGES], empty[STAGES];
    uint64_t acc_full[BUFS], acc_empty[BUFS];
    uint64_t drain;                                          // the MMAs that an abandoned step left in flight
    uint32_t tmem_base;
    volatile int abort_flag;
    alignas(16) float4 par[GROUPS][MAX_TOK];                 // a token's parameters (make_code)
    float2 ext[GROUPS][GROUP_WARPS * MAX_TOK];               // extremes: [warp][token] over its rows of the token
    unsigned char nan[GROUPS][GROUP_WARPS * MAX_TOK];        // one of the rows has a NaN
};
constexpr size_t SMEM_BYTES = 1024 + H_BYTES + STAGES * STAGE_BYTES + sizeof(Ctl);
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");

struct Params {
    int M, K, nb, T, steps, mode;
    float scale_mul;                                         // token_params_f32
    uint8_t* codes; float* scale; int32_t* zp; int* status;
};

// Waits for this thread's TMEM loads; as operands, the loaded registers cannot be read ahead of it.
#define LRQ_W4(r, i) "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3])
#define LRQ_W8(r, i) LRQ_W4(r, i), LRQ_W4(r, i + 4)
__device__ __forceinline__ void tc_wait_ld32(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : LRQ_W8(r, 0), LRQ_W8(r, 8), LRQ_W8(r, 16), LRQ_W8(r, 24) :: "memory");
}

// Four consecutive columns of the warp's 32 TMEM lanes, loaded (not waited for) and stored.
__device__ __forceinline__ void tc_ld4(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_st4(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// The maximum of three, or NaN when one of them is.
__device__ __forceinline__ float max3_nan(float a, float b, float c) { float d; asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d; }

// Barrier of a group's warps that also returns the OR of `pred`.
__device__ __forceinline__ bool group_bar_or(int id, bool pred) {
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 q, %1, 0;\nbar.red.or.pred p, %2, %3, q;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(r) : "r"((uint32_t)pred), "r"(id), "n"(GROUP_WARPS * 32) : "memory");
    return r != 0;
}

// How a token's values become codes.  fast: every value lies between the token's extremes, and both of these have their codes within
// 0 .. 2^b - 1 (and there is nothing else in the token): then no value needs the clamp, and y / s - z, rounded to fp32, plus 1.5 * 2^23 is
// the code in the low bits of a float.  Either way a code is the same one, that of the other kernels, whatever tokens are beside it.
// x: 1 / s, y: -z, z: from that float to the operand, w: fast.
constexpr float MAGIC = 12582912.f;
__device__ __forceinline__ float4 make_code(TokenQ q, float mn, float mx, float qmax, bool plain) {
    const float c = fminf(fmaxf(q.negz, 0.f), qmax);
    const float lo = fmaf(mn, q.inv, q.negz) + MAGIC, hi = fmaf(mx, q.inv, q.negz) + MAGIC;
    return make_float4(q.inv, q.negz, -MAGIC - c, plain && lo >= MAGIC && hi <= MAGIC + qmax ? 1.f : 0.f);
}

__device__ __forceinline__ f32x2 pair_of(const uint32_t* r) { return pack2(__uint_as_float(r[0]), __uint_as_float(r[1])); }
// Two values -> the code floats (in the low bits), or for OUT16 the operand's.
template <bool OUT16>
__device__ __forceinline__ void code_fast(const uint32_t* r, const float4& q, uint32_t& a, uint32_t& b) {
    f32x2 v = add2(fma2(pair_of(r), pack2(q.x, q.x), pack2(q.y, q.y)), pack2(MAGIC, MAGIC));
    if (OUT16) v = add2(v, pack2(q.z, q.z));
    float x, y;
    unpack2(v, x, y);
    a = __float_as_uint(x); b = __float_as_uint(y);
}
// whole numbers up to 256: the upper half of the float is the bf16 number
__device__ __forceinline__ uint32_t upper_halves(uint32_t a, uint32_t b) { return lrq_dec::prmt(a, b, 0x7632u); }
__device__ __forceinline__ uint32_t low_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return lrq_dec::prmt(lrq_dec::prmt(a, b, 0x0040u), lrq_dec::prmt(c, d, 0x0040u), 0x5410u);
}

// 32 consecutive channels of a row -> codes (8-bit: 32 bytes, 4-bit: 16) or the operand (64 bytes).
template <int A_BITS, bool OUT16>
__device__ __forceinline__ void code_row32(const uint32_t* r, const float4& q, bool fast, uint32_t* o) {
    if (fast) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t x[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) code_fast<OUT16>(r + 8 * i + 2 * j, q, x[2 * j], x[2 * j + 1]);
            if (OUT16) {
#pragma unroll
                for (int j = 0; j < 4; ++j) o[4 * i + j] = upper_halves(x[2 * j], x[2 * j + 1]);
            } else if (A_BITS == 8) {
                o[2 * i] = low_bytes(x[0], x[1], x[2], x[3]);
                o[2 * i + 1] = low_bytes(x[4], x[5], x[6], x[7]);
            } else {
                o[i] = low_bytes(x[0] + (x[1] << 4), x[2] + (x[3] << 4), x[4] + (x[5] << 4), x[6] + (x[7] << 4));
            }
        }
        return;
    }
    const f32x2 INV = pack2(q.x, q.x), NEGZ = pack2(q.y, q.y);
    if constexpr (OUT16) {
        const Centre<A_BITS> ctr(q.y);
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = centred_bf16x2(fma2(pair_of(r + 2 * i), INV, NEGZ), ctr);
    } else {
        int n[32];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float x, y;
            unpack2(fma2(pair_of(r + 2 * i), INV, NEGZ), x, y);
            n[2 * i] = __float2int_rn(x); n[2 * i + 1] = __float2int_rn(y);
        }
        if (A_BITS == 8) {
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] = pack_u8x4(n[4 * i], n[4 * i + 1], n[4 * i + 2], n[4 * i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = pack_u4x8(n + 8 * i);
        }
    }
}
__device__ __forceinline__ void stg256(uint8_t* p, const uint32_t* o) {
    asm volatile("st.global.v8.u32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "l"(p), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]) : "memory");
}

// Bounded wait of the unwinding after an abort; what it waits for was issued long ago.
__device__ __forceinline__ void drain(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity) && clock64() - t0 < kWaitCycles / 8) {}
}

template <int A_BITS, bool OUT16>
__global__ void __launch_bounds__(NUM_THREADS, 1)
rotq_tc_kernel(const __grid_constant__ CUtensorMap tmX, const Params p, const LrqExpand ex) {
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    const uint32_t sH = smem_u32(base), sX = sH + H_BYTES;
    Ctl* ctl = reinterpret_cast<Ctl*>(base + H_BYTES + STAGES * STAGE_BYTES);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(smem_u32(&ctl->full[s]), 1); mbar_init(smem_u32(&ctl->empty[s]), 1); }
        for (int b = 0; b < BUFS; ++b) { mbar_init(smem_u32(&ctl->acc_full[b]), 1); mbar_init(smem_u32(&ctl->acc_empty[b]), GROUP_WARPS); }
        mbar_init(smem_u32(&ctl->drain), 1);
        ctl->abort_flag = 0;
        mbar_init_fence();
        tma_prefetch_desc(&tmX);
    }
    // H_16 as a K-major operand, 128-byte swizzle: H[r][k] = (-1)^popc(r & k)
    if (threadIdx.x < 32) {
        const int r = threadIdx.x >> 1, c = threadIdx.x & 1;
        // signs of eight k at once: row r & 7 of H_8, all turned in the lower right quarter
        uint32_t m = (uint32_t)(0x963C5AF066CCAA00ull >> (8 * (r & 7))) & 0xFFu;
        if ((r >> 3) & c) m ^= 0xFFu;
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = 0x3F803F80u | ((m << (15 - 2 * j)) & 0x8000u) | ((m << (30 - 2 * j)) & 0x80000000u);
        *reinterpret_cast<uint4*>(base + r * 128 + ((c ^ (r & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    fence_async_smem();
    if (warp == MMA_WARP) tmem_alloc(smem_u32(&ctl->tmem_base), BUFS * COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    lrq_pdl_trigger();
    lrq_pdl_wait();                      // X may be the previous kernel's output; the code buffer may still be read by it

    const int mine = (int)blockIdx.x < p.steps ? (p.steps - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;   // this CTA's steps
    bool lead = false;                   // the thread of the TMA or MMA warp that issues
    int issued = 0;                      // steps that it has issued
    if (warp >= TMA_WARP) {
        if (warp == TMA_WARP) {
            lead = elect_one();
            int s = 0;
            uint32_t ph = 1;
            for (int i = 0; i < mine; ++i) {
                if (!mbar_wait_warp(smem_u32(&ctl->empty[s]), ph, &ctl->abort_flag, p.status, 51)) break;
                if (lead) {
                    const int m0 = ((int)blockIdx.x + i * (int)gridDim.x) * p.T;
                    const uint32_t bar = smem_u32(&ctl->full[s]), dst = sX + s * STAGE_BYTES;
                    mbar_arrive_expect_tx(bar, (uint32_t)(p.T * p.nb) * 256u);
                    tma_load_3d(dst, &tmX, 0, 0, m0, bar);
                    tma_load_3d(dst + HALF_BYTES, &tmX, 64, 0, m0, bar);
                }
                __syncwarp();
                ++issued;
                if (++s == STAGES) { s = 0; ph ^= 1; }
            }
            __syncwarp();
        } else if (warp == MMA_WARP) {
            lead = elect_one();
            // the tokens' blocks are the 128 lanes, the channels of a block the columns
            const uint64_t h0 = umma_desc_sw128(sH, 16, 1024), x0 = umma_desc_sw128(sX, 16, 1024);
            const uint32_t idesc = umma_idesc_bf16(128, 16, false, false);
            int s = 0;
            uint32_t ph = 0;
            for (int i = 0; i < mine; ++i) {
                const int b = i % BUFS;
                if (!mbar_wait_warp(smem_u32(&ctl->acc_empty[b]), ((i / BUFS) & 1) ^ 1, &ctl->abort_flag, p.status, 52)) break;
                if (!mbar_wait_warp(smem_u32(&ctl->full[s]), ph, &ctl->abort_flag, p.status, 53)) break;
                tc_fence_after();
                const uint32_t d = tmem_base + b * COLS;
                const uint64_t x1 = x0 + (uint64_t)(s * (STAGE_BYTES >> 4));     // descriptors count 16 bytes
                if (lead) {
                    // sixteen channels each, into columns of their own
#pragma unroll
                    for (int c = 0; c < 8; ++c) tc_mma_f16(d + 16 * c, x1 + (c >> 2) * (HALF_BYTES >> 4) + 2 * (c & 3), h0, idesc, 0u);
                    tc_commit(smem_u32(&ctl->empty[s]));
                    tc_commit(smem_u32(&ctl->acc_full[b]));
                }
                __syncwarp();
                ++issued;
                if (++s == STAGES) { s = 0; ph ^= 1; }
            }
            __syncwarp();
        }
    } else {
        const int g = warp / GROUP_WARPS, quad = warp % GROUP_WARPS, gt = threadIdx.x % (GROUP_WARPS * 32);
        const double nrm = 1.0 / sqrt(128.0);
        constexpr float qmax = (float)((1 << A_BITS) - 1);
        constexpr int ES2 = OUT16 ? 4 : A_BITS / 4;          // half bytes of a result
        const int nb = p.nb;
        const size_t pitch = (size_t)p.K * ES2 / 2;
        // the token of this thread's row (one past the last for rows that are none), the lanes of the warp that share it, and for
        // the thread that works out a token's parameters the warps that hold rows of it
        const int my_tok = min(gt / nb, p.T);
        const unsigned seg = __match_any_sync(0xffffffffu, my_tok);
        const bool seg_first = lane == __ffs(seg) - 1 && my_tok < p.T;
        const int w_first = (gt * nb) >> 5, w_last = (gt * nb + nb - 1) >> 5;
        float2* ext = ctl->ext[g];
        const float4* par = ctl->par[g];
        for (int i = g; i < mine; i += GROUPS) {
            const int m0 = ((int)blockIdx.x + i * (int)gridDim.x) * p.T, tokens = min(p.T, p.M - m0);
            const int b = i % BUFS;
            const uint32_t acc = tmem_base + ((uint32_t)(quad * 32) << 16) + b * COLS;
            const bool ok = mbar_wait_warp<32>(smem_u32(&ctl->acc_full[b]), (i / BUFS) & 1, &ctl->abort_flag, p.status, 54);
            tc_fence_after();
            const bool busy = quad * 32 < tokens * nb;       // the warp has rows of a token
            if (ok && busy) {
                float mn4[4] = {INFINITY, INFINITY, INFINITY, INFINITY}, mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                // the last three stages: butterflies between the sums of the eight sixteens, four columns of each at a time
#pragma unroll 1
                for (int c = 0; c < 16; c += 4) {
                    uint32_t r[32];
#pragma unroll
                    for (int j = 0; j < 8; ++j) tc_ld4(acc + 16 * j + c, r + 4 * j);
                    tc_wait_ld32(r);
                    f32x2 v[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = pair_of(r + 2 * i);
#pragma unroll
                    for (int h = 2; h < 16; h <<= 1)
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (!(i & h)) { const f32x2 a = v[i], b = v[i | h]; v[i] = add2(a, b); v[i | h] = sub2(a, b); }
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        float x, y;
                        unpack2(v[i], x, y);
                        mn4[i & 3] = min3(mn4[i & 3], x, y);
                        mx4[i & 3] = max3_nan(mx4[i & 3], x, y);
                        r[2 * i] = __float_as_uint(x); r[2 * i + 1] = __float_as_uint(y);
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) tc_st4(acc + 16 * j + c, r + 4 * j);
                }
                tc_wait_st();
                float mn = fminf(min3(mn4[0], mn4[1], mn4[2]), mn4[3]), mx = max3_nan(max3_nan(mx4[0], mx4[1], mx4[2]), mx4[3], mx4[3]);
                const bool nan = mx != mx && my_tok < p.T;       // (rows that are none hold what was there)
                if (__any_sync(0xffffffffu, nan)) {
                    // it has no part in the range: once more without it
                    mx = -INFINITY;
#pragma unroll 1
                    for (int c = 0; c < COLS; c += 32) {
                        uint32_t r[32];
                        tc_ld32(acc + c, r);
                        tc_wait_ld32(r);
#pragma unroll
                        for (int j = 0; j < 16; ++j) mx = max3(mx, __uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                    }
                }
                float lo, hi;
                asm volatile("redux.sync.min.f32 %0, %1, %2;" : "=f"(lo) : "f"(mn), "r"(seg));
                asm volatile("redux.sync.max.f32 %0, %1, %2;" : "=f"(hi) : "f"(mx), "r"(seg));
                const bool any_nan = __any_sync(seg, nan);
                if (seg_first) { ext[quad * MAX_TOK + my_tok] = make_float2(lo, hi); ctl->nan[g][quad * MAX_TOK + my_tok] = any_nan; }
            }
            if (group_bar_or(1 + g, !ok || ctl->abort_flag != 0)) break;      // the group's warps leave together
            if (gt < tokens) {
                float mn = INFINITY, mx = -INFINITY;
                bool nan = false;
#pragma unroll 1
                for (int w = w_first; w <= w_last; ++w) {
                    const float2 e = ext[w * MAX_TOK + gt];
                    mn = fminf(mn, e.x); mx = fmaxf(mx, e.y);
                    nan = nan || ctl->nan[g][w * MAX_TOK + gt];
                }
                const bool plain = !nan && mn > -INFINITY && mx < INFINITY;
                if (mn > mx) mn = mx = NAN;          // a token of NaN alone: an empty range, as in rotq_blk.cu
                float sc; int32_t z;
                const TokenQ q = token_params_f32<A_BITS>(mn, mx, p.mode, p.scale_mul, nrm, &sc, &z);
                const float4 code = make_code(q, mn, mx, qmax, plain);
                ctl->par[g][gt] = code;
                p.scale[m0 + gt] = sc;
                p.zp[m0 + gt] = OUT16 ? z + (int)(-MAGIC - code.z) : z;
            }
            asm volatile("bar.sync %0, %1;" :: "r"(1 + g), "n"(GROUP_WARPS * 32) : "memory");
            if (busy) {
                const bool live = gt < tokens * nb;
                const float4 q = par[live ? my_tok : 0];
                const bool fast = __all_sync(0xffffffffu, q.w != 0.f);
                uint8_t* row = p.codes + (size_t)m0 * pitch + (size_t)gt * (128 * ES2 / 2);
                constexpr int W32 = 8 * ES2 / 2;         // words of 32 results
                constexpr int STEP = W32 >= 8 ? 32 : 64; // channels that fill a 256-bit store
#pragma unroll 1
                for (int c = 0; c < COLS; c += STEP) {
                    uint32_t o[STEP / 32 * W32];
#pragma unroll
                    for (int h = 0; h < STEP / 32; ++h) {
                        uint32_t r[32];
                        tc_ld32(acc + c + 32 * h, r);
                        tc_wait_ld32(r);
                        code_row32<A_BITS, OUT16>(r, q, fast, o + h * W32);
                    }
                    if (live)
#pragma unroll
                        for (int j = 0; j < STEP / 32 * W32; j += 8) stg256(row + c * ES2 / 2 + 4 * j, o + j);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
        }
    }
    __syncwarp();
    if (ex.out) lrq_dec::expand_share(ex);
    tc_fence_before();
    __syncthreads();
    if (ctl->abort_flag) {
        // A wait ran out, in whatever role, so that copies may still write this CTA's shared memory and MMAs its TMEM: both
        // end (bounded) before either is given back.  Otherwise every copy and MMA has been waited for above.
        if (lead && warp == TMA_WARP)
            for (int i = max(issued - STAGES, 0); i < issued; ++i) drain(smem_u32(&ctl->full[i % STAGES]), (uint32_t)(i / STAGES) & 1u);
        if (lead && warp == MMA_WARP && issued) {
            tc_commit(smem_u32(&ctl->drain));
            drain(smem_u32(&ctl->drain), 0);
        }
        __syncthreads();
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, BUFS * COLS);
    }
}

template <int A_BITS, bool OUT16>
lrq_status launch_tc(const CUtensorMap& tm, const Params& p, int grid, int dev, const LrqExpand& ex, cudaStream_t st) {
    auto kern = rotq_tc_kernel<A_BITS, OUT16>;
    // the shared-memory opt-in is a per-device function attribute: set once per device and kernel variant
    static std::mutex mu;
    static bool configured[LRQ_MAX_DEVICES] = {};
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!configured[dev]) {
            LRQ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES));
            configured[dev] = true;
        }
    }
    LRQ_CUDA_TRY(lrq_launch_pdl(kern, dim3(grid), dim3(NUM_THREADS), SMEM_BYTES, st, tm, p, ex));
    return LRQ_OK;
}

}  // namespace

// Returns LRQ_ERR_UNSUPPORTED for calls this kernel does not take (the caller then uses the other kernels).  The line between them, with
// us of rotq_blk.cu / here (L2 flushed): the start and the rounds of long steps cost 1 to 3 us, the rate is up to 1.5 times theirs.
//   codes, M * K >= 24 million and K >= 768: 20834 x 1152 21.5 / 20.1, 11719 x 2048 18.9 / 19.1, 7813 x 3072 20.0 / 18.9, 5209 x 4608 22.7 / 18.9,
//     2885 x 8320 (65 of a step's 128 lanes in use) 24.2 / 23.7, 32553 x 4608 105.4 / 77.1; below, 11285 x 1152 14.2 / 14.9, 6348 x 2048
//     12.9 / 14.7, 1547 x 6144 11.7 / 15.1; narrower, 62501 x 512 24.6 / 25.7.
//   the operand, where both are bound by what they write, M * K >= 30 million and only where the other kernel has five sub-groups an SM
//     or fewer: 26042 x 1152 30.4 / 29.1, 86806 x 1152 77.0 / 75.7, 19532 x 1536 32.5 / 28.9, 6511 x 4608 34.2 / 30.3, 32553 x 4608 115.8 / 111.1,
//     18029 x 8320 132.0 / 125.6, 2442 x 12288 40.5 / 36.4; its six to ten short sub-groups are as fast or faster: 48829 x 2048 69.0 / 76.7,
//     32553 x 3072 73.7 / 78.0, 24415 x 4096 72.3 / 76.5, 16277 x 6144 75.9 / 79.8 (but 17756 x 5632 81.5 / 77.3).
lrq_status lrq_launch_rotq_tc(const void* X, int M, int K, long ldx, int B, int a_bits, int mode, int out16, const float* prescale,
                              uint8_t* codes, float* scale, int32_t* zp, const LrqExpand& ex, cudaStream_t st) {
    if (prescale || B != 128 || K % 128 || K < MIN_BLOCKS * 128 || K > 128 * COLS) return LRQ_ERR_UNSUPPORTED;
    if ((long)M * K < (out16 ? 30000000 : 24000000) || (out16 && lrq_rotq_blk_subgroups(M, K) > 5)) return LRQ_ERR_UNSUPPORTED;
    if ((ldx % 8) || !lrq_aligned(X, 16) || !lrq_aligned(codes, 32)) return LRQ_ERR_UNSUPPORTED;
    int dev = 0, sms = 0;
    if (lrq_current_device(&dev, &sms) != LRQ_OK) return LRQ_ERR_CUDA;
    Params p = {};
    const int nb = K / 128;
    p.M = M; p.K = K; p.nb = nb; p.mode = mode;
    // Tokens per step: the groups' rounds of steps, each with the latency of some 40 rows' work besides its own
    long best = -1;
    for (int t = 1; t <= COLS / nb; ++t) {
        const long rounds = (((long)M + t - 1) / t + GROUPS * sms - 1) / (GROUPS * sms), cost = rounds * (t * nb + 40);
        if (best < 0 || cost < best) { best = cost; p.T = t; }
    }
    p.steps = (M + p.T - 1) / p.T;
    const double qsteps = mode == LRQ_ACT_ASYM ? (double)((1 << a_bits) - 1) : (double)((1 << (a_bits - 1)) - 1);
    p.scale_mul = (float)(1.0 / (sqrt((double)B) * qsteps));
    p.codes = codes; p.scale = scale; p.zp = zp; p.status = lrq_status_word();
    const int grid = lrq_quant_grid(p.steps, sms, NUM_THREADS / 32, ex);
    CUtensorMap tm;
    if (!lrq_tma::make_map_blocks_bf16(&tm, X, (uint64_t)M, (uint64_t)nb, (uint64_t)ldx, (uint32_t)p.T)) return LRQ_ERR_UNSUPPORTED;
    if (out16) return a_bits == 8 ? launch_tc<8, true>(tm, p, grid, dev, ex, st) : launch_tc<4, true>(tm, p, grid, dev, ex, st);
    return a_bits == 8 ? launch_tc<8, false>(tm, p, grid, dev, ex, st) : launch_tc<4, false>(tm, p, grid, dev, ex, st);
}
