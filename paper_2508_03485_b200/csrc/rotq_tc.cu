// Rotation + per-token activation quantization (Sec. 4.2 Eq. 12, first case; Sec. 3.1 Eq. 1) for long batches and Hadamard blocks of
// 128, 2048 and 4096 channels: the first seven stages of the transform are a product on the tensor cores.
//
//   y = x . blockdiag(H_B),  H_B = H_(B/128) (x) H_128
//
// Inputs are bf16 numbers and H_128 is +-1, so every product is exact and the accumulator is the fp32 sum that butterflies make.  What
// bounds the CUDA-core kernels are the instructions of an element (11 for B = 128, 22 for B = 4096: shared-memory reads, unpacking,
// adds, exchanges); here a thread finds finished sums in TMEM, folds their extremes, and when the token's parameters are known reads
// them a second time and codes them: 3 instructions for B = 128.
//   * One persistent CTA per SM.  A warp brings steps of T whole tokens (up to 128 blocks of 128 channels) to a ring of stages by
//     TMA, one issues a step's eight MMAs, four groups of four warps take the steps in turn, each with an accumulator of 128
//     columns, so that one group's barriers and reductions lie under the others' arithmetic and a stage is free as soon
//     as its MMAs are done.
//   * B = 128 (ROWS): the tokens' blocks are the accumulator's lanes, the channels of a block its columns; a thread codes 128
//     consecutive channels.
//   * B >= 2048: channels are lanes and blocks columns, so that the remaining stages are butterflies between a thread's registers,
//     32 columns at a time; the results go back to TMEM.  Neighbouring lanes exchange halves to store 64 bytes of a block.
// Loops over 32 columns are kept rolled: with 128 values a thread in registers between the passes and everything unrolled (8 warps of
// 200 registers) the warps waited for instructions, 32768 x 4608 8-bit codes 107 us.  Measured, us before (rotq_blk.cu, rotq_big_kernel)
// and here: 32768 x 4608 B = 128 8-bit codes 107.5 -> 85 (5.3 TB/s), the operand 116.5 -> 112 (5.4); 32768 x 1152 33.7 -> 29.5, 35.7 ->
// 31.9; 4608 x 12288 B = 4096 codes 64.5 -> 46, the operand 72 -> 49; 4429 x 6144 B = 2048 34.5 -> 30.  It is bound by memory for
// B = 128 (0.82 of the copy rate in codes), by instructions and the latency of a step above.
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
constexpr int MAX_TOK = 32;                                  // tokens of a step, and more than its transform blocks of 2048 channels
constexpr int MAX_STAGES = 8;
constexpr int H_BYTES = 128 * 128 * 2;
constexpr size_t RING_BYTES = 168 * 1024;

struct __align__(16) Ctl {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES];
    uint64_t acc_full[BUFS], acc_empty[BUFS];
    uint32_t tmem_base;
    volatile int abort_flag;
    alignas(16) float4 par[GROUPS][MAX_TOK];                 // a token's parameters (make_code)
    float2 ext[GROUPS][GROUP_WARPS * MAX_TOK];               // extremes: [warp][token] over its rows of the token (ROWS), [warp][transform block] over its channels
    unsigned char none[GROUPS][GROUP_WARPS * MAX_TOK];       // ROWS: one of the rows has no numbers
};
constexpr size_t SMEM_MAX = 1024 + H_BYTES + RING_BYTES + sizeof(Ctl);
static_assert(SMEM_MAX <= 227 * 1024, "shared memory budget");

struct Params {
    int M, K, nb, T, steps, stages, mode, log2B, a_bits;
    uint32_t half_bytes;                                     // bytes of one 64-channel half of a stage
    uint8_t* codes; float* scale; int32_t* zp; int* status;
};

#define LRQ_I4(r, i) "r"(r[i]), "r"(r[i + 1]), "r"(r[i + 2]), "r"(r[i + 3])
#define LRQ_I8(r, i) LRQ_I4(r, i), LRQ_I4(r, i + 4)
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
                 "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 :: "r"(taddr), LRQ_I8(r, 0), LRQ_I8(r, 8), LRQ_I8(r, 16), LRQ_I8(r, 24) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Waits for this thread's TMEM loads; as operands, the loaded registers cannot be read ahead of it.
#define LRQ_W4(r, i) "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3])
#define LRQ_W8(r, i) LRQ_W4(r, i), LRQ_W4(r, i + 4)
__device__ __forceinline__ void tc_wait_ld32(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : LRQ_W8(r, 0), LRQ_W8(r, 8), LRQ_W8(r, 16), LRQ_W8(r, 24) :: "memory");
}

// Stages 7 .. 6 + LOGU of the transform over 32 blocks: butterflies between a thread's columns.
template <int LOGU>
__device__ __forceinline__ void butterflies(uint32_t* r) {
    f32x2 v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float a = __uint_as_float(r[2 * i]), b = __uint_as_float(r[2 * i + 1]);
        v[i] = pack2(a + b, a - b);
    }
#pragma unroll
    for (int h = 1; 2 * h < (1 << LOGU); h <<= 1)
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (!(i & h)) { const f32x2 a = v[i], b = v[i | h]; v[i] = add2(a, b); v[i | h] = sub2(a, b); }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        float a, b;
        unpack2(v[i], a, b);
        r[2 * i] = __float_as_uint(a); r[2 * i + 1] = __float_as_uint(b);
    }
}

// Barrier of a group's warps that also returns the OR of `pred`.
__device__ __forceinline__ bool group_bar_or(int id, bool pred) {
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 q, %1, 0;\nbar.red.or.pred p, %2, %3, q;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(r) : "r"((uint32_t)pred), "r"(id), "n"(GROUP_WARPS * 32) : "memory");
    return r != 0;
}

// How a token's values become codes.  fast: every value lies between the token's extremes, and both of these have their codes within
// 0 .. 2^b - 1 (and there is nothing else in the token): then no value needs the clamp, and y / s - z + 1.5 * 2^23, one fused
// multiply-add, is the code in the low bits of a float, rounded once (elsewhere y / s - z is rounded to fp32 first: of 2048 x 4608
// codes of 8 bits 47 were off the fp64 ones, 6 are now).  x: 1 / s, y: -z, z: from that float to the operand, w: 1.5 * 2^23 - z, or
// 0: not fast.
constexpr float MAGIC = 12582912.f;
__device__ __forceinline__ float4 make_code(TokenQ q, float mn, float mx, float qmax, bool plain) {
    const float c = fminf(fmaxf(q.negz, 0.f), qmax), w = MAGIC + q.negz;
    const float lo = fmaf(mn, q.inv, w) - MAGIC, hi = fmaf(mx, q.inv, w) - MAGIC;
    const bool fast = plain && fabsf(q.negz) < 1048576.f && lo >= 0.f && hi <= qmax;
    return make_float4(q.inv, q.negz, -MAGIC - c, fast ? w : 0.f);
}

__device__ __forceinline__ f32x2 pair_of(const uint32_t* r) { return pack2(__uint_as_float(r[0]), __uint_as_float(r[1])); }
// Two values -> the code floats (in the low bits), or for OUT16 the operand's.
template <bool OUT16>
__device__ __forceinline__ void code_fast(const uint32_t* r, const float4& q, uint32_t& a, uint32_t& b) {
    f32x2 v = fma2(pair_of(r), pack2(q.x, q.x), pack2(q.w, q.w));
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
__device__ __forceinline__ void code_row32(const uint32_t* r, const float4& q, bool fast, int a_bits, uint32_t* o) {
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
        if (a_bits == 8) {
            const Centre<8> ctr(q.y);
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = centred_bf16x2(fma2(pair_of(r + 2 * i), INV, NEGZ), ctr);
        } else {
            const Centre<4> ctr(q.y);
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = centred_bf16x2(fma2(pair_of(r + 2 * i), INV, NEGZ), ctr);
        }
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

// V blocks of one token (this lane's channel of each) -> the contraction's operand.  Neighbouring lanes swap halves, so that
// each stores two channels of one block as a word: 64 bytes of a block per store and half warp.
template <int V>
__device__ __forceinline__ void store16(const uint32_t* r, const float4& q, int a_bits, uint8_t* dst, int lane) {
    const uint32_t sel = lane & 1 ? 0x3276u : 0x5410u;
    uint8_t* d = dst + (lane & 1) * 256 + (lane >> 1) * 4;
    uint32_t h[V / 2];
    if (q.w != 0.f) {
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            uint32_t a, b;
            code_fast<true>(r + 2 * i, q, a, b);
            h[i] = upper_halves(a, b);
        }
    } else {
        const f32x2 INV = pack2(q.x, q.x), NEGZ = pack2(q.y, q.y);
        const Centre<8> c8(q.y);
        const Centre<4> c4(q.y);
#pragma unroll
        for (int i = 0; i < V / 2; ++i) h[i] = a_bits == 8 ? centred_bf16x2(fma2(pair_of(r + 2 * i), INV, NEGZ), c8) : centred_bf16x2(fma2(pair_of(r + 2 * i), INV, NEGZ), c4);
    }
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
        const uint32_t o = __shfl_xor_sync(0xffffffffu, h[i], 1);
        asm volatile("st.global.u32 [%0], %1;" :: "l"(d + 512 * i), "r"(lrq_dec::prmt(h[i], o, sel)) : "memory");
    }
}
// The same as codes: four blocks of four lanes (8-bit) or eight of eight (4-bit) are transposed by two or three exchanges.
template <int V, int A_BITS>
__device__ __forceinline__ void store_codes(const uint32_t* r, const float4& q, uint8_t* dst, int lane) {
    const bool fast = q.w != 0.f;
    uint32_t n[V];
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
        float x, y;
        unpack2(fma2(pair_of(r + 2 * i), pack2(q.x, q.x), fast ? pack2(q.w, q.w) : pack2(q.y, q.y)), x, y);
        n[2 * i] = __float_as_uint(x); n[2 * i + 1] = __float_as_uint(y);
    }
    if (!fast) {
#pragma unroll
        for (int i = 0; i < V; ++i) n[i] = (uint32_t)min(max(__float2int_rn(__uint_as_float(n[i])), 0), (1 << A_BITS) - 1);
    }
    auto halves = [&](uint32_t w, int m) { return lrq_dec::prmt(w, __shfl_xor_sync(0xffffffffu, w, m), lane & m ? 0x3276u : 0x5410u); };
    auto bytes = [&](uint32_t w, int m) { return lrq_dec::prmt(w, __shfl_xor_sync(0xffffffffu, w, m), lane & m ? 0x3715u : 0x6240u); };
    if (A_BITS == 8) {
        uint8_t* d = dst + (lane & 3) * 128 + (lane >> 2) * 4;
#pragma unroll
        for (int i = 0; i < V / 4; ++i)
            asm volatile("st.global.u32 [%0], %1;" :: "l"(d + 512 * i), "r"(halves(bytes(low_bytes(n[4 * i], n[4 * i + 1], n[4 * i + 2], n[4 * i + 3]), 1), 2)) : "memory");
    } else {
        uint8_t* d = dst + (lane & 7) * 64 + (lane >> 3) * 4;
#pragma unroll
        for (int i = 0; i < V / 8; ++i) {
            const uint32_t* c = n + 8 * i;
            const uint32_t w = bytes(halves(low_bytes(c[0] + (c[1] << 4), c[2] + (c[3] << 4), c[4] + (c[5] << 4), c[6] + (c[7] << 4)), 4), 2);
            const uint32_t o = __shfl_xor_sync(0xffffffffu, w, 1);
            const uint32_t v = lane & 1 ? ((o >> 4) & 0x0F0F0F0Fu) | (w & 0xF0F0F0F0u) : (w & 0x0F0F0F0Fu) | ((o & 0x0F0F0F0Fu) << 4);
            asm volatile("st.global.u32 [%0], %1;" :: "l"(d + 512 * i), "r"(v) : "memory");
        }
    }
}

// LOGU: log2 of the blocks of 128 channels that a transform block has.
template <int LOGU, int A_BITS, bool OUT16>
__global__ void __launch_bounds__(NUM_THREADS, 1)
rotq_tc_kernel(const __grid_constant__ CUtensorMap tmX, const Params p, const LrqExpand ex) {
    constexpr bool ROWS = LOGU == 0;
    constexpr int V = 1 << LOGU;             // columns of a transform block, whose extremes are folded together (not ROWS)
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    const uint32_t stage_bytes = 2 * p.half_bytes;
    const uint32_t sH = smem_u32(base), sX = sH + H_BYTES;
    Ctl* ctl = reinterpret_cast<Ctl*>(base + H_BYTES + (size_t)p.stages * stage_bytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&ctl->full[s]), 1); mbar_init(smem_u32(&ctl->empty[s]), 1); }
        for (int b = 0; b < BUFS; ++b) { mbar_init(smem_u32(&ctl->acc_full[b]), 1); mbar_init(smem_u32(&ctl->acc_empty[b]), GROUP_WARPS); }
        ctl->abort_flag = 0;
        mbar_init_fence();
        tma_prefetch_desc(&tmX);
    }
    // H_128 as a K-major operand, two halves of 64 k, 128-byte swizzle: H[r][k] = (-1)^popc(r & k)
    for (int i = threadIdx.x; i < H_BYTES / 16; i += NUM_THREADS) {
        const int h = i >> 10, r = (i >> 3) & 127, c = i & 7;
        // signs of eight k at once: row r & 7 of H_8, all turned when the upper bits of r and k have an odd number in common
        uint32_t m = (uint32_t)(0x963C5AF066CCAA00ull >> (8 * (r & 7))) & 0xFFu;
        if (__popc((r >> 3) & (8 * h + c)) & 1) m ^= 0xFFu;
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = 0x3F803F80u | ((m << (15 - 2 * j)) & 0x8000u) | ((m << (30 - 2 * j)) & 0x80000000u);
        *reinterpret_cast<uint4*>(base + h * (H_BYTES / 2) + r * 128 + ((c ^ (r & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
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
    if (warp >= TMA_WARP) {
        if (warp == TMA_WARP) {
            const bool lead = elect_one();
            int s = 0, issued = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (int i = 0; i < mine; ++i) {
                ok = mbar_wait_warp(smem_u32(&ctl->empty[s]), ph, &ctl->abort_flag, p.status, 51);
                if (!ok) break;
                if (lead) {
                    const int m0 = ((int)blockIdx.x + i * (int)gridDim.x) * p.T;
                    const uint32_t bar = smem_u32(&ctl->full[s]), dst = sX + s * stage_bytes;
                    mbar_arrive_expect_tx(bar, (uint32_t)(p.T * p.nb) * 256u);
                    tma_load_3d(dst, &tmX, 0, 0, m0, bar);
                    tma_load_3d(dst + p.half_bytes, &tmX, 64, 0, m0, bar);
                }
                __syncwarp();
                ++issued;
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            if (!ok && issued) {
                // copies in flight still write this CTA's shared memory: a millisecond to land before the CTA ends
                const long long t0 = clock64();
                while (clock64() - t0 < 2000000) __nanosleep(1000);
            }
            __syncwarp();
        } else if (warp == MMA_WARP) {
            const bool lead = elect_one();
            // rows: the tokens' blocks are the 128 lanes and the channels of a block the columns; otherwise the other way round
            const uint64_t h0 = umma_desc_sw128(sH, 16, 1024), x0 = umma_desc_sw128(sX, 16, 1024);
            const uint32_t idesc = umma_idesc_bf16(128, ROWS ? 128 : (p.T * p.nb + 15) / 16 * 16, false, false);
            const uint32_t half_units = p.half_bytes >> 4, stage_units = 2 * half_units;      // descriptors count 16 bytes
            int s = 0;
            uint32_t ph = 0;
            for (int i = 0; i < mine; ++i) {
                const int b = i % BUFS;
                if (!mbar_wait_warp(smem_u32(&ctl->acc_empty[b]), ((i / BUFS) & 1) ^ 1, &ctl->abort_flag, p.status, 52)) break;
                if (!mbar_wait_warp(smem_u32(&ctl->full[s]), ph, &ctl->abort_flag, p.status, 53)) break;
                tc_fence_after();
                const uint32_t d = tmem_base + b * COLS;
                const uint64_t x1 = x0 + (uint64_t)(s * stage_units), x2 = x1 + half_units, h1 = h0 + (H_BYTES / 2 >> 4);
                if (lead) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) tc_mma_f16(d, (ROWS ? x1 : h0) + 2 * k, (ROWS ? h0 : x1) + 2 * k, idesc, k ? 1u : 0u);
#pragma unroll
                    for (int k = 0; k < 4; ++k) tc_mma_f16(d, (ROWS ? x2 : h1) + 2 * k, (ROWS ? h1 : x2) + 2 * k, idesc, 1u);
                    tc_commit(smem_u32(&ctl->empty[s]));
                    tc_commit(smem_u32(&ctl->acc_full[b]));
                }
                __syncwarp();
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
            __syncwarp();
        }
    } else {
        const int g = warp / GROUP_WARPS, quad = warp % GROUP_WARPS, gt = threadIdx.x % (GROUP_WARPS * 32);
        const double nrm = 1.0 / sqrt((double)(1 << p.log2B));
        const int a_bits = OUT16 ? p.a_bits : A_BITS;
        const float qmax = (float)((1 << a_bits) - 1);
        constexpr int ES2 = OUT16 ? 4 : A_BITS / 4;          // half bytes of a result
        const int nb = p.nb, upt = ROWS ? 1 : nb / V;        // transform blocks of a token
        const size_t pitch = (size_t)p.K * ES2 / 2;
        // rows: the token of this thread's row (one past the last for rows that are none), the lanes of the warp that share it, and for
        // the thread that works out a token's parameters the warps that hold rows of it
        const int my_tok = ROWS ? min(gt / nb, p.T) : 0;
        const unsigned seg = ROWS ? __match_any_sync(0xffffffffu, my_tok) : 0u;
        const bool seg_first = ROWS && lane == __ffs(seg) - 1 && my_tok < p.T;
        const int w_first = (gt * nb) >> 5, w_last = (gt * nb + nb - 1) >> 5;
        float2* ext = ctl->ext[g];
        const float4* par = ctl->par[g];
        for (int i = g; i < mine; i += GROUPS) {
            const int m0 = ((int)blockIdx.x + i * (int)gridDim.x) * p.T, tokens = min(p.T, p.M - m0);
            const int b = i % BUFS;
            const uint32_t acc = tmem_base + ((uint32_t)(quad * 32) << 16) + b * COLS;
            const bool ok = mbar_wait_warp<32>(smem_u32(&ctl->acc_full[b]), (i / BUFS) & 1, &ctl->abort_flag, p.status, 54);
            tc_fence_after();
            const int cols = ROWS ? (quad * 32 < tokens * nb ? COLS : 0) : tokens * nb;      // of this warp's accumulator
            if constexpr (ROWS) {
                if (ok && cols) {
                    float mn4[4] = {INFINITY, INFINITY, INFINITY, INFINITY}, mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                    for (int c = 0; c < COLS; c += 32) {
                        uint32_t r[32];
                        tc_ld32(acc + c, r);
                        tc_wait_ld32(r);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            mn4[j & 3] = min3(mn4[j & 3], __uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                            mx4[j & 3] = max3(mx4[j & 3], __uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                        }
                    }
                    const float mn = fminf(min3(mn4[0], mn4[1], mn4[2]), mn4[3]), mx = fmaxf(max3(mx4[0], mx4[1], mx4[2]), mx4[3]);
                    float lo, hi;
                    asm volatile("redux.sync.min.f32 %0, %1, %2;" : "=f"(lo) : "f"(mn), "r"(seg));
                    asm volatile("redux.sync.max.f32 %0, %1, %2;" : "=f"(hi) : "f"(mx), "r"(seg));
                    const bool none = __any_sync(seg, !(mn <= mx));           // a row without numbers
                    if (seg_first) { ext[quad * MAX_TOK + my_tok] = make_float2(lo, hi); ctl->none[g][quad * MAX_TOK + my_tok] = none; }
                }
            } else {
#pragma unroll 1
                for (int c = 0; ok && c < cols; c += 32) {
                        uint32_t r[32];
                        tc_ld32(acc + c, r);
                        tc_wait_ld32(r);
                        butterflies<LOGU>(r);
                        tc_st32(acc + c, r);
#pragma unroll
                        for (int u = 0; u < 32; u += V) {
                            float mn = INFINITY, mx = -INFINITY;
#pragma unroll
                            for (int j = u; j < u + V; j += 2) {
                                mn = min3(mn, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
                                mx = max3(mx, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
                            }
                            asm volatile("redux.sync.min.f32 %0, %0, 0xffffffff;" : "+f"(mn));
                            asm volatile("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(mx));
                            if (lane == 0) ext[quad * MAX_TOK + (c + u) / V] = make_float2(mn, mx);
                        }
                }
                tc_wait_st();
            }
            if (group_bar_or(1 + g, !ok || ctl->abort_flag != 0)) break;      // the group's warps leave together
            if (gt < tokens) {
                float mn = INFINITY, mx = -INFINITY;
                bool none = false;
                auto fold = [&](float2 e) { mn = fminf(mn, e.x); mx = fmaxf(mx, e.y); none = none || !(e.x <= e.y); };
                if constexpr (ROWS) {
#pragma unroll 1
                    for (int w = w_first; w <= w_last; ++w) { fold(ext[w * MAX_TOK + gt]); none = none || ctl->none[g][w * MAX_TOK + gt]; }
                } else {
#pragma unroll 1
                    for (int u = gt * upt; u < (gt + 1) * upt; ++u)
#pragma unroll
                        for (int w = 0; w < GROUP_WARPS; ++w) fold(ext[w * MAX_TOK + u]);
                }
                // A NaN among a transform block's inputs is in all of its outputs.  Blocks of 128 channels: it is kept out of the token's range, as
                // rotq_blk.cu does for tokens of more than a warp; larger ones: it makes the range one, as in rotq_big_kernel.  A token
                // of nothing else has no range in either.
                const bool plain = !none && mn > -INFINITY && mx < INFINITY;
                if (none && (!ROWS || mn > mx)) { mx = NAN; if (mn == INFINITY) mn = NAN; }
                float sc; int32_t z;
                const TokenQ q = token_params_fast(mn, mx, a_bits, p.mode, nrm, &sc, &z);
                const float4 code = make_code(q, mn, mx, qmax, plain);
                ctl->par[g][gt] = code;
                p.scale[m0 + gt] = sc;
                p.zp[m0 + gt] = OUT16 ? z + (int)(-MAGIC - code.z) : z;
            }
            asm volatile("bar.sync %0, %1;" :: "r"(1 + g), "n"(GROUP_WARPS * 32) : "memory");
            if constexpr (ROWS) {
                if (cols) {
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
                            code_row32<A_BITS, OUT16>(r, q, fast, a_bits, o + h * W32);
                        }
                        if (live)
#pragma unroll
                            for (int j = 0; j < STEP / 32 * W32; j += 8) stg256(row + c * ES2 / 2 + 4 * j, o + j);
                    }
                }
            } else {
                uint8_t* dst = p.codes + (size_t)m0 * pitch + quad * 32 * ES2 / 2;
                int tok = 0, left = upt;
#pragma unroll 1
                for (int c = 0; c < cols; c += 32) {
                    uint32_t r[32];
                    tc_ld32(acc + c, r);
                    tc_wait_ld32(r);
#pragma unroll
                    for (int u = 0; u < 32; u += V)
                        if (c + u < cols) {
                            const float4 q = par[tok];
                            if constexpr (OUT16) store16<V>(r + u, q, a_bits, dst, lane);
                            else store_codes<V, A_BITS>(r + u, q, dst, lane);
                            dst += V * 128 * ES2 / 2;        // a row of the results ends where the next one starts
                            if (--left == 0) { left = upt; ++tok; }
                        }
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
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, BUFS * COLS);
    }
}

template <int LOGU, int A_BITS, bool OUT16>
lrq_status launch_tc(const CUtensorMap& tm, const Params& p, int grid, size_t smem, int dev, const LrqExpand& ex, cudaStream_t st) {
    auto kern = rotq_tc_kernel<LOGU, A_BITS, OUT16>;
    // the shared-memory opt-in is a per-device function attribute: set once per device and kernel variant, to the most it can need
    static std::mutex mu;
    static bool configured[LRQ_MAX_DEVICES] = {};
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!configured[dev]) {
            LRQ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
            configured[dev] = true;
        }
    }
    LRQ_CUDA_TRY(lrq_launch_pdl(kern, dim3(grid), dim3(NUM_THREADS), smem, st, tm, p, ex));
    return LRQ_OK;
}

}  // namespace

// Returns LRQ_ERR_UNSUPPORTED for calls this kernel does not take (the caller then uses the other kernels).  The line between them:
// its start (H_128, TMEM, the chain copy - product - two passes) costs 1 to 2 us more than theirs and its rate is 1.2 to 1.5 times
// theirs.  us there / here, operand with the decode of 1536 rows of weights: B = 128 4096 x 1152 10.8 / 11.4, 8192 x 1152 15.7 / 14.7,
// 1024 x 4608 13.3 / 13.3, 2048 x 4608 18.3 / 16.8, 4096 x 4608 25.6 / 22.3; B >= 2048 1024 x 6144 16.7 / 16.6, 2048 x 6144 22.4 / 21.4,
// 4096 x 2048 15.6 / 15.3 (codes 12.0 / 13.3), 1024 x 12288 27.5 / 25.2, 4096 x 4096 25.8 / 21.1.  Blocks of 256 to 1024 channels are
// no faster here (16384 x 1536 B = 512 36 / 39, 4608 x 3072 B = 1024 19.9 / 20.9): a column group's extremes cost as much as
// its butterflies.
lrq_status lrq_launch_rotq_tc(const void* X, int M, int K, long ldx, int B, int a_bits, int mode, int out16, const float* prescale,
                              uint8_t* codes, float* scale, int32_t* zp, const LrqExpand& ex, cudaStream_t st) {
    if (prescale || (B != 128 && B != 2048 && B != 4096) || K % 128 || K < COLS / MAX_TOK * 128 || K > 128 * COLS) return LRQ_ERR_UNSUPPORTED;
    if ((long)M * K < (B == 128 ? 9000000 : 12000000)) return LRQ_ERR_UNSUPPORTED;
    if ((ldx % 8) || !lrq_aligned(X, 16) || !lrq_aligned(codes, 32)) return LRQ_ERR_UNSUPPORTED;
    int dev = 0, sms = 0;
    if (lrq_current_device(&dev, &sms) != LRQ_OK) return LRQ_ERR_CUDA;
    Params p = {};
    const int nb = K / 128;
    p.M = M; p.K = K; p.nb = nb; p.mode = mode; p.a_bits = a_bits;
    while ((1 << p.log2B) < B) ++p.log2B;
    // Tokens per step: the groups' rounds of steps, each with the latency of some 40 columns' work besides its own
    long best = -1;
    for (int t = 1; t <= COLS / nb; ++t) {
        const long rounds = (((long)M + t - 1) / t + GROUPS * sms - 1) / (GROUPS * sms), cost = rounds * (t * nb + 40);
        if (best < 0 || cost < best) { best = cost; p.T = t; }
    }
    p.steps = (M + p.T - 1) / p.T;
    // rows that the products read: 128, or the columns in sixteens
    p.half_bytes = B == 128 ? 128 * 128 : (uint32_t)(p.T * nb + 15) / 16 * 16 * 128;
    const int fit = (int)(RING_BYTES / (2 * p.half_bytes));
    p.stages = fit < MAX_STAGES ? fit : MAX_STAGES;
    p.codes = codes; p.scale = scale; p.zp = zp; p.status = lrq_status_word();
    const size_t smem = 1024 + H_BYTES + (size_t)p.stages * 2 * p.half_bytes + sizeof(Ctl);
    const int grid = lrq_quant_grid(p.steps, sms, NUM_THREADS / 32, ex);
    CUtensorMap tm;
    if (!lrq_tma::make_map_blocks_bf16(&tm, X, (uint64_t)M, (uint64_t)nb, (uint64_t)ldx, (uint32_t)p.T)) return LRQ_ERR_UNSUPPORTED;
    const int form = p.log2B == 7 ? 0 : p.log2B == 11 ? 1 : 2;
    switch (form * 4 + (out16 ? 2 : 0) + (a_bits == 8)) {
        case 0: return launch_tc<0, 4, false>(tm, p, grid, smem, dev, ex, st);
        case 1: return launch_tc<0, 8, false>(tm, p, grid, smem, dev, ex, st);
        case 2: case 3: return launch_tc<0, 8, true>(tm, p, grid, smem, dev, ex, st);       // (of the operand, only the slow form asks for the bits)
        case 4: return launch_tc<4, 4, false>(tm, p, grid, smem, dev, ex, st);
        case 5: return launch_tc<4, 8, false>(tm, p, grid, smem, dev, ex, st);
        case 6: case 7: return launch_tc<4, 8, true>(tm, p, grid, smem, dev, ex, st);
        case 8: return launch_tc<5, 4, false>(tm, p, grid, smem, dev, ex, st);
        case 9: return launch_tc<5, 8, false>(tm, p, grid, smem, dev, ex, st);
        case 10: case 11: return launch_tc<5, 8, true>(tm, p, grid, smem, dev, ex, st);
    }
    return LRQ_ERR_UNSUPPORTED;
}
