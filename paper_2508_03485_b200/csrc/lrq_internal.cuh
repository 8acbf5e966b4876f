// Internal declarations shared by the translation units of the CUDA library.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include "../../include/lrq.h"

#define LRQ_CUDA_TRY(expr)                                   \
    do {                                                     \
        cudaError_t e__ = (expr);                            \
        if (e__ != cudaSuccess) { (void)cudaGetLastError(); return LRQ_ERR_CUDA; } \
    } while (0)

static inline bool lrq_is_pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }
static inline bool lrq_aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
static inline size_t lrq_round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

#include <cuda.h>

struct lrq_layer {
    int N, K, w_bits, group;          // group == K for per-channel tables
    int packed3;                      // 1: codes are true 3-bit packed (8 codes in 3 bytes, row pitch 3K/8 bytes)
    const uint8_t* codes;
    const float* levels;
    const float* wsum;
    const float* wscale;
    const float* bias;
    lrq_act_params act;
    // what does not change from call to call, prepared once by lrq_layer_create (read-only afterwards, so
    // concurrent calls on one layer need no lock): TMA descriptors of the weight codes for the two tile widths
    // of the tensor-core contraction.  have_tm_w is false when the shape takes the CUDA-core kernel, or when no
    // driver was present at creation (the launch then encodes the descriptors itself).
    bool have_tm_w;
    CUtensorMap tm_w_wide, tm_w_narrow;
};

constexpr int LRQ_MAX_DEVICES = 64;

// Current device and its SM count (queried once per device, thread-safe).
lrq_status lrq_current_device(int* dev, int* sms);

// Device status word: written by a kernel whose bounded wait expired.  A file-scope device variable of the
// library image; this returns its address on the current device.
int* lrq_status_word();

// Launch with programmatic stream serialization: the kernel may become resident while its predecessor in the
// stream is still draining; it must execute lrq_pdl_wait() before its first access to global memory.
template <typename... KArgs, typename... Args>
inline cudaError_t lrq_launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                  Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// A layer's weight decode (codes -> bf16 [N,K] at `out`, tlq_decode.cuh), done by the quantizer kernels' warps when they have no
// tokens left: the two are independent, and a launch of its own costs three microseconds on a short batch.  out ==
// nullptr: nothing to decode.  fmt: 4, 3, 2 nibble layout, 13 packed 3-bit.
struct LrqExpand {
    const uint8_t* codes; const float* levels; int N, K, G, fmt; void* out;
    // a row's shares (tlq_decode.cuh): the row itself, or with grouped tables runs of up to 32 / 2^bits words of eight codes a lane
    __host__ __device__ int segments() const {
        const int most = 32 << (fmt == 4 ? 1 : fmt == 2 ? 3 : 2);
        return G == K ? 1 : (K / 8 + most - 1) / most;
    }
};

// CTAs of a quantizer grid: `need` for its tokens, or more (up to `resident`) when there are weight rows for them.
static inline int lrq_quant_grid(int need, int resident, int warps_per_cta, const LrqExpand& ex) {
    int g = need < resident ? need : resident;
    if (ex.out) {
        const long want = g + ((long)ex.N * ex.segments() + warps_per_cta - 1) / warps_per_cta;
        g = want < resident ? (int)want : resident;
    }
    return g;
}

// Quantizers: out16 == 0 writes packed 8- or 4-bit codes, out16 == 1 the contraction's operand instead, bf16 [M,K] of
// the codes less the token's centre c (rotq_common.cuh; 16-byte aligned rows), from the same arithmetic, and z + c in zp.
// rotq.cu
lrq_status lrq_launch_rotq_hadamard(const void* X, int M, int K, long ldx, int B, int a_bits, int mode, int out16, const float* prescale,
                                    uint8_t* codes, float* scale, int32_t* zp, const LrqExpand& ex, cudaStream_t st);
// rotq_blk.cu : the same for blocks of 8..128 channels with K a multiple of 128; LRQ_ERR_UNSUPPORTED otherwise
lrq_status lrq_launch_rotq_blk(const void* X, int M, int K, long ldx, int B, int a_bits, int mode, int out16, const float* prescale,
                               uint8_t* codes, float* scale, int32_t* zp, const LrqExpand& ex, cudaStream_t st);
int lrq_rotq_blk_subgroups(int M, int K);        // independent sub-groups of its CTA at this shape, without multipliers
// rotq_tc.cu : the same for long batches of blocks of 128 channels, without multipliers; LRQ_ERR_UNSUPPORTED otherwise
lrq_status lrq_launch_rotq_tc(const void* X, int M, int K, long ldx, int B, int a_bits, int mode, int out16, const float* prescale,
                              uint8_t* codes, float* scale, int32_t* zp, const LrqExpand& ex, cudaStream_t st);
// Where a rotation product leaves each row's extremes: over each tile's columns as a pair of floats (minimum, maximum), tile j of
// row m at rows + m * pitch + 8 j; when a row is one tile, in row_min[m] and row_max[m].  All null: not wanted.
struct LrqRowExt { unsigned char* rows; size_t pitch; float* row_min; float* row_max; };
constexpr int LRQ_ROT_TILE = 128;     // columns per tile
// qgemm_bf16.cu : Y[M,K] (fp32) = X[M,K] (bf16) . R[K,K] (bf16) on the tensor cores
lrq_status lrq_launch_rotgemm(const void* X, int M, int K, long ldx, const void* R, float* Y, const LrqRowExt& ext, cudaStream_t st);
// rotgemm.cu : the dual transformation, R1 and R2 bf16 [K/128][128][128].  For M a multiple of 8: U3 = the three bf16 terms of
// (x . R1hat . P)^T, [3K][M], then Y[M,K] (fp32) = their sum . R2hat; an entry of perm outside 0 .. K-1 is read as 0 and
// recorded (status 31)
lrq_status lrq_launch_dual_first(const void* X, int M, int K, long ldx, const void* R1, const int32_t* perm, void* U3, cudaStream_t st);
lrq_status lrq_launch_dual_second(const void* U3, int M, int K, const void* R2, float* Y, const LrqRowExt& ext, cudaStream_t st);
// For any M: Y[M,K] (fp32) = sum over the `parts` column panels of A[M, parts*K] (bf16) of panel . blockdiag(Rblk)
lrq_status lrq_launch_bdiag_gemm(const void* A, int M, int K, long lda, int parts, const void* Rblk, float* Y, const LrqRowExt& ext,
                                 cudaStream_t st);
// rotdual.cu : V3 bf16 [M,3K], panel p = p-th bf16 term of U[m, perm[i]] (the reordering between the two)
lrq_status lrq_launch_dual_gather_split(const float* U, int M, int K, const int32_t* perm, void* V3, cudaStream_t st);
// rotq.cu : per-token quantization of fp32 rows whose extremes a rotation product has left, per tile of LRQ_ROT_TILE columns at
// the start of the row's own part of `codes` (8 bytes a tile; the codes overwrite them, and are longer for every K above
// one tile), for one tile in scale[m] and zp[m].
lrq_status lrq_launch_quantize_f32_ext(const float* Y, int M, int K, int a_bits, int mode, int out16, uint8_t* codes,
                                       float* scale, int32_t* zp, const LrqExpand& ex, cudaStream_t st);

// rotq.cu : fluctuation metric J (Eq. 11) and the kind Eq. 12 picks; acc is one double of device scratch
lrq_status lrq_launch_ars_metric(const void* X, int M, int K, long ldx, double thr, float* J, int* kind, double* acc,
                                 cudaStream_t st);

// wrot.cu : W diag(colmul) R in fp64, rounded to fp32 (Eq. 2, weight side)
lrq_status lrq_launch_rotate_weights(const float* W, int N, int K, long ldw, const float* colmul, int kind,
                                     int had_block, const void* R, float* out, long ldo, cudaStream_t st);
// wrot_i8.cu : the dense case on the int8 tensor cores, to the same accuracy; 0 bytes: the shape is not taken
size_t lrq_wrot_i8_workspace(int N, int K);
lrq_status lrq_launch_rotate_weights_i8(const float* W, int N, int K, long ldw, const float* colmul, const void* R, float* out, long ldo,
                                        void* workspace, cudaStream_t st);
lrq_status lrq_launch_rotate_weights_dual(const float* W, int N, int K, long ldw, const float* colmul, int Bd, const void* R1,
                                          const int32_t* perm, const void* R2, float* out, long ldo, cudaStream_t st);

#ifdef __CUDACC__
// Programmatic dependent launch.  Every hot kernel lets its successor in the stream start early (the successor's
// prologue - barrier set-up, TMEM allocation, descriptor prefetch - overlaps this kernel's tail) and, before its
// own first global access, waits until its predecessor has completed and its writes are visible.  Both are
// no-ops for a launch without the attribute.
__device__ __forceinline__ void lrq_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void lrq_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Order-preserving map between fp32 and int32 (and back), so that integer min/max reductions serve floats.
__device__ __forceinline__ int lrq_ordered_int(float f) { const int i = __float_as_int(f); return i ^ ((i >> 31) & 0x7fffffff); }
__device__ __forceinline__ float lrq_ordered_float(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }
#endif
// qgemm_simple.cu / qgemm_tc.cu
lrq_status lrq_launch_qgemm_simple(const lrq_layer* L, const uint8_t* a_codes, const float* a_scale,
                                   const int32_t* a_zp, int M, void* Y, lrq_dtype dt, long ldy, cudaStream_t st);
// qgemm_simple.cu : the integer form of Eq. 10 (mantissa products, shifts, exact integer accumulation) on the CUDA cores
lrq_status lrq_launch_qgemm_shift(const lrq_layer* L, const uint8_t* a_codes, const float* a_scale,
                                  const int32_t* a_zp, int M, void* Y, lrq_dtype dt, long ldy, cudaStream_t st);
bool lrq_qgemm_tc_takes(const lrq_layer* L);
lrq_status lrq_launch_qgemm_tc(const lrq_layer* L, const uint8_t* a_codes, const float* a_scale,
                               const int32_t* a_zp, int M, void* Y, lrq_dtype dt, long ldy, cudaStream_t st);
// qgemm_small.cu : 128 x 32 tiles, one CTA each; lrq_qgemm_codes only
lrq_status lrq_launch_qgemm_small(const lrq_layer* L, const uint8_t* a_codes, const float* a_scale,
                                  const int32_t* a_zp, int M, void* Y, lrq_dtype dt, long ldy, cudaStream_t st);
// qgemm_bf16.cu : contraction of bf16 operands, A [M,K] of centred codes (a_zp with them), W [N,K] of decoded levels (both 16-byte aligned)
lrq_status lrq_launch_qgemm_bf16(const lrq_layer* L, const void* A, const void* W, const float* a_scale, const int32_t* a_zp, int M,
                                 void* Y, lrq_dtype dt, long ldy, cudaStream_t st);
// fills the layer's cached TMA descriptors (called once by lrq_layer_create; never fails: without a driver, or for
// shapes the tensor-core kernel does not take, the layer is simply left without them)
void lrq_qgemm_tc_prepare(lrq_layer* L);
