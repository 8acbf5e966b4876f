// Weight side of the rotation identity (Sec. 3.2, Eq. 2: (X R)(W R)^T = X W^T) with the smoothing of
// Sec. 5.1 folded in: W_rot = W diag(colmul) R, evaluated in fp64 and rounded once to fp32, which is what
// the TLQ quantizer reads.
//
// Offline step.  Hadamard: butterflies in registers, up to four stages between two trips through shared memory, by warps of their own
// (blocks of 16 to 256 channels) or one CTA per weight row.  Dense: an fp64 matrix product on the fp64 tensor cores, 64 x 64 output tiles, for small
// layers and for callers without scratch (wrot_i8.cu otherwise); R is the layer's stored bf16 matrix (exact in fp64), so both
// sides of Eq. 2 use the same R.  Dual transformation (R = R1hat P R2hat, Sec. 4.2): one CTA per row, the
// row in shared memory as fp64, block-diagonal product, gather through the index map, second product.
#include "lrq_internal.cuh"

#include <cuda_bf16.h>
#include <cmath>

namespace {

// The result may stand in the place of W (but for the dense product): an element is read by the threads that write it, ahead of that.
// NB butterfly stages (index bits bit .. bit + NB - 1) of the row: a thread takes the 2^NB elements that differ in these
// bits, from global memory in the first pass, to global memory in the last.  Elements lie in shared memory with one
// pad after every 16, which makes both the first pass (runs of 16 per thread) and the later ones (neighbouring
// threads, neighbouring elements) conflict-free.  Stages run in the order of increasing bits whatever NB is, so the
// result does not depend on how they are grouped.
template <int NB>
__device__ __forceinline__ void hadamard_pass(double* row, int K, int bit, const float* w, const float* colmul, float* o, double norm) {
    constexpr int E = 1 << NB;
    for (int g = threadIdx.x; g < (K >> NB); g += blockDim.x) {
        const int low = g & ((1 << bit) - 1), base = ((g - low) << NB) | low;
        double v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = base + (e << bit);
            v[e] = w ? (double)w[k] * (colmul ? (double)colmul[k] : 1.0) : row[k + (k >> 4)];
        }
#pragma unroll
        for (int h = 1; h < E; h <<= 1)
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (!(e & h)) { const double a = v[e], b = v[e | h]; v[e] = a + b; v[e | h] = a - b; }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = base + (e << bit);
            if (o) o[k] = (float)(v[e] * norm); else row[k + (k >> 4)] = v[e];
        }
    }
    __syncthreads();
}

// Any block, any alignment: a CTA per row.
__global__ void __launch_bounds__(128)
wrot_hadamard_kernel(const float* W, int N, int K, long ldw, const float* __restrict__ colmul, int log2B,
                     float* out, long ldo) {
    extern __shared__ double row[];                // [K + K / 16]
    const int n = blockIdx.x;
    const float* w = W + (size_t)n * ldw;
    // 1/sqrt(B): a power of two for even log2(B), else a power of two times 1/sqrt(2)
    const double norm = ldexp((log2B & 1) ? 0.70710678118654752440 : 1.0, -(log2B >> 1));
    float* o = out + (size_t)n * ldo;
    lrq_pdl_trigger();
    lrq_pdl_wait();
    int bit = 0;
    do {
        const int left = log2B - bit, nb = left < 4 ? left : 4;
        const float* src = bit == 0 ? w : nullptr;
        float* dst = nb == left ? o : nullptr;
        if (nb == 4) hadamard_pass<4>(row, K, bit, src, colmul, dst, norm);
        else if (nb == 3) hadamard_pass<3>(row, K, bit, src, colmul, dst, norm);
        else if (nb == 2) hadamard_pass<2>(row, K, bit, src, colmul, dst, norm);
        else if (nb == 1) hadamard_pass<1>(row, K, bit, src, colmul, dst, norm);
        else hadamard_pass<0>(row, K, bit, src, colmul, dst, norm);
        bit += nb;
    } while (bit < log2B);
}

// Blocks of 16 to 256 channels: a warp by itself takes 512 consecutive elements of the matrix (whole blocks, of one row or two), a
// lane 16 of them with 128-bit loads: stages 0-3 in its registers, one exchange through the warp's shared memory (a pad after
// every 16 doubles: conflict-free both ways), the other one to four stages at stride 16.  The kernel above keeps a CTA per row,
// whose 128 threads a row of 1152 fills to 0.56, and has barriers.  The same additions in the same order, the same results.
// 4608 x 1152, B = 128: 27.5 us there with a cold L2, 15.2 here (2.8 TB/s); 2600 x 6144 61.4 and 30.7 (4.2 TB/s); 9216 x 1728, B = 64
// 58 and 36; 1024 x 3072, B = 256 17.8 and 12.3; 512 x 512 8.2 both.  Bound by the fp64 conversions and additions on the way.
template <int LOG2B>
__global__ void __launch_bounds__(256)
wrot_hadamard_warp_kernel(const float* W, unsigned items, unsigned items_per_row, long ldw, const float* __restrict__ colmul,
                          double norm, float* out, long ldo) {
    constexpr int NB = LOG2B - 4, E = 1 << NB;
    __shared__ double smem[8][32 * 17];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* s = smem[warp];
    lrq_pdl_trigger();
    lrq_pdl_wait();
    for (unsigned first = (blockIdx.x * 8 + warp) * 32; first < items; first += gridDim.x * 256) {
        const unsigned item = first + lane;
        double v[16];
        if (item < items) {
            const unsigned n = item / items_per_row, k = (item - n * items_per_row) * 16;
            const float4* w = reinterpret_cast<const float4*>(W + n * ldw + k);
            float4 f[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) f[i] = w[i];
#pragma unroll
            for (int i = 0; i < 4; ++i) { v[4 * i] = f[i].x; v[4 * i + 1] = f[i].y; v[4 * i + 2] = f[i].z; v[4 * i + 3] = f[i].w; }
            if (colmul) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 c = __ldg(reinterpret_cast<const float4*>(colmul + k) + i);
                    v[4 * i] *= (double)c.x; v[4 * i + 1] *= (double)c.y; v[4 * i + 2] *= (double)c.z; v[4 * i + 3] *= (double)c.w;
                }
            }
#pragma unroll
            for (int h = 1; h < 16; h <<= 1)
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    if (!(e & h)) { const double a = v[e], b = v[e | h]; v[e] = a + b; v[e | h] = a - b; }
#pragma unroll
            for (int e = 0; e < 16; ++e) s[lane * 17 + e] = v[e];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 16 / E; ++q) {
            const int id = q * 32 + lane, i = id & 15, r = (id >> 4) * E;      // element i of items r .. r + E - 1: one block
            if (first + r < items) {
                double u[E];
#pragma unroll
                for (int e = 0; e < E; ++e) u[e] = s[(r + e) * 17 + i];
#pragma unroll
                for (int h = 1; h < E; h <<= 1)
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (!(e & h)) { const double a = u[e], b = u[e | h]; u[e] = a + b; u[e | h] = a - b; }
                const unsigned n = (first + r) / items_per_row, k = (first + r - n * items_per_row) * 16 + i;
                float* o = out + n * ldo + k;
#pragma unroll
                for (int e = 0; e < E; ++e) o[16 * e] = (float)(u[e] * norm);
            }
        }
        __syncwarp();                              // read before the next elements are written
    }
}

// Dense rotation: out[N,K] = (W diag(colmul)) . R in fp64 on the tensor cores (mma m8n8k4).  A CTA of four warps owns a
// 64 x 64 tile, a warp 32 x 32 of it (4 x 4 fragments, 64 accumulator registers): per 4-deep step 8 fragment loads feed
// 16 MMAs, a quarter of the shared-memory traffic that 4 x 4 accumulators per thread needed.  Both operands are
// widened to fp64 on their way into shared memory, double-buffered, the next 16-deep block in flight in registers.
// Bound by the fp64 pipe.  4608 x 1536 x 1536: 1924 us on the CUDA cores (11 TFLOP/s), 660 now (33 TFLOP/s).
constexpr int TM = 64, TN = 64, TK = 16;
constexpr int A_PITCH = TK + 4, B_PITCH = TN + 4;   // doubles; 4 mod 16: a fragment's 4 x 4 half-warp hits 16 bank pairs

__device__ __forceinline__ void dmma(double* d, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

__global__ void __launch_bounds__(128)
wrot_dense_kernel(const float* __restrict__ W, int N, int K, long ldw, const float* __restrict__ colmul,
                  const __nv_bfloat16* __restrict__ R, float* __restrict__ out, long ldo, int vec_w, int vec_r) {
    __shared__ __align__(16) double sA[2][TM * A_PITCH];
    __shared__ __align__(16) double sB[2][TK * B_PITCH];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int ar = tid >> 1, ak = (tid & 1) * 8;               // W: row of the tile, first of eight k
    const int bk = tid >> 3, bn = (tid & 7) * 8;               // R: k of the block, first of eight columns
    lrq_pdl_trigger();
    lrq_pdl_wait();
    const float* wrow = W + (size_t)(n0 + ar) * ldw;
    const bool row_ok = n0 + ar < N;
    float fa[8], fc[8];
    uint32_t fb[4];
    auto fetch = [&](int k0) {
        const int k = k0 + ak;
        if (vec_w && row_ok && k + 8 <= K) {
            const float4 x = *reinterpret_cast<const float4*>(wrow + k), y = *reinterpret_cast<const float4*>(wrow + k + 4);
            fa[0] = x.x; fa[1] = x.y; fa[2] = x.z; fa[3] = x.w; fa[4] = y.x; fa[5] = y.y; fa[6] = y.z; fa[7] = y.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) fa[i] = row_ok && k + i < K ? wrow[k + i] : 0.f;
        }
        if (colmul) {
#pragma unroll
            for (int i = 0; i < 8; ++i) fc[i] = k + i < K ? colmul[k + i] : 0.f;
        }
        const int kr = k0 + bk, c = j0 + bn;
        if (vec_r && kr < K && c + 8 <= K) {
            const uint4 x = *reinterpret_cast<const uint4*>(R + (size_t)kr * K + c);
            fb[0] = x.x; fb[1] = x.y; fb[2] = x.z; fb[3] = x.w;
        } else {
            const unsigned short* r = reinterpret_cast<const unsigned short*>(R) + (size_t)kr * K + c;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t lo = kr < K && c + 2 * i < K ? r[2 * i] : 0u, hi = kr < K && c + 2 * i + 1 < K ? r[2 * i + 1] : 0u;
                fb[i] = lo | (hi << 16);
            }
        }
    };
    auto stage = [&](int s) {
        double2* a = reinterpret_cast<double2*>(&sA[s][ar * A_PITCH + ak]);
        double2* b = reinterpret_cast<double2*>(&sB[s][bk * B_PITCH + bn]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            double x = (double)fa[2 * i], y = (double)fa[2 * i + 1];
            if (colmul) { x *= (double)fc[2 * i]; y *= (double)fc[2 * i + 1]; }
            a[i] = make_double2(x, y);
            b[i] = make_double2((double)__uint_as_float(fb[i] << 16), (double)__uint_as_float(fb[i] & 0xffff0000u));
        }
    };
    double acc[4][4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    fetch(0);
    stage(0);
    __syncthreads();
    for (int k0 = 0, s = 0; k0 < K; k0 += TK, s ^= 1) {
        const bool more = k0 + TK < K;
        if (more) fetch(k0 + TK);
        const double* a = &sA[s][(wm + (lane >> 2)) * A_PITCH + (lane & 3)];
        const double* b = &sB[s][(lane & 3) * B_PITCH + wn + (lane >> 2)];
#pragma unroll
        for (int k = 0; k < TK; k += 4) {
            double x[4], y[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { x[i] = a[8 * i * A_PITCH + k]; y[i] = b[k * B_PITCH + 8 * i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dmma(acc[i][j], x[i], y[j]);
        }
        if (more) stage(s ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int n = n0 + wm + 8 * i + (lane >> 2);
        if (n >= N) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = j0 + wn + 8 * j + 2 * (lane & 3);
            if (c < K) out[(size_t)n * ldo + c] = (float)acc[i][j][0];
            if (c + 1 < K) out[(size_t)n * ldo + c + 1] = (float)acc[i][j][1];
        }
    }
}

// out[n] = ((w[n] * colmul) . blockdiag(R1)) gathered through perm, then . blockdiag(R2); blocks of Bd x Bd, row-major
__global__ void __launch_bounds__(256)
wrot_dual_kernel(const float* W, int N, int K, long ldw, const float* __restrict__ colmul, int Bd,
                 const __nv_bfloat16* __restrict__ R1, const int32_t* __restrict__ perm, const __nv_bfloat16* __restrict__ R2,
                 float* out, long ldo) {
    extern __shared__ double rows2[];              // a[K], b[K]
    double* a = rows2;
    double* b = rows2 + K;
    const int n = blockIdx.x, tid = threadIdx.x;
    const float* w = W + (size_t)n * ldw;
    for (int k = tid; k < K; k += 256) a[k] = (double)w[k] * (colmul ? (double)colmul[k] : 1.0);
    __syncthreads();
    for (int c = tid; c < K; c += 256) {           // b = a . blockdiag(R1)
        const int j = c / Bd, i = c - j * Bd;
        const __nv_bfloat16* r = R1 + (size_t)j * Bd * Bd + i;
        const double* x = a + j * Bd;
        double acc = 0.0;
        for (int l = 0; l < Bd; ++l) acc = fma(x[l], (double)__bfloat162float(r[(size_t)l * Bd]), acc);
        b[c] = acc;
    }
    __syncthreads();
    for (int c = tid; c < K; c += 256) {           // a = b . P
        const int p = perm[c];
        a[c] = (uint32_t)p < (uint32_t)K ? b[p] : b[0];
    }
    __syncthreads();
    float* o = out + (size_t)n * ldo;
    for (int c = tid; c < K; c += 256) {           // out = a . blockdiag(R2)
        const int j = c / Bd, i = c - j * Bd;
        const __nv_bfloat16* r = R2 + (size_t)j * Bd * Bd + i;
        const double* x = a + j * Bd;
        double acc = 0.0;
        for (int l = 0; l < Bd; ++l) acc = fma(x[l], (double)__bfloat162float(r[(size_t)l * Bd]), acc);
        o[c] = (float)acc;
    }
}

__global__ void wrot_scale_kernel(const float* W, int N, int K, long ldw, const float* __restrict__ colmul,
                                  float* out, long ldo) {
    const size_t total = (size_t)N * K;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t n = i / K, k = i % K;
        out[n * ldo + k] = (float)((double)W[n * ldw + k] * (colmul ? (double)colmul[k] : 1.0));
    }
}

}  // namespace

lrq_status lrq_launch_rotate_weights(const float* W, int N, int K, long ldw, const float* colmul, int kind,
                                     int had_block, const void* R, float* out, long ldo, cudaStream_t st) {
    if (kind == LRQ_ROT_HADAMARD) {
        int log2B = 0;
        while ((1 << log2B) < had_block) ++log2B;
        // 16-byte aligned rows of whole blocks of 16 to 256 channels; the result may stand in the place of W
        if (log2B >= 4 && log2B <= 8 && ldw % 4 == 0 && lrq_aligned(W, 16) && (!colmul || lrq_aligned(colmul, 16)) && (long)N * (K / 16) < (1l << 31)) {
            static constexpr decltype(&wrot_hadamard_warp_kernel<4>) kerns[] = {wrot_hadamard_warp_kernel<4>, wrot_hadamard_warp_kernel<5>, wrot_hadamard_warp_kernel<6>,
                                                                                wrot_hadamard_warp_kernel<7>, wrot_hadamard_warp_kernel<8>};
            int sms = 0;
            if (lrq_current_device(nullptr, &sms) != LRQ_OK) return LRQ_ERR_CUDA;
            const unsigned items = (unsigned)N * (unsigned)(K / 16), ctas = (items + 255) / 256, most = (unsigned)sms * 5;
            const double norm = ldexp((log2B & 1) ? 0.70710678118654752440 : 1.0, -(log2B >> 1));
            LRQ_CUDA_TRY(lrq_launch_pdl(kerns[log2B - 4], dim3(ctas < most ? ctas : most), dim3(256), 0, st, W, items, (unsigned)(K / 16), ldw, colmul, norm, out, ldo));
            return LRQ_OK;
        }
        // one pad after every 16 elements; the opt-in is the same for every K, since another host thread's call sets it too
        constexpr int MAX_K = 25600;
        auto row_bytes = [](int k) { return (size_t)(k + k / 16 + 1) * sizeof(double); };
        const size_t smem = row_bytes(K);
        if (K > MAX_K) return LRQ_ERR_UNSUPPORTED;
        if (smem > 40 * 1024)
            LRQ_CUDA_TRY(cudaFuncSetAttribute(wrot_hadamard_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_bytes(MAX_K)));
        LRQ_CUDA_TRY(lrq_launch_pdl(wrot_hadamard_kernel, dim3(N), dim3(128), smem, st, W, N, K, ldw, colmul, log2B, out, ldo));
    } else if (kind == LRQ_ROT_DENSE) {
        const dim3 grid((K + TN - 1) / TN, (N + TM - 1) / TM);
        const int vec_w = lrq_aligned(W, 16) && ldw % 4 == 0, vec_r = lrq_aligned(R, 16) && K % 8 == 0;
        LRQ_CUDA_TRY(lrq_launch_pdl(wrot_dense_kernel, grid, dim3(128), 0, st, W, N, K, ldw, colmul, static_cast<const __nv_bfloat16*>(R),
                                    out, ldo, vec_w, vec_r));
    } else {
        const size_t total = (size_t)N * K;
        const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
        wrot_scale_kernel<<<blocks, 256, 0, st>>>(W, N, K, ldw, colmul, out, ldo);
    }
    LRQ_CUDA_TRY(cudaGetLastError());
    return LRQ_OK;
}

lrq_status lrq_launch_rotate_weights_dual(const float* W, int N, int K, long ldw, const float* colmul, int Bd, const void* R1,
                                          const int32_t* perm, const void* R2, float* out, long ldo, cudaStream_t st) {
    const size_t smem = (size_t)K * 2 * sizeof(double);
    constexpr size_t MAX_SMEM = 200 * 1024;
    if (smem > MAX_SMEM) return LRQ_ERR_UNSUPPORTED;
    if (smem > 40 * 1024)                                    // (the same for every K, as above)
        LRQ_CUDA_TRY(cudaFuncSetAttribute(wrot_dual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MAX_SMEM));
    wrot_dual_kernel<<<N, 256, smem, st>>>(W, N, K, ldw, colmul, Bd, static_cast<const __nv_bfloat16*>(R1), perm,
                                           static_cast<const __nv_bfloat16*>(R2), out, ldo);
    LRQ_CUDA_TRY(cudaGetLastError());
    return LRQ_OK;
}
