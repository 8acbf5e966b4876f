// TLQ weight codes -> bf16, once per call (Sec. 4.1, Eqs. 7-9: every level is exactly a bf16 number).
//
// A layer meets each weight in M/256 tiles of the contraction; decoded there, a weight costs 2.6 lane-operations and a trip
// through shared memory in every one of them.  Decoded here it costs one pass over 2.5 bytes per weight, whose
// results the contraction then reads mostly from L2.  Bound by those bytes.
//
// A warp takes a row at a time, so that a per-channel table is loaded once; a lane turns eight codes (4 bytes, 3 when
// packed) into one 16-byte store, eight of them in flight, so a warp reads and writes whole lines.  With grouped tables a
// lane reloads its table when its group changes.
#include "lrq_internal.cuh"
#include "tlq_decode.cuh"

namespace {
using namespace lrq_dec;
constexpr int WARPS = 8, UNROLL = 8;

template <int W_BITS, bool PACKED3>
__global__ void __launch_bounds__(WARPS * 32)
expand_w_kernel(const uint8_t* __restrict__ codes, const float* __restrict__ levels, int N, int K, int G, uint4* __restrict__ out) {
    constexpr int NLEV = 1 << W_BITS;
    const int lane = threadIdx.x & 31, n = blockIdx.x * WARPS + (threadIdx.x >> 5);
    const int words = K >> 3, ngrp = K / G, wpg = G >> 3;          // groups of eight codes: per row, per table
    lrq_pdl_trigger();
    lrq_pdl_wait();                                                // the destination may still be read by the previous kernel
    if (n >= N) return;
    const size_t pitch = PACKED3 ? (size_t)K * 3 / 8 : (size_t)K / 2;
    const uint8_t* row = codes + (size_t)n * pitch;
    const uint8_t* end = codes + (size_t)N * pitch;
    const float* tab = levels + (size_t)n * ngrp * NLEV;
    uint4* dst = out + (size_t)n * words;
    Lut L;
    int held = -1;
    if (ngrp == 1) { load_lut<W_BITS>(L, tab); held = 0; }
    for (int j0 = lane; j0 < words; j0 += 32 * UNROLL) {
        uint32_t w[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int j = j0 + 32 * u;
            w[u] = 0;
            if (j < words) w[u] = PACKED3 ? fetch_packed3(row + 3 * (size_t)j, end) : __ldg(reinterpret_cast<const uint32_t*>(row) + j);
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int j = j0 + 32 * u;
            if (j >= words) break;
            if (ngrp > 1) {
                const int g = j / wpg;
                if (g != held) { load_lut<W_BITS>(L, tab + (size_t)g * NLEV); held = g; }
            }
            uint32_t o[4];
            decode_w<W_BITS>(PACKED3 ? spread3(w[u]) : w[u], L, o);
            dst[j] = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}
}  // namespace

lrq_status lrq_launch_expand_w(const lrq_layer* L, void* out, cudaStream_t st) {
    auto kern = L->packed3 ? expand_w_kernel<3, true> : L->w_bits == 4 ? expand_w_kernel<4, false> : L->w_bits == 3 ? expand_w_kernel<3, false> : expand_w_kernel<2, false>;
    LRQ_CUDA_TRY(lrq_launch_pdl(kern, dim3((L->N + WARPS - 1) / WARPS), dim3(WARPS * 32), 0, st, L->codes, L->levels, L->N, L->K, L->group,
                                static_cast<uint4*>(out)));
    return LRQ_OK;
}
