// Register-resident decode of TLQ weight codes: the row's level table as two byte planes, looked up with byte permutes.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "lrq_internal.cuh"

namespace lrq_dec {

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// Level table of one (row, group): low and high byte of each bf16 entry, 16 entries = 4 + 4 registers.  Levels are
// exact bf16 numbers stored as fp32: the upper two bytes of each word are the entry.
struct Lut { uint32_t lo[4], hi[4]; };

template <int W_BITS>
__device__ __forceinline__ void load_lut(Lut& L, const float* __restrict__ tab) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (j < (1 << W_BITS) / 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(tab) + j);
            const uint32_t t01 = prmt(__float_as_uint(v.x), __float_as_uint(v.y), 0x7632u);
            const uint32_t t23 = prmt(__float_as_uint(v.z), __float_as_uint(v.w), 0x7632u);
            L.lo[j] = prmt(t01, t23, 0x6420u);
            L.hi[j] = prmt(t01, t23, 0x7531u);
        } else {
            L.lo[j] = 0; L.hi[j] = 0;
        }
    }
}

// Eight codes as nibbles (one word) -> four registers of two bf16 each, in k order.
template <int W_BITS>
__device__ __forceinline__ void decode_w(uint32_t w, const Lut& L, uint32_t* o) {
    const uint32_t selA = w & 0x77777777u, selB = selA >> 16;
    uint32_t loA, hiA, loB, hiB;                   // codes 0-3 and 4-7, one byte each
    if (W_BITS == 4) {
        const uint32_t x0 = w << 4;
        const uint32_t mA = prmt(x0, w, 0xD9C8u), mB = prmt(x0, w, 0xFBEAu);    // 0xFF where the code's top bit is set
        loA = (prmt(L.lo[0], L.lo[1], selA) & ~mA) | (prmt(L.lo[2], L.lo[3], selA) & mA);
        hiA = (prmt(L.hi[0], L.hi[1], selA) & ~mA) | (prmt(L.hi[2], L.hi[3], selA) & mA);
        loB = (prmt(L.lo[0], L.lo[1], selB) & ~mB) | (prmt(L.lo[2], L.lo[3], selB) & mB);
        hiB = (prmt(L.hi[0], L.hi[1], selB) & ~mB) | (prmt(L.hi[2], L.hi[3], selB) & mB);
    } else {                                       // at most 8 entries: one permute per plane
        loA = prmt(L.lo[0], L.lo[1], selA); hiA = prmt(L.hi[0], L.hi[1], selA);
        loB = prmt(L.lo[0], L.lo[1], selB); hiB = prmt(L.hi[0], L.hi[1], selB);
    }
    o[0] = prmt(loA, hiA, 0x5140u); o[1] = prmt(loA, hiA, 0x7362u);
    o[2] = prmt(loB, hiB, 0x5140u); o[3] = prmt(loB, hiB, 0x7362u);
}

// eight 3-bit codes in the low 24 bits -> eight nibbles
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
    x = (x & 0x00000FFFu) | ((x & 0x00FFF000u) << 4);        // two groups of four codes, one per 16-bit half
    x = (x & 0x003F003Fu) | ((x & 0x0FC00FC0u) << 2);        // four groups of two codes, one per byte
    return (x & 0x07070707u) | ((x & 0x38383838u) << 1);     // one code per nibble
}

// The eight packed 3-bit codes at byte address `a` (any alignment): the 32-bit window that starts there, from the two
// aligned words around it; never reads at or past `end`, the end of the code matrix.
__device__ __forceinline__ uint32_t fetch_packed3(const uint8_t* a, const uint8_t* end) {
    const uintptr_t ai = reinterpret_cast<uintptr_t>(a);
    const uint32_t* w0 = reinterpret_cast<const uint32_t*>(ai & ~uintptr_t(3));
    const uint32_t lo = __ldg(w0);
    const uint32_t hi = (reinterpret_cast<const uint8_t*>(w0 + 2) <= end) ? __ldg(w0 + 1) : 0u;
    return __funnelshift_r(lo, hi, 8 * (uint32_t)(ai & 3)) & 0x00FFFFFFu;
}

// Weight rows first, first + stride, ... of a layer decoded to bf16 [N,K], by one warp.  A layer meets each weight in M/256
// tiles of the contraction; decoded there, a weight costs 2.6 lane-operations and a trip through shared memory in every
// one of them.  Decoded here it costs one pass over 2.5 bytes per weight, whose results the contraction then reads
// mostly from L2.  Bound by those bytes.  A warp takes a row at a time, so that a per-channel table is loaded once; a lane
// turns eight codes (4 bytes, 3 when packed) into one 16-byte store, UNROLL of them in flight, so a warp reads and
// writes whole lines.  With grouped tables a lane reloads its table when its group changes.
template <int W_BITS, bool PACKED3>
__device__ __forceinline__ void expand_rows(const LrqExpand& e, int first, int stride) {
    constexpr int NLEV = 1 << W_BITS, UNROLL = 6;
    const int lane = threadIdx.x & 31;
    const int words = e.K >> 3, ngrp = e.K / e.G, wpg = e.G >> 3;  // groups of eight codes: per row, per table
    const size_t pitch = PACKED3 ? (size_t)e.K * 3 / 8 : (size_t)e.K / 2;
    const uint8_t* end = e.codes + (size_t)e.N * pitch;
    for (int n = first; n < e.N; n += stride) {
        const uint8_t* row = e.codes + (size_t)n * pitch;
        const float* tab = e.levels + (size_t)n * ngrp * NLEV;
        uint4* dst = static_cast<uint4*>(e.out) + (size_t)n * words;
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
}

// The weight decode that rides on a quantizer kernel: called by every warp of the grid when it has no tokens left.  Rows are
// dealt from the last warp of the grid backwards, so that those of a short batch go to CTAs that had none.
static __device__ __noinline__ void expand_share(const LrqExpand e) {
    const int wpc = blockDim.x >> 5, total = gridDim.x * wpc, first = total - 1 - (int)(blockIdx.x * wpc + (threadIdx.x >> 5));
    if (e.fmt == 4) expand_rows<4, false>(e, first, total);
    else if (e.fmt == 3) expand_rows<3, false>(e, first, total);
    else if (e.fmt == 13) expand_rows<3, true>(e, first, total);
    else expand_rows<2, false>(e, first, total);
}

}  // namespace lrq_dec
