// Embedding lookup from a quantised table (paper Section 4.2: in the mixed 8/4/4 scheme the embedding
// table is stored with int4 weights, like the feed-forward layers): y[t, :] = fp16(s * q[ids[t], :]).
//
// The table is an ordinary packed layer (N = vocabulary, K = hidden size), so the LM head and the
// embedding can share one blob.  A CTA serves one token: its threads walk the 16-byte pieces of the
// token's row (one piece = the row's weights of one lane column in one K chunk), unpack them with the
// same routine the decode and prefill kernels use, and multiply by the scale: one fp16 multiplication of
// an exact integer is the correctly rounded product.  A piece holds runs of 8 consecutive k, which leave
// as 16-byte stores.  Bound: HBM (2048 rows of 4096 from a table of 128256: 21.5 MB, 3.3 us at the measured
// copy rate).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dequant.cuh"
#include "layout.h"

namespace ql {

struct EmbedParams {
    const uint8_t* body;
    const __half* chan_scales;           // nullptr when grouped
    const int32_t* ids;                  // [n] row numbers; rows outside [0, N) give zeros
    __half* y;                           // [n, K]
    int32_t n, N, K, n_kc, block_bytes;
};

template <int BITS, bool GROUPED>
__global__ void __launch_bounds__(128) embed_kernel(const EmbedParams p)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");                  // ids and the output buffer may be the previous kernel's
    const int t = blockIdx.x;
    const int row = p.ids[t];
    __half* yrow = p.y + (int64_t)t * p.K;
    constexpr int CHUNK_K = BITS == 4 ? 64 : 32;
    if (row < 0 || row >= p.N) {
        for (int k = threadIdx.x * 8; k < p.K; k += blockDim.x * 8) *reinterpret_cast<uint4*>(yrow + k) = make_uint4(0, 0, 0, 0);
        return;
    }
    const int rsb = row / kRsbRows, rb = (row % kRsbRows) / kRbRows;
    const int r16 = row % kRbRows, g = r16 & 7, hi = r16 >> 3;          // lane group and row half inside the row-block
    const uint8_t* base = p.body + (int64_t)rsb * p.n_kc * p.block_bytes + rb * 512 + g * 64;
    uint32_t s2[2];                                                     // scales of the chunk's two groups, in both halves
    s2[0] = s2[1] = GROUPED ? 0u : 0x10001u * (uint32_t)__half_as_ushort(p.chan_scales[row]);
    for (int piece = threadIdx.x; piece < p.n_kc * 4; piece += blockDim.x) {
        const int kc = piece >> 2, c = piece & 3;
        const uint8_t* blk = base + (int64_t)kc * p.block_bytes;
        const uint4 w = *reinterpret_cast<const uint4*>(blk + c * 16);
        if (GROUPED) {
            const uint32_t s = *reinterpret_cast<const uint32_t*>(blk - (rb * 512 + g * 64) + kWeightBlockBytes + rb * 64 + g * 8 + 4 * hi);
            s2[0] = __byte_perm(s, 0, 0x1010);
            s2[1] = __byte_perm(s, 0, 0x3232);
        }
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
        constexpr int RUNS = BITS == 4 ? 2 : 1;                          // runs of 8 consecutive k in a piece: 16 bytes of output each
#pragma unroll
        for (int h = 0; h < RUNS; ++h) {
            uint32_t o[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                uint32_t a[4];
                if (BITS == 4) unpack_int4_word(ww[2 * h + i], a);
                else unpack_int8_words(ww[2 * i], ww[2 * i + 1], a);
                o[2 * i] = h2_mul(hi ? a[1] : a[0], s2[h]);              // registers hi and hi + 2 hold this row; one rounding
                o[2 * i + 1] = h2_mul(hi ? a[3] : a[2], s2[h]);
            }
            const int k = kc * CHUNK_K + 32 * h + 8 * c;                 // (K is a multiple of 32: a run lies inside or outside)
            if (k < p.K) *reinterpret_cast<uint4*>(yrow + k) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

}  // namespace ql
