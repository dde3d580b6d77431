// Embedding lookup from a quantised table (paper Section 4.2: in the mixed 8/4/4 scheme the embedding
// table is stored with int4 weights, like the feed-forward layers): y[t, :] = fp16(s * q[ids[t], :]).
//
// The table is an ordinary packed layer (N = vocabulary, K = hidden size), so the LM head and the
// embedding can share one blob.  A CTA serves one token (short rows: several): its threads walk the 16-byte pieces of the
// token's row (one piece = the row's weights of one lane column in one K chunk), unpack them with the
// same routine the decode and prefill kernels use, and multiply by the scale: one fp16 multiplication of
// an exact integer is the correctly rounded product.  A piece holds runs of 8 consecutive k, which leave
// as 16-byte stores.  Bound: HBM (2048 rows of 4096 from a table of 128256: 21.5 MB, 3.3 us at the measured
// copy rate); with short rows the CTAs themselves, each with its wait for the kernel before
// (8192 rows of 32 9.1 us with a CTA per token, 5.9 without the programmatic launch, 2.1 with 8 tokens to a CTA; 8192 rows of 512 9.1, 7.6, 3.4).
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
    int32_t log2_tokens;                 // 1 << log2_tokens tokens per CTA, 128 >> log2_tokens threads each
};

// SEVERAL: tokens per CTA (else one).  U: pieces of a thread that are requested together: 2 where it has more than one.  The table
// comes from HBM, the rows of one prompt all over it (64 rows of 4096, the table not in L2, 3.6 -> 3.1 us, of 8192 5.2 -> 4.3; 2048 rows of 4096 11.5 both ways,
// their scattered 64-byte reads and the writes are the bound there; with one piece per thread the second one's tests cost 0.1).
template <int BITS, bool GROUPED, bool SEVERAL, int U = 1>
__global__ void __launch_bounds__(128) embed_kernel(const EmbedParams p)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");                  // ids and the output buffer may be the previous kernel's
    // (unsigned: with a signed stride the compiler unrolls the loop below, 0.2 us more at two pieces per thread)
    const unsigned lanes = SEVERAL ? 128u >> p.log2_tokens : blockDim.x, first = SEVERAL ? threadIdx.x & (lanes - 1) : threadIdx.x;
    const int t = SEVERAL ? (blockIdx.x << p.log2_tokens) + (threadIdx.x >> (7 - p.log2_tokens)) : blockIdx.x;
    if (SEVERAL && t >= p.n) return;
    const int row = p.ids[t];
    __half* yrow = p.y + (int64_t)t * p.K;
    constexpr int CHUNK_K = BITS == 4 ? 64 : 32;
    if (row < 0 || row >= p.N) {
        for (int k = (int)first * 8; k < p.K; k += lanes * 8) *reinterpret_cast<uint4*>(yrow + k) = make_uint4(0, 0, 0, 0);
        return;
    }
    const int rsb = row / kRsbRows, rb = (row % kRsbRows) / kRbRows;
    const int r16 = row % kRbRows, g = r16 & 7, hi = r16 >> 3;          // lane group and row half inside the row-block
    const uint8_t* base = p.body + (int64_t)rsb * p.n_kc * p.block_bytes + rb * 512 + g * 64;
    uint32_t s2[2];                                                     // scales of the chunk's two groups, in both halves
    s2[0] = s2[1] = GROUPED ? 0u : 0x10001u * (uint32_t)__half_as_ushort(p.chan_scales[row]);
    for (int piece0 = (int)first; piece0 < p.n_kc * 4; piece0 += U * lanes) {
        uint4 w[U];
        uint32_t s[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int piece = piece0 + j * (int)lanes;
            if (piece >= p.n_kc * 4) break;
            const uint8_t* blk = base + (int64_t)(piece >> 2) * p.block_bytes;
            w[j] = *reinterpret_cast<const uint4*>(blk + (piece & 3) * 16);
            if (GROUPED) s[j] = *reinterpret_cast<const uint32_t*>(blk - (rb * 512 + g * 64) + kWeightBlockBytes + rb * 64 + g * 8 + 4 * hi);
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int piece = piece0 + j * (int)lanes, kc = piece >> 2, c = piece & 3;
            if (piece >= p.n_kc * 4) break;
            if (GROUPED) {
                s2[0] = __byte_perm(s[j], 0, 0x1010);
                s2[1] = __byte_perm(s[j], 0, 0x3232);
            }
            const uint32_t ww[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
            constexpr int RUNS = BITS == 4 ? 2 : 1;                      // runs of 8 consecutive k in a piece: 16 bytes of output each
#pragma unroll
            for (int h = 0; h < RUNS; ++h) {
                uint32_t o[4];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    uint32_t a[4];
                    if (BITS == 4) unpack_int4_word(ww[2 * h + i], a);
                    else unpack_int8_words(ww[2 * i], ww[2 * i + 1], a);
                    o[2 * i] = h2_mul(hi ? a[1] : a[0], s2[h]);          // registers hi and hi + 2 hold this row; one rounding
                    o[2 * i + 1] = h2_mul(hi ? a[3] : a[2], s2[h]);
                }
                const int k = kc * CHUNK_K + 32 * h + 8 * c;             // (K is a multiple of 32: a run lies inside or outside)
                if (k < p.K) *reinterpret_cast<uint4*>(yrow + k) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    }
}

}  // namespace ql
