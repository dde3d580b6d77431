// Kernel for int8 layers with a SHORT K (2, 4 or 8 chunks of 32) and more than 8 tokens: the score product of a prompt's
// queries over a KV cache (paper Section 3.8: the K cache is a layer with O = cache positions and I = d_h), for up to 8 KV
// heads of a layer in one launch.
//
// Bound: the outputs.  At d_h = 128 a score costs 128 multiply-adds and 2 bytes of HBM; 8 heads x 1024 query rows x 4096
// positions write 67 MB (10.3 us at the measured copy rate) and keep the warp-level tensor core busy for 15 us (8.05 cycles per
// m16n8k16 and SM quarter).  In the prefill kernel such a tile has 2 k-steps and an epilogue that nothing hides.
//
// Work decomposition: the tiles (row super-block of 128 positions x 8 NT tokens) of all layers are numbered through, token
// blocks innermost, and every CTA of a grid that fills the GPU once takes an equal contiguous range.  A warp keeps the packed
// weights of its row-block, the whole K, in registers while the super-block lasts (4 NKC registers) and unpacks them per tile;
// the x tile of the next token block is in flight (two cp.async buffers) while it works on the current one.  Results leave
// through shared memory: stmatrix turns the accumulator fragments, which hold pairs of tokens of one position, into rows of
// 128 positions, which go out as 256-byte pieces.
//
// Measured: 8 heads x 1024 rows x 4096 positions, d_h = 128: 35 us (1.9 TB/s written), 72 us as eight launches of the prefill
// kernel; 8 heads x 64 rows 4.4 us against 42; 8 heads of 256 x 256 rows 18.6 us against 50.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dequant.cuh"
#include "layout.h"

namespace ql {

constexpr int kRowsMaxLayers = 8;

struct GemmRowsParams {
    const uint8_t* body[kRowsMaxLayers];
    const __half* chan_scales[kRowsMaxLayers];
    const __half* x[kRowsMaxLayers];             // [M, K] each
    __half* y[kRowsMaxLayers];                   // [M, N_i]
    int32_t N[kRowsMaxLayers];
    int32_t rsb_end[kRowsMaxLayers];             // row super-blocks of layers 0..i
    int32_t n_layers, M, n_tb, n_tiles;
};

template <int NKC, int NT>
struct GemmRowsSmem {
    static constexpr int kTokens = 8 * NT;
    static constexpr int kXBytes = kTokens * NKC * 64;
    static constexpr int kOutStride = 272;       // bytes per token of the output tile: 128 positions and a pad that spreads 8 rows over all banks
    static constexpr int kTotal = 2 * kXBytes + kTokens * kOutStride;
};

template <int NKC, int NT>
__global__ void __launch_bounds__(256, 2) gemm_rows_kernel(const GemmRowsParams p)
{
    using S = GemmRowsSmem<NKC, NT>;
    constexpr int UNITS = NKC * 4;                                       // 16-byte pieces of a token
    constexpr int K = 32 * NKC;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem_raw), out0 = smem0 + 2 * S::kXBytes;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, c = lane & 3;
    const int i0 = (int)((int64_t)blockIdx.x * p.n_tiles / gridDim.x), i1 = (int)((int64_t)(blockIdx.x + 1) * p.n_tiles / gridDim.x);

    auto layer_of = [&](int rsb) {
        int ly = 0;
#pragma unroll
        for (int i = 1; i < kRowsMaxLayers; ++i)
            if (i < p.n_layers && rsb >= p.rsb_end[i - 1]) ly = i;
        return ly;
    };
    auto load_x = [&](int i, int buf) {
        if (i < i1) {
            const int rsb = i / p.n_tb, m0 = (i - rsb * p.n_tb) * S::kTokens;
            const __half* x = p.x[layer_of(rsb)];
            const uint32_t dst = smem0 + buf * S::kXBytes;
#pragma unroll
            for (int e0 = 0; e0 < S::kTokens * UNITS; e0 += 256) {
                const int e = e0 + t;
                if (S::kTokens * UNITS % 256 == 0 || e < S::kTokens * UNITS) {
                    const int tok = e / UNITS, u = e % UNITS;
                    const uint32_t sz = m0 + tok < p.M ? 16u : 0u;       // beyond M: zeros
                    // pieces of odd tokens swapped in pairs of four: the 8 lanes of a read phase touch all 32 banks
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + tok * (UNITS * 16) + ((u ^ ((tok & 1) << 2)) << 4)),
                                 "l"(sz ? x + (int64_t)(m0 + tok) * K + u * 8 : x), "r"(sz) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_x(i0, 0);

    uint4 w[NKC];
    float s0 = 0.f, s1 = 0.f;
    int cur = -1, ly = 0, row_base = 0;
    const uint32_t xl[2] = {(uint32_t)(g * UNITS * 16 + (g & 1) * 64 + c * 16), (uint32_t)(g * UNITS * 16 + ((g & 1) ^ 1) * 64 + c * 16)};
    for (int i = i0; i < i1; ++i) {
        const int rsb = i / p.n_tb, m0 = (i - rsb * p.n_tb) * S::kTokens;
        load_x(i + 1, (i - i0 + 1) & 1);
        if (rsb != cur) {                                                // (uniform) the next super-block's weights
            cur = rsb;
            ly = layer_of(rsb);
            const int r = rsb - (ly ? p.rsb_end[ly - 1] : 0);
            const uint8_t* src = p.body[ly] + (int64_t)r * NKC * kWeightBlockBytes + t * 16;
#pragma unroll
            for (int kc = 0; kc < NKC; ++kc) w[kc] = __ldcg(reinterpret_cast<const uint4*>(src + kc * kWeightBlockBytes));
            row_base = r * kRsbRows;
            const int row = row_base + warp * 16 + g;
            s0 = row < p.N[ly] ? __half2float(__ldcg(p.chan_scales[ly] + row)) : 0.f;
            s1 = row + 8 < p.N[ly] ? __half2float(__ldcg(p.chan_scales[ly] + row + 8)) : 0.f;
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                                                 // this tile's x has landed; the output tile has been sent
        float acc[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
        const uint32_t xs = smem0 + ((i - i0) & 1) * S::kXBytes;
#pragma unroll
        for (int kc = 0; kc < NKC; ++kc) {
            uint32_t a0[4], a1[4];
            unpack_int8_words(w[kc].x, w[kc].y, a0);
            unpack_int8_words(w[kc].z, w[kc].w, a1);
            const uint32_t xa = xs + xl[kc & 1] + (kc >> 1) * 128;
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                uint4 b;
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "r"(xa + n * 8 * UNITS * 16));
                mma_16816_pure(acc[n], a0, b.x, b.y);
                mma_16816_pure(acc[n], a1, b.z, b.w);
            }
        }
        // Four 8 x 8 matrices per store: positions 0..7 and 8..15 of the row-block, tokens of columns n and n + 1; lane L gives the
        // address of row L % 8 (a token) of matrix L / 8.
        const uint32_t oa = out0 + (lane & 7) * S::kOutStride + ((lane >> 4) & 1) * 8 * S::kOutStride + warp * 32 + ((lane >> 3) & 1) * 16;
#pragma unroll
        for (int n = 0; n < NT; n += 2) {
            uint32_t r[4];
            const __half2 h0 = __floats2half2_rn(acc[n][0] * s0, acc[n][1] * s0), h1 = __floats2half2_rn(acc[n][2] * s1, acc[n][3] * s1);
            const __half2 h2 = __floats2half2_rn(acc[n + 1][0] * s0, acc[n + 1][1] * s0), h3 = __floats2half2_rn(acc[n + 1][2] * s1, acc[n + 1][3] * s1);
            r[0] = *reinterpret_cast<const uint32_t*>(&h0);
            r[1] = *reinterpret_cast<const uint32_t*>(&h1);
            r[2] = *reinterpret_cast<const uint32_t*>(&h2);
            r[3] = *reinterpret_cast<const uint32_t*>(&h3);
            asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(oa + n * 8 * S::kOutStride), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
        }
        __syncthreads();
        const int N = p.N[ly];
        __half* y = p.y[ly];
#pragma unroll
        for (int e0 = 0; e0 < S::kTokens * 16; e0 += 256) {
            const int e = e0 + t, tok = e >> 4, q = e & 15;              // 16 bytes = 8 positions (N is a multiple of 8)
            if ((S::kTokens * 16 % 256 == 0 || e < S::kTokens * 16) && m0 + tok < p.M && row_base + 8 * q < N) {
                uint4 v;
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(out0 + tok * S::kOutStride + q * 16));
                *reinterpret_cast<uint4*>(y + (int64_t)(m0 + tok) * N + row_base + 8 * q) = v;
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

}  // namespace ql
