// Kernel for int8 layers with a SHORT K (2, 4 or 8 chunks of 32) and more than 8 tokens: the score product of a prompt's
// queries over a KV cache (paper Section 3.8: the K cache is a layer with O = cache positions and I = d_h), for up to 8 KV
// heads of a layer in one launch.
//
// Bound: the outputs.  At d_h = 128 a score costs 128 multiply-adds and 2 bytes of HBM; 8 heads x 256 query rows x 4096
// positions write 17 MB (2.6 us at the measured copy rate) and keep the warp-level tensor core busy for 3.8 us (8.05 cycles per
// m16n8k16 and SM quarter).  In the prefill kernel such a tile has 2 k-steps and an epilogue that nothing hides.
//
// Work decomposition: the tiles (row super-block of 128 positions x 8 NT tokens) of all layers are numbered through, token
// blocks innermost, and every CTA of a grid that fills the GPU once takes an equal contiguous range.  A warp keeps the packed
// weights of its row-block, the whole K, in registers while the super-block lasts (4 NKC registers) and unpacks them per tile;
// the x tile of the next token block is in flight (two cp.async buffers) while it works on the current one.  Results leave
// through shared memory: stmatrix turns the accumulator fragments, which hold pairs of tokens of one position, into rows of
// 128 positions, which go out as 256-byte pieces.
//
// Measured, d_h = 128, 8 heads: 256 rows x 4096 positions 11.6 us (1.4 TB/s written), 128 rows 7.1, 256 rows x 2048 positions 7.1, 64 rows 4.0; 8
// heads of 256, 128 rows x 4096 positions 10.6.  (As eight launches of the prefill kernel 42 us for 64 rows x 4096 positions, 4.4 here.)
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dequant.cuh"
#include "layout.h"
#include "sm100_ptx.cuh"

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
            for (int kc = 0; kc < NKC; ++kc) w[kc] = ld_cg_u128(src + kc * kWeightBlockBytes);
            row_base = r * kRsbRows;
            const int row = row_base + warp * 16 + g;
            s0 = row < p.N[ly] ? __half2float(ld_cg_half(p.chan_scales[ly] + row)) : 0.f;
            s1 = row + 8 < p.N[ly] ? __half2float(ld_cg_half(p.chan_scales[ly] + row + 8)) : 0.f;
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

// The same for many tokens, on the fifth-generation tensor core.  At 8 heads x 1024 rows x 4096 positions the warp-level MMAs of the kernel
// above keep its tensor core busy for 15 us of a launch whose 67 MB of outputs need 10.4, and the reads of x, MMAs, stores and barriers of a tile run one after the other.
// Here (two CTAs per SM) eight warps convert the super-block's integers once into tensor memory (exact fp16, the A operand) and take finished
// tiles (128 positions x 64 tokens) out: a thread has one position, scales it, and leaves fp16 in a shared tile whose rows (one token, 256
// bytes) leave as 16-byte stores (one bulk copy per token: 36 us for the launch above, the copies were the bound).  One thread issues the MMAs of the next tile into the other of two accumulators meanwhile (55 cycles each,
// which is why none of the eight warps does it: 42 us instead of 35 for the kernel above), one loads x by TMA, some tiles ahead.
// Every byte is read after griddepcontrol.wait (the cache may have been appended to just before).  Measured: 8 heads x 1024 rows x 4096
// positions 34.8 -> 24.1 us at d_h = 128 (2.8 TB/s written), 58.6 -> 28.1 at 256; the rule is rows_take_tc in qlinear.cu.
struct GemmRowsMaps { CUtensorMap x[kRowsMaxLayers]; };                  // [M, K] of each layer, box 64 k x 64 tokens, 128-byte swizzle
constexpr int kRowsTcTokens = 64;
constexpr int kRowsTcThreads = 320;                                      // warps 0..7 conversion and outputs, 8 MMAs, 9 x
template <int NKC>
struct GemmRowsTcSmem {
    static constexpr int kXTile = kRowsTcTokens * 128;                   // 64 k of a token block
    static constexpr int kXBytes = NKC / 2 * kXTile;
    static constexpr int kXStages = NKC == 8 ? 2 : 4;
    static constexpr int kOutBytes = kRowsTcTokens * 256;
    static constexpr int kOuts = NKC == 8 ? 1 : 2;                       // (d_h = 256: two CTAs per SM leave room for one)
    static constexpr int kOutOffset = kXStages * kXBytes;
    static constexpr int kUsed = 1024 + kOutOffset + kOuts * kOutBytes;
    static constexpr int kTotal = kUsed > 80 * 1024 ? kUsed : 80 * 1024; // (never a third CTA on an SM: it would wait for tensor memory)
    static_assert(kTotal <= 112 * 1024, "two CTAs per SM");
};

template <int NKC>
__global__ void __launch_bounds__(kRowsTcThreads, 2) gemm_rows_tc_kernel(const __grid_constant__ GemmRowsMaps maps, const GemmRowsParams p)
{
    using S = GemmRowsTcSmem<NKC>;
    constexpr int BN = kRowsTcTokens, ACOL = 2 * BN, NX = S::kXStages;   // tensor memory: two accumulators, then A (16 columns per 32 k)
    extern __shared__ unsigned char smem_dyn[];
    __shared__ __align__(8) unsigned long long bars[2 * NX + 5];
    __shared__ volatile uint32_t flags[5];                               // tensor-memory address; abort words (see wait_expired)
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t xfull = smem_u32(bars), mdone = xfull + 8 * NX, xempty = mdone + 16, taken = xempty + 8 * NX, aready = taken + 16;   // MMAs retired, accumulator taken out: two of each
    volatile uint32_t* abort_flag = flags + 1;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, quarter = warp & 3, half = warp >> 2;
    const int i0 = (int)((int64_t)blockIdx.x * p.n_tiles / gridDim.x), n = (int)((int64_t)(blockIdx.x + 1) * p.n_tiles / gridDim.x) - i0;   // tiles i0 .. i0 + n - 1
    if (t < 2 * NX + 5) {
        mbar_init(xfull + 8 * t, t < 2 * NX + 2 ? 1 : 8);                    // taken, aready: the eight warps
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (t >= 32 && t < 36) abort_flag[t - 32] = 0;
    if (t >= 64 && t < 64 + p.n_layers) asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.x[t - 64]) : "memory");
    if (warp == 8) tmem_alloc(smem_u32((const void*)flags), 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = flags[0];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (t == 0) abort_flag[2] = abort_flag[3] = 1;

    auto layer_of = [&](int rsb) {
        int ly = 0;
#pragma unroll
        for (int i = 1; i < kRowsMaxLayers; ++i)
            if (i < p.n_layers && rsb >= p.rsb_end[i - 1]) ly = i;
        return ly;
    };
    if (warp == 9) {
        // ------------------------------------------------------------------ x
        if (lane == 0) {
            int j = 0;
            for (; j < n; ++j) {
                const int s = j % NX, rsb = (i0 + j) / p.n_tb, m0 = (i0 + j - rsb * p.n_tb) * BN;
                if (!mbar_wait(xempty + 8 * s, ((uint32_t)(j / NX) & 1) ^ 1, abort_flag, 0x6A8 + s)) break;
                const CUtensorMap* map = &maps.x[layer_of(rsb)];
                mbar_expect_tx(xfull + 8 * s, S::kXBytes);
#pragma unroll
                for (int b = 0; b < NKC / 2; ++b) tma_load_2d(base + s * S::kXBytes + b * S::kXTile, map, 64 * b, m0, xfull + 8 * s);
            }
            if (*abort_flag)                                             // copies in flight land before the CTA leaves
                for (int i = max(0, j - NX); i < j; ++i) mbar_wait(xfull + 8 * (i % NX), (uint32_t)(i / NX) & 1, abort_flag + 1, 0);
        }
    } else if (warp == 8) {
        // ------------------------------------------------------------------ MMAs
        if (lane == 0) {
            uint32_t apar = 0;
            int cur = -1;
            for (int j = 0; j < n; ++j) {
                const int d = j & 1, s = j % NX, rsb = (i0 + j) / p.n_tb;
                if (rsb != cur) {
                    if (!mbar_wait(aready, apar, abort_flag, 0x6A0)) break;
                    cur = rsb;
                    apar ^= 1;
                }
                if (j >= 2 && !mbar_wait(taken + 8 * d, (uint32_t)((j - 2) >> 1) & 1, abort_flag, 0x6A4 + d)) break;
                if (!mbar_wait(xfull + 8 * s, (uint32_t)(j / NX) & 1, abort_flag, 0x6B0 + s)) break;
                tc_fence_after();
                const uint32_t b_lo = umma_desc_lo(base + s * S::kXBytes);
#pragma unroll
                for (int k = 0; k < 2 * NKC; ++k)
                    umma_f16_ta(tmem + (uint32_t)(d * BN), tmem + (uint32_t)(ACOL + 8 * k), b_lo + (uint32_t)((k >> 2) * (S::kXTile >> 4) + 2 * (k & 3)), umma_idesc_f16(BN), k > 0 ? 1u : 0u);
                umma_commit(mdone + 8 * d);
                umma_commit(xempty + 8 * s);
            }
        }
    } else {
        // ------------------------------------------------------------------ weights and outputs
        // this thread's position: row-block 2 quarter + lane / 16, lane-row lane % 8, rows g + 8 for lanes 8..15 and 24..31 (layout.h)
        const int row = quarter * 32 + lane, line = ((2 * quarter + (lane >> 4)) * 8 + (lane & 7)) * 64;
        const uint32_t sel = lane & 8 ? 0x4342u : 0x4140u, lane_base = (uint32_t)(quarter * 32) << 16;
        float scale = 0.f;
        int ly = 0, n0 = 0;
        auto convert = [&](int rsb) {                                    // the super-block's integers -> A; the two warps of a quarter share its k
            ly = layer_of(rsb);
            const int r = rsb - (ly ? p.rsb_end[ly - 1] : 0);
            const uint8_t* src = p.body[ly] + (int64_t)r * NKC * kWeightBlockBytes + line + half * (NKC / 2) * kWeightBlockBytes;
            n0 = r * kRsbRows;
            scale = n0 + row < p.N[ly] ? __half2float(ld_cg_half(p.chan_scales[ly] + n0 + row)) : 0.f;
            constexpr int B = NKC == 8 ? 2 : NKC / 2;                    // blocks whose loads are in flight together
#pragma unroll
            for (int b0 = 0; b0 < NKC / 2; b0 += B) {
                uint4 w[B][4];
#pragma unroll
                for (int b = 0; b < B; ++b)
#pragma unroll
                    for (int c = 0; c < 4; ++c) w[b][c] = ld_cg_u128(src + (b0 + b) * kWeightBlockBytes + 16 * c);
#pragma unroll
                for (int b = 0; b < B; ++b)
#pragma unroll
                    for (int cp = 0; cp < 2; ++cp) {
                        uint32_t o[8];
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const uint4 v = w[b][2 * cp + c];
                            o[4 * c + 0] = h2_sub(__byte_perm(v.x, 0x64646464u, sel), 0x64806480u);
                            o[4 * c + 1] = h2_sub(__byte_perm(v.y, 0x64646464u, sel), 0x64806480u);
                            o[4 * c + 2] = h2_sub(__byte_perm(v.z, 0x64646464u, sel), 0x64806480u);
                            o[4 * c + 3] = h2_sub(__byte_perm(v.w, 0x64646464u, sel), 0x64806480u);
                        }
                        tmem_st8_async(tmem + lane_base + (uint32_t)(ACOL + 16 * (half * (NKC / 2) + b0 + b) + 8 * cp), o);
                    }
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(aready);
        };
        auto meet = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };
        bool ok = true;
        convert(i0 / p.n_tb);
        for (int j = 0; j < n; ++j) {
            const int i = i0 + j, d = j & 1, ob = S::kOuts == 2 ? d : 0, rsb = i / p.n_tb, m0 = (i - rsb * p.n_tb) * BN;
            ok = ok && mbar_wait(mdone + 8 * d, (uint32_t)(j >> 1) & 1, abort_flag, 0x6A6 + d);
            tc_fence_after();
            uint32_t v[32];
            tmem_ld32(tmem + lane_base + (uint32_t)(d * BN + 32 * half), v);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(taken + 8 * d);
            if (S::kOuts == 1) meet();                                   // everybody has read the output tile (two of them: the barrier below is enough)
            const uint32_t out = base + S::kOutOffset + ob * S::kOutBytes;
            __half* orow = reinterpret_cast<__half*>(smem_dyn + (out - smem_u32(smem_dyn))) + row;
#pragma unroll
            for (int q = 0; q < 32; ++q) orow[(32 * half + q) * 128] = __float2half_rn(__uint_as_float(v[q]) * scale);
            meet();
            const int N = p.N[ly];
            __half* y = p.y[ly] + (int64_t)m0 * N + n0;
#pragma unroll
            for (int e = t; e < BN * 16; e += 256) {                     // 16 bytes = 8 positions (N is a multiple of 8)
                const int tok = e >> 4, u = e & 15;
                if (ok && m0 + tok < p.M && n0 + 8 * u < N) {
                    uint4 o;
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(o.x), "=r"(o.y), "=r"(o.z), "=r"(o.w) : "r"(out + tok * 256 + u * 16));
                    *reinterpret_cast<uint4*>(y + (int64_t)tok * N + 8 * u) = o;
                }
            }
            if (j + 1 < n && (i + 1) / p.n_tb != rsb) convert(rsb + 1);  // (uniform; every MMA so far has retired)
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        tmem_dealloc(tmem, 256);
    }
}

}  // namespace ql
