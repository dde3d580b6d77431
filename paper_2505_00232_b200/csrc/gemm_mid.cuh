// Kernel for a batch of 9 to 64 tokens on few weights (gemm_narrow.cuh takes more: gemm_route in qlinear.cu), and for products with few output channels and any number of tokens (the
// value product of an attention over a KV cache held as weights: N = d_h).  Between the two stages of paper Section 3.7:
// too many tokens for the 8 MMA columns of the decode kernel, too few to fill the 256-token tiles of the prefill kernel,
// which then multiplies padding and, with few tiles, leaves most SMs without work.
//
// Bound: none of the limits is reached.  Llama gate + up (66 MB of int4 in groups) needs 10.3 us of HBM, and at 8.05 cycles per m16n8k16 and SM
// quarter (measured, independent MMAs) 6.6 us of MMAs at 16 tokens, 13.1 at 32; at 32 tokens it takes 37, with the tensor pipe active 32 % and
// DRAM 19 % of the time and 12 warps per SM resident: reads of x, unpack, MMAs and the waits between them add up.
//
// Work decomposition: a CTA takes one row super-block (128 channels, one row-block of 16 per warp), one block of 8 NT
// tokens and one part of K; the K parts of a tile are the CTAs of a thread-block cluster and add their fp32 partial sums
// through distributed shared memory in rank order (deterministic, no scratch in global memory).  Packed weights and x
// arrive through one ring of cp.async stages (2 chunks of weights per stage: 128 k of int4, 64 k of int8).  A weight goes
// from the packed block to the MMA's A fragment in registers, the layout's fragment order needs no exchange; x is the B
// operand, read as 16-byte pieces (8 k of one token: two MMAs' fragments), pieces of odd tokens swapped in pairs of four
// so that the 8 lanes of a shared-memory phase touch all 32 banks.  Arithmetic of the prefill kernels: exact integers,
// fp16(s * q) for grouped weights, fp32 sums, the per-channel scale on the fp32 result.
//
// Measured, weights out of HBM, against the 256-token-tile kernel that served these sizes: Llama gate + up 25.9 us at 16 tokens (47.3 before),
// 37.0 at 32 (48.9); down (33 MB) 13.7 (26.6), 18.9 (28.7); q + k + v (25 MB of int8) 8.9 (19.2), 12.4 (20.5); one 2304 x 2304 int8 layer 4.5
// (11.7), 6.0 (13.7).  Against gemm_narrow.cuh: see gemm_route in qlinear.cu.  Value product of 1024 rows over 4096 positions,
// d_h = 128: a pass over the probabilities for the scales and a single-CTA matmul on 8 CTAs 38.5 us, now 9.5; its tiles: value_tokens in qlinear.cu.
#pragma once
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dequant.cuh"
#include "layout.h"

namespace ql {

constexpr int kMidThreads = 256;
constexpr int kMidMaxLayers = 8;

struct MidParams {
    // Row units are numbered through the layers: row super-blocks, or (gated) half super-blocks of ONE layer.
    const uint8_t* body[kMidMaxLayers];
    const __half* chan_scales[kMidMaxLayers];    // nullptr when grouped
    const __half* x[kMidMaxLayers];              // [M, K] each
    // KSCALE form: fp16 factor per k, x'[m, k] = fp16(x[m, k] * kscale[k]) on the way to the tensor core (the per-token scales of
    // a value cache, as in the decode kernel).  All 8 warps repeat the products; they fit beside the MMAs.
    const __half* kscale[kMidMaxLayers];
    __half* y[kMidMaxLayers];                    // [M, N_i]
    int32_t N[kMidMaxLayers];
    int32_t unit_end[kMidMaxLayers];             // row units of layers 0..i
    int32_t n_layers, M, K, n_kc, n_steps, n_tb, cl, act;
    int32_t late;                                // the weights may come from the previous kernel (a KV cache): nothing of them is read before griddepcontrol.wait
};

template <int BITS, bool GROUPED, int NT>
struct MidSmem {
    static constexpr int kKStep = 2 * (BITS == 4 ? 64 : 32);             // k per stage: two chunks
    static constexpr int kTokens = 8 * NT;
    static constexpr int kXBytes = kTokens * kKStep * 2;
    static constexpr int kWBytes = 2 * kWeightBlockBytes;
    static constexpr int kSBytes = GROUPED ? 2 * kScaleBlockBytes : 0;
    static constexpr int kKsBytes = BITS == 8 ? kKStep * 2 : 0;          // per-k factors (KSCALE form)
    static constexpr int kStage = kXBytes + kWBytes + kSBytes + kKsBytes;
    static constexpr int kStages = 100 * 1024 / kStage < 8 ? 100 * 1024 / kStage : 8;   // two CTAs per SM
    static constexpr int kPartStride = 132;                              // floats per token of a partial tile: 2 * 132 = 8 mod 32 banks
    static constexpr int kPartBytes = kTokens * kPartStride * 4;
    static constexpr int kTotal = kStages * kStage > kPartBytes ? kStages * kStage : kPartBytes;
    static_assert(kStages >= 3 && kTotal <= 112 * 1024, "two CTAs per SM");
};

template <int BITS, bool GROUPED, int NT, bool GATED, bool KSCALE>
__global__ void __launch_bounds__(kMidThreads, 2) gemm_mid_kernel(const MidParams p)
{
    static_assert(!KSCALE || (BITS == 8 && !GATED), "the per-k factor exists for int8 layers");
    namespace cg = cooperative_groups;
    using S = MidSmem<BITS, GROUPED, NT>;
    constexpr int NS = S::kStages, CHUNK_K = BITS == 4 ? 64 : 32, BB = kWeightBlockBytes + (GROUPED ? kScaleBlockBytes : 0);
    constexpr int UNITS = S::kKStep / 8;                                 // 16-byte pieces of a token's stage
    // Warps that share a tile's tokens, each with as many row-blocks: what a warp reads of x from shared memory halves.  (The value product, whose
    // x needs arithmetic as well, 4096 rows of 4096 positions 22.8 -> 21.3 us; elsewhere the second unpacking of the weights costs more.)
    constexpr int WT = KSCALE && NT >= 4 && NT % 2 == 0 ? 2 : 1, NTW = NT / WT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, c = lane & 3;

    uint32_t crank_u, cid_u;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank_u));
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(cid_u));
    const int crank = (int)crank_u, cid = (int)cid_u;
    const int unit = cid / p.n_tb, m0 = (cid - unit * p.n_tb) * S::kTokens;
    int ly = 0;
    if (!GATED) {
#pragma unroll
        for (int i = 1; i < kMidMaxLayers; ++i)
            if (i < p.n_layers && unit >= p.unit_end[i - 1]) ly = i;
    }
    const int lunit = unit - (ly ? p.unit_end[ly - 1] : 0);
    const int rsb = GATED ? lunit >> 1 : lunit;
    const int wly = GATED ? warp >> 2 : ly;                              // layer and row-block this warp works on
    const int wrb = GATED ? (lunit & 1) * 4 + (warp & 3) : warp;
    const int st0 = (int)((int64_t)crank * p.n_steps / p.cl), st1 = (int)((int64_t)(crank + 1) * p.n_steps / p.cl);
    const uint8_t* wbase = p.body[wly] + (int64_t)rsb * p.n_kc * BB + wrb * 512 + lane * 16;
    const uint8_t* sbase = p.body[wly] + (int64_t)rsb * p.n_kc * BB + kWeightBlockBytes + wrb * 64 + (lane & 3) * 16;
    const __half* x = p.x[ly];

    auto copy16 = [](uint32_t dst, const void* src, bool in_range) {     // out of range: reads nothing, writes zeros
        const uint32_t sz = in_range ? 16u : 0u;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
    };
    auto load_weights = [&](int step, int stage) {
        const uint32_t dst = smem0 + stage * S::kStage + S::kXBytes;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int kc = 2 * step + i;
            const bool in = kc < p.n_kc;
            copy16(dst + i * kWeightBlockBytes + t * 16, wbase + (int64_t)(in ? kc : 0) * BB, in);
        }
        if (GROUPED && lane < 8) {
            const int kc = 2 * step + (lane >> 2);
            const bool in = kc < p.n_kc;
            copy16(dst + S::kWBytes + (lane >> 2) * kScaleBlockBytes + warp * 64 + (lane & 3) * 16, sbase + (int64_t)(in ? kc : 0) * BB, in);
        }
    };
    auto load_x = [&](int step, int stage) {
        const uint32_t dst = smem0 + stage * S::kStage;
#pragma unroll
        for (int i0 = 0; i0 < S::kTokens * UNITS; i0 += kMidThreads) {
            const int i = i0 + t;
            if (S::kTokens * UNITS % kMidThreads == 0 || i < S::kTokens * UNITS) {
                const int tok = i / UNITS, u = i % UNITS;
                const int k = step * S::kKStep + u * 8;
                const bool in = m0 + tok < p.M && k < p.K;
                copy16(dst + tok * (S::kKStep * 2) + ((u ^ ((tok & 1) << 2)) << 4), in ? x + (int64_t)(m0 + tok) * p.K + k : x, in);
            }
        }
        if (KSCALE && t < UNITS) {
            const int k = step * S::kKStep + t * 8;
            copy16(dst + S::kXBytes + S::kWBytes + S::kSBytes + t * 16, p.kscale[ly] + (k < p.K ? k : 0), k < p.K);
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

    // Weights do not depend on the previous kernel: those of the first stages are requested before waiting for it.
    if (p.late) asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
    for (int s = 0; s < NS - 1; ++s)
        if (st0 + s < st1) load_weights(st0 + s, s);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // Output element of this thread: 4 channels (the same in every pass over the tokens); their scales are weights too.
    constexpr int QUADS = GATED ? 16 : 32;
    const int quad = t % QUADS;
    const int row0 = GATED ? rsb * kRsbRows + (lunit & 1) * 64 + quad * 4 : rsb * kRsbRows + quad * 4;
    const int N = p.N[GATED ? 0 : ly];
    uint2 cs[2] = {make_uint2(0x3C003C00u, 0x3C003C00u), make_uint2(0x3C003C00u, 0x3C003C00u)};
    if (!GROUPED && row0 < N) {
        cs[0] = ld_cg_u64(p.chan_scales[GATED ? 0 : ly] + row0);
        if (GATED) cs[1] = ld_cg_u64(p.chan_scales[1] + row0);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
    for (int s = 0; s < NS - 1; ++s) {
        if (st0 + s < st1) load_x(st0 + s, s);
        commit();
    }

    const int rb0 = WT == 1 ? warp : WT * (warp & 3), n0 = WT == 1 ? 0 : (warp >> 2) * NTW;   // this warp's row-blocks and groups of 8 tokens
    float acc[WT][NTW][4];
#pragma unroll
    for (int j = 0; j < WT; ++j)
#pragma unroll
        for (int n = 0; n < NTW; ++n) acc[j][n][0] = acc[j][n][1] = acc[j][n][2] = acc[j][n][3] = 0.f;
    auto lds128 = [](uint32_t addr) {
        uint4 v;
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
        return v;
    };
    // 32-k group G of the stage: this lane's piece of token 8 n + g
    const uint32_t x_warp = (uint32_t)(n0 * 8 * S::kKStep * 2);
    const uint32_t xl[2] = {x_warp + (uint32_t)(g * S::kKStep * 2 + (g & 1) * 64 + c * 16), x_warp + (uint32_t)(g * S::kKStep * 2 + ((g & 1) ^ 1) * 64 + c * 16)};
    auto group = [&](uint32_t xs, int G, const uint32_t a0[WT][4], const uint32_t a1[WT][4], const uint4& f) {
        const uint32_t xa = xs + xl[G & 1] + (G >> 1) * 128;
#pragma unroll
        for (int n = 0; n < NTW; ++n) {
            uint4 b = lds128(xa + n * 8 * S::kKStep * 2);
            if (KSCALE) b = make_uint4(h2_mul(b.x, f.x), h2_mul(b.y, f.y), h2_mul(b.z, f.z), h2_mul(b.w, f.w));
#pragma unroll
            for (int j = 0; j < WT; ++j) {
                mma_16816_pure(acc[j][n], a0[j], b.x, b.y);
                mma_16816_pure(acc[j][n], a1[j], b.z, b.w);
            }
        }
    };
    int stage = 0;
    for (int step = st0; step < st1; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
        __syncthreads();                                                 // the stage has landed; everybody is done with the one refilled next
        {
            const int nxt = step + NS - 1, ns = stage == 0 ? NS - 1 : stage - 1;
            if (nxt < st1) { load_weights(nxt, ns); load_x(nxt, ns); }
            commit();
        }
        const uint32_t xs = smem0 + stage * S::kStage, ws = xs + S::kXBytes;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
            if (BITS == 4) {
                const uint4 w = lds128(ws + ch * kWeightBlockBytes + t * 16);
                const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
                uint2 sc = make_uint2(0, 0);
                if (GROUPED) asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(sc.x), "=r"(sc.y) : "r"(ws + S::kWBytes + ch * kScaleBlockBytes + warp * 64 + g * 8));
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t a0[WT][4], a1[WT][4];
                    unpack_int4_word(ww[2 * h], a0[0]);
                    unpack_int4_word(ww[2 * h + 1], a1[0]);
                    if (GROUPED) {
                        const uint32_t lo = __byte_perm(sc.x, 0, h ? 0x3232 : 0x1010), hi = __byte_perm(sc.y, 0, h ? 0x3232 : 0x1010);
                        a0[0][0] = h2_mul(a0[0][0], lo); a0[0][1] = h2_mul(a0[0][1], hi); a0[0][2] = h2_mul(a0[0][2], lo); a0[0][3] = h2_mul(a0[0][3], hi);
                        a1[0][0] = h2_mul(a1[0][0], lo); a1[0][1] = h2_mul(a1[0][1], hi); a1[0][2] = h2_mul(a1[0][2], lo); a1[0][3] = h2_mul(a1[0][3], hi);
                    }
                    group(xs, 2 * ch + h, a0, a1, make_uint4(0, 0, 0, 0));
                }
            } else {
                uint32_t a0[WT][4], a1[WT][4];
#pragma unroll
                for (int j = 0; j < WT; ++j) {
                    const uint4 w = lds128(ws + ch * kWeightBlockBytes + (rb0 + j) * 512 + lane * 16);
                    unpack_int8_words(w.x, w.y, a0[j]);
                    unpack_int8_words(w.z, w.w, a1[j]);
                }
                uint4 f = make_uint4(0, 0, 0, 0);
                if (KSCALE) f = lds128(ws + S::kWBytes + S::kSBytes + ch * CHUNK_K * 2 + c * 16);
                group(xs, ch, a0, a1, f);
            }
        }
        if (++stage == NS) stage = 0;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                                     // the ring is free: the partial tile takes its place

    float* part = reinterpret_cast<float*>(smem_raw);                    // [token][channel]
#pragma unroll
    for (int j = 0; j < WT; ++j)
#pragma unroll
        for (int n = 0; n < NTW; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) part[(8 * (n0 + n) + 2 * c + (i & 1)) * S::kPartStride + (rb0 + j) * 16 + g + 8 * (i >> 1)] = acc[j][n][i];
    cg::cluster_group cluster = cg::this_cluster();
    if (p.cl > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else __syncthreads();
    // rank r finishes tokens r, r + cl, ... of the tile
    const float sc0[4] = {__low2float(*reinterpret_cast<__half2*>(&cs[0].x)), __high2float(*reinterpret_cast<__half2*>(&cs[0].x)),
                          __low2float(*reinterpret_cast<__half2*>(&cs[0].y)), __high2float(*reinterpret_cast<__half2*>(&cs[0].y))};
    const float sc1[4] = {__low2float(*reinterpret_cast<__half2*>(&cs[1].x)), __high2float(*reinterpret_cast<__half2*>(&cs[1].x)),
                          __low2float(*reinterpret_cast<__half2*>(&cs[1].y)), __high2float(*reinterpret_cast<__half2*>(&cs[1].y))};
    for (int tok = crank + (t / QUADS) * p.cl; tok < S::kTokens && m0 + tok < p.M; tok += (kMidThreads / QUADS) * p.cl) {
        float v[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f};
        const float* src = part + tok * S::kPartStride + quad * 4;
        for (int r = 0; r < p.cl; ++r) {
            const float* s = p.cl > 1 ? cluster.map_shared_rank(src, r) : src;
            const float4 a = *reinterpret_cast<const float4*>(s);
            v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
            if (GATED) {
                const float4 b = *reinterpret_cast<const float4*>(s + 64);
                u[0] += b.x; u[1] += b.y; u[2] += b.z; u[3] += b.w;
            }
        }
        if (!GROUPED) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { v[i] *= sc0[i]; if (GATED) u[i] *= sc1[i]; }
        }
        if (GATED) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = gate_activation(v[i], p.act) * u[i];
        }
        if (row0 < N) {                                                  // (N is a multiple of 8: the four channels exist together)
            uint2 o;
            *reinterpret_cast<__half2*>(&o.x) = __floats2half2_rn(v[0], v[1]);
            *reinterpret_cast<__half2*>(&o.y) = __floats2half2_rn(v[2], v[3]);
            *reinterpret_cast<uint2*>(p.y[GATED ? 0 : ly] + (int64_t)(m0 + tok) * N + row0) = o;
        }
    }
    // peers keep their partial tile alive until it has been read: a rendezvous only
    if (p.cl > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

}  // namespace ql
