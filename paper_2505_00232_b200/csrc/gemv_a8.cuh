// Decode kernel with int8 activations (paper Section 3.7: in the memory-bound decode stage the quantisation of
// the input activations is done INSIDE the fully-connected kernel, and the products with the pre-quantised
// weights use integer instructions, with the dequantisation applied to the output).
//
// Steps, in the order the section gives them:
//   1. quantise x per token:  amax = max |x[m,:]|,  r = 127 / amax,  xq = round-half-even(x * r) clamped to
//      [-127, 127],  scale_x = amax / 127  (IEEE fp32 operations, one rounding each; a zero row: scale 1, xq 0)
//   2. integer dot products of xq with the stored weight integers on the tensor cores
//      (mma.m16n8k32, u8 x s8 -> s32): exact
//   3. dequantise the output:  y = scale_x[m] * sum_g s[n,g] * acc[m,n,g]   (fp32), rounded once to fp16
//
// Work decomposition, ring and reductions are those of gemv.cuh: a warp owns one row-block and one K slice.  The
// weights are stored with an offset (q + 8, q + 128), so the products come out as sum (q + off) * xq; the term
// off * sum xq is known per token and 32-k group once x is quantised, and enters the MMA as its accumulator input.
// The quantisation stands between the stream dependency and the first product, in every CTA, so it is kept short: the token
// count is a template parameter, all tokens' loads of a turn are in flight together, the maximum is taken on packed fp16
// and by one warp reduction, every thread forms the reciprocals itself, and short rows are quantised from the registers they
// were measured in.  Measured (weights out of HBM, before / after): 4096 x 4096 int8 at 1 token 8.0 / 7.1 us, at 4 tokens
// 11.9 / 8.4; 14336 x 4096 int4 per channel 10.7 / 9.4 and 17.6 / 12.4; 4096 x 14336 int4 12.0 / 10.3 and 24.0 / 23.5 (two
// reads of rows that long).  Since then the chunks go in pairs and a warp adds the offset terms of its groups across its lanes (one after the
// other they were a chain of shared-memory loads at the end): 7.1 / 6.5, 9.3 / 8.2 and 10.3 / 9.4 at 1 token.  Tried and not better: the
// maxima of a cluster's K ranges through distributed shared memory, rounding by an addition instead of a conversion.
// int4 unpack is two logic operations per 8 weights (the low and the high nibbles of a word are the 4-byte
// operand registers of rows g and g + 8), against nine for the fp16 path.
#pragma once
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemv.cuh"
#include "layout.h"

namespace ql {

struct GemvA8Params {
    const uint8_t* body;
    const __half* chan_scales;           // per-channel scales (nullptr when grouped)
    const __half* x;                     // [M, K] fp16
    __half* y;                           // [M, N]
    int32_t M, N, K;
    int32_t n_rb, n_kc, block_bytes;
    int32_t ks_cta, ks_cta_log2, cl, cps;
    int32_t xq_stride;                   // bytes between tokens in the shared xq slab (span + 32: rows land 8 banks apart)
    int32_t xq_bytes;                    // bytes of the slab
    int32_t sg_bytes;                    // bytes of the per-group sums that follow it
};

// D = A (16 x 32, u8: stored weight integers) . B (32 x 8, s8: quantised activations) + C, exact in s32.
__device__ __forceinline__ void imma_16832(int d[4], const uint32_t a[4], uint32_t b0, uint32_t b1, const int c[4])
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]));
}

// Step 1 for one value, bit for bit as stated above.  |x| <= amax gives |x * r| <= 127 (1 + 2^-22), which rounds
// into [-127, 127] by itself: the clamp of the definition never acts, and is left to the byte packing's saturation.
__device__ __forceinline__ int quantize_one(float x, float r) { return __float2int_rn(__fmul_rn(x, r)); }

// Four s32 values in [-128, 127] as the four bytes of a word (lowest byte first).
__device__ __forceinline__ uint32_t pack_s8x4(int b0, int b1, int b2, int b3)
{
    uint32_t hi, out;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(b3), "r"(b2));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(out) : "r"(b1), "r"(b0), "r"(hi));
    return out;
}
// Sum of the four signed bytes of a word.
__device__ __forceinline__ int sum_s8x4(uint32_t w) { return __dp4a((int)w, 0x01010101, 0); }

// What the planner counts on: the CTAs per SM that the registers allow, and a CTA's shared memory beside the dynamic part
// (static arrays, and the 1 KB that the system keeps per CTA).
constexpr int kGemvA8MaxResident = 4;
constexpr int kGemvA8OtherSmem = 5 * 1024 + 1024;

// T: 1, 2, 4 or 8, at least M: the quantisation steps are unrolled over the tokens that exist, not over all 8 columns.
template <int BITS, bool GROUPED, int T>
__global__ void __launch_bounds__(kGemvThreads, kGemvA8MaxResident) gemv_a8_kernel(const GemvA8Params p)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kGemvWarps][128];                                 // per-warp results: s32, or fp32 bits when GROUPED
    __shared__ int part[128];
    __shared__ float amax_w[kGemvWarps][8];
    __shared__ float scale_x[8];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, c = lane & 3;
    constexpr int CHUNK_K = BITS == 4 ? 64 : 32;
    constexpr int OFFSET = BITS == 4 ? 8 : 128;                          // storage offset of the weight integers

    uint32_t crank_u, rb_group_u;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank_u));
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(rb_group_u));
    const int crank = (int)crank_u, rb_group = (int)rb_group_u;
    const int rb_per_cta = kGemvWarps >> p.ks_cta_log2;
    const int ks_local = warp & (p.ks_cta - 1);
    const int rb = rb_group * rb_per_cta + (warp >> p.ks_cta_log2);
    const bool rb_live = rb < p.n_rb;
    const int ks = crank * p.ks_cta + ks_local;
    const int kc0 = min(ks * p.cps, p.n_kc);
    const int kc1 = rb_live ? min(kc0 + p.cps, p.n_kc) : kc0;
    const int kc_cta0 = min(crank * p.ks_cta * p.cps, p.n_kc);           // first chunk of this CTA's K range
    const int kc_cta1 = min(kc_cta0 + p.ks_cta * p.cps, p.n_kc);
    const int k_cta0 = kc_cta0 * CHUNK_K, span = (kc_cta1 - kc_cta0) * CHUNK_K;

    signed char* xq = reinterpret_cast<signed char*>(smem_raw);          // [M][xq_stride], int4: each 4 k stored in order 0, 2, 1, 3
    int* sg = reinterpret_cast<int*>(smem_raw + p.xq_bytes);             // [32-k groups of the span][8 tokens]: -OFFSET * sum xq
    constexpr int WARP_SMEM = kGemvRing * 512 + (GROUPED ? 2 * 512 : 0);
    unsigned char* ring = smem_raw + p.xq_bytes + p.sg_bytes + warp * WARP_SMEM;
    unsigned char* sbuf = ring + kGemvRing * 512;
    const uint32_t ring_u32 = (uint32_t)__cvta_generic_to_shared(ring) + lane * 16;
    const uint32_t sbuf_u32 = (uint32_t)__cvta_generic_to_shared(sbuf) + lane * 16;
    const uint8_t* blk = p.body + ((int64_t)(rb >> 3) * p.n_kc + kc0) * p.block_bytes;
    const uint8_t* wsrc = blk + (rb & 7) * 512 + lane * 16;
    const int s_off = (lane >> 2) * p.block_bytes + kWeightBlockBytes - (rb & 7) * 448 + (lane & 3) * 16 - lane * 16;

    auto copy16 = [](uint32_t dst, const void* src, bool in_range) {     // out of range: reads nothing, writes zeros
        const uint32_t sz = in_range ? 16u : 0u;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

    // Weights do not depend on the previous kernel: fill the ring before waiting for it.
    if (GROUPED) copy16(sbuf_u32, wsrc + s_off, kc0 + (lane >> 2) < kc1);
#pragma unroll
    for (int d = 0; d < kGemvRing; ++d) {                                // one commit group per pair of chunks
        copy16(ring_u32 + d * 512, wsrc, kc0 + d < kc1);
        if (d & 1) commit();
        wsrc += p.block_bytes;
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // One token: the per-channel scales of the (at most 4) outputs that this thread will store, which are weights too, are requested now, so that
    // their latency does not sit at the very end (4096 x 4096 int8 7.0 -> 6.5 us; with more tokens their registers are worth more, 8 tokens 12.0 -> 12.4).
    constexpr bool EARLY_SCALES = T == 1 && !GROUPED;
    const int t = threadIdx.x;
    [[maybe_unused]] unsigned short pre_scale[4];
    if (EARLY_SCALES) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int idx = t + k * kGemvThreads;
            const int row = (rb_group * rb_per_cta + (idx >> 7)) * kRbRows + ((idx & 127) >> 4) + 8 * ((idx >> 1) & 1);
            pre_scale[k] = idx < (p.cl > 1 ? 128 : rb_per_cta * 128) && row < p.N ? __half_as_ushort(p.chan_scales[row]) : 0;
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- step 1a: amax of every token over its WHOLE row (every CTA needs it, whatever its K range)
    // A thread's eight vectors in flight are J of each token; rows of up to 2048 J values stay in registers for step 1b.
    constexpr int J = 8 / T;
    const int vec_per_row = p.K >> 3;
    const bool keep = vec_per_row <= J * kGemvThreads;
    uint4 u[8];                                                          // [j][m]
    float recip[T];
    {
        __half2 mx[T];
#pragma unroll
        for (int m = 0; m < T; ++m) mx[m] = __float2half2_rn(0.f);
        for (int v0 = threadIdx.x; v0 < vec_per_row; v0 += J * kGemvThreads) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int m = i % T, v = v0 + (i / T) * kGemvThreads;
                u[i] = m < p.M && v < vec_per_row ? reinterpret_cast<const uint4*>(p.x + (int64_t)m * p.K)[v] : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const __half2* h = reinterpret_cast<const __half2*>(&u[i]);
#pragma unroll
                for (int k = 0; k < 4; ++k) mx[i % T] = __hmax2(mx[i % T], __habs2(h[k]));
            }
        }
        uint32_t am[T];                                                  // bits of a non-negative float: ordered like unsigned integers
#pragma unroll
        for (int m = 0; m < T; ++m) {
            const float2 f = __half22float2(mx[m]);
            am[m] = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(f.x, f.y)));
        }
        if (lane < T) {
            uint32_t mine = am[0];
#pragma unroll
            for (int m = 1; m < T; ++m) mine = lane == m ? am[m] : mine;
            amax_w[warp][lane] = __uint_as_float(mine);
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < T; ++m) {                                    // (every thread: cheaper than a second barrier)
            float a = amax_w[0][m];
#pragma unroll
            for (int w = 1; w < kGemvWarps; ++w) a = fmaxf(a, amax_w[w][m]);
            const bool live = a > 0.f;
            const float safe = live ? a : 1.f;
            recip[m] = __fdiv_rn(127.f, safe);
            if (threadIdx.x == m) scale_x[m] = live ? __fdiv_rn(safe, 127.f) : 1.f;
        }
    }
    // ---- step 1b: quantise this CTA's K range, and -OFFSET * (sum of xq) per token and 32-k group
    // (8 values per thread and turn, the 4 threads of a 32-k group are neighbours)
    auto quantise8 = [&](const uint4& x8, float r, int m, int v, bool in) {   // v: vector inside the CTA's range
        const __half2* h = reinterpret_cast<const __half2*>(&x8);
        int q8[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(h[j]);
            q8[2 * j] = quantize_one(f.x, r);
            q8[2 * j + 1] = quantize_one(f.y, r);
        }
        uint2 out;
        if (BITS == 4) { out.x = pack_s8x4(q8[0], q8[2], q8[1], q8[3]); out.y = pack_s8x4(q8[4], q8[6], q8[5], q8[7]); }
        else { out.x = pack_s8x4(q8[0], q8[1], q8[2], q8[3]); out.y = pack_s8x4(q8[4], q8[5], q8[6], q8[7]); }
        if (in) *reinterpret_cast<uint2*>(xq + m * p.xq_stride + v * 8) = out;
        int s8 = sum_s8x4(out.x) + sum_s8x4(out.y);
        s8 += __shfl_xor_sync(0xffffffffu, s8, 1);
        s8 += __shfl_xor_sync(0xffffffffu, s8, 2);
        if (in && (lane & 3) == 0) sg[(v >> 2) * 8 + m] = -OFFSET * s8;
    };
    const int vec_span = span >> 3;
    if (keep) {
        // (a thread whose vectors all lie beyond the row has loaded nothing into u: nothing of it is stored)
        const int v_first = k_cta0 >> 3, v_end = max(0, min(vec_span, vec_per_row - v_first));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = i / T, m = i % T, v = (int)threadIdx.x + j * kGemvThreads - v_first;
            if (m < p.M && j * kGemvThreads < v_first + vec_span && (j + 1) * kGemvThreads > v_first) quantise8(u[i], recip[m], m, v, v >= 0 && v < v_end);
        }
        // the last chunk of int4 can be half padding: 32 k of zeros, which the MMAs multiply by whatever the blob holds there
        if (BITS == 4 && v_end < vec_span && (int)threadIdx.x < 4 * p.M) {   // (whole chunks: v_end = vec_span - 4)
            const int m = threadIdx.x >> 2, v = v_end + (threadIdx.x & 3);
            *reinterpret_cast<uint2*>(xq + m * p.xq_stride + v * 8) = make_uint2(0, 0);
            if ((threadIdx.x & 3) == 0) sg[(v >> 2) * 8 + m] = 0;
        }
    } else {
        constexpr int LOG = T == 8 ? 3 : T == 4 ? 2 : T == 2 ? 1 : 0;
        const int total = vec_span << LOG;
        constexpr int B = 4;                                             // turns whose loads are issued together
        for (int i0 = warp * 32; i0 < total; i0 += B * kGemvThreads) {
            uint4 xb[B];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int i = i0 + b * kGemvThreads + lane, m = (i >> 2) & (T - 1), v = ((i >> (2 + LOG)) << 2) | (i & 3);
                const int k = k_cta0 + v * 8;
                xb[b] = make_uint4(0, 0, 0, 0);
                if (i < total && m < p.M && k < p.K) xb[b] = *reinterpret_cast<const uint4*>(p.x + (int64_t)m * p.K + k);
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                if (i0 + b * kGemvThreads >= total) break;               // (warp-uniform)
                const int i = i0 + b * kGemvThreads + lane, m = (i >> 2) & (T - 1), v = ((i >> (2 + LOG)) << 2) | (i & 3);
                float r = recip[0];
#pragma unroll
                for (int mm = 1; mm < T; ++mm) r = m == mm ? recip[mm] : r;
                quantise8(xb[b], r, m, v, i < total && m < p.M);
            }
        }
    }
    __syncthreads();

    // ---- steps 2 and 3 over this warp's chunks
    float ftotal[4] = {0.f, 0.f, 0.f, 0.f};                              // GROUPED: sum_g s * acc, fp32
    int itotal[4] = {0, 0, 0, 0};                                        // per channel: the integer sum (offset term added below)
    const signed char* xrow = xq + min(g, p.M - 1) * p.xq_stride + 8 * c;   // columns g >= M copy the last token, never stored
    [[maybe_unused]] const uint32_t sc_u32 = sbuf_u32 - lane * 16 + g * 8;   // (read by the grouped form only)
    int sflip = 0;
    auto chunk_math = [&](const uint4& w, const uint2& sc, int kl) {     // kl: first k of the chunk inside the CTA's range
        if (BITS == 4) {
            const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int h = 0; h < 2; ++h) {                                // the chunk's two 32-k groups
                uint32_t a[4];
                a[0] = ww[2 * h] & 0x0F0F0F0Fu;                          // row g:     k 8c + {0, 2, 1, 3}
                a[1] = (ww[2 * h] >> 4) & 0x0F0F0F0Fu;                   // row g + 8
                a[2] = ww[2 * h + 1] & 0x0F0F0F0Fu;                      // row g:     k 8c + 4 + {0, 2, 1, 3}
                a[3] = (ww[2 * h + 1] >> 4) & 0x0F0F0F0Fu;
                const uint2 xb = *reinterpret_cast<const uint2*>(xrow + kl + 32 * h);
                if (GROUPED) {
                    const int2 off = *reinterpret_cast<const int2*>(sg + ((kl >> 5) + h) * 8 + 2 * c);
                    const int cin[4] = {off.x, off.y, off.x, off.y};
                    int acc[4];
                    imma_16832(acc, a, xb.x, xb.y, cin);
                    const __half2 s_lo = *reinterpret_cast<const __half2*>(&sc.x);      // row g:   G0, G1
                    const __half2 s_hi = *reinterpret_cast<const __half2*>(&sc.y);      // row g+8: G0, G1
                    const float s0 = h == 0 ? __low2float(s_lo) : __high2float(s_lo);
                    const float s8 = h == 0 ? __low2float(s_hi) : __high2float(s_hi);
                    ftotal[0] = fmaf(s0, (float)acc[0], ftotal[0]);
                    ftotal[1] = fmaf(s0, (float)acc[1], ftotal[1]);
                    ftotal[2] = fmaf(s8, (float)acc[2], ftotal[2]);
                    ftotal[3] = fmaf(s8, (float)acc[3], ftotal[3]);
                } else {
                    imma_16832(itotal, a, xb.x, xb.y, itotal);
                }
            }
        } else {
            uint32_t a[4];
            a[0] = __byte_perm(w.x, w.y, 0x5410);                        // row g:     k 8c + 0..3
            a[1] = __byte_perm(w.x, w.y, 0x7632);                        // row g + 8
            a[2] = __byte_perm(w.z, w.w, 0x5410);                        // row g:     k 8c + 4..7
            a[3] = __byte_perm(w.z, w.w, 0x7632);
            const uint2 xb = *reinterpret_cast<const uint2*>(xrow + kl);
            imma_16832(itotal, a, xb.x, xb.y, itotal);
        }
    };
    for (int kc = kc0; kc < kc1; kc += kGemvRing) {
#pragma unroll
        for (int d = 0; d < kGemvRing; d += 2) {                         // two chunks read and their slots refilled before the math
            if (kc + d >= kc1) break;
            asm volatile("cp.async.wait_group %0;" ::"n"(kGemvRing / 2 - 1) : "memory");
            if (GROUPED && d == 0) {
                __syncwarp();                                            // scales of this pass visible; last pass's reads done
                copy16(sbuf_u32 + (sflip ^ 1) * 512, wsrc + s_off, kc + kGemvRing + (lane >> 2) < kc1);
            }
            const uint4 w0 = *reinterpret_cast<const uint4*>(ring + d * 512 + lane * 16);
            const uint4 w1 = *reinterpret_cast<const uint4*>(ring + (d + 1) * 512 + lane * 16);
            uint2 sc0 = make_uint2(0, 0), sc1 = make_uint2(0, 0);
            if (GROUPED) {
                sc0 = *reinterpret_cast<const uint2*>(sbuf + sflip * 512 + d * 64 + g * 8);
                sc1 = *reinterpret_cast<const uint2*>(sbuf + sflip * 512 + (d + 1) * 64 + g * 8);
            }
            copy16(ring_u32 + d * 512, wsrc, kc + d + kGemvRing < kc1);
            copy16(ring_u32 + (d + 1) * 512, wsrc + p.block_bytes, kc + d + 1 + kGemvRing < kc1);
            commit();
            wsrc += 2 * (int64_t)p.block_bytes;
            const int kl = (kc + d - kc_cta0) * CHUNK_K;
            chunk_math(w0, sc0, kl);
            if (kc + d + 1 < kc1) chunk_math(w1, sc1, kl + CHUNK_K);
        }
        sflip ^= 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (!GROUPED) {                                                      // the offset term of this warp's K slice, per token column
        // (lane (g, c) takes every eighth group of its two columns)
        const int g0 = ((kc0 - kc_cta0) * CHUNK_K) >> 5, g1 = ((kc1 - kc_cta0) * CHUNK_K) >> 5;
        int o0 = 0, o1 = 0;
        for (int gi = g0 + g; gi < g1; gi += 8) {
            const int2 off = *reinterpret_cast<const int2*>(sg + gi * 8 + 2 * c);
            o0 += off.x; o1 += off.y;
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) { o0 += __shfl_xor_sync(0xffffffffu, o0, o); o1 += __shfl_xor_sync(0xffffffffu, o1, o); }
        itotal[0] += o0; itotal[1] += o1; itotal[2] += o0; itotal[3] += o1;
    }

    // ---- K reduction across warps (shared memory), then across the cluster (distributed shared memory)
    if (GROUPED) *reinterpret_cast<float4*>(&red[warp][lane * 4]) = make_float4(ftotal[0], ftotal[1], ftotal[2], ftotal[3]);
    else *reinterpret_cast<int4*>(&red[warp][lane * 4]) = make_int4(itotal[0], itotal[1], itotal[2], itotal[3]);
    __syncthreads();

    // element e of a row-block's 128 results: lane e / 4, register e % 4
    auto store_out = [&](int rbl, int e, float fsum, int isum, float early) {
        const int out_rb = rb_group * rb_per_cta + rbl;
        const int el = e >> 2, i = e & 3;
        const int row = out_rb * kRbRows + (el >> 2) + 8 * (i >> 1);
        const int tok = 2 * (el & 3) + (i & 1);
        if (row < p.N && tok < p.M) {
            const float v = GROUPED ? fsum : (EARLY_SCALES ? early : __half2float(p.chan_scales[row])) * (float)isum;
            p.y[(int64_t)tok * p.N + row] = __float2half_rn(scale_x[tok] * v);
        }
    };
    auto add = [](float& f, int& i, int bits) {
        if (GROUPED) f += __int_as_float(bits); else i += bits;
    };

    if (p.cl > 1) {                                                      // ks_cta == 8: one row-block per CTA
        cg::cluster_group cluster = cg::this_cluster();
        if (t < 128) {
            float f = 0.f; int i = 0;
            for (int s = 0; s < kGemvWarps; ++s) add(f, i, red[s][t]);
            part[t] = GROUPED ? __float_as_int(f) : i;
        }
        cluster.sync();
        if (crank == 0 && t < 128) {
            float f = 0.f; int i = 0;
            for (int r = 0; r < p.cl; ++r) add(f, i, *cluster.map_shared_rank(&part[t], r));
            store_out(0, t, f, i, EARLY_SCALES ? __half2float(__ushort_as_half(pre_scale[0])) : 0.f);
        }
        // peers keep `part` alive until it has been read: a rendezvous only (relaxed arrive, plain wait)
        asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    } else {
        // (rb_per_cta <= 8: at most 4 elements per thread)
        auto finish = [&](int idx, unsigned short early) {
            const int rbl = idx >> 7, e = idx & 127;
            float f = 0.f; int i = 0;
            for (int s = 0; s < p.ks_cta; ++s) add(f, i, red[rbl * p.ks_cta + s][e]);
            store_out(rbl, e, f, i, EARLY_SCALES ? __half2float(__ushort_as_half(early)) : 0.f);
        };
        if constexpr (EARLY_SCALES) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (t + k * kGemvThreads < rb_per_cta * 128) finish(t + k * kGemvThreads, pre_scale[k]);
        } else {
            for (int idx = t; idx < rb_per_cta * 128; idx += kGemvThreads) finish(idx, 0);
        }
    }
}

// The quantisation kernel of the prefill stage (Section 3.7): x fp16 [M, K] -> xq int8 [M, K] and one fp32
// scale per token, by the same steps as above; rowsum (may be null) receives the sum of each quantised row, which
// the integer matmul needs to remove the weights' storage offset.  One CTA per token.
__global__ void __launch_bounds__(256) quantize_activations_kernel(const __half* x, signed char* xq, float* scale, int32_t* rowsum, int M, int K)
{
    __shared__ float wmax[8];
    __shared__ int wsum[8];
    __shared__ float recip;
    // the matmul behind it may set up and request its weights; it reads what is written here, in scratch that the matmul before may still be
    // reading, past its own wait (its epilogue with loads that pass L1 by; the form that reads it as constant data starts when this grid is complete)
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
    const int m = blockIdx.x;
    const uint4* row = reinterpret_cast<const uint4*>(x + (int64_t)m * K);
    float am = 0.f;
    for (int v = threadIdx.x; v < (K >> 3); v += 256) {
        const uint4 u = row[v];
        const __half2* h = reinterpret_cast<const __half2*>(&u);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(h[j]);
            am = fmaxf(am, fmaxf(fabsf(f.x), fabsf(f.y)));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = am;
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = 0.f;
        for (int w = 0; w < 8; ++w) a = fmaxf(a, wmax[w]);
        const bool live = a > 0.f;
        const float safe = live ? a : 1.f;
        recip = __fdiv_rn(127.f, safe);
        scale[m] = live ? __fdiv_rn(safe, 127.f) : 1.f;
    }
    __syncthreads();
    const float r = recip;
    int total = 0;
    for (int v = threadIdx.x; v < (K >> 3); v += 256) {
        const uint4 u = row[v];
        const __half2* h = reinterpret_cast<const __half2*>(&u);
        int q8[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(h[j]);
            q8[2 * j] = quantize_one(f.x, r);
            q8[2 * j + 1] = quantize_one(f.y, r);
        }
        uint2 out;
        out.x = pack_s8x4(q8[0], q8[1], q8[2], q8[3]);
        out.y = pack_s8x4(q8[4], q8[5], q8[6], q8[7]);
        *reinterpret_cast<uint2*>(xq + (int64_t)m * K + v * 8) = out;
        total += sum_s8x4(out.x) + sum_s8x4(out.y);
    }
    if (rowsum) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = total;
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
            for (int w = 0; w < 8; ++w) t += wsum[w];
            rowsum[m] = t;
        }
    }
}

}  // namespace ql
