// The KV cache held as weights (paper Section 3.8, "GPU-Optimized KV Cache Layout"): the K cache is a layer with
// O = cache positions and I = head dimension (it stands for K^T in Q K^T), the V cache a layer with O = head
// dimension and I = cache positions, so that both attention products are calls of the linear kernels and the
// second one comes out as [query rows, d_h].  Both caches are int8 blobs in the layout of layout.h.
//
// This kernel appends tokens: it quantises each new key and value vector with one scale per TOKEN,
//     s = fp16(amax / 127)  (fp32 division, rounded to fp16),   q = round-half-even(v / s) clamped to [-127, 127]
// (a vector whose scale rounds to zero is stored as zeros with scale 1), and writes the integers to the places the
// layout gives them.  For K a token is an output channel, so s is that channel's scale in the blob.  For V a token
// is an INPUT channel; its scale cannot live in the blob (a channel scale there would span all tokens), so it goes
// to a side array and is folded into the attention probabilities before the product:
//     out[r, d] = sum_t (prob[r, t] * s_v[t]) * q_v[t, d].
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "layout.h"

namespace ql {

// Byte offset, from the start of the body, of int8 weight (row, k) of a layer with n_kc chunks of 32.
__host__ __device__ __forceinline__ int64_t int8_weight_offset(int row, int k, int n_kc)
{
    const int rsb = row >> 7, rb = (row & 127) >> 4, g = row & 7, upper = (row >> 3) & 1;
    const int kc = k >> 5, c = (k & 31) >> 3, r8 = k & 7;
    const int w = ((r8 >> 2) << 1) | ((r8 >> 1) & 1), b = (r8 & 1) | (upper << 1);
    return ((int64_t)rsb * n_kc + kc) * kWeightBlockBytes + rb * 512 + ((g << 2) | c) * 16 + w * 4 + b;
}

constexpr int kKvMaxHeads = 16;          // KV heads (cache pairs of equal shape) that one append launch serves

struct KvAppendParams {
    // per head (blockIdx.y)
    uint8_t* k_body[kKvMaxHeads];        // K cache: N = cache positions, K = d_h
    __half* k_scales[kKvMaxHeads];       // its per-channel (= per-token) scales
    uint8_t* v_body[kKvMaxHeads];        // V cache: N = d_h, K = cache positions
    __half* v_scale[kKvMaxHeads];        // [cache positions] per-token scales of V (side array)
    const __half* k_new;                 // element (head h, new token i, dimension j) at h * head_stride + i * token_stride + j
    const __half* v_new;
    int64_t head_stride, token_stride;
    int32_t d_h, cache_size, pos, n_new;
    int32_t k_n_kc, v_n_kc;
};

// One CTA per new token and head, d_h <= 1024, a multiple of 32; warps in pairs, one for the key and one for the value vector, each pair
// for the 32 E dimensions of its slice.  Bound: the chain of latencies (previous kernel -> vector -> amax -> scale -> bytes); with many
// tokens and wide heads the stores, a sector of its own for every byte of V.  Every warp takes the amax of the whole vector itself (it is
// in L1 for all but the first), so there is no barrier and no shared memory.  The dependents are released only after the wait: whoever
// runs beside this kernel then knows that every kernel before it is complete, and that only the bytes of these tokens may still change.
// Measured, us, 128 threads striding over both vectors with two barriers / a warp per vector, four dimensions in a row per lane / this: one
// token of 8 heads of 128 1.81 / 1.62 / 1.62, of 1024 3.67 / 3.54 / 2.32; 256 tokens of 8 heads of 128 3.67 / 4.07 / 3.40, of 256 5.20 / 6.57 / 4.38, of
// 1024 12.0 / 19.6 / 11.4; 2048 tokens of 8 heads of 128 18.5 / 17.7 / 17.5, of 1024 60.6 / 85.3 / 71.3 (every warp reads the whole vector).
template <int E, bool SPREAD>
__global__ void __launch_bounds__(E == 2 ? 1024 : 512) kv_append_kernel(const KvAppendParams p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int i = blockIdx.x, t = p.pos + i, hd = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool value = warp & 1;
    const __half* src = (value ? p.v_new : p.k_new) + hd * p.head_stride + i * p.token_stride;
    // This lane's dimensions: E in a row for K (their bytes lie in a word or two).  For V 32 apart (SPREAD), so that the lanes of a store are
    // consecutive rows, 8 lines of 128 bytes (with 4 in a row per lane 16 lines: 2048 vectors of 1024 14.8 us instead of 11.4), or, for few
    // vectors, in a row too: one load instead of E.
    const bool apart = SPREAD && value;
    const int own = (warp >> 1) * 32 * E + (apart ? lane : lane * E), step = apart ? 32 : 1;
    __align__(2 * E) __half h[E];
    if (apart) {
#pragma unroll
        for (int e = 0; e < E; ++e) h[e] = own + 32 * e < p.d_h ? src[own + 32 * e] : __float2half_rn(0.f);
    } else if (own < p.d_h) {
        if constexpr (E == 4) *reinterpret_cast<uint2*>(h) = *reinterpret_cast<const uint2*>(src + own);
        else *reinterpret_cast<uint32_t*>(h) = *reinterpret_cast<const uint32_t*>(src + own);
    }
    __half2 mx = __float2half2_rn(0.f);
    uint4 u[4];                                                          // the whole vector, 8 values per lane and piece
#pragma unroll
    for (int j = 0; j < 4; ++j) u[j] = (lane + 32 * j) * 8 < p.d_h ? *reinterpret_cast<const uint4*>(src + (lane + 32 * j) * 8) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __half2* v = reinterpret_cast<const __half2*>(&u[j]);
        mx = __hmax2(mx, __hmax2(__hmax2(__habs2(v[0]), __habs2(v[1])), __hmax2(__habs2(v[2]), __habs2(v[3]))));
    }
    const float2 m = __half22float2(mx);
    // (bits of a non-negative float: ordered like unsigned integers)
    const float amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(m.x, m.y))));
    const __half h0 = __float2half_rn(__fdiv_rn(amax, 127.f));
    const bool dead = __half2float(h0) == 0.f;                           // a zero vector, or a scale below fp16's range: zeros, scale 1
    const float sc = dead ? 1.f : __half2float(h0);
    if (threadIdx.x < 64 && lane == 0) (value ? p.v_scale[hd] : p.k_scales[hd])[t] = __float2half_rn(sc);
    uint32_t q[E];                                                       // as stored: q + 128
#pragma unroll
    for (int e = 0; e < E; ++e) q[e] = dead ? 128u : (uint32_t)(max(-127, min(127, __float2int_rn(__fdiv_rn(__half2float(h[e]), sc)))) + 128);
    if (value) {                                                         // V: row = dimension, k = token
#pragma unroll
        for (int e = 0; e < E; ++e)                                      // (next row: 64 bytes; 32 rows: two row-blocks of 512; a slice lies in one super-block)
            if (own + step * e < p.d_h) p.v_body[hd][int8_weight_offset(own, t, p.v_n_kc) + (SPREAD ? 1024 : 64) * e] = (uint8_t)q[e];
    } else if (own < p.d_h) {                                            // K: row = token, k = dimension: pairs of k in each of a lane's words
        uint8_t* dst = p.k_body[hd] + int8_weight_offset(t, own, p.k_n_kc);
#pragma unroll
        for (int e = 0; e < E / 2; ++e) *reinterpret_cast<uint16_t*>(dst + 4 * e) = (uint16_t)(q[2 * e] | q[2 * e + 1] << 8);
    }
}

// x'[r, t] = fp16(prob[r, t] * s_v[t]): the per-token scales of V folded into the probabilities.
__global__ void __launch_bounds__(256) kv_scale_probs_kernel(const __half* prob, const __half* v_scale, __half* out, int64_t n, int T)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        out[i] = __float2half_rn(__half2float(prob[i]) * __half2float(v_scale[i % T]));
}

}  // namespace ql
