// Decode kernel for int8 layers with FEW rows and a LONG K whose input is scaled per k: the value product over a KV cache
// (paper Section 3.8: the V cache is a layer with O = d_h and I = cache positions), for all KV heads of a layer at once:
//
//   y[m, n] = sum_k fp16(x[m, k] * xscale[k]) * w[n, k]        (one rounding per product, as a separate pass would make it)
//
// Bound: latency at ordinary lengths (one head's values are 1 MB at 8192 positions), HBM beyond.  What the general kernel
// (gemv.cuh) pays here: clusters of 8 CTAs and two cluster-wide barriers to spread so few row-blocks over the GPU, and one
// trip to L2 per pair of chunks for x and its scales, because no other row-block of the CTA has brought them into L1.
// Here a CTA of 16 warps takes ONE row-block (16 rows), a warp a contiguous slice of K, and everything a chunk needs
// (weights, x, scales) travels in one ring of cp.async slots, kColsRing chunks per warp ahead: x and weights miss
// together, once.  One CTA per SM; K is split over a cluster only where the row-blocks leave SMs idle and the slices
// keep 2 chunks per warp (cols_split in qlinear.cu).  Sums: tensor core, then the 16 warps in order, then the cluster's ranks in order.
//
// Measured, append + scores + values of one layer (8 heads of 128, 4 query rows each, caches rotated past L2), with the
// general kernel / with this one: 6.0 / 5.5 us at 1280 positions, 9.0 / 8.5 at 4096, 10.7 / 10.7 at 8192, 25.5 / 21.4 at 32768.
#pragma once
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dequant.cuh"
#include "gemv.cuh"
#include "layout.h"

namespace ql {

constexpr int kColsWarps = 16;
constexpr int kColsThreads = kColsWarps * 32;
constexpr int kColsRing = 8;                     // chunks in flight per warp
constexpr int kColsSlot = 512 + 512 + 64;        // weights, x of 8 tokens, scales of one 32-k chunk
constexpr int kColsSmem = kColsWarps * kColsRing * kColsSlot;

struct GemvColsParams {
    const uint8_t* body[kGemvMaxBatch];
    const __half* chan_scales[kGemvMaxBatch];
    const __half* x[kGemvMaxBatch];              // [M, K]
    const __half* xscale[kGemvMaxBatch];         // [K]
    __half* y[kGemvMaxBatch];                    // [M, N]
    int32_t n_layers, M, N, K, n_rb, n_kc, cl, cps;   // layers of equal shape: n_rb row-blocks each
    int32_t hold0, hold1;                        // chunks that the kernel before this one may be writing (a KV cache): read after griddepcontrol.wait only
    int32_t late;                                // all of them (see GemvRowsParams)
};

__global__ void __launch_bounds__(kColsThreads, 1) gemv_cols_kernel(const GemvColsParams p)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float red[kColsWarps][128];
    __shared__ float part[128];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, c = lane & 3;
    uint32_t crank_u, cid_u;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank_u));
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(cid_u));
    const int crank = (int)crank_u, ly = (int)cid_u / p.n_rb, rb = (int)cid_u - ly * p.n_rb;
    const int ks = crank * kColsWarps + warp;
    const int kc0 = min(ks * p.cps, p.n_kc), kc1 = min(kc0 + p.cps, p.n_kc);
    const uint8_t* wsrc = p.body[ly] + ((int64_t)(rb >> 3) * p.n_kc) * kWeightBlockBytes + (rb & 7) * 512 + lane * 16;
    const __half* x = p.x[ly] + (int64_t)min(g, p.M - 1) * p.K + 8 * c;  // (K is a whole number of 32-k chunks)
    const __half* xs = p.xscale[ly] + 8 * c;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem_raw) + warp * kColsRing * kColsSlot;
    auto copy16 = [](uint32_t dst, const void* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); };
    auto copy_w = [&](int kc) {
        if (kc < kc1) copy16(ring + ((kc - kc0) & (kColsRing - 1)) * kColsSlot + lane * 16, wsrc + (int64_t)kc * kWeightBlockBytes);
    };
    auto copy_x = [&](int kc) {
        if (kc < kc1) {
            const uint32_t dst = ring + ((kc - kc0) & (kColsRing - 1)) * kColsSlot;
            if (g < p.M) copy16(dst + 512 + lane * 16, x + 32 * kc);
            if (g == 0) copy16(dst + 1024 + c * 16, xs + 32 * kc);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");             // (an empty group keeps the count in step)
    };
    auto held = [&](int kc) { return kc >= p.hold0 && kc < p.hold1; };
    if (p.late) asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = 0; i < kColsRing; ++i)
        if (!held(kc0 + i)) copy_w(kc0 + i);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = 0; i < kColsRing; ++i) {
        if (held(kc0 + i)) copy_w(kc0 + i);
        copy_x(kc0 + i);                                                 // (commits the chunk's group; what was requested earlier is part of the first)
    }

    auto lds128 = [](uint32_t addr) {
        uint4 v;
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
        return v;
    };
    float total[4] = {0.f, 0.f, 0.f, 0.f};
    for (int kc = kc0; kc < kc1; ++kc) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kColsRing - 1) : "memory");
        __syncwarp();                                                    // the scales were copied by four of the lanes
        const uint32_t slot = ring + ((kc - kc0) & (kColsRing - 1)) * kColsSlot;
        const uint4 w = lds128(slot + lane * 16), s = lds128(slot + 1024 + c * 16);
        uint4 b = make_uint4(0, 0, 0, 0);
        if (g < p.M) b = lds128(slot + 512 + lane * 16);
        __syncwarp();                                                    // everybody has read the slot
        copy_w(kc + kColsRing);
        copy_x(kc + kColsRing);
        uint32_t a[4];
        unpack_int8_words(w.x, w.y, a);
        mma_16816_pure(total, a, h2_mul(b.x, s.x), h2_mul(b.y, s.y));
        unpack_int8_words(w.z, w.w, a);
        mma_16816_pure(total, a, h2_mul(b.z, s.z), h2_mul(b.w, s.w));
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    *reinterpret_cast<float4*>(&red[warp][lane * 4]) = make_float4(total[0], total[1], total[2], total[3]);
    __syncthreads();
    // element t of the row-block: lane t / 4, register t % 4 of the accumulator fragment
    const int row = rb * kRbRows + (t >> 4) + 8 * ((t & 3) >> 1), tok = 2 * ((t >> 2) & 3) + (t & 1);
    auto store = [&](float v) {
        if (row < p.N && tok < p.M) p.y[ly][(int64_t)tok * p.N + row] = __float2half_rn(v * __half2float(p.chan_scales[ly][row]));
    };
    float v = 0.f;
    if (t < 128)
#pragma unroll
        for (int s = 0; s < kColsWarps; ++s) v += red[s][t];
    if (p.cl == 1) {
        if (t < 128) store(v);
        return;
    }
    cg::cluster_group cluster = cg::this_cluster();
    if (t < 128) part[t] = v;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // (as in gemv.cuh: only the reading CTA acquires)
    if (crank == 0) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (crank == 0 && t < 128) {
        v = 0.f;
        for (int r = 0; r < p.cl; ++r) v += *cluster.map_shared_rank(&part[t], r);
        store(v);
    }
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

}  // namespace ql
