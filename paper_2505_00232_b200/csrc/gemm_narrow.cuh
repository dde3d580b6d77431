// Kernel for a batch of tokens on the fifth-generation tensor core, and for prompts on layers too small to fill the CTA-pair tiles of
// the prefill kernel.  Between the two stages of paper Section 3.7.
//
// Why beside gemm_mid.cuh, the same with warp-level MMAs: there every 8 tokens cost another MMA per weight fragment and another read of x
// (8.05 cycles per m16n8k16 and SM quarter: 13 us of Llama gate + up at 32 tokens, 26 at 64); here the weights are unpacked once into tensor
// memory, one instruction multiplies 128 channels by up to 64 tokens, and the time is flat in the number of tokens.
//
// Work decomposition: a CTA takes one row super-block (128 channels; gated: of both layers), one block of up to 64 tokens and one part of
// K; the K parts of a tile are the CTAs of a cluster and add their fp32 partial sums through distributed shared memory in rank order
// (deterministic, no scratch in global memory, calls on several streams do not meet).  A step is 128 k.  Warps: one thread loads packed
// weights and one x, by TMA, into rings of their own; groups of four warps take turns at the steps: a thread unpacks its channel (its
// tensor-memory lane) and stores fp16(s * q), or the exact integers, as the A operand; two threads issue the MMAs, even and odd weight
// tiles, each into its own accumulator (gated: gate and up), which are added at the end.  Two CTAs per SM; every wait is bounded.
//
// Ownership: a weight stage, an A slot and its barriers belong to one group, and a "slot written" barrier to one issuer, because a wait by
// parity is only sound for a thread that sees every phase (the host keeps the ring lengths multiples of what that takes).
//
// What bounds it: the chain of a step inside a group (wait, unpack, store, signal: 1560 cycles per 128 k, half of them unpacking), of which
// 4 to 6 are in flight per SM; issuing an MMA costs its thread 55 cycles whatever its width up to 64 (measured), which is why there are
// two issuers (one: 25.0 / 15.7 us instead of 24.2 / 14.0 on Llama gate + up / down at 32 tokens).  One CTA per SM with 24 unpacking
// warps: 30.9 / 17.6.  Of 112 or 224 tiles on 148 SMs some SMs get two and some one: about a quarter of the time of gate + up.
// Measured, us, weights out of HBM, the route before (gemm_mid.cuh to about 64 tokens, then the prefill kernels) / this one, int4 in groups
// (qkv, o int8): Llama gate + up at 32 tokens 37.0 / 23.5, at 64 43.8 / 26.0; down 18.8 / 14.0, 27.9 / 15.8, at 128 29.3 / 22.7; q + k + v 12.3 /
// 9.6, 18.1 / 11.9, 19.4 / 16.3; o at 128 tokens 19.1 / 12.2; Gemma2-2B down 12.8 / 9.6, 20.8 / 11.5, at 256 27.6 / 23.3; 1024 x 1024 at 128
// tokens 12.4 / 5.4, at 512 16.0 / 7.3; a gated pair of 2688 x 1024 at 128 28.8 / 9.6.  The rule that picks it: gemm_route in qlinear.cu.
#pragma once
#include "gemm_pair_ta.cuh"

namespace ql {

constexpr int kNarrowFirstWorker = 4;        // warps 0 weight producer, 1 and 3 MMA issuers, 2 x producer, 4.. dequantise and epilogue
constexpr int kNarrowKStep = 128;
constexpr int kNarrowCols = 256;             // tensor memory of a CTA (two per SM): two accumulators and the slots
constexpr int kNarrowMaxW = 6, kNarrowMaxX = 6, kNarrowMaxSlots = 6;    // barriers exist for this many stages and slots
constexpr int kNarrowSmem = 112 * 1024;      // most that two CTAs per SM leave for one (and never less: at most two fit, whose tensor memory fits too)
constexpr int kNarrowTail = 1024;            // barriers and flags
constexpr int kNarrowRing = kNarrowSmem - 1024 - kNarrowTail;        // weight and x stages (1024: alignment)
constexpr int kNarrowPartStride = 132;       // floats per token of a partial tile
// G groups of four dequantise warps take turns at the steps, each with two A slots of 64 k (32 columns) of its own.
constexpr int narrow_threads(int G) { return 32 * kNarrowFirstWorker + 128 * G; }

struct NarrowMaps {
    CUtensorMap x;                           // [M, K] fp16, box 64 k x bn tokens, 128-byte swizzle
    CUtensorMap w[kGemmMaxGroup];            // packed body of each layer (w_tensor_map)
};

struct NarrowParams {
    const __half* chan_scales[kGemmMaxGroup];    // nullptr when grouped
    __half* y[kGemmMaxGroup];                    // [M, N_i]
    int32_t N[kGemmMaxGroup];
    int32_t unit_end[kGemmMaxGroup];             // row super-blocks of layers 0..i
    int32_t n_layers, M, K, n_kc, w_rows, n_steps, n_tb, cl, act, bn, nw, nx, a_col;
    int32_t late;                                // the weights may come from the previous kernel (a KV cache): nothing of them is read before griddepcontrol.wait
};

// 64 consecutive k of one row -> 32 registers, the 32 columns of the row's tensor-memory lane.  Per-thread constants as in
// DequantRowTa; a 16-byte piece holds both 32-k halves (int4), so it is read once.
struct DequantRow64 {
    int off[4], s_off;
    uint32_t mask, mul, add, sel;
    __device__ DequantRow64(int quarter, int lane)
    {
        const int rb = 2 * quarter + (lane >> 4), g = lane & 7, hi = (lane >> 3) & 1;
        for (int c = 0; c < 4; ++c) off[c] = (rb * 8 + g) * 64 + ((c ^ ((g >> 1) & 3)) << 4);
        s_off = kWeightBlockBytes + rb * 64 + (((g >> 1) ^ quarter) << 4) + (g & 1) * 8 + hi * 4;
        mask = hi ? 0x00F000F0u : 0x000F000Fu;
        mul = hi ? 0x2C002C00u : 0x3C003C00u;
        add = hi ? 0xD480D480u : 0xE408E408u;
        sel = hi ? 0x4342u : 0x4140u;
        for (int c = 0; c < 4; ++c) asm volatile("" : "+r"(off[c]));
        asm volatile("" : "+r"(s_off), "+r"(mask), "+r"(mul), "+r"(add), "+r"(sel));
    }
    // 64 k at wp (a half of a stage) -> the 32 columns of the slot, in pieces of 8 columns (16 k, one MMA's share), so that few registers
    // are live and the stores run under the conversion of the next piece.
    template <int BITS, bool GROUPED>
    __device__ __forceinline__ void convert(uint32_t wp, uint32_t slot) const
    {
        if (BITS == 4) {
            uint32_t s2[2] = {0, 0};
            if (GROUPED) {
                uint32_t s;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(s) : "r"(wp + s_off));
                s2[0] = __byte_perm(s, 0, 0x1010);
                s2[1] = __byte_perm(s, 0, 0x3232);
            }
#pragma unroll
            for (int cp = 0; cp < 2; ++cp) {
                uint32_t r[2][8];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const uint4 w = lds_u128(wp + off[2 * cp + c]);
                    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {                        // word i: 32-k half i / 2, k 8c + 4 (i % 2) ..
                        uint32_t* o = r[i >> 1] + 4 * c + 2 * (i & 1);
                        o[0] = h2_fma(lop3_and_or(ww[i], mask, 0x64006400u), mul, add);
                        o[1] = h2_fma(lop3_and_or(ww[i] >> 8, mask, 0x64006400u), mul, add);
                        if (GROUPED) { o[0] = h2_mul(o[0], s2[i >> 1]); o[1] = h2_mul(o[1], s2[i >> 1]); }
                    }
                }
                tmem_st8_async(slot + 8 * cp, r[0]);
                tmem_st8_async(slot + 16 + 8 * cp, r[1]);
            }
        } else {
#pragma unroll
            for (int b = 0; b < 2; ++b)                                  // packed blocks of 32 k
#pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                    uint32_t r[8];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const uint4 w = lds_u128(wp + b * kWeightBlockBytes + off[2 * cp + c]);
                        r[4 * c + 0] = h2_sub(__byte_perm(w.x, 0x64646464u, sel), 0x64806480u);
                        r[4 * c + 1] = h2_sub(__byte_perm(w.y, 0x64646464u, sel), 0x64806480u);
                        r[4 * c + 2] = h2_sub(__byte_perm(w.z, 0x64646464u, sel), 0x64806480u);
                        r[4 * c + 3] = h2_sub(__byte_perm(w.w, 0x64646464u, sel), 0x64806480u);
                    }
                    tmem_st8_async(slot + 16 * b + 8 * cp, r);
                }
        }
    }
};

template <int BITS, bool GROUPED, bool GATED, int G>
__global__ void __launch_bounds__(narrow_threads(G), 2) gemm_narrow_kernel(const __grid_constant__ NarrowMaps maps, const NarrowParams p)
{
    namespace cg = cooperative_groups;
    constexpr int R = GATED ? 2 : 1;                                     // row super-blocks per step: gate and up
    constexpr int CHUNKS = BITS == 4 ? 2 : 4;                            // packed blocks of a step
    constexpr int W_BYTES = CHUNKS * (kWeightBlockBytes + (GROUPED ? kScaleBlockBytes : 0));
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
    const int bn = p.bn, NW = p.nw, NX = p.nx;
    const uint32_t x_half = (uint32_t)bn * 128, x_bytes = 2 * x_half;        // two tiles of 64 k
    const uint32_t x0 = base + (uint32_t)NW * W_BYTES, tail = base + kNarrowRing;
    const uint32_t wfull0 = tail, wempty0 = wfull0 + 8 * kNarrowMaxW, xfull0 = wempty0 + 8 * kNarrowMaxW, xempty0 = xfull0 + 8 * kNarrowMaxX;
    const uint32_t afull0 = xempty0 + 8 * kNarrowMaxX, aempty0 = afull0 + 16 * kNarrowMaxSlots, tfull_bar = aempty0 + 8 * kNarrowMaxSlots;
    constexpr int kBars = 2 * kNarrowMaxW + 2 * kNarrowMaxX + 3 * kNarrowMaxSlots + 1;
    static_assert(8 * kBars <= 512 && 512 + 20 <= kNarrowTail, "tail");
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + (tail - base) + 512);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t crank_u, cid_u;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank_u));
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(cid_u));
    const int crank = (int)crank_u, cid = (int)cid_u;
    const int unit = cid / p.n_tb, m0 = (cid - unit * p.n_tb) * bn;
    int ly = 0;
    if (!GATED) {
#pragma unroll
        for (int i = 1; i < kGemmMaxGroup; ++i)
            if (i < p.n_layers && unit >= p.unit_end[i - 1]) ly = i;
    }
    const int rsb = unit - (ly ? p.unit_end[ly - 1] : 0);
    const int st0 = (int)((int64_t)crank * p.n_steps / p.cl), st1 = (int)((int64_t)(crank + 1) * p.n_steps / p.cl);
    const int total = (st1 - st0) * R;                                   // weight tiles of this CTA

    // (one thread per barrier: one after the other they took more than half a microsecond)
    if (threadIdx.x < kBars) {
        const int i = threadIdx.x;
        const bool workers = (i >= kNarrowMaxW && i < 2 * kNarrowMaxW) || (i >= 2 * (kNarrowMaxW + kNarrowMaxX) && i < 2 * (kNarrowMaxW + kNarrowMaxX + kNarrowMaxSlots));
        const bool issuers = i == kBars - 1 || (R == 2 && i >= 2 * kNarrowMaxW + kNarrowMaxX && i < 2 * (kNarrowMaxW + kNarrowMaxX));
        mbar_init(wfull0 + 8 * i, workers ? 4 : issuers ? 2 : 1);        // wempty and afull: the four warps of a group; tfull and (gated) xempty: both issuers
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 64) {
        abort_flag[0] = abort_flag[1] = abort_flag[2] = abort_flag[3] = 0;
        asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.x) : "memory");
    }
    if (threadIdx.x == 96) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.w[ly]) : "memory");
        if (GATED) asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.w[1]) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32((const void*)tmem_slot), kNarrowCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // The per-channel scales of the four channels whose sums over the K parts this thread finishes: requested here unless the kernel before
    // may be writing them, so that their latency does not follow the cluster's barrier (Llama q + k + v at 32 tokens 9.5 -> 9.2 us, o 8.2 -> 7.9, at
    // 16 tokens 8.9 -> 8.45; a gated pair, twice the registers, 24.3 -> 24.6).
    constexpr bool EARLY_SCALES = !GROUPED && !GATED;
    [[maybe_unused]] uint2 early = make_uint2(0, 0);
    [[maybe_unused]] auto load_early = [&] {
        const int row = rsb * kRsbRows + lane * 4;                       // (N is a multiple of 8: the four channels exist together)
        if (row < p.N[ly]) asm volatile("ld.global.cg.v2.u32 {%0,%1}, [%2];" : "=r"(early.x), "=r"(early.y) : "l"(p.chan_scales[ly] + row) : "memory");
    };
    if constexpr (EARLY_SCALES)
        if (p.cl > 1 && !p.late && warp >= kNarrowFirstWorker) load_early();

    bool ok = true;
    if (warp == 0) {
        // ------------------------------------------------------------------ weights
        if (lane == 0) {
            if (p.late) asm volatile("griddepcontrol.wait;" ::: "memory");
            int s = 0, g = 0;
            uint32_t par = 1;
            for (int it = st0; ok && it < st1; ++it)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (!mbar_wait(wempty0 + 8 * s, par, abort_flag, 0x600 + s)) { ok = false; break; }
                    mbar_expect_tx(wfull0 + 8 * s, W_BYTES);
                    // (blocks beyond K: what follows in the blob, or zeros; they are not multiplied)
                    tma_load_2d(base + s * W_BYTES, &maps.w[GATED ? r : ly], 0, (rsb * p.n_kc + it * CHUNKS) * p.w_rows, wfull0 + 8 * s);
                    ++g;
                    if (++s == NW) { s = 0; par ^= 1; }
                }
            if (*abort_flag)
                for (int j = max(0, g - NW); j < g; ++j) mbar_wait(wfull0 + 8 * (j % NW), (j / NW) & 1, abort_flag + 1, 0);
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ x
        if (lane == 0) {
            asm volatile("griddepcontrol.wait;" ::: "memory");           // x may come from the previous kernel
            abort_flag[2] = 1;                                           // from here on, waiting counts against the time limit
            abort_flag[3] = 1;
            int s = 0, g = 0;
            uint32_t par = 1;
            for (int it = st0; it < st1; ++it, ++g) {
                if (!mbar_wait(xempty0 + 8 * s, par, abort_flag, 0x620 + s)) break;
                const int k = it * kNarrowKStep;
                mbar_expect_tx(xfull0 + 8 * s, x_bytes);
                tma_load_2d(x0 + s * x_bytes, &maps.x, k, m0, xfull0 + 8 * s);
                tma_load_2d(x0 + s * x_bytes + x_half, &maps.x, k + 64, m0, xfull0 + 8 * s);   // (beyond K: zeros)
                if (++s == NX) { s = 0; par ^= 1; }
            }
            if (*abort_flag)
                for (int j = max(0, g - NX); j < g; ++j) mbar_wait(xfull0 + 8 * (j % NX), (j / NX) & 1, abort_flag + 1, 0);
        }
    } else if (warp == 1 || warp == 3) {
        // ------------------------------------------------------------------ MMA issuers: they take turns at the weight tiles, each with an accumulator of its own
        if (lane == 0) {
            const uint32_t idesc = umma_idesc_f16(bn), x_lo0 = umma_desc_lo(x0), x_lo_half = x_half >> 4;
            const int who = warp >> 1;
            const uint32_t d = tmem_base + (uint32_t)(who * bn);
            int s = R == 1 ? who : 0;
            uint32_t xpar = 0, apar = 0;
            // A slot's barrier exists once per issuer: with three groups its uses alternate between the issuers, and a wait by parity
            // is only sound for one that sees every phase.
            const uint32_t afull = afull0 + (uint32_t)(8 * kNarrowMaxSlots * who);
            int wg = who, turn = 0;                                      // group that dequantises step g
            bool live = true;
            for (int g = who; live && g < total; g += 2) {
                const int it = R == 1 ? st0 + g : st0 + (g >> 1);
                if (!mbar_wait(xfull0 + 8 * s, xpar, abort_flag, 0x630 + s)) break;
                const uint32_t b_lo = x_lo0 + (uint32_t)s * (x_bytes >> 4);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int a = 2 * wg + h;
                    if (!mbar_wait(afull + 8 * a, apar, abort_flag, 0x640 + a)) { live = false; break; }
                    tc_fence_after();
                    const uint32_t ta = tmem_base + (uint32_t)(p.a_col + a * kTaSlotCols);
                    if (h == 0 || it * kNarrowKStep + 64 < p.K) {        // (else the step's second 64 k lie beyond the layer)
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4) umma_f16_ta(d, ta + 8 * k4, b_lo + h * x_lo_half + 2 * k4, idesc, (g >= 2 || h > 0 || k4 > 0) ? 1u : 0u);
                    }
                    umma_commit(aempty0 + 8 * a);
                }
                if (live) umma_commit(xempty0 + 8 * s);
                s += R == 1 ? 2 : 1; if (s >= NX) { s -= NX; xpar ^= 1; }
                wg += 2; if (wg >= G) wg -= G;
                if (++turn == ((G & 1) ? G : G / 2)) { turn = 0; apar ^= 1; }
            }
            umma_commit(tfull_bar);
        }
    } else if (warp >= kNarrowFirstWorker) {
        // ------------------------------------------------------------------ dequantise: the groups of four warps take turns
        const int quarter = warp & 3, wg = (warp - kNarrowFirstWorker) >> 2;
        const DequantRow64 dq(quarter, lane);
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        int s = wg;                                                      // (NW is a multiple of G: a stage belongs to one group)
        uint32_t wpar = 0, apar = 1;
        const uint32_t slot0 = tmem_base + lane_base + (uint32_t)(p.a_col + 2 * wg * kTaSlotCols), ae0 = aempty0 + 16 * wg;
        for (int g = wg; ok && g < total; g += G, apar ^= 1) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 0 && !mbar_wait(wfull0 + 8 * s, wpar, abort_flag, 0x650 + s)) { ok = false; break; }
                if (!mbar_wait(ae0 + 8 * h, apar, abort_flag, 0x670 + 2 * wg + h)) { ok = false; break; }
                tc_fence_after();
                dq.template convert<BITS, GROUPED>(base + s * W_BYTES + h * (W_BYTES / 2), slot0 + h * kTaSlotCols);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (h == 1) mbar_arrive(wempty0 + 8 * s);
                    mbar_arrive(afull0 + (uint32_t)(8 * (kNarrowMaxSlots * (g & 1) + 2 * wg + h)));
                }
            }
            s += G; if (s >= NW) { s -= NW; wpar ^= 1; }
        }
        // ------------------------------------------------------------------ epilogue: a thread has one channel, the groups take turns at 8 tokens
        const int n = rsb * kRsbRows + quarter * 32 + lane, N = p.N[GATED ? 0 : ly];
        float sc0 = 1.f, sc1 = 1.f;
        auto load_scales = [&] {
            if (!GROUPED && p.cl == 1 && n < N) {
                sc0 = __half2float(ld_cg_half(p.chan_scales[GATED ? 0 : ly] + n));
                if (GATED) sc1 = __half2float(ld_cg_half(p.chan_scales[1] + n));
            }
        };
        // Early, unless the kernel before this one may still be writing them: a group without a step of its own has waited for nothing
        // so far.  (The accumulators are complete only past the x producer's griddepcontrol.wait.)
        if (!p.late) load_scales();
        ok = ok && mbar_wait(tfull_bar, 0, abort_flag, 0x680);
        if (ok) {
            if (p.late) load_scales();
            tc_fence_after();
            float* part = reinterpret_cast<float*>(base_ptr) + quarter * 32 + lane;   // [layer of the pair][token][channel]
            __half* yc = p.y[GATED ? 0 : ly] + (int64_t)m0 * N + n;
            const bool two = R == 2 || total > 1;                        // both issuers had work
            for (int cc = 8 * wg; cc < bn; cc += 8 * G) {
                uint32_t v[2][8];
                tmem_ld8(tmem_base + lane_base + (uint32_t)cc, v[0]);
                if (two) {
                    tmem_ld8(tmem_base + lane_base + (uint32_t)(bn + cc), v[1]);
                    if (R == 1)
#pragma unroll
                        for (int q = 0; q < 8; ++q) v[0][q] = __float_as_uint(__uint_as_float(v[0][q]) + __uint_as_float(v[1][q]));
                }
                if (p.cl > 1) {
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int q = 0; q < 8; ++q) part[(r * bn + cc + q) * kNarrowPartStride] = __uint_as_float(v[r][q]);
                } else if (n < N) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float o = __uint_as_float(v[0][q]) * sc0;
                        if (GATED) o = gate_activation(o, p.act) * (__uint_as_float(v[R - 1][q]) * sc1);
                        if (m0 + cc + q < p.M) yc[(int64_t)(cc + q) * N] = __float2half_rn(o);
                    }
                }
            }
            tc_fence_before();
        }
    }
    __syncwarp();
    if (p.cl > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (warp >= kNarrowFirstWorker && ok) {
            // rank r finishes tokens r, r + cl, ... of the tile, 4 channels per thread
            cg::cluster_group cluster = cg::this_cluster();
            const int t = threadIdx.x - 32 * kNarrowFirstWorker, quad = t & 31, row0 = rsb * kRsbRows + quad * 4, N = p.N[GATED ? 0 : ly];
            const float* part = reinterpret_cast<const float*>(base_ptr) + quad * 4;
            float sc[R][4];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int i = 0; i < 4; ++i) sc[r][i] = !GROUPED && !EARLY_SCALES && row0 < N ? __half2float(ld_cg_half(p.chan_scales[GATED ? r : ly] + row0 + i)) : 1.f;
            if constexpr (EARLY_SCALES) {
                if (p.late) load_early();
                const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&early.x)), hi = __half22float2(*reinterpret_cast<const __half2*>(&early.y));
                sc[0][0] = lo.x; sc[0][1] = lo.y; sc[0][2] = hi.x; sc[0][3] = hi.y;
            }
            for (int tok = crank + (t >> 5) * p.cl; tok < bn && m0 + tok < p.M; tok += 4 * G * p.cl) {
                float v[R][4];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r][0] = v[r][1] = v[r][2] = v[r][3] = 0.f;
                for (int k = 0; k < p.cl; ++k) {
                    const float* src = cluster.map_shared_rank(part, k);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 f = *reinterpret_cast<const float4*>(src + (r * bn + tok) * kNarrowPartStride);
                        v[r][0] += f.x; v[r][1] += f.y; v[r][2] += f.z; v[r][3] += f.w;
                    }
                }
                if (row0 < N) {                                          // (N is a multiple of 8: the four channels exist together)
                    float o[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        o[i] = v[0][i] * sc[0][i];
                        if (GATED) o[i] = gate_activation(o[i], p.act) * (v[R - 1][i] * sc[R - 1][i]);
                    }
                    uint2 u;
                    *reinterpret_cast<__half2*>(&u.x) = __floats2half2_rn(o[0], o[1]);
                    *reinterpret_cast<__half2*>(&u.y) = __floats2half2_rn(o[2], o[3]);
                    *reinterpret_cast<uint2*>(p.y[GATED ? 0 : ly] + (int64_t)(m0 + tok) * N + row0) = u;
                }
            }
        }
        __syncwarp();
        // peers keep their partial tile alive until it has been read: a rendezvous only
        asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    } else __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kNarrowCols);
    }
}

}  // namespace ql
