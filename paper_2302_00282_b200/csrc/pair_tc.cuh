// Two linked convolutions, the second one 1x1 (Table 1 of the Xenos paper, row ConvX -> ConvY: Conv k x k -> Conv 1x1, with
// the shortcut row's identity branch in the last epilogue), in one kernel: the first one's result never leaves the SM.
//
// A CTA walks over tiles of 128 consecutive output pixels (im2col boxes, as in conv_tc.cuh):
//   GEMM 1   im2col boxes x weight blocks -> accumulator 1 (all Cmid <= 256 channels of the tile)
//   middle   eight epilogue warps: bias, activation, bf16, written to shared memory in the K-major swizzled operand layout
//            that the second product reads (Section 4.1: the producer writes in the order the consumer reads)
//   GEMM 2   that buffer x 128-row blocks of the second weight matrix -> accumulator 2, 128 output channels at a time, two
//            accumulators so that the store of one block of channels overlaps the product of the next
//   final    bias, activation [, + shortcut, activation], bf16, 32-row boxes by bulk tensor stores; the shortcut's boxes
//            arrive by the copy engine in the buffers the results leave from
// Operand blocks live in two rings of 16 KB slots: A (one im2col box) and B (up to 128 weight rows x 64), so that the
// second product's blocks follow the first one's without a gap.  Where both weight matrices fit beside four A slots (64
// middle channels) they are loaded once per CTA.  With at most 128 middle channels accumulator 1 exists twice and GEMM 1 of
// the next tile is issued before GEMM 2 of this one, which waits for the middle epilogue.
// A tile moves 144 / 288 / 576 KB of input, shortcut and output for 64 / 128 / 256 middle channels through HBM and 0 / 426 /
// 1700 KB of weights from L2.  Reached, 512 x 512 images, batch 64: 260 / 183 / 161 us a launch, 0.71 and 0.51 of the HBM rate
// and 0.51 of the tensor rate (counters at batch 8: tensor pipe 14 to 18 %, DRAM 6 to 29 %, issue slots 19 to 27 %): no unit is
// full.  At 256 middle channels first product, middle and second product of a tile follow one another.
// One thread per role issues all requests; every wait is bounded.
#pragma once

#include "conv_tc.cuh"

namespace xk {

constexpr int kPairMaxSlots = 8;

struct PairParams {
    ConvSegment seg;                   // first convolution
    const float *bias1, *bias2;
    unsigned int *status;
    FastDiv d_rpi, d_q;
    int rows, tiles, n1pad, n1_slots, kblocks2, n2_blocks, npad2;
    int a_slots, b_slots, resident, dbl;      // dbl: two first accumulators
    int s_slots;                    // staging boxes per epilogue warp
    int act1, act2, act3;
    uint32_t idesc1, idesc2;
    int off_b, off_mid, off_stage, off_bias, off_bar;
    int launch_id;
};

struct PairRing {
    int s, n;
    uint32_t ph, ready;      // ready: as in ConvRing
    __device__ __forceinline__ void next() { if (++s == n) { s = 0; ph ^= 1u; } }
};

// The products of one tile's first convolution.
__device__ __forceinline__ bool pair_gemm1(const PairParams &g, PairRing &ra, PairRing &rb, uint32_t sbase, uint32_t a_full, uint32_t b_full, uint32_t d1) {
    const uint32_t idesc = in_reg(g.idesc1);
    const int n = in_reg(g.seg.kblocks), slots = in_reg(g.n1_slots), resident = in_reg(g.resident), n1pad = in_reg(g.n1pad);
    constexpr uint32_t hi = 64u | (1u << 14) | (2u << 29);
    const uint32_t b0 = sbase + g.off_b;
    uint32_t acc = 0u;
#pragma unroll 1
    for (int kb = 0; kb < n; ++kb) {
        if (!ra.ready && !mbar_wait(a_full + 8u * ra.s, ra.ph)) return false;
        const uint32_t a4 = 0x10000u | ((sbase + ra.s * kABytes) >> 4), a_used = a_full + 8u * (kPairMaxSlots + ra.s);
        ra.next();
        ra.ready = 0u;
#pragma unroll 1
        for (int h = 0; h < slots; ++h) {
            uint32_t b4, b_used = 0u;
            if (resident) b4 = 0x10000u | ((b0 + kb * n1pad * 128) >> 4);
            else {
                if (!rb.ready && !mbar_wait(b_full + 8u * rb.s, rb.ph)) return false;
                b4 = 0x10000u | ((b0 + rb.s * kABytes) >> 4);
                b_used = b_full + 8u * (kPairMaxSlots + rb.s);
                rb.next();
            }
            const uint32_t d = d1 + h * 128;
            // (resident weights: one block per activation slot, whose successor is asked for; else the next weight slot)
            if (resident) ra.ready = umma_block(d, hi, a4, 2u, 4u, 6u, hi, b4, idesc, acc, 4, a_used, a_full + 8u * ra.s, ra.ph);
            else rb.ready = umma_block(d, hi, a4, 2u, 4u, 6u, hi, b4, idesc, acc, 4, b_used, b_full + 8u * rb.s, rb.ph);
        }
        if (!resident) umma_commit(a_used);
        acc = 1u;
    }
    return true;
}

template <bool kSkip>
__global__ void __launch_bounds__(kCvThreads, 1)
pair_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmB2,
               const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmS, const __grid_constant__ PairParams g) {
    extern __shared__ uint8_t smem_raw[];
    pdl_launch_dependents();
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (sbase - raw);
    const uint32_t bar = sbase + g.off_bar;
    const uint32_t a_full = bar, b_full = bar + 8u * 2 * kPairMaxSlots, d_bar = bar + 8u * 4 * kPairMaxSlots;
    // d_bar: first accumulator full [2] / empty [2], second full [2] / empty [2], middle full, middle empty, resident weights
    const uint32_t d1f = d_bar, d1e = d_bar + 16u, d2f = d_bar + 32u, d2e = d_bar + 48u, midf = d_bar + 64u, mide = d_bar + 72u, bres = d_bar + 80u;
    const uint32_t skip0 = d_bar + 96u;                                           // kMaxSkipSlots per epilogue warp
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + g.off_bar + 8 * (4 * kPairMaxSlots + 12 + kMaxSkipSlots * kCvEpiWarps));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        // (a lane per barrier; d1e, d2e and midf count the epilogue warps)
        constexpr int d0 = 4 * kPairMaxSlots, n_bars = d0 + 12 + kMaxSkipSlots * kCvEpiWarps;
        for (int i = lane; i < n_bars; i += 32) {
            const int d = i - d0;
            mbar_init(bar + 8u * i, d == 2 || d == 3 || (d >= 6 && d <= 8) ? kCvEpiWarps : 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        if (lane == 1) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB1) : "memory");
    }
    if (warp == 3) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp >= 4) {
        float *dst = reinterpret_cast<float *>(sm + g.off_bias);
        for (int i = threadIdx.x - 128; i < g.n1pad; i += 256) dst[i] = __ldg(g.bias1 + i);
        for (int i = threadIdx.x - 128; i < g.npad2; i += 256) dst[g.n1pad + i] = __ldg(g.bias2 + i);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // columns: first accumulator(s) [0, 256), second accumulators [256, 384) and [384, 512)
    const unsigned gave_up = kStatusTimeout | (((unsigned)g.launch_id & 0xfffu) << 12);
    bool ok = true;
    if (warp == 0) {
        if (elect_one()) {
            // ---- A: im2col boxes of the first convolution ----
            pdl_wait();
            PairRing ra = {0, in_reg(g.a_slots), 0u, 0u};
            int fresh = ra.n;      // slots that nothing has been put in yet
            const int tiles = in_reg(g.tiles), n_kb = in_reg(g.seg.kblocks), cend = in_reg(g.seg.cblocks * kTileK), k = in_reg(g.seg.k);
#pragma unroll 1
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
                const int m0 = t * kTileM;
                const int n = (int)g.d_rpi.div((uint32_t)m0), rem = m0 - n * (int)g.d_rpi.d;
                const int p = (int)g.d_q.div((uint32_t)rem), q = rem - p * (int)g.d_q.d;
                const int h0 = p * g.seg.stride + g.seg.low, w0 = q * g.seg.stride + g.seg.low;
                const bool im2col = g.seg.im2col != 0;
                int c = 0, r = 0, s = 0;
#pragma unroll 1
                for (int kb = 0; kb < n_kb; ++kb) {
                    const uint32_t fb = a_full + 8u * ra.s;
                    ok = --fresh >= 0 || mbar_wait(fb + 8u * kPairMaxSlots, ra.ph ^ 1u);
                    if (!ok) break;
                    mbar_arrive_expect_tx(fb, kABytes);
                    if (im2col) tma_load_im2col(sbase + ra.s * kABytes, &tmA, c, w0, h0, n, fb, s, r);
                    else tma_load_2d(sbase + ra.s * kABytes, &tmA, c, m0, fb);
                    ra.next();
                    c += kTileK;
                    if (c == cend) { c = 0; if (++s == k) { s = 0; ++r; } }
                }
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (1u << 8));
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // ---- B: weight blocks, in the order the MMA thread uses them ----
            const uint32_t b0 = sbase + g.off_b;
            const int n_kb = in_reg(g.seg.kblocks), n1pad = in_reg(g.n1pad), slots = in_reg(g.n1_slots), kb2n = in_reg(g.kblocks2), n2 = in_reg(g.n2_blocks);
            if (g.resident) {
                mbar_arrive_expect_tx(bres, (uint32_t)(n_kb * n1pad + kb2n * n2 * 128) * 128u);
#pragma unroll 1
                for (int kb = 0; kb < n_kb; ++kb) tma_load_2d(b0 + kb * n1pad * 128, &tmB1, kb * kTileK, 0, bres);
#pragma unroll 1
                for (int c = 0; c < n2; ++c)
#pragma unroll 1
                    for (int kb = 0; kb < kb2n; ++kb) tma_load_2d(b0 + n_kb * n1pad * 128 + (c * kb2n + kb) * kABytes, &tmB2, kb * kTileK, c * 128, bres);
            } else {
                PairRing rb = {0, in_reg(g.b_slots), 0u, 0u};
                int fresh = rb.n;
                const uint32_t bytes1 = (uint32_t)min(n1pad, 128) * 128u;
                auto first = [&]() {
#pragma unroll 1
                    for (int kb = 0; kb < n_kb && ok; ++kb)
#pragma unroll 1
                        for (int h = 0; h < slots; ++h) {
                            const uint32_t fb = b_full + 8u * rb.s;
                            ok = --fresh >= 0 || mbar_wait(fb + 8u * kPairMaxSlots, rb.ph ^ 1u);
                            if (!ok) break;
                            mbar_arrive_expect_tx(fb, bytes1);
                            tma_load_2d(b0 + rb.s * kABytes, &tmB1, kb * kTileK, h * 128, fb);
                            rb.next();
                        }
                };
                auto second = [&]() {
#pragma unroll 1
                    for (int c = 0; c < n2 && ok; ++c)
#pragma unroll 1
                        for (int kb = 0; kb < kb2n; ++kb) {
                            const uint32_t fb = b_full + 8u * rb.s;
                            ok = --fresh >= 0 || mbar_wait(fb + 8u * kPairMaxSlots, rb.ph ^ 1u);
                            if (!ok) break;
                            mbar_arrive_expect_tx(fb, kABytes);
                            tma_load_2d(b0 + rb.s * kABytes, &tmB2, kb * kTileK, c * 128, fb);
                            rb.next();
                        }
                };
                const int step = gridDim.x;
                if (g.dbl) first();
#pragma unroll 1
                for (int t = blockIdx.x; t < g.tiles && ok; t += step) {
                    if (!g.dbl || t + step < g.tiles) first();
                    if (ok) second();
                }
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (1u << 8));
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ---- MMA ----
            PairRing ra = {0, in_reg(g.a_slots), 0u, 0u}, rb = {0, in_reg(g.b_slots), 0u, 0u};
            const int tiles = in_reg(g.tiles), step = gridDim.x, kb2n = in_reg(g.kblocks2), n2 = in_reg(g.n2_blocks), resident = in_reg(g.resident), dbl = in_reg(g.dbl);
            const uint32_t idesc2 = in_reg(g.idesc2), mid = sbase + g.off_mid, b0 = sbase + g.off_b, b2 = b0 + g.seg.kblocks * g.n1pad * 128;
            constexpr uint32_t hi = 64u | (1u << 14) | (2u << 29);
            int i1 = 0, c2 = 0;      // first products issued; second-accumulator uses
            auto first = [&]() {
                const int b = dbl ? i1 & 1 : 0, use = dbl ? i1 >> 1 : i1;
                if (!mbar_wait(d1e + 8u * b, (use & 1) ^ 1u)) return false;      // the middle epilogue has read this accumulator
                tc_fence_after();
                if (!pair_gemm1(g, ra, rb, sbase, a_full, b_full, tmem_base + b * 128)) return false;
                umma_commit(d1f + 8u * b);
                ++i1;
                return true;
            };
            if (resident) ok = mbar_wait(bres, 0u);
            if (ok && dbl && (int)blockIdx.x < tiles) ok = first();
            int i = 0;
#pragma unroll 1
            for (int t = blockIdx.x; t < tiles && ok; t += step, ++i) {
                if (!dbl || t + step < tiles) { ok = first(); if (!ok) break; }
                ok = mbar_wait(midf, i & 1);
#pragma unroll 1
                for (int c = 0; c < n2 && ok; ++c, ++c2) {
                    const int b = c2 & 1;
                    ok = mbar_wait(d2e + 8u * b, ((c2 >> 1) & 1) ^ 1u);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d = tmem_base + 256 + b * 128;
#pragma unroll 1
                    for (int kb = 0; kb < kb2n; ++kb) {
                        const uint32_t a4 = 0x10000u | ((mid + kb * kABytes) >> 4);
                        uint32_t b4, b_used = 0u;
                        if (resident) b4 = 0x10000u | ((b2 + (c * kb2n + kb) * kABytes) >> 4);
                        else {
                            ok = rb.ready || mbar_wait(b_full + 8u * rb.s, rb.ph);
                            if (!ok) break;
                            b4 = 0x10000u | ((b0 + rb.s * kABytes) >> 4);
                            b_used = b_full + 8u * (kPairMaxSlots + rb.s);
                            rb.next();
                        }
                        // (resident weights have no slot to give back)
                        if (!resident) rb.ready = umma_block(d, hi, a4, 2u, 4u, 6u, hi, b4, idesc2, kb > 0 ? 1u : 0u, 4, b_used, b_full + 8u * rb.s, rb.ph);
                        else {
                            const uint64_t h64 = (uint64_t)hi << 32;
                            umma_bf16(d, h64 | a4, h64 | b4, idesc2, kb > 0 ? 1u : 0u);
                            umma_bf16_acc(d, h64 | (a4 + 2), h64 | (b4 + 2), idesc2);
                            umma_bf16_acc(d, h64 | (a4 + 4), h64 | (b4 + 4), idesc2);
                            umma_bf16_acc(d, h64 | (a4 + 6), h64 | (b4 + 6), idesc2);
                        }
                    }
                    if (ok) umma_commit(d2f + 8u * b);
                }
                if (ok) umma_commit(mide);
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (2u << 8));
        }
    } else if (warp >= 4) {
        // ---- epilogues: warp w reads tensor-memory lanes 32 * (w % 4) .., alternate 32-column chunks ----
        pdl_wait();
        const int e = warp - 4, quarter = warp & 3, half = e >> 2, row = quarter * 32 + lane;
        const uint32_t t_warp = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t bias1 = sbase + g.off_bias, bias2 = bias1 + (uint32_t)g.n1pad * 4u;
        const uint32_t mid = sbase + g.off_mid, stage0 = sbase + g.off_stage + (uint32_t)(g.s_slots * e) * 2048u;
        const uint32_t lo1 = g.act1 >= 1 ? 0u : 0xff80ff80u, hi1 = g.act1 == 2 ? 0x40c040c0u : 0x7f807f80u;
        const int last_act = kSkip ? g.act3 : g.act2;
        const uint32_t lo2 = last_act >= 1 ? 0u : 0xff80ff80u, hi2 = last_act == 2 ? 0x40c040c0u : 0x7f807f80u;
        const float flo = act_lo(g.act2), fhi = act_hi(g.act2);
        const bool mid_act = kSkip && g.act2 != 0;
        const int tiles = in_reg(g.tiles), step = gridDim.x, n1pad = in_reg(g.n1pad), n2 = in_reg(g.n2_blocks), dbl = in_reg(g.dbl);
        auto bias_pairs = [&](const float *v, uint32_t sb, float2 *t) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 bz = ld_shared_f4(sb + (uint32_t)q * 16u);
                t[2 * q] = __fadd2_rn(make_float2(v[4 * q], v[4 * q + 1]), make_float2(bz.x, bz.y));
                t[2 * q + 1] = __fadd2_rn(make_float2(v[4 * q + 2], v[4 * q + 3]), make_float2(bz.z, bz.w));
            }
        };
        // Shortcut boxes are asked for s_slots - 1 ahead of their use: with one box of 2 KB ahead every box cost a warp the whole
        // latency of the load (3.5 TB/s of traffic at best).  (at, ac, aj): the next box to ask for.
        const int depth = in_reg(g.s_slots), step_c = n2;
        int at = blockIdx.x, ac = 0, aj = 0;
        auto ask_skip = [&](int slot) {
            const uint32_t sb = skip0 + 8u * (kMaxSkipSlots * e + slot);
            mbar_arrive_expect_tx(sb, 2048u);
            tma_load_2d(stage0 + (uint32_t)slot * 2048u, &tmS, ac * 128 + (half * 2 + aj) * 32, at * kTileM + quarter * 32, sb);
        };
        auto advance = [&]() {
            if (++aj == 2) { aj = 0; if (++ac == step_c) { ac = 0; at += step; } }
        };
        int i = 0, c2 = 0, slot = 0;
        uint32_t sph = 0;
        if (kSkip)
            for (int d = 0; d + 1 < depth && at < tiles; ++d, advance()) {
                if (elect_one()) ask_skip(d);
                __syncwarp();
            }
#pragma unroll 1
        for (int t = blockIdx.x; t < tiles && ok; t += step, ++i) {
            // middle: first accumulator -> operand layout of the second product
            const int b1 = dbl ? i & 1 : 0, use = dbl ? i >> 1 : i;
            ok = mbar_wait(mide, (i & 1) ^ 1u) && mbar_wait(d1f + 8u * b1, use & 1);      // GEMM 2 has read the previous tile's middle
            if (!ok) break;
            tc_fence_after();
#pragma unroll 1
            for (int j = half; j < (n1pad >> 5); j += 2) {
                float v[32];
                tmem_ld32(t_warp + b1 * 128 + j * 32, v);
                const uint32_t blk = mid + (uint32_t)(j >> 1) * kABytes;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 s[8];
                    uint32_t pk[8];
                    bias_pairs(v + 16 * h, bias1 + (uint32_t)(j * 32 + 16 * h) * 4u, s);
#pragma unroll
                    for (int q = 0; q < 8; ++q) pk[q] = clamp_bf16x2(pack2(s[q].x, s[q].y), lo1, hi1);
                    const int piece = (j & 1) * 4 + 2 * h;
                    st_shared16(a_chunk_addr(blk, row, piece), make_uint4(pk[0], pk[1], pk[2], pk[3]));
                    st_shared16(a_chunk_addr(blk, row, piece + 1), make_uint4(pk[4], pk[5], pk[6], pk[7]));
                }
            }
            tc_fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) { mbar_arrive(d1e + 8u * b1); mbar_arrive(midf); }
            // final
#pragma unroll 1
            for (int c = 0; c < n2 && ok; ++c, ++c2) {
                const int b = c2 & 1;
                ok = mbar_wait(d2f + 8u * b, (c2 >> 1) & 1);
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int j = 0; j < 2; ++j) {
                    const uint32_t buf = stage0 + (uint32_t)slot * 2048u;
                    const int col = (half * 2 + j) * 32;
                    if (kSkip) {
                        ok = mbar_wait(skip0 + 8u * (kMaxSkipSlots * e + slot), sph);
                        if (!ok) break;
                    } else {
                        if (elect_one()) bulk_wait_read<1>();
                        __syncwarp();
                    }
                    float v[32];
                    tmem_ld32(t_warp + 256 + b * 128 + col, v);
                    if (j == 1) {
                        tc_fence_before();
                        warp_arrive(d2e + 8u * b, lane);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float2 s[8];
                        uint32_t pk[8];
                        bias_pairs(v + 16 * h, bias2 + (uint32_t)(c * 128 + col + 16 * h) * 4u, s);
                        const uint32_t p0 = buf + box_piece(32, lane, 2 * h), p1 = buf + box_piece(32, lane, 2 * h + 1);
                        if (kSkip) {
                            const uint4 k0 = ld_shared16(p0), k1 = ld_shared16(p1);
                            const uint32_t sk[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                if (mid_act) { s[q].x = fminf(fmaxf(s[q].x, flo), fhi); s[q].y = fminf(fmaxf(s[q].y, flo), fhi); }
                                s[q] = __fadd2_rn(s[q], make_float2(__uint_as_float(sk[q] << 16), __uint_as_float(sk[q] & 0xffff0000u)));
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 8; ++q) pk[q] = clamp_bf16x2(pack2(s[q].x, s[q].y), lo2, hi2);
                        st_shared16(p0, make_uint4(pk[0], pk[1], pk[2], pk[3]));
                        st_shared16(p1, make_uint4(pk[4], pk[5], pk[6], pk[7]));
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (elect_one()) {
                        tma_store_2d(&tmO, buf, c * 128 + col, t * kTileM + quarter * 32);
                        bulk_commit();
                        // the next shortcut box goes where the box before this one was, once that one's store has left it
                        if (kSkip && at < tiles) { bulk_wait_read<1>(); ask_skip(slot ? slot - 1 : depth - 1); }
                    }
                    if (kSkip && at < tiles) advance();
                    if (++slot == depth) { slot = 0; sph ^= 1u; }
                    __syncwarp();
                }
            }
        }
        if (elect_one()) bulk_wait_read<0>();
        __syncwarp();
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (5u << 8));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 3) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

}  // namespace xk
