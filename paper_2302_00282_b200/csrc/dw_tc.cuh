// Depthwise 3x3 -> pointwise 1x1 (Sections 2.2 and 4.1 of the Xenos paper: the depthwise result is produced in the layout
// the pointwise product reads and never leaves the SM), with a store, global-average or reduction-split epilogue.
//
// A CTA walks over tiles of ni images x rh x rw <= 128 output pixels (rw a multiple of 4) x n_acc * tile_n channels.
//   warp 0     copies the tile's input window of each 64-channel block (zero fill = padding) into the halo ring
//   warp 1     tensor memory; tcgen05.mma: depthwise block x weight block -> accumulator
//   warps 2-17 workers: the stencils of the next batch of tiles, then the epilogues of this one (all of them do both, so that
//              neither half of the CTA idles in chains with one tile per CTA).  nothing of the stencil stays in registers across an
//              epilogue: spilled values were reloaded from L2, since the shared memory leaves no L1 to speak of
//   warp 18    copies the weight blocks into their ring (or once, when a CTA meets several tiles and they fit: b_resident)
// The workers form G groups; a (tile, channel block) item is the work of one group, items are dealt in turn (a batch has at least one item per group: with one
// channel block per tile several tiles form a batch, each with its own accumulator pair), and a group's
// slots of the rings are its own (ring sizes are multiples of G: a group meets every phase of its slots' barriers).  A
// thread owns BR x 4 pixels of a channel pair; G is chosen so that a group covers a tile: small tiles have all their channel
// blocks under way at once, large ones two, which hides the shared-memory latency of the stencil.
// Bound: issue slots (4 x 4 pixels: some 400 instructions of a warp for 1024 results; a result box some 120 per 32 columns; the
// walk over a batch's tiles by all workers the rest of the first chain's 16.7 million), and at small batches the latencies of
// one tile: window, stencil, products, box.  MobileNet at batch 32: issue slots 58 % busy in the first chain, 28 to 53 % in the
// others.  A launch on 14 x 14 x 512 at batch 1 takes 5 to 6 us between its predecessor's end and its own, 5.8 to 7.2 before
// operand slots became as short as the tile (all of a tile's blocks fit, so the stencils do not wait for the products), weights
// stayed in shared memory and the products of a block were issued in one sequence (umma_block; 750 cycles a block before).
#pragma once

#include "pair_tc.cuh"

namespace xk {

constexpr int kDwWorkers = 16;
constexpr int kDwThreads = 96 + 32 * kDwWorkers;
constexpr int kDwMaxSlots = 8;
enum { DE_STORE = 0, DE_GAP = 1, DE_SPLIT = 2 };

struct DwParams {
    const float *dw_w, *dw_b, *bias;
    void *out;
    unsigned int *status;
    FastDiv d_nt, d_ks, d_tx, d_ty;
    int batch, P, Q, C, stride, pad, dw_act;
    int ni, rh, rw, tile_rows;
    int total, kblocks, last_steps, tile_n, n_acc, N, kb_per;
    int groups, wpg_log2, pairs;              // worker groups, log2(warps per group), lanes (channel pairs) per block
    int batch_tiles, n_bufs;                  // tiles per batch; accumulator buffers (2 per tile of a batch; 1 when a tile takes all columns)
    int a_stride;                             // distance of operand slots: tiles of few rows have short ones (see layout_dw)
    int a_slots, b_slots, h_slots, b_resident, halo_bytes, halo_stride, halo_h, halo_w, halo_cb;
    int acc_stride, tmem_cols;
    int chunk, nchunks, box_bytes, out_bufs;
    int act, out_ctot, out_f32;
    uint32_t idesc;
    int off_b, off_halo, off_dww, off_stage, off_bias, off_bar;
    int gap_imgs, gap_area, gap_rpi;
    int ksplit, split_ld;
    long long split_stride;
    float *split_part;
    unsigned int *split_cnt;
    int launch_id;
};

__device__ __forceinline__ void tma_store_4d(const CUtensorMap *tm, uint32_t src, int c, int x, int y, int n) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(tm), "r"(src), "r"(c), "r"(x), "r"(y), "r"(n) : "memory");
}

struct DwTile { int mt, nt, ks, kb0, kb1, n0, y0, x0; };      // first image, output row and column of the tile
__device__ __forceinline__ DwTile dw_tile(const DwParams &g, int ti) {
    DwTile t;
    const uint32_t pair = g.d_ks.div((uint32_t)ti);
    t.ks = ti - (int)(pair * g.d_ks.d);
    t.mt = (int)g.d_nt.div(pair);
    t.nt = (int)pair - t.mt * (int)g.d_nt.d;
    t.kb0 = t.ks * g.kb_per;
    t.kb1 = min(g.kblocks, t.kb0 + g.kb_per);
    const uint32_t rows = g.d_tx.div((uint32_t)t.mt), img = g.d_ty.div(rows);
    t.x0 = (t.mt - (int)(rows * g.d_tx.d)) * g.rw;
    t.y0 = (int)(rows - img * g.d_ty.d) * g.rh;
    t.n0 = (int)img * g.ni;
    return t;
}

// A worker thread's unit of a tile: BR x 4 pixels of a channel pair; the lanes of a warp take the pairs of one block of pixels
// (of two blocks when a channel block has at most 32 channels).
// a_row, a_step: where its first pixel's row of the operand block starts and how far the next block row is; a_piece: its
// channel pair in that row (K-major, 128-byte swizzle: bits 4..6 of an address are xor-ed with the row's low bits; rows start on
// multiples of four, so pixel b of a block row has piece ^ (b << 4), and an odd block row of an odd number of fours the other 64)
struct DwWork { int q, base, nrows, live; uint32_t a_row, a_step, a_piece; };
__device__ __forceinline__ uint32_t dw_flip(const DwWork &u) { return (u.a_step >> 3) & 64u; }

// The tap weights and bias of a thread's two channels.
struct DwTaps { float2 w[9], b; };
__device__ __forceinline__ float2 ld_shared_f2(uint32_t src) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(src));
    return v;
}
__device__ __forceinline__ void dw_load_taps(DwTaps &t, uint32_t dww, int C, int c0) {
#pragma unroll
    for (int i = 0; i < 9; ++i) t.w[i] = ld_shared_f2(dww + (uint32_t)(i * C + c0) * 4u);
    t.b = ld_shared_f2(dww + (uint32_t)(9 * C + c0) * 4u);
}

// Depthwise 3x3 + bias + activation of one unit, rounded to bf16 and stored in the operand layout.  Every input pair is read
// once per unit (one 128-byte row per warp and read) and feeds up to 9 results.
// kCB: channels of a window block where they are known at compile time (the loads of a row are then one address and
// immediate offsets), 0 otherwise.
template <int S, int BR, int kCB>
__device__ __forceinline__ void dw_stencil(const DwTaps &t, const DwWork &u, uint32_t halo, uint32_t a_base, int row_bytes, int cb,
                                           uint32_t lo, uint32_t hi) {
    const int cbytes = kCB ? 2 * kCB : 2 * cb;
    float2 acc[BR][4];
#pragma unroll
    for (int a = 0; a < BR; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = t.b;
    uint32_t rowp = halo + u.base;
#pragma unroll
    for (int iy = 0; iy < (BR - 1) * S + 3; ++iy, rowp += row_bytes) {
#pragma unroll
        for (int ci = 0; ci < 3 * S + 3; ++ci) {
            uint32_t v;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(rowp + ci * cbytes));
            const float2 x = make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
#pragma unroll
            for (int ry = 0; ry < 3; ++ry) {
                if ((iy - ry) % S != 0 || iy - ry < 0 || (iy - ry) / S >= BR) continue;      // resolved at compile time
#pragma unroll
                for (int sx = 0; sx < 3; ++sx) {
                    if ((ci - sx) % S != 0 || ci - sx < 0 || (ci - sx) / S >= 4) continue;
                    acc[(iy - ry) / S][(ci - sx) / S] = __ffma2_rn(x, t.w[ry * 3 + sx], acc[(iy - ry) / S][(ci - sx) / S]);
                }
            }
        }
    }
    // (rounding, then clamping: the bounds 0 and 6 are bf16 values and rounding is monotonic)
    uint32_t row = a_base + u.a_row, piece = u.a_piece;
    asm volatile("" : "+r"(piece));      // (the addresses are made here, not kept through the sums)
#pragma unroll
    for (int a = 0; a < BR; ++a, row += u.a_step, piece ^= dw_flip(u)) {
        if (a >= u.nrows) break;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(row + b * 128 + (piece ^ (b << 4))), "r"(clamp_bf16x2(pack2(acc[a][b].x, acc[a][b].y), lo, hi)) : "memory");
    }
}
// Output pixel of tile row r, -1 when the row lies outside the map or the batch.
__device__ __forceinline__ long long dw_pixel(const DwParams &g, const DwTile &t, int r) {
    const int area = g.rh * g.rw, img = r / area, rem = r - img * area, dy = rem / g.rw, dx = rem - dy * g.rw;
    const int n = t.n0 + img, y = t.y0 + dy, x = t.x0 + dx;
    if (img >= g.ni || n >= g.batch || y >= g.P || x >= g.Q) return -1;
    return ((long long)n * g.P + y) * g.Q + x;
}

// kS, kBR: stride and block rows of the stencil (an instance carries one stencil: instruction fetch is what a launch with one
// tile per CTA spends most of its time on)
template <int kEpi, int kS, int kBR, int kCB>
__global__ void __launch_bounds__(kDwThreads, 1)
dw_tc_kernel(const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmO,
             const __grid_constant__ DwParams g) {
    extern __shared__ uint8_t smem_raw[];
    pdl_launch_dependents();
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (sbase - raw);
    const uint32_t bar = sbase + g.off_bar;
    const uint32_t a_full = bar, b_full = bar + 8u * 2 * kDwMaxSlots, h_full = bar + 8u * 4 * kDwMaxSlots;      // "empty" follows each
    constexpr uint32_t kEmpty = 8u * kDwMaxSlots;
    const uint32_t accf = bar + 8u * 6 * kDwMaxSlots, acce = accf + 64u, bres = accf + 128u, dww_bar = accf + 136u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + g.off_bar + 8 * (6 * kDwMaxSlots + 18));
    volatile int *fail_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        // (a lane per barrier: a_full, empty, b_full, empty, h_full, empty, accf, acce of 8 each, bres, dww_bar)
        for (int i = lane; i < 8 * kDwMaxSlots + 2; i += 32) {
            const int kind = i / kDwMaxSlots;
            mbar_init(bar + 8u * i, kind == 0 || kind == 5 ? 1u << g.wpg_log2 : kind == 7 ? (kEpi == DE_STORE ? 4u * g.nchunks : kDwWorkers) : 1u);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncwarp();
    }
    if (warp == 0 && elect_one()) {
        fail_flag[0] = 0;
        // depthwise taps [9][C] and bias [C]: constants, awaited by the workers before their first stencil
        const uint32_t C = (uint32_t)g.C;
        mbar_arrive_expect_tx(dww_bar, 40u * C);
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(sbase + g.off_dww), "l"(g.dw_w), "r"(36u * C), "r"(dww_bar) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(sbase + g.off_dww + 36u * C), "l"(g.dw_b), "r"(4u * C), "r"(dww_bar) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmH) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp >= 2) {
        const int wt = threadIdx.x - 64, npad = (int)g.d_nt.d * g.n_acc * g.tile_n;
        float4 *dst = reinterpret_cast<float4 *>(sm + g.off_bias);
        for (int i = wt; i < (npad >> 2); i += 32 * kDwWorkers) dst[i] = __ldg(reinterpret_cast<const float4 *>(g.bias) + i);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const unsigned gave_up = kStatusTimeout | (((unsigned)g.launch_id & 0xfffu) << 12);
    bool ok = true;

    if (warp == 0) {
        if (elect_one()) {
            // ---- input windows (those of the first tile that find a fresh slot are asked for by the worker groups) ----
            PairRing rh = {0, in_reg(g.h_slots), 0u, 0u};
            const int total = in_reg(g.total), step = gridDim.x, stride = in_reg(g.stride), pad = in_reg(g.pad), hstride = in_reg(g.halo_stride);
            const uint32_t hbytes = in_reg((uint32_t)g.halo_bytes), dst0 = sbase + g.off_halo;
            pdl_wait();
            bool first = true;
            int fresh = rh.n;      // slots that nothing has been put in yet: no need to ask for room
#pragma unroll 1
            for (int ti = blockIdx.x; ti < total && ok; ti += step) {
                const DwTile t = dw_tile(g, ti);
                const int hy = t.y0 * stride - pad, hx = t.x0 * stride - pad;
                int kb = t.kb0;
                if (first) {
                    first = false;
                    const int n = min(rh.n, t.kb1 - t.kb0);
                    kb += n;
                    fresh -= n;
                    rh.s = n;
                    if (n == rh.n) { rh.s = 0; rh.ph = 1u; }
                }
#pragma unroll 1
                for (; kb < t.kb1; ++kb) {
                    const uint32_t fb = h_full + 8u * rh.s;
                    ok = --fresh >= 0 || mbar_wait(fb + kEmpty, rh.ph ^ 1u);
                    if (!ok) break;
                    mbar_arrive_expect_tx(fb, hbytes);
                    tma_load_4d(dst0 + rh.s * hstride, &tmH, kb * kTileK, hx, hy, t.n0, fb);
                    rh.next();
                }
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (1u << 8));
        }
    } else if (warp == kDwThreads / 32 - 1) {
        if (elect_one()) {
            // ---- weights: constants, so nothing here waits for the predecessor kernel.  A slot holds one block of tile_n columns ----
            const int total = in_reg(g.total), step = gridDim.x, tile_n = in_reg(g.tile_n), n_acc = in_reg(g.n_acc), cols = tile_n * n_acc;
            const uint32_t part = (uint32_t)tile_n * 128u, b0 = sbase + g.off_b;
            if (g.b_resident) {
                const int nt = dw_tile(g, blockIdx.x).nt;
                mbar_arrive_expect_tx(bres, part * n_acc * g.kblocks);
#pragma unroll 1
                for (int kb = 0; kb < g.kblocks; ++kb)
#pragma unroll 1
                    for (int h = 0; h < n_acc; ++h) tma_load_2d(b0 + (kb * n_acc + h) * part, &tmB, kb * kTileK, nt * cols + h * tile_n, bres);
            } else {
                PairRing rb = {0, in_reg(g.b_slots), 0u, 0u};
                int fresh = rb.n;
#pragma unroll 1
                for (int ti = blockIdx.x; ti < total && ok; ti += step) {
                    const DwTile t = dw_tile(g, ti);
#pragma unroll 1
                    for (int kb = t.kb0; kb < t.kb1 && ok; ++kb)
#pragma unroll 1
                        for (int h = 0; h < n_acc; ++h) {
                            const uint32_t fb = b_full + 8u * rb.s;
                            ok = --fresh >= 0 || mbar_wait(fb + kEmpty, rb.ph ^ 1u);
                            if (!ok) break;
                            mbar_arrive_expect_tx(fb, part);
                            tma_load_2d(b0 + rb.s * part, &tmB, kb * kTileK, t.nt * cols + h * tile_n, fb);
                            rb.next();
                        }
                }
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (1u << 8));
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ---- MMA ----
            PairRing ra = {0, in_reg(g.a_slots), 0u, 0u}, rb = {0, in_reg(g.b_slots), 0u, 0u};
            const int total = in_reg(g.total), step = gridDim.x, kblocks = in_reg(g.kblocks), last = in_reg(g.last_steps), n_acc = in_reg(g.n_acc), resident = in_reg(g.b_resident), a_stride = in_reg(g.a_stride);
            const uint32_t idesc = in_reg(g.idesc), part = (uint32_t)in_reg(g.tile_n) * 128u, bytes = part * n_acc, b0 = sbase + g.off_b, acc_stride = in_reg((uint32_t)g.acc_stride);
            constexpr uint32_t hi = 64u | (1u << 14) | (2u << 29);
            PairRing rc = {0, in_reg(g.n_bufs), 0u, 0u};      // accumulators
            int fresh = rc.n;
            if (resident) ok = mbar_wait(bres, 0u);
            const uint32_t a_last = a_full + 8u * (uint32_t)(ra.n - 1), a_step = (uint32_t)a_stride >> 4, a0 = 0x10000u | (sbase >> 4), b_step = bytes >> 4, w0 = 0x10000u | (b0 >> 4);
            uint32_t af = a_full, a4 = a0, ready = 0u;      // the operand slot at hand: its barrier, its address, what is known of it
#pragma unroll 1
            for (int ti = blockIdx.x; ti < total && ok; ti += step) {
                int kb0 = 0, kb1 = kblocks;
                if (kEpi == DE_SPLIT) { const DwTile t = dw_tile(g, ti); kb0 = t.kb0; kb1 = t.kb1; }
                const int b = rc.s;
                ok = --fresh >= 0 || mbar_wait(acce + 8u * b, rc.ph ^ 1u);
                if (!ok) break;
                rc.next();
                tc_fence_after();
                const uint32_t d = tmem_base + b * acc_stride;
                uint32_t acc = 0u, b4 = w0 + kb0 * b_step;
                // (few instructions and no branches in here: a lone thread needs some eight cycles for each)
#pragma unroll 1
                for (int kb = kb0; kb < kb1; ++kb) {
                    const int steps = kb == kblocks - 1 ? last : 4;
                    if (!ready) {
                        ok = mbar_wait(af, ra.ph);
                        if (!ok) break;
                    }
                    const uint32_t now = a4, used = af + kEmpty;
                    const bool wrap = af == a_last;
                    af = wrap ? a_full : af + 8u;
                    a4 = wrap ? a0 : a4 + a_step;
                    ra.ph ^= wrap ? 1u : 0u;
                    if (resident) {
                        ready = umma_block(d, hi, now, 2u, 4u, 6u, hi, b4, idesc, acc, steps, used, af, ra.ph);
                        b4 += b_step;
                    } else {
                        ready = 0u;
#pragma unroll 1
                        for (int h = 0; h < n_acc; ++h) {
                            ok = rb.ready || mbar_wait(b_full + 8u * rb.s, rb.ph);
                            if (!ok) break;
                            const uint32_t bs = 0x10000u | ((b0 + rb.s * part) >> 4), b_used = b_full + kEmpty + 8u * rb.s;
                            rb.next();
                            rb.ready = umma_block(d + h * acc_stride, hi, now, 2u, 4u, 6u, hi, bs, idesc, acc, steps, b_used, b_full + 8u * rb.s, rb.ph);
                        }
                        if (!ok) break;
                        umma_commit(used);
                    }
                    acc = 1u;
                }
                if (ok) umma_commit(accf + 8u * b);
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (2u << 8));
        }
    } else {
        // ---- workers ----
        const int wk = warp - 2, wt = threadIdx.x - 64, wpg_log2 = in_reg(g.wpg_log2), groups = in_reg(g.groups);
        const int grp = wk >> wpg_log2, pt = wt - (grp << (wpg_log2 + 5));      // group; thread inside the group
        const int pairs = in_reg(g.pairs), cb = in_reg(g.halo_cb), rw = in_reg(g.rw), kblocks = in_reg(g.kblocks);
        const int row_bytes = in_reg(g.halo_w * g.halo_cb * 2), C = in_reg(g.C), a_stride = in_reg(g.a_stride);
        DwWork u;
        {
            u.q = pt & (pairs - 1);
            const int blk = pt / pairs, upr = g.rw >> 2, upi = ((g.rh + kBR - 1) / kBR) * upr;      // (image, block row, block column)
            const int img = blk / upi, rem = blk - img * upi, uy = rem / upr, ux = rem - uy * upr;
            u.live = img < g.ni && u.q * 2 < ((cb + 15) & ~15);
            u.base = ((img * g.halo_h + kBR * uy * kS) * g.halo_w + 4 * ux * kS) * cb * 2 + u.q * 4;
            const int row0 = img * g.rh * g.rw + kBR * uy * g.rw + 4 * ux;      // (a multiple of 4)
            u.a_row = (uint32_t)row0 * 128u; u.a_step = in_reg((uint32_t)g.rw * 128u);
            u.a_piece = ((((uint32_t)(u.q >> 2) ^ (row0 & 4))) << 4) | ((u.q & 3) << 2);
            u.nrows = min(kBR, max(0, g.rh - kBR * uy));
        }
        const uint32_t dlo = g.dw_act >= 1 ? 0u : 0xff80ff80u, dhi = g.dw_act == 2 ? 0x40c040c0u : 0x7f807f80u;
        const uint32_t plo = g.act >= 1 ? 0u : 0xff80ff80u, phi = g.act == 2 ? 0x40c040c0u : 0x7f807f80u;
        const uint32_t dww = sbase + g.off_dww, halo0 = sbase + g.off_halo;
        const int a_per = in_reg(g.a_slots) / groups, h_per = in_reg(g.h_slots) / groups, hstride = in_reg(g.halo_stride);
        PairRing ra = {0, a_per, 0u, 0u}, rh = {0, h_per, 0u, 0u};      // this group's slots: grp + groups * s
        int fresh = a_per;
        int base = 0;      // items before the tile at hand, modulo groups
        if ((wk & ((1 << wpg_log2) - 1)) == 0) {
            // The first tile's windows, asked for by one warp per group (its own slots): a request is some 250 to 400 cycles of the
            // thread that makes it, so one thread brought the last of eight windows 2800 cycles after the first.
            const DwTile t = dw_tile(g, blockIdx.x);
            const int hy = t.y0 * kS - g.pad, hx = t.x0 * kS - g.pad, n = min(g.h_slots, t.kb1 - t.kb0);
            pdl_wait();
            if (elect_one())
#pragma unroll 1
                for (int i = grp; i < n; i += groups) {
                    mbar_arrive_expect_tx(h_full + 8u * i, (uint32_t)g.halo_bytes);
                    tma_load_4d(halo0 + i * hstride, &tmH, (t.kb0 + i) * kTileK, hx, hy, t.n0, h_full + 8u * i);
                }
            __syncwarp();
        }
        ok = mbar_wait(dww_bar, 0u);
        auto stencil = [&](int kb0, int kb1) {
#pragma unroll 1
            for (int kb = kb0 + ((grp - base) & (groups - 1)); kb < kb1; kb += groups) {
                const int as = grp + groups * ra.s, hs = grp + groups * rh.s;
                // (both barriers are asked at once; the first round's operand slots are free)
                const uint32_t got = --fresh >= 0 ? 1u : mbar_test(a_full + kEmpty + 8u * as, ra.ph ^ 1u), win = mbar_test(h_full + 8u * hs, rh.ph);
                ok = ok && (got || mbar_wait(a_full + kEmpty + 8u * as, ra.ph ^ 1u)) && (win || mbar_wait(h_full + 8u * hs, rh.ph));
                if (!ok) return;
                const int c0 = kb * kTileK + u.q * 2;
                const uint32_t halo = halo0 + hs * hstride, a_base = sbase + as * a_stride;
                if (u.live && c0 < C) {
                    DwTaps taps;
                    dw_load_taps(taps, dww, C, c0);
                    dw_stencil<kS, kBR, kCB>(taps, u, halo, a_base, row_bytes, cb, dlo, dhi);
                } else if (u.live && c0 < ((C + 15) & ~15)) {
                    // the last K = 16 step reads up to 8 channels beyond C: zeros (their weights are zeros too)
#pragma unroll 1
                    for (int x = 0; x < u.nrows * 4; ++x)
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(a_base + u.a_row + (x >> 2) * u.a_step + (((x & 4) ? dw_flip(u) : 0u) ^ u.a_piece ^ (uint32_t)((x & 3) << 4)) + (x & 3) * 128u), "r"(0u) : "memory");
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) { mbar_arrive(a_full + 8u * as); mbar_arrive(h_full + kEmpty + 8u * hs); }
                ra.next(); rh.next();
            }
            base = (base + kb1 - kb0) & (groups - 1);
        };
        const int total = in_reg(g.total), step = gridDim.x, nb = in_reg(g.batch_tiles);
        const int quarter = warp & 3, cgroup = wk >> 2, row = quarter * 32 + lane;      // accumulator lanes; which column chunks
        const uint32_t bias_s = sbase + g.off_bias, t_warp = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const int chunk = in_reg(g.chunk), nchunks = in_reg(g.nchunks), cols = g.n_acc * g.tile_n;
        PairRing rc = {0, in_reg(g.n_bufs), 0u, 0u};      // accumulators
        int ts = blockIdx.x, te = -1, cnt = 0;
        // the stencils of the next batch of tiles, then the epilogues of this one (one copy of either)
#pragma unroll 1
        for (;;) {
#pragma unroll 1
            for (int j = 0, tj = ts; j < nb && tj < total; ++j, tj += step) {
                if (kEpi == DE_SPLIT) { const DwTile t = dw_tile(g, tj); stencil(t.kb0, t.kb1); }
                else stencil(0, kblocks);
            }
            if (te >= 0) {
#pragma unroll 1
              for (int j = 0, tj = te, unit = 0; j < nb && tj < total; ++j, tj += step) {
                const DwTile t = dw_tile(g, tj);      // (a store needs all of it in one thread only)
                const int b = rc.s, n0 = t.nt * cols;
                const uint32_t ph = rc.ph, t_acc = t_warp + b * g.acc_stride;
                rc.next();
                if (kEpi == DE_STORE) {
                    // this thread's row of a result box and the swizzle of its 16-byte pieces (box_piece), made anew per tile
                    int r = row;
                    asm volatile("" : "+r"(r));
                    const bool live_rows = quarter * 32 < g.tile_rows;
                    const uint32_t box_row = (uint32_t)(r * chunk * 2), box_xor = chunk == 64 ? (r & 7u) << 4 : chunk == 32 ? ((r >> 1) & 3u) << 4 : ((r >> 2) & 1u) << 4;
                    // (tile, column chunk) pairs are dealt to the four column groups in turn
#pragma unroll 1
                    for (int c = (cgroup - unit) & 3; c < nchunks; c += 4) {
                        const uint32_t buf = sbase + g.off_stage + (uint32_t)(cgroup * g.out_bufs + (g.out_bufs == 2 ? (cnt & 1) : 0)) * g.box_bytes;
                        // (the group's warps meet twice per box: all know whether to go on, and the box is free)
                        ok = ok && mbar_wait(accf + 8u * b, ph);
                        if (quarter == 0) {
                            if (elect_one()) { if (g.out_bufs == 2) bulk_wait_read<1>(); else bulk_wait_read<0>(); }
                            __syncwarp();
                        }
                        if (!ok && lane == 0) fail_flag[0] = 1;
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + cgroup) : "memory");
                        if (fail_flag[0]) { ok = false; break; }
                        tc_fence_after();
                        // (a quarter of the accumulator's lanes behind the tile's rows has nothing to store)
                        if (!live_rows) warp_arrive(acce + 8u * b, lane);
#pragma unroll 1
                        for (int c0 = 0; live_rows && c0 < chunk; c0 += 32) {
                            const bool wide = chunk - c0 >= 32;
                            float v[32];
                            if (wide) tmem_ld32(t_acc + c * chunk + c0, v); else tmem_ld16(t_acc + c * chunk + c0, v);
                            if (c0 + 32 >= chunk) { tc_fence_before(); warp_arrive(acce + 8u * b, lane); }
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if (h == 1 && !wide) break;
                                uint32_t pk[8];
#pragma unroll
                                for (int q4 = 0; q4 < 16; q4 += 4) {
                                    const float4 bz = ld_shared_f4(bias_s + (uint32_t)(n0 + c * chunk + c0 + 16 * h + q4) * 4u);
                                    const float2 t0 = __fadd2_rn(make_float2(v[16 * h + q4], v[16 * h + q4 + 1]), make_float2(bz.x, bz.y));
                                    const float2 t1 = __fadd2_rn(make_float2(v[16 * h + q4 + 2], v[16 * h + q4 + 3]), make_float2(bz.z, bz.w));
                                    pk[q4 / 2] = clamp_bf16x2(pack2(t0.x, t0.y), plo, phi);
                                    pk[q4 / 2 + 1] = clamp_bf16x2(pack2(t1.x, t1.y), plo, phi);
                                }
                                const uint32_t piece = (uint32_t)(c0 * 2 + 32 * h);      // bytes in front of it, before the swizzle
                                st_shared16(buf + box_row + (piece ^ box_xor), make_uint4(pk[0], pk[1], pk[2], pk[3]));
                                st_shared16(buf + box_row + ((piece + 16u) ^ box_xor), make_uint4(pk[4], pk[5], pk[6], pk[7]));
                            }
                        }
                        fence_proxy_async();
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + cgroup) : "memory");
                        if (quarter == 0) {
                            if (elect_one()) {
                                if (n0 + c * chunk < g.N) tma_store_4d(&tmO, buf, n0 + c * chunk, t.x0, t.y0, t.n0);
                                bulk_commit();
                            }
                            __syncwarp();
                        }
                        ++cnt;
                    }
                    unit += nchunks;
                    if (!ok) break;
                    continue;
                }
                if (ok) ok = mbar_wait(accf + 8u * b, ph);
                // (the workers share named barriers below, so they agree on giving up before any of them can miss one)
                if (!ok && lane == 0) fail_flag[0] = 1;
                asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwWorkers) : "memory");
                if (fail_flag[0]) { ok = false; break; }
                tc_fence_after();
                if (kEpi == DE_GAP) {
                    // global average of whole images: per pass every column group parks the activated fp32 rows of 32 columns in
                    // its slab; (slab, image, column, part) items sum the rows part, part + parts, ... in ascending order, then
                    // the parts in ascending order
                    float *slab0 = reinterpret_cast<float *>(sm + g.off_stage), *slab = slab0 + cgroup * (kTileM * 33), *parts_mem = slab0 + 4 * (kTileM * 33);
                    const float lo1 = act_lo(g.act), hi1 = act_hi(g.act);
                    const int per = 4 * g.gap_imgs * 32, parts = per * 4 <= 512 ? 4 : (per * 2 <= 512 ? 2 : 1);
                    const bool valid = dw_pixel(g, t, row) >= 0;
#pragma unroll 1
                    for (int p0 = 0; p0 < nchunks; p0 += 4) {
                        const int j = p0 + cgroup;
                        if (j < nchunks) {
                            float v[32];
                            const int ncols = min(32, cols - j * 32);
                            if (ncols == 32) tmem_ld32(t_acc + j * 32, v); else { tmem_ld16(t_acc + j * 32, v); for (int q = 16; q < 32; ++q) v[q] = 0.0f; }
#pragma unroll
                            for (int q4 = 0; q4 < 32; q4 += 4) {
                                float4 bz = make_float4(0.f, 0.f, 0.f, 0.f);
                                if (q4 < ncols) bz = ld_shared_f4(bias_s + (uint32_t)(n0 + j * 32 + q4) * 4u);
                                slab[row * 33 + q4] = valid ? fminf(fmaxf(v[q4] + bz.x, lo1), hi1) : 0.0f;
                                slab[row * 33 + q4 + 1] = valid ? fminf(fmaxf(v[q4 + 1] + bz.y, lo1), hi1) : 0.0f;
                                slab[row * 33 + q4 + 2] = valid ? fminf(fmaxf(v[q4 + 2] + bz.z, lo1), hi1) : 0.0f;
                                slab[row * 33 + q4 + 3] = valid ? fminf(fmaxf(v[q4 + 3] + bz.w, lo1), hi1) : 0.0f;
                            }
                        }
                        if (p0 + 4 >= nchunks) { tc_fence_before(); warp_arrive(acce + 8u * b, lane); }
                        asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwWorkers) : "memory");
#pragma unroll 1
                        for (int item = wt; item < per * parts; item += 32 * kDwWorkers) {
                            const int c = item & 31, rest = item >> 5, pa = rest % parts, tri = rest / parts, sl = tri & 3, img = tri >> 2;
                            const float *src = slab0 + sl * (kTileM * 33);
                            float acc = 0.0f;
                            for (int r = pa; r < g.gap_area; r += parts) acc += src[(img * g.gap_area + r) * 33 + c];
                            parts_mem[item] = acc;
                        }
                        asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwWorkers) : "memory");
#pragma unroll 1
                        for (int item = wt; item < per; item += 32 * kDwWorkers) {
                            const int c = item & 31, tri = item >> 5, sl = tri & 3, img = tri >> 2, n = t.n0 + img, nc = n0 + (p0 + sl) * 32 + c;
                            if ((p0 + sl) * 32 + c >= cols || n >= g.batch || nc >= g.N) continue;
                            float acc = 0.0f;
                            for (int pa = 0; pa < parts; ++pa) acc += parts_mem[((tri * parts + pa) << 5) + c];
                            acc /= (float)g.gap_rpi;
                            const size_t oi = (size_t)n * g.out_ctot + nc;
                            if (g.out_f32) reinterpret_cast<float *>(g.out)[oi] = acc;
                            else reinterpret_cast<__nv_bfloat16 *>(g.out)[oi] = __float2bfloat16_rn(acc);
                        }
                        // (the slabs were last read before the barrier above; the next pass's sums wait for its own barrier)
                    }
                } else {
                    // reduction split: as in conv_tc.cuh (fp32 partial sums, every chunk's CTA adds its share of the rows in
                    // ascending chunk order)
                    const long long pix = dw_pixel(g, t, row);
#pragma unroll 1
                    for (int j = cgroup; j < nchunks; j += 4) {
                        float v[16];
                        tmem_ld16(t_acc + j * 16, v);
                        if (pix >= 0)
#pragma unroll
                            for (int q4 = 0; q4 < 16; q4 += 4)
                                __stcg(reinterpret_cast<float4 *>(g.split_part + t.ks * g.split_stride + pix * g.split_ld + n0 + j * 16 + q4), make_float4(v[q4], v[q4 + 1], v[q4 + 2], v[q4 + 3]));
                    }
                    tc_fence_before();
                    warp_arrive(acce + 8u * b, lane);
                    __threadfence();
                    asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwWorkers) : "memory");
                    unsigned int *arr = g.split_cnt + 2 * ((size_t)t.mt * g.d_nt.d + t.nt);
                    if (wt == 0) {
                        atomicAdd(arr, 1u);
                        int seen = 0;
#pragma unroll 1
                        for (int spin = 0; spin < (1 << 22); ++spin) {
                            if (*reinterpret_cast<volatile unsigned int *>(arr) >= (unsigned int)g.ksplit) { seen = 1; break; }
                            __nanosleep(32);
                        }
                        fail_flag[1] = seen;
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwWorkers) : "memory");
                    if (!fail_flag[1]) { ok = false; break; }
                    __threadfence();
                    const float lo1 = act_lo(g.act), hi1 = act_hi(g.act);
                    const int rows_per = (g.tile_rows + g.ksplit - 1) / g.ksplit, r0 = t.ks * rows_per, r1 = min(g.tile_rows, r0 + rows_per), c4n = cols >> 2;
#pragma unroll 1
                    for (int idx = wt; idx < (r1 - r0) * c4n; idx += 32 * kDwWorkers) {
                        const int rr = r0 + idx / c4n, c4 = idx % c4n, nc = n0 + c4 * 4;
                        const long long px = dw_pixel(g, t, rr);
                        if (px < 0 || nc >= g.N) continue;
                        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                        for (int sp = 0; sp < g.ksplit; ++sp) {
                            const float4 x4 = __ldcg(reinterpret_cast<const float4 *>(g.split_part + sp * g.split_stride + px * g.split_ld + nc));
                            a.x += x4.x; a.y += x4.y; a.z += x4.z; a.w += x4.w;
                        }
                        const float4 bz = ld_shared_f4(bias_s + (uint32_t)nc * 4u);
                        *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(g.out) + px * g.out_ctot + nc) =
                            make_uint2(pack2(fminf(fmaxf(a.x + bz.x, lo1), hi1), fminf(fmaxf(a.y + bz.y, lo1), hi1)),
                                       pack2(fminf(fmaxf(a.z + bz.z, lo1), hi1), fminf(fmaxf(a.w + bz.w, lo1), hi1)));
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(32 * kDwWorkers) : "memory");
                    if (wt == 0) {
                        __threadfence();
                        const unsigned int old = atomicAdd(arr + 1, 1u);
                        if (old == (unsigned int)(g.ksplit - 1)) { arr[0] = 0u; arr[1] = 0u; }
                    }
                }
              }
            }
            if (ts >= total || !ok) break;
            te = ts;
            ts += nb * step;
        }
        if (kEpi == DE_STORE && quarter == 0) {
            if (elect_one()) bulk_wait_read<0>();
            __syncwarp();
        }
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (3u << 8));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols) : "memory");
    }
}

}  // namespace xk
