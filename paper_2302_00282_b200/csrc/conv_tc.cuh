// Convolution, pointwise product and fully connected layer as an implicit GEMM on the 5th-generation tensor cores
// (sm_100a) whose every operand and result is moved by the copy engine (x.conv / x.matmul of Table 3 of the Xenos paper,
// with the shortcut, concat and global-average tails of its Table 1 in the epilogue).
//
//   D [output pixels][output channels] = A [pixels][(tap, channel)] x B [(tap, channel)][channels]
//
// A CTA walks over tiles of 128 consecutive output pixels (numbered image, row, column: a tile may span rows and images,
// so no row of the MMA is padding except in the last tile) x tile_n <= 256 channels (Section 4.2.1's split).
//   warp 0      A operand (with warp 3 where a block takes several boxes): one box per 64-channel block and tap.  A 1x1 stride-1 product reads rows of the [pixels][C]
//               matrix; every other window is fetched in the copy engine's im2col form, which walks the output pixels
//               with the convolution's stride and fills padding with zeros.  No thread computes an address per element.
//   warp 1      tcgen05.mma into one of two tensor-memory accumulators
//   warp 2      B operand: streamed with A, or, when a CTA keeps one channel tile and its weights fit beside the ring,
//               loaded once and kept (b_resident).  Weights are constants, so this warp does not wait for the
//               predecessor kernel: the first stages' weights arrive while that kernel drains.
//   warps 4-11  epilogue of tile i while tile i + 1 is multiplied: two warps per quarter of the accumulator's lanes take
//               alternate column chunks: bias, activation [, + shortcut, activation], bf16, a swizzled 32-row box in
//               shared memory, one bulk tensor store.  A shortcut tile arrives in the same boxes the result leaves from.
// A role is one elected lane.  Measured: a request with its announcement takes that lane 50 to 120 cycles, the look at a barrier
// 190 (mbar_test), other work some eight cycles an instruction; an MMA takes the pipe 40-48 cycles (M = 128, N <= 64; 64 at N =
// 128, 128 at N = 256).  The copy engine brings 16 KB of A in 150 to 180 cycles alone and in 200 to 256 with all SMs at it.
// What bounds it: at N = 64 the products' issue (some 260 cycles a block, 400 before umma_block and the early look at the ring)
// and shared memory, which an MMA of N <= 128 reads at its full 128 B per cycle while the copies write; at N = 256 the tensor
// pipe (550 of 512 cycles at 72 blocks of a 3 x 3 window over 512 channels); for 1x1 products HBM.
//
// Channels: C in (32, 64] and above uses 64-channel boxes (128-byte swizzle), C <= 32 and C <= 16 use boxes of 32 and 16
// channels (64- and 32-byte swizzle; 2 or 4 taps share a stage), and MMA steps over channels beyond C are not issued.
#pragma once

#include "gemm_tc.cuh"

namespace xk {

constexpr int kCvEpiWarps = 8;
constexpr int kCvThreads = 128 + 32 * kCvEpiWarps;
constexpr int kCvMaxStages = 6;
enum { CE_STORE = 0, CE_SKIP = 1, CE_VEC = 2, CE_GAP = 3, CE_SPLIT = 4, CE_CLUSTER = 5 };
constexpr int kCvMaxCluster = 8;
constexpr int kMaxSkipSlots = 4;         // shortcut / result boxes per epilogue warp
constexpr int kGapFloats = 4352;         // column sums of an average, per half of the epilogue

// Exact division of n < 2^31 by a constant of the launch: multiplication by a rounded-up reciprocal and a shift (Granlund and
// Montgomery, Division by Invariant Integers using Multiplication, 1994).
struct FastDiv {
    uint32_t mul, shift, d;
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return (__umulhi(n, mul) + n) >> shift; }
};
inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f;
    f.d = d; f.shift = 0;
    while ((1ull << f.shift) < d) ++f.shift;
    f.mul = (uint32_t)((((1ull << f.shift) - d) << 32) / d + 1);
    return f;
}

struct ConvSegment {
    int im2col;                    // 0: rows of the [pixels][C] matrix; 1: im2col boxes
    int k, stride, low;            // window size, stride, first input coordinate of output 0 (= -padding)
    int cblocks, last_steps;       // 64-channel boxes per tap; K = 16 steps of the last one
    int per_stage, spb;            // boxes per stage (1, 2, 4); K = 16 steps per box (4, 2, 1)
    int taps, kblocks;             // taps of the window, stages of this segment
    uint32_t box_bytes, box_stride;      // bytes a box delivers; distance of the boxes of one stage
    uint32_t desc_hi;              // upper half of the operand descriptor (swizzle mode and group stride)
};

struct ConvParams {
    ConvSegment seg[2];
    const float *bias;
    void *out;
    unsigned int *status;
    FastDiv d_rpi, d_q, d_nt, d_ks;
    int rows, tile_rows;           // output pixels of this run; pixels a tile advances
    int total, tile_n, npad, N;
    int kblocks, stages, stage_bytes, b_resident, b_group;
    int acc_stride, tmem_cols;
    int chunk, nchunks, box_bytes; // epilogue: columns per chunk, chunks per tile, bytes of one 32-row staging box
    int s_slots;                   // boxes per epilogue warp
    int act, act2, out_ctot, out_f32;
    uint32_t idesc;
    int off_b, off_stage, off_bias, off_bar;
    int launch_id;
    // global average (CE_GAP): whole images per tile, or gap_parts tiles per image
    int gap_imgs, gap_rpi, gap_parts, batch;
    // reduction split (CE_SPLIT)
    int ksplit, kb_per, split_ld;
    long long split_stride;
    float *split_part;
    unsigned int *split_cnt;
    const __nv_bfloat16 *skip;     // CE_SPLIT: identity shortcut, read directly
    int skip_ctot;
};

__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// c must be a multiple of 8 channels; w, h may be negative; (s, r) is the tap
__device__ __forceinline__ void tma_load_im2col(uint32_t dst, const CUtensorMap *tm, int c, int w, int h, int n, uint32_t bar, int s, int r) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"((unsigned short)s), "h"((unsigned short)r) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *tm, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(tm), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory"); }

// A role's copy of the tile walk: tile index -> (pixel tile, channel tile, K range).
struct ConvTile { int mt, nt, ks, kb0, kb1; };
__device__ __forceinline__ ConvTile conv_tile(const ConvParams &g, int ti) {
    ConvTile t;
    const uint32_t pair = g.d_ks.div((uint32_t)ti);
    t.ks = ti - (int)(pair * g.d_ks.d);
    t.mt = (int)g.d_nt.div(pair);
    t.nt = (int)pair - t.mt * (int)g.d_nt.d;
    t.kb0 = t.ks * g.kb_per;
    t.kb1 = min(g.kblocks, t.kb0 + g.kb_per);
    return t;
}
// first output pixel of a tile (a global average over several tiles per image cuts every image anew)
__device__ __forceinline__ int conv_row0(const ConvParams &g, int mt) {
    if (g.gap_parts > 1) { const int img = mt / g.gap_parts; return img * g.gap_rpi + (mt - img * g.gap_parts) * kTileM; }
    return mt * g.tile_rows;
}

// A launch constant kept in a register.  The role loops below contain asm volatile statements that clobber memory, across
// which the compiler reloads parameters from constant memory; each such load is some 40 cycles on the issuing thread's path.
__device__ __forceinline__ int in_reg(int x) { asm volatile("" : "+r"(x)); return x; }
__device__ __forceinline__ uint32_t in_reg(uint32_t x) { asm volatile("" : "+r"(x)); return x; }

// The ring as a thread that walks all of it sees it: the slot's barrier, data and phase; ready: what is known of its barrier,
// which is asked as early as possible (see mbar_test).  No branches: a lone thread needs some eight cycles an instruction and
// more for a branch.
struct ConvRing {
    uint32_t ph, fb, data, fb0, data0, fb_last, step, ready;
    __device__ __forceinline__ void init(const ConvParams &g, uint32_t sbase, uint32_t bar) {
        step = in_reg((uint32_t)g.stage_bytes); ph = 0u; ready = 0u;
        fb = fb0 = in_reg(bar); data = data0 = in_reg(sbase);
        fb_last = in_reg(bar + 8u * (uint32_t)(g.stages - 1));
    }
    __device__ __forceinline__ uint32_t empty() const { return fb + 8u * kCvMaxStages; }
    __device__ __forceinline__ bool full() const { return ready || mbar_wait(fb, ph); }
    __device__ __forceinline__ void next() {
        const bool wrap = fb == fb_last;
        fb = wrap ? fb0 : fb + 8u;
        data = wrap ? data0 : data + step;
        ph ^= wrap ? 1u : 0u;
    }
};

// A filling thread's view of the ring: every turn-th slot.  Two threads bring the activation operand where a stage takes several
// boxes (16 or 32 channels: some 180 cycles a box, 720 a stage); else one does (it gets a 64-channel block in 250, as often as
// the products ask for one, and a second thread's look at the barriers costs more than it brings: ResNet-18 at batch 32 250 us
// against 248; SqueezeNet, whose expands have such stages, 162 with two threads against 165).
struct ConvFill {
    int s, n, turn, skip;              // skip: blocks of the next stretch before this thread's first one
    uint32_t ph, fresh, fb, data, step, back;
    __device__ __forceinline__ void init(const ConvParams &g, uint32_t sbase, uint32_t bar, int which) {
        turn = in_reg(g.seg[0].per_stage > 1 ? 2 : 1);
        s = skip = which; n = in_reg(g.stages); ph = 0u; fresh = 1u;
        step = in_reg((uint32_t)g.stage_bytes); back = (uint32_t)n * step;
        fb = bar + 8u * which; data = sbase + step * which;
    }
    // (nothing has been put into the slots of the first round yet: no need to ask for room)
    __device__ __forceinline__ bool room() const { return fresh || mbar_wait(fb + 8u * kCvMaxStages, ph ^ 1u); }
    __device__ __forceinline__ void next() {
        s += turn; fb += 8u * turn; data += (uint32_t)turn * step;
        const bool wrap = s >= n;
        s -= wrap ? n : 0; fb -= wrap ? 8u * (uint32_t)n : 0u; data -= wrap ? back : 0u;
        ph ^= wrap ? 1u : 0u; fresh = wrap ? 0u : fresh;
    }
};

// One thread's copies of a segment's K blocks [kb0, kb1) of a tile.  kSeg is a compile-time index: fields of g.seg[i] with a
// run-time i are indexed constant loads.
template <int kSeg>
__device__ __forceinline__ bool conv_load_a(const ConvParams &g, const CUtensorMap *tm, ConvFill &st, int kb0, int kb1, int m0, int n, int p, int q) {
    const ConvSegment &sg = g.seg[kSeg];
    const uint32_t box = in_reg(sg.box_bytes);
    int kb = kb0 + st.skip;
    if (!sg.im2col && sg.per_stage == 1) {
#pragma unroll 1
        for (; kb < kb1; kb += st.turn) {
            if (!st.room()) return false;
            mbar_arrive_expect_tx(st.fb, box);
            tma_load_2d(st.data, tm, kb * kTileK, m0, st.fb);
            st.next();
        }
        st.skip = kb - kb1;
        return true;
    }
    const int h0 = p * sg.stride + sg.low, w0 = q * sg.stride + sg.low;
    const int k = in_reg(sg.k);
    if (sg.per_stage == 1) {
        const int cend = in_reg(sg.cblocks * kTileK);
        int c = 0, r = 0, s = 0;
        auto advance = [&]() {
            c += kTileK;
            const bool tap = c == cend;
            c = tap ? 0 : c;
            s += tap ? 1 : 0;
            const bool row = s == k;
            s = row ? 0 : s;
            r += row ? 1 : 0;
        };
        if (kb0) {
            const int tap = kb0 / sg.cblocks;
            c = (kb0 - tap * sg.cblocks) * kTileK; r = tap / k; s = tap - r * k;
        }
        if (st.skip) advance();
#pragma unroll 1
        for (; kb < kb1; kb += st.turn) {
            if (!st.room()) return false;
            mbar_arrive_expect_tx(st.fb, box);
            tma_load_im2col(st.data, tm, c, w0, h0, n, st.fb, s, r);
            st.next();
            advance();
            if (st.turn == 2) advance();
        }
        st.skip = kb - kb1;
        return true;
    }
    // several taps of 16 or 32 channels share a stage
    const int per = in_reg(sg.per_stage), taps = in_reg(sg.taps);
    const uint32_t stride = in_reg(sg.box_stride);
    int tap = kb * per, r = tap / k, s = tap - r * k;
#pragma unroll 1
    for (; kb < kb1; kb += st.turn) {
        const int nb = min(per, taps - tap);
        if (!st.room()) return false;
        mbar_arrive_expect_tx(st.fb, box * nb);
#pragma unroll 1
        for (int b = 0; b < nb; ++b) {
            if (sg.im2col) tma_load_im2col(st.data + b * stride, tm, 0, w0, h0, n, st.fb, s, r);
            else tma_load_2d(st.data + b * stride, tm, 0, m0, st.fb);
            if (++s == k) { s = 0; ++r; }
        }
        tap += st.turn * per;
        s += (st.turn - 1) * per;
        while (s >= k) { s -= k; ++r; }
        st.next();
    }
    st.skip = kb - kb1;
    return true;
}

__device__ __forceinline__ void umma_bf16_acc(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.eq.u32 p, 0, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(da), "l"(db), "r"(idesc) : "memory");
}

// One thread's products of a segment's K blocks [kb0, kb1) of a tile.  kRes: the weights are resident, block kb at b_res +
// kb * tile bytes (bseen: how many of their four arrival groups have been waited for); else they arrive in the ring behind
// the activation block.
template <int kSeg, bool kRes>
__device__ __forceinline__ bool conv_mma(const ConvParams &g, ConvRing &st, uint32_t bar, int kb0, int kb1, int kb_off, uint32_t d_tmem, uint32_t acc,
                                         int &bseen, uint32_t b_res) {
    const ConvSegment &sg = g.seg[kSeg];
    constexpr uint32_t b_hi = 64u | (1u << 14) | (2u << 29);      // 128-byte swizzle, 1024-byte groups
    const uint32_t a_hi = in_reg(sg.desc_hi);
    const uint32_t idesc = in_reg(g.idesc), tile16 = in_reg((uint32_t)g.tile_n * 8u);
    const int per = in_reg(sg.per_stage);
    if (kRes && bseen < 4)
        while (bseen < 4 && bseen * g.b_group < kb1 + kb_off) {
            // (a CTA's first tile waits for all of its weights here; the ring fills meanwhile)
            if (!mbar_wait(bar + 8u * (2 * kCvMaxStages + 4 + bseen), 0u)) return false;
            ++bseen;
        }
    uint32_t b4 = 0x10000u | ((b_res >> 4) + kb0 * tile16);
    if (per == 1) {
        const int cblocks = in_reg(sg.cblocks), last = in_reg(sg.last_steps);
        int cb = kb0 ? kb0 % cblocks : 0;
#pragma unroll 1
        for (int kb = kb0; kb < kb1; ++kb) {
            const uint32_t a4 = 0x10000u | (st.data >> 4), used = st.empty();      // (shared addresses are below 2^18)
            if (!kRes) b4 = a4 + (kABytes >> 4);
            const bool end = ++cb == cblocks;
            const int steps = end ? last : 4;
            cb = end ? 0 : cb;
            if (!st.full()) return false;
            st.next();
            st.ready = umma_block(d_tmem, a_hi, a4, 2u, 4u, 6u, b_hi, b4, idesc, acc, steps, used, st.fb, st.ph);
            acc = 1u;
            if (kRes) b4 += tile16;
        }
    } else {
        // descriptor advance per K = 16 step, in 16-byte units: a box holds one step (16 channels) or two (32)
        const int spb = in_reg(sg.spb);
        const uint32_t box16 = in_reg(sg.box_stride >> 4);
        const uint32_t s1 = spb == 1 ? box16 : 2u, s2 = spb == 1 ? 2 * box16 : box16;
        int left = sg.taps - kb0 * per;
#pragma unroll 1
        for (int kb = kb0; kb < kb1; ++kb) {
            const uint32_t a4 = 0x10000u | (st.data >> 4), used = st.empty();
            if (!kRes) b4 = a4 + (kABytes >> 4);
            const int steps = min(per, left) * spb;
            left -= per;
            if (!st.full()) return false;
            st.next();
            st.ready = umma_block(d_tmem, a_hi, a4, s1, s2, s1 + s2, b_hi, b4, idesc, acc, steps, used, st.fb, st.ph);
            acc = 1u;
            if (kRes) b4 += tile16;
        }
    }
    return true;
}
template <bool kRes>
__device__ __forceinline__ bool conv_mma_loop(const ConvParams &g, uint32_t sbase, uint32_t bar, uint32_t tmem_base) {
    ConvRing st;
    st.init(g, sbase, bar);
    int i = 0, bseen = 0;
    const int k0 = in_reg(g.seg[0].kblocks), total = in_reg(g.total);
    const uint32_t b_res = sbase + g.off_b, acc_stride = in_reg((uint32_t)g.acc_stride), accf = bar + 8u * (2 * kCvMaxStages);
#pragma unroll 1
    for (int ti = blockIdx.x; ti < total; ti += gridDim.x, ++i) {
        const int b = i & 1;
        const ConvTile t = conv_tile(g, ti);
        if (i > 1 && !mbar_wait(accf + 8u * (2 + b), ((i >> 1) & 1) ^ 1u)) return false;      // the epilogue has drained this accumulator
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + b * acc_stride;
        if (t.kb0 < k0 && !conv_mma<0, kRes>(g, st, bar, t.kb0, min(t.kb1, k0), 0, d_tmem, 0u, bseen, b_res)) return false;
        if (t.kb1 > k0 && !conv_mma<1, kRes>(g, st, bar, max(t.kb0 - k0, 0), t.kb1 - k0, k0, d_tmem, t.kb0 < k0 ? 1u : 0u, bseen, b_res + k0 * g.tile_n * 128)) return false;
        umma_commit(accf + 8u * b);
    }
    return true;
}

// Byte offset of 16-byte piece j of row r in a box of `cols` bf16 columns (64, 32 or 16), in the swizzle of its width.
__device__ __forceinline__ uint32_t box_piece(int cols, int r, int j) {
    if (cols == 64) return (uint32_t)(r * 128 + ((j ^ (r & 7)) << 4));
    if (cols == 32) return (uint32_t)(r * 64 + ((j ^ ((r >> 1) & 3)) << 4));
    return (uint32_t)(r * 32 + ((j ^ ((r >> 2) & 1)) << 4));
}

// 16 accumulator columns of one row: bias, activation [, shortcut, second activation], rounded to bf16 pairs.  The last
// activation is a clamp on the pairs (0 and 6 are bf16 values and rounding is monotonic: clamping first gives the same).
template <bool kSkip>
__device__ __forceinline__ void conv_finish16(const ConvParams &g, const float *v, uint32_t sbias, const uint32_t *sk, uint32_t *pk,
                                              uint32_t plo, uint32_t phi) {
    const float lo1 = act_lo(g.act), hi1 = act_hi(g.act);
#pragma unroll
    for (int q4 = 0; q4 < 16; q4 += 4) {
        const float4 bz = ld_shared_f4(sbias + (uint32_t)q4 * 4u);
        float2 t0 = __fadd2_rn(make_float2(v[q4], v[q4 + 1]), make_float2(bz.x, bz.y));
        float2 t1 = __fadd2_rn(make_float2(v[q4 + 2], v[q4 + 3]), make_float2(bz.z, bz.w));
        if (kSkip) {
            if (g.act) {
                t0.x = fminf(fmaxf(t0.x, lo1), hi1); t0.y = fminf(fmaxf(t0.y, lo1), hi1);
                t1.x = fminf(fmaxf(t1.x, lo1), hi1); t1.y = fminf(fmaxf(t1.y, lo1), hi1);
            }
            const uint32_t s0 = sk[q4 / 2], s1 = sk[q4 / 2 + 1];
            t0 = __fadd2_rn(t0, make_float2(__uint_as_float(s0 << 16), __uint_as_float(s0 & 0xffff0000u)));
            t1 = __fadd2_rn(t1, make_float2(__uint_as_float(s1 << 16), __uint_as_float(s1 & 0xffff0000u)));
        }
        pk[q4 / 2] = clamp_bf16x2(pack2(t0.x, t0.y), plo, phi);
        pk[q4 / 2 + 1] = clamp_bf16x2(pack2(t1.x, t1.y), plo, phi);
    }
}

// 16 columns of one row in fp32, for the epilogues that do not store bf16 boxes.
__device__ __forceinline__ void conv_act16(const ConvParams &g, float *v, uint32_t sbias) {
    const float lo1 = act_lo(g.act), hi1 = act_hi(g.act);
#pragma unroll
    for (int q4 = 0; q4 < 16; q4 += 4) {
        const float4 bz = ld_shared_f4(sbias + (uint32_t)q4 * 4u);
        v[q4] = fminf(fmaxf(v[q4] + bz.x, lo1), hi1); v[q4 + 1] = fminf(fmaxf(v[q4 + 1] + bz.y, lo1), hi1);
        v[q4 + 2] = fminf(fmaxf(v[q4 + 2] + bz.z, lo1), hi1); v[q4 + 3] = fminf(fmaxf(v[q4 + 3] + bz.w, lo1), hi1);
    }
}

// Sums of 32 columns over the 32 rows of a warp: lane l holds a row's 32 values and gets the sum of column l.  Each exchange
// halves the columns a lane carries: 31 shuffles, a fixed order.
__device__ __forceinline__ float column_sum(const float (&v)[32], bool mine, int lane) {
    float w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float a = mine ? v[i] : 0.0f, b = mine ? v[i + 16] : 0.0f;
        const bool up = lane & 16;
        w[i] = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
    }
#pragma unroll
    for (int n = 8; n >= 1; n >>= 1)
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const bool up = lane & n;
            const float keep = up ? w[i + n] : w[i], send = up ? w[i] : w[i + n];
            w[i] = keep + __shfl_xor_sync(0xffffffffu, send, n);
        }
    return w[0];
}

// Global average.  A warp sums 32 columns of its 32 rows in registers, once per image that its rows meet; the sums of a
// quarter and an image go to slot image + quarter of a small buffer (no two pairs share one), and the quarters are added in
// ascending order: a fixed order.  Images of more than 128 pixels take gap_parts tiles each: a tile leaves its column sums in
// the split scratch, and the tile that arrives last at the image's counter adds the parts in ascending order.  (With the
// activated rows parked in shared memory and summed column by column the epilogue took longer than the product: 512 -> 1000
// channels, 13 x 13, batch 32, 33.7 us; 23.4 us in this form.)
__device__ __forceinline__ bool conv_epilogue_gap(const ConvParams &g, uint8_t *sm, uint32_t bar, uint32_t tmem_base, volatile int *fail_flag) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e = warp - 4, quarter = warp & 3, half = e >> 2;
    const int row = quarter * 32 + lane, ht = quarter * 32 + lane;                 // thread of the half
    float *part = reinterpret_cast<float *>(sm + g.off_stage) + half * kGapFloats;
    const int slots = g.gap_imgs + 3, group = max(1, kGapFloats / (32 * slots));     // chunks of a half between two barriers
    const uint32_t bias_s = smem_u32(sm) + g.off_bias;
    const uint32_t t_warp = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const bool parted = g.gap_parts > 1;
    const float lo2 = act_lo(g.act2), hi2 = act_hi(g.act2);
    auto store = [&](int img, int col, float sum) {
        sum /= (float)g.gap_rpi;
        const size_t oi = (size_t)img * g.out_ctot + col;
        if (g.out_f32) reinterpret_cast<float *>(g.out)[oi] = sum;
        else reinterpret_cast<__nv_bfloat16 *>(g.out)[oi] = __float2bfloat16_rn(sum);
    };
    int i = 0;
#pragma unroll 1
    for (int ti = blockIdx.x; ti < g.total; ti += gridDim.x, ++i) {
        const ConvTile t = conv_tile(g, ti);
        const int b = i & 1, n0 = t.nt * g.tile_n;
        const int img0 = parted ? t.mt / g.gap_parts : t.mt * g.gap_imgs, gp = parted ? t.mt - img0 * g.gap_parts : 0;
        const int area = parted ? kTileM : g.gap_rpi;      // rows of the tile that one image's sum takes
        const bool valid = parted ? gp * kTileM + row < g.gap_rpi : row < g.tile_rows;
        const size_t pix = (size_t)conv_row0(g, t.mt) + row;
        if (!mbar_wait(bar + 8u * (2 * kCvMaxStages + b), (i >> 1) & 1) && lane == 0) fail_flag[0] = 1;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (fail_flag[0]) return false;
        tc_fence_after();
        const int img_lo = quarter * 32 / area, img_hi = min(g.gap_imgs - 1, (quarter * 32 + 31) / area), my = row / area;
#pragma unroll 1
        for (int jg = half; jg < g.nchunks; jg += 2 * group) {
            const int jend = min(g.nchunks, jg + 2 * group);
#pragma unroll 1
            for (int j = jg; j < jend; j += 2) {
                float v[32];
                const int ncols = min(32, g.tile_n - j * 32), nc0 = n0 + j * 32;
                const uint32_t ta = t_warp + b * g.acc_stride + j * 32;
                if (ncols == 32) tmem_ld32(ta, v); else tmem_ld16(ta, v);
                if (j + 2 >= g.nchunks) {
                    tc_fence_before();
                    warp_arrive(bar + 8u * (2 * kCvMaxStages + 2 + b), lane);
                }
                conv_act16(g, v, bias_s + (uint32_t)nc0 * 4u);
                if (ncols == 32) conv_act16(g, v + 16, bias_s + (uint32_t)(nc0 + 16) * 4u);
                else
#pragma unroll
                    for (int c = 16; c < 32; ++c) v[c] = 0.0f;
                if (g.skip && valid && pix < (size_t)g.rows)
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        if (h * 8 < ncols && nc0 + h * 8 + 8 <= g.N) {
                            const f8 s = unpack8(__ldg(reinterpret_cast<const uint4 *>(g.skip + pix * g.skip_ctot + nc0 + h * 8)));
#pragma unroll
                            for (int c = 0; c < 8; ++c) v[h * 8 + c] += s.v[c];
                        }
                if (g.act2)
#pragma unroll
                    for (int c = 0; c < 32; ++c) v[c] = fminf(fmaxf(v[c], lo2), hi2);
                const int jl = (j - jg) >> 1;
#pragma unroll 1
                for (int img = img_lo; img <= img_hi; ++img)
                    part[((img + quarter) * group + jl) * 32 + lane] = column_sum(v, valid && my == img, lane);
            }
            asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory");
            const int nj = (jend - jg + 1) >> 1;
#pragma unroll 1
            for (int item = ht; item < nj * g.gap_imgs * 32; item += 128) {
                const int c = item & 31, rest = item >> 5, img = rest / nj, jl = rest - img * nj, col = (jg + 2 * jl) * 32 + c;
                if (col >= g.tile_n || n0 + col >= g.N || img0 + img >= g.batch) continue;
                float acc = 0.0f;
                for (int q = img * area >> 5; q <= (img * area + area - 1) >> 5; ++q) acc += part[((img + q) * group + jl) * 32 + c];
                if (parted) __stcg(g.split_part + (size_t)t.mt * g.split_ld + n0 + col, acc);
                else store(img0 + img, n0 + col, acc);
            }
            asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory");
        }
        if (half >= g.nchunks) warp_arrive(bar + 8u * (2 * kCvMaxStages + 2 + b), lane);
        if (parted) {
            __threadfence();
            asm volatile("bar.sync 1, 256;" ::: "memory");
            unsigned int *cnt = g.split_cnt + 2 * ((size_t)img0 * g.d_nt.d + t.nt);
            if (e == 0 && lane == 0) fail_flag[1] = atomicAdd(cnt, 1u) == (unsigned int)(g.gap_parts - 1) ? 1 : 0;
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (fail_flag[1]) {
                __threadfence();
                for (int col = threadIdx.x - 128; col < g.tile_n; col += 256) {
                    if (n0 + col >= g.N || img0 >= g.batch) continue;
                    float acc = 0.0f;
#pragma unroll 1
                    for (int q = 0; q < g.gap_parts; ++q) acc += __ldcg(g.split_part + ((size_t)img0 * g.gap_parts + q) * g.split_ld + n0 + col);
                    store(img0, n0 + col, acc);
                }
                if (e == 0 && lane == 0) *cnt = 0u;      // ready for the next run
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");      // (fail_flag[1] is read before the next tile rewrites it)
        }
    }
    return true;
}

// Four adjacent columns of one output pixel behind a split reduction: bias, activation, identity shortcut, second
// activation, store.
// (sk: the shortcut's four elements, asked for by the caller)
__device__ __forceinline__ uint2 conv_skip4(const ConvParams &g, int nc, size_t pix) {
    return g.skip ? __ldg(reinterpret_cast<const uint2 *>(g.skip + pix * g.skip_ctot + nc)) : make_uint2(0u, 0u);
}
__device__ __forceinline__ void conv_finish_store4(const ConvParams &g, float4 a, const float4 bz, int nc, size_t pix, const uint2 sk) {
    const float lo1 = act_lo(g.act), hi1 = act_hi(g.act), lo2 = act_lo(g.act2), hi2 = act_hi(g.act2);
    float v[4] = {a.x + bz.x, a.y + bz.y, a.z + bz.z, a.w + bz.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = fminf(fmaxf(v[c], lo1), hi1);
    if (g.skip) {
        v[0] += __uint_as_float(sk.x << 16); v[1] += __uint_as_float(sk.x & 0xffff0000u);
        v[2] += __uint_as_float(sk.y << 16); v[3] += __uint_as_float(sk.y & 0xffff0000u);
    }
    if (g.act2) {
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = fminf(fmaxf(v[c], lo2), hi2);
    }
    if (g.out_f32 || (g.out_ctot & 7)) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (nc + c < g.N) {
                if (g.out_f32) reinterpret_cast<float *>(g.out)[pix * g.out_ctot + nc + c] = v[c];
                else reinterpret_cast<__nv_bfloat16 *>(g.out)[pix * g.out_ctot + nc + c] = __float2bfloat16_rn(v[c]);
            }
    } else {
        *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(g.out) + pix * g.out_ctot + nc) = make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
    }
}

// Reduction split (Section 4.2.2: the C / R / S split, which needs an additional reduction): chunk ks of a tile parks its
// fp32 partial sums [pixel][channel] in the workspace; when all chunks of the tile have arrived, every chunk's CTA adds
// them, in ascending chunk order, for its share of the tile's rows.  The chunks of a tile are consecutive tiles of the walk:
// a wait never points at a later tile of its own CTA, so waits cannot form a cycle; they are bounded all the same.
__device__ __forceinline__ bool conv_epilogue_split(const ConvParams &g, uint8_t *sm, uint32_t bar, uint32_t tmem_base, volatile int *fail_flag) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e = warp - 4, quarter = warp & 3, half = e >> 2;
    const int row = quarter * 32 + lane, et = threadIdx.x - 128;
    const uint32_t bias_s = smem_u32(sm) + g.off_bias;
    const uint32_t t_warp = tmem_base + ((uint32_t)(quarter * 32) << 16);
    int i = 0;
#pragma unroll 1
    for (int ti = blockIdx.x; ti < g.total; ti += gridDim.x, ++i) {
        const ConvTile t = conv_tile(g, ti);
        const int b = i & 1, n0 = t.nt * g.tile_n, m0 = t.mt * g.tile_rows;
        if (!mbar_wait(bar + 8u * (2 * kCvMaxStages + b), (i >> 1) & 1) && lane == 0) fail_flag[0] = 1;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (fail_flag[0]) return false;
        tc_fence_after();
        float *part = g.split_part + (size_t)t.ks * g.split_stride + (size_t)(m0 + row) * g.split_ld + n0;
#pragma unroll 1
        for (int j = half; j < g.nchunks; j += 2) {
            float v[16];
            tmem_ld16(t_warp + b * g.acc_stride + j * 16, v);
            if (m0 + row < g.rows)
#pragma unroll
                for (int q4 = 0; q4 < 16; q4 += 4) __stcg(reinterpret_cast<float4 *>(part + j * 16 + q4), make_float4(v[q4], v[q4 + 1], v[q4 + 2], v[q4 + 3]));
        }
        tc_fence_before();
        warp_arrive(bar + 8u * (2 * kCvMaxStages + 2 + b), lane);
        __threadfence();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        unsigned int *cnt = g.split_cnt + 2 * ((size_t)t.mt * g.d_nt.d + t.nt);      // [arrived, reduced]
        if (et == 0) {
            atomicAdd(cnt, 1u);
            int seen = 0;
#pragma unroll 1
            for (int spin = 0; spin < (1 << 22); ++spin) {
                if (*reinterpret_cast<volatile unsigned int *>(cnt) >= (unsigned int)g.ksplit) { seen = 1; break; }
                __nanosleep(32);
            }
            fail_flag[1] = seen;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (!fail_flag[1]) return false;
        __threadfence();
        const int live = min(kTileM, g.rows - m0), rows_per = (live + g.ksplit - 1) / g.ksplit;
        const int r0 = t.ks * rows_per, r1 = min(live, r0 + rows_per), c4n = g.tile_n >> 2;
#pragma unroll 1
        for (int idx = et; idx < (r1 - r0) * c4n; idx += 256) {
            const int rr = r0 + idx / c4n, c4 = idx - (rr - r0) * c4n, nc = n0 + c4 * 4;
            if (nc >= g.N) continue;
            const size_t px = (size_t)(m0 + rr);
            const float *src = g.split_part + px * g.split_ld + nc;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int sp = 0; sp < g.ksplit; ++sp) {
                const float4 x4 = __ldcg(reinterpret_cast<const float4 *>(src + (size_t)sp * g.split_stride));
                a.x += x4.x; a.y += x4.y; a.z += x4.z; a.w += x4.w;
            }
            conv_finish_store4(g, a, ld_shared_f4(bias_s + (uint32_t)nc * 4u), nc, px, conv_skip4(g, nc, px));
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (et == 0) {
            __threadfence();
            const unsigned int old = atomicAdd(cnt + 1, 1u);
            if (old == (unsigned int)(g.ksplit - 1)) { cnt[0] = 0u; cnt[1] = 0u; }      // all have read: ready for the next run
        }
    }
    return true;
}

__device__ __forceinline__ uint32_t cluster_addr(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Reduction split over a thread-block cluster: the chunks of a tile are the CTAs of one cluster (rank = chunk).  Each CTA owns
// an equal share of the tile's rows.  A CTA parks its fp32 partial sums [row][tile_n + 4] in the operand ring, which is free by
// then, and sends every other owner its rows, which are contiguous, as one bulk copy into chunk t.ks of that owner's exchange
// buffer [chunk][row of the share][tile_n + 4]; the owner adds the chunks in ascending order and stores.  (The 4 words of padding
// spread a warp's rows over the banks; "arrived" counts the bytes.)
// Measured at batch 1: through global memory and counters the exchange took 5 us, as much as the product.  As 16-byte stores to
// distributed shared memory by all threads it took 4400 to 6000 cycles for 18 KB a CTA (of which 1100 to 2700 for the release
// behind the stores) and 8900 for 57 KB.
__device__ __forceinline__ bool conv_epilogue_cluster(const ConvParams &g, uint8_t *sm, uint32_t bar, uint32_t tmem_base, uint32_t arrived) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e = warp - 4, quarter = warp & 3, half = e >> 2;
    const int row = quarter * 32 + lane, et = threadIdx.x - 128;
    const uint32_t sbase = smem_u32(sm), bias_s = sbase + g.off_bias, buf = sbase + g.off_stage;
    const ConvTile t = conv_tile(g, blockIdx.x);
    const int n0 = t.nt * g.tile_n, m0 = t.mt * g.tile_rows;
    const int live = min(kTileM, g.rows - m0), per = (live + g.ksplit - 1) / g.ksplit;
    const uint32_t pitch = (uint32_t)(g.tile_n + 4) * 4u;
    const int r0 = t.ks * per, mine = max(0, min(per, live - r0)), c4n = g.tile_n >> 2, items = mine * c4n;
    if (et == 0) mbar_arrive_expect_tx(arrived, (uint32_t)((g.ksplit - 1) * mine) * pitch);
    // this thread's first four columns of the result, and its shortcut elements, which are asked for before the exchange
    int rr = et / c4n, c4 = et - rr * c4n;
    const int step_r = 32 * kCvEpiWarps / c4n, step_c = 32 * kCvEpiWarps - step_r * c4n;
    uint2 sk = make_uint2(0u, 0u);
    if (et < items && n0 + c4 * 4 < g.N) sk = conv_skip4(g, n0 + c4 * 4, (size_t)(m0 + r0 + rr));
    const bool ok = mbar_wait(bar + 8u * (2 * kCvMaxStages), 0u);
    if (ok) {
        tc_fence_after();
        const uint32_t dst = sbase + (uint32_t)row * pitch;
#pragma unroll 1
        for (int j = half; j < g.nchunks; j += 2) {
            float v[16];
            tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + j * 16, v);
            if (row < live)
#pragma unroll
                for (int q4 = 0; q4 < 16; q4 += 4)
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(j * 16 + q4) * 4u), "f"(v[q4]), "f"(v[q4 + 1]),
                                 "f"(v[q4 + 2]), "f"(v[q4 + 3]) : "memory");
        }
        tc_fence_before();
        fence_proxy_async();
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    // warp e sends owner e its rows (also after a wait that gave up: nobody waits in vain for this CTA)
    const int theirs = min(per, live - e * per);
    if (e < g.ksplit && e != t.ks && theirs > 0 && elect_one())
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(cluster_addr(buf, (uint32_t)e) + (uint32_t)(t.ks * per) * pitch), "r"(sbase + (uint32_t)(e * per) * pitch), "r"((uint32_t)theirs * pitch),
                     "r"(cluster_addr(arrived, (uint32_t)e)) : "memory");
    __syncwarp();
    // (behind a wait that gave up, too: the other CTAs' copies are on their way into this CTA's buffer until they have arrived)
    bool seen = false;
#pragma unroll 1
    for (int i = 0; i < kSpinLimit && !seen; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0, %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(arrived), "r"(kSuspendHintNs) : "memory");
        seen = done != 0;
    }
    if (!ok || !seen) return false;
#pragma unroll 1
    for (int idx = et; idx < items; idx += 32 * kCvEpiWarps) {
        const int nc = n0 + c4 * 4;
        const size_t px = (size_t)(m0 + r0 + rr);
        int rn = rr + step_r, cn = c4 + step_c;
        if (cn >= c4n) { cn -= c4n; ++rn; }
        uint2 next = make_uint2(0u, 0u);
        if (idx + 32 * kCvEpiWarps < items && n0 + cn * 4 < g.N) next = conv_skip4(g, n0 + cn * 4, (size_t)(m0 + r0 + rn));
        if (nc < g.N) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int s = 0; s < g.ksplit; ++s) {
                const float4 x = ld_shared_f4(s == t.ks ? sbase + (uint32_t)(r0 + rr) * pitch + (uint32_t)c4 * 16u : buf + (uint32_t)(s * per + rr) * pitch + (uint32_t)c4 * 16u);
                a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
            }
            conv_finish_store4(g, a, ld_shared_f4(bias_s + (uint32_t)nc * 4u), nc, px, sk);
        }
        rr = rn; c4 = cn; sk = next;
    }
    return true;
}

template <int kEpi>
__global__ void __launch_bounds__(kCvThreads, kEpi == CE_GAP ? 1 : 2)
conv_tc_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmS, const __grid_constant__ ConvParams g) {
    extern __shared__ uint8_t smem_raw[];
    pdl_launch_dependents();
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (sbase - raw);
    const uint32_t bar = sbase + g.off_bar;
    auto accf_bar = [&](int b) { return bar + 8u * (2 * kCvMaxStages + b); };
    auto acce_bar = [&](int b) { return bar + 8u * (2 * kCvMaxStages + 2 + b); };
    auto bres_bar = [&](int q) { return bar + 8u * (2 * kCvMaxStages + 4 + q); };                       // 4
    auto skip_bar = [&](int e, int b) { return bar + 8u * (2 * kCvMaxStages + 8 + kMaxSkipSlots * e + b); };
    const uint32_t arrived = skip_bar(0, 0);      // (a split has no shortcut boxes)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + g.off_bar + 8 * (2 * kCvMaxStages + 8 + kMaxSkipSlots * kCvEpiWarps));
    volatile int *fail_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);      // [0] give-up, [1], [2] agreement of a split / average

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        // (a lane per barrier: one thread takes half a microsecond for all of them)
        constexpr int acce = 2 * kCvMaxStages + 2, first_skip = 2 * kCvMaxStages + 8, n_bars = kEpi == CE_SKIP ? first_skip + kMaxSkipSlots * kCvEpiWarps : first_skip + 1;
        for (int i = lane; i < n_bars; i += 32)
            mbar_init(bar + 8u * i, i < kCvMaxStages ? (g.b_resident ? 1u : 2u) : i == acce || i == acce + 1 ? kCvEpiWarps : 1u);
        if (lane == 0) fail_flag[0] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA0) : "memory");
        if (lane == 1) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
    if (warp == 3) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp >= 4) {
        float4 *dst = reinterpret_cast<float4 *>(sm + g.off_bias);
        for (int i = threadIdx.x - 128; i < (g.npad >> 2); i += 32 * kCvEpiWarps) dst[i] = __ldg(reinterpret_cast<const float4 *>(g.bias) + i);
    }
    tc_fence_before();
    __syncthreads();
    if (kEpi == CE_CLUSTER) cluster_sync();      // every CTA's "arrived" barrier exists
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    bool ok = true;

    const unsigned gave_up = kStatusTimeout | (((unsigned)g.launch_id & 0xfffu) << 12);
    if (warp == 0 || (warp == 3 && g.seg[0].per_stage > 1)) {
        // ---- A operand ----
        if (elect_one()) {
            ConvFill st;
            st.init(g, sbase, bar, warp ? 1 : 0);
            const int k0 = in_reg(g.seg[0].kblocks), total = in_reg(g.total);
            bool waited = false;
#pragma unroll 1
            for (int ti = blockIdx.x; ti < total && ok; ti += gridDim.x) {
                const ConvTile t = conv_tile(g, ti);
                const int m0 = conv_row0(g, t.mt);
                const int n = (int)g.d_rpi.div((uint32_t)m0), rem = m0 - n * (int)g.d_rpi.d;
                const int p = (int)g.d_q.div((uint32_t)rem), q = rem - p * (int)g.d_q.d;
                if (!waited) { pdl_wait(); waited = true; }      // (behind the first tile's divisions)
                if (t.kb0 < k0) ok = conv_load_a<0>(g, &tmA0, st, t.kb0, min(t.kb1, k0), m0, n, p, q);
                if (ok && t.kb1 > k0) ok = conv_load_a<1>(g, &tmA1, st, max(t.kb0 - k0, 0), t.kb1 - k0, m0, n, p, q);
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (1u << 8));
        }
    } else if (warp == 1) {
        // ---- MMA ----
        if (elect_one()) {
            ok = g.b_resident ? conv_mma_loop<true>(g, sbase, bar, tmem_base) : conv_mma_loop<false>(g, sbase, bar, tmem_base);
            if (!ok) atomicCAS(g.status, 0u, gave_up | (2u << 8));
        }
    } else if (warp == 2) {
        // ---- B operand ----
        if (elect_one()) {
            const uint32_t bytes = in_reg((uint32_t)g.tile_n * 128u);
            const int tile_n = in_reg(g.tile_n);
            if (g.b_resident) {
                const ConvTile t = conv_tile(g, blockIdx.x);
                for (int q = 0; q < 4; ++q) {
                    const int k0 = q * g.b_group, k1 = min(g.kblocks, k0 + g.b_group);
                    mbar_arrive_expect_tx(bres_bar(q), k1 > k0 ? (uint32_t)(k1 - k0) * bytes : 0u);
#pragma unroll 1
                    for (int kb = k0; kb < k1; ++kb) tma_load_2d(sbase + g.off_b + kb * bytes, &tmB, kb * kTileK, t.nt * tile_n, bres_bar(q));
                }
            } else {
                ConvRing st;
                st.init(g, sbase, bar);
                const int total = in_reg(g.total);
                int fresh = in_reg(g.stages);      // slots that nothing has been put in yet
#pragma unroll 1
                for (int ti = blockIdx.x; ti < total && ok; ti += gridDim.x) {
                    const ConvTile t = conv_tile(g, ti);
                    const int row = t.nt * tile_n;
#pragma unroll 1
                    for (int kb = t.kb0; kb < t.kb1; ++kb) {
                        ok = --fresh >= 0 || mbar_wait(st.empty(), st.ph ^ 1u);
                        if (!ok) break;
                        mbar_arrive_expect_tx(st.fb, bytes);
                        tma_load_2d(st.data + kABytes, &tmB, kb * kTileK, row, st.fb);
                        st.next();
                    }
                }
            }
            if (!ok) atomicCAS(g.status, 0u, gave_up | (1u << 8));
        }
    } else if (warp >= 4) {
        // ---- epilogue: warp w reads tensor-memory lanes 32 * (w % 4) .., column chunks half, half + 2, ... ----
        pdl_wait();
        const int e = warp - 4, quarter = warp & 3, half = e >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t t_warp = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t bias_s = sbase + g.off_bias;
        if (kEpi == CE_STORE || kEpi == CE_SKIP) {
            const int last_act = (kEpi == CE_SKIP) ? g.act2 : g.act;
            const uint32_t plo = last_act >= 1 ? 0u : 0xff80ff80u, phi = last_act == 2 ? 0x40c040c0u : 0x7f807f80u;
            const uint32_t stage0 = sbase + g.off_stage + (uint32_t)(g.s_slots * e) * g.box_bytes;
            const int depth = in_reg(g.s_slots);
            int i = 0, slot = 0;
            // Shortcut boxes are asked for s_slots - 1 ahead of their use: with one ahead every box cost a warp the whole latency
            // of the load.  (ati, aj): the next box to ask for.
            uint32_t sph = 0;
            int ati = half < g.nchunks ? (int)blockIdx.x : g.total, aj = half;
            auto ask_skip = [&](int to) {
                const ConvTile u = conv_tile(g, ati);
                mbar_arrive_expect_tx(skip_bar(e, to), (uint32_t)g.box_bytes);
                tma_load_2d(stage0 + (uint32_t)to * g.box_bytes, &tmS, u.nt * g.tile_n + aj * g.chunk, u.mt * g.tile_rows + quarter * 32, skip_bar(e, to));
            };
            auto advance = [&]() {
                aj += 2;
                if (aj >= g.nchunks) { aj = half; ati += (int)gridDim.x; }
            };
            if (kEpi == CE_SKIP)
                for (int d = 0; d + 1 < depth && ati < g.total; ++d, advance()) {
                    if (elect_one()) ask_skip(d);
                    __syncwarp();
                }
#pragma unroll 1
            for (int ti = blockIdx.x; ti < g.total && ok; ti += gridDim.x, ++i) {
                const ConvTile t = conv_tile(g, ti);
                const int b = i & 1, y = t.mt * g.tile_rows + quarter * 32;
                if (!mbar_wait(accf_bar(b), (i >> 1) & 1)) { ok = false; break; }
                tc_fence_after();
                const uint32_t t_acc = t_warp + b * g.acc_stride;
#pragma unroll 1
                for (int j = half; j < g.nchunks; j += 2) {
                    const uint32_t buf = stage0 + (uint32_t)slot * g.box_bytes;
                    const int x = t.nt * g.tile_n + j * g.chunk;
                    const uint32_t sb = bias_s + (uint32_t)x * 4u;
                    if (kEpi == CE_STORE) {
                        if (elect_one()) bulk_wait_read<1>();      // the store before last has left this box
                        __syncwarp();
                    } else {
                        ok = mbar_wait(skip_bar(e, slot), sph);
                        if (!ok) break;
                    }
#pragma unroll 1
                    for (int c0 = 0; c0 < g.chunk; c0 += 32) {
                        const bool wide = g.chunk - c0 >= 32;
                        float v[32];
                        if (wide) tmem_ld32(t_acc + j * g.chunk + c0, v); else tmem_ld16(t_acc + j * g.chunk + c0, v);
                        if (j + 2 >= g.nchunks && c0 + 32 >= g.chunk) {
                            tc_fence_before();
                            warp_arrive(acce_bar(b), lane);
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (h == 1 && !wide) break;
                            const int piece = (c0 >> 3) + 2 * h;
                            const uint32_t p0 = buf + box_piece(g.chunk, lane, piece), p1 = buf + box_piece(g.chunk, lane, piece + 1);
                            uint32_t pk[8];
                            if (kEpi == CE_SKIP) {
                                const uint4 s0 = ld_shared16(p0), s1 = ld_shared16(p1);
                                const uint32_t sk[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
                                conv_finish16<true>(g, v + 16 * h, sb + (uint32_t)(c0 + 16 * h) * 4u, sk, pk, plo, phi);
                            } else {
                                conv_finish16<false>(g, v + 16 * h, sb + (uint32_t)(c0 + 16 * h) * 4u, nullptr, pk, plo, phi);
                            }
                            st_shared16(p0, make_uint4(pk[0], pk[1], pk[2], pk[3]));
                            st_shared16(p1, make_uint4(pk[4], pk[5], pk[6], pk[7]));
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (elect_one()) { tma_store_2d(&tmO, buf, x, y); bulk_commit(); }
                    __syncwarp();
                    // (into the box before this one, once that one's store has left it)
                    if (kEpi == CE_SKIP && ati < g.total) {
                        if (elect_one()) { bulk_wait_read<1>(); ask_skip(slot ? slot - 1 : depth - 1); }
                        __syncwarp();
                        advance();
                    }
                    if (++slot == depth) { slot = 0; sph ^= 1u; }
                }
                if (half >= g.nchunks && ok) warp_arrive(acce_bar(b), lane);      // a warp without a chunk in so narrow a tile
            }
            if (elect_one()) bulk_wait_read<0>();
            __syncwarp();
        } else if (kEpi == CE_VEC) {
            // vectors (fp32 results, channel counts that are no multiple of 8): plain stores
            int i = 0;
#pragma unroll 1
            for (int ti = blockIdx.x; ti < g.total && ok; ti += gridDim.x, ++i) {
                const ConvTile t = conv_tile(g, ti);
                const int b = i & 1, m = t.mt * g.tile_rows + row;
                if (!mbar_wait(accf_bar(b), (i >> 1) & 1)) { ok = false; break; }
                tc_fence_after();
#pragma unroll 1
                for (int j = half; j < g.nchunks; j += 2) {
                    const int x = t.nt * g.tile_n + j * 16;
                    float v[16];
                    tmem_ld16(t_warp + b * g.acc_stride + j * 16, v);
                    conv_act16(g, v, bias_s + (uint32_t)x * 4u);
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        if (m < g.rows && x + c < g.N) {
                            if (g.out_f32) reinterpret_cast<float *>(g.out)[(size_t)m * g.out_ctot + x + c] = v[c];
                            else reinterpret_cast<__nv_bfloat16 *>(g.out)[(size_t)m * g.out_ctot + x + c] = __float2bfloat16_rn(v[c]);
                        }
                }
                tc_fence_before();
                warp_arrive(acce_bar(b), lane);
            }
        } else {
            ok = kEpi == CE_GAP ? conv_epilogue_gap(g, sm, bar, tmem_base, fail_flag)
               : kEpi == CE_CLUSTER ? conv_epilogue_cluster(g, sm, bar, tmem_base, arrived)
               : conv_epilogue_split(g, sm, bar, tmem_base, fail_flag);
        }
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (5u << 8));
    }
    tc_fence_before();
    __syncthreads();
    // (a cluster barrier does not wait for bulk copies: every CTA has seen all that was announced to it arrive, so nothing is on its
    // way into its buffer, and behind the barrier nothing out of its ring either)
    if (kEpi == CE_CLUSTER) cluster_sync();
    if (warp == 3) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols) : "memory");
    }
}

}  // namespace xk
