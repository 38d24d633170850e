// The first layer: a k x k convolution of an NCHW image with few channels (fp32 or bf16) as an implicit product on the
// 5th-generation tensor cores, alone or with a linked max pool.
//
// Eight adjacent image elements hold every tap of one window row (k <= 8), so the operand of a K chunk of 8 is, for output
// column q, the 16 bytes that start at element q * stride - pad of an image row.  These 16-byte pieces are laid out once per
// (image row, channel, q); with no swizzle the tensor core addresses 8-row groups and K chunks by two free strides, so every
// window row of every output row reads the same pieces in place: an im2col operand would be 3.5 times the shared-memory
// stores for a 7 x 7 window of stride 2.  Products (K = 16, two chunks each) pair two window rows of a channel; the last row
// of an odd window pairs two channels, and a last single chunk is paired with zeros kept behind the ring.
// A piece holds zeros outside its window: those elements meet zero weights, but an infinity or a NaN times zero would reach
// columns whose window does not hold it (the zeros cost the producers 1 us of ResNet-18's 255 at batch 32).
//
// A CTA walks down a column block of the image: image rows enter a ring of row slots (slot R repeats slot 0, so that a pair
// of rows is contiguous wherever the ring wraps), one step per two convolution rows (one where a CTA has few rows or the ring does
// not hold two steps of two).
//   warps 0..7   : epilogue: bias, activation, bf16; stores, or the running maximum of the pool's rows in registers, staged
//   warps 8..13  : image rows -> operand pieces (8..14 for seven channels)
//   warps 14, 15 : issue the products of every second step each (15 all of them for seven channels); a convolution row is one
//                  accumulator per 128 columns
//   warps 16..19 : with a pool: the maximum over columns, from the staged rows to the output
// What bounds it: instructions.  A scheduler's ALU takes two cycles for most of what the roles do, a waiting warp's polls among
// them, and an mbarrier's answer 60 to 250 cycles: with one row a step, one barrier per image row, one issuing thread and the pool's
// columns behind barriers of the whole epilogue a convolution row of 128 columns took 1650 (3 x 3) to 2300 cycles (7 x 7).  Products
// read 6 KB of shared memory each for 64 channels (48 cycles), 11 per 128 columns for a 7 x 7 window of 3 channels; at 512 x 512
// images they are half of the time.  Before and after, us in a stream of launches, batch 32, 224 x 224, bf16: 3 x 3 to 32 channels
// 21.8 -> 17.6; 7 x 7 to 64 29.1 -> 26.2, with the pool 33.0 -> 26.6; 3 x 3 to 64 with the pool 28.9 -> 24.1; 512 x 512, 7 x 7 with the
// pool, batch 64: 198 -> 150.  At batch 1 (224 x 224, pool): 7 x 7 7.95 -> 8.5, 3 x 3 6.7 -> 6.7.
// Measured and slower: 24 warps at 80 registers with 12 of producers (19.4 against 17.6) or 16 of the epilogue (29.0 against 26.6);
// waits without a time hint (17.9) or with sleeps between polls (18.0).
#pragma once

#include "conv_tc.cuh"

namespace xk {

constexpr int kStEpiWarps = 8, kStMaxProd = 7, kStColWarps = 4, kStThreads = 512;      // (and kStColWarps more with a pool)
constexpr int kStMaxSteps = 8, kStMaxSets = 4;

struct StemParams {
    const void *src;
    const uint4 *w;                 // [pair of chunks][2][tile_n] pieces of 8 weights, per channel tile
    const float *bias;
    void *out;
    unsigned int *status;
    int units;                      // (image, column block, row) triples; rows of the output or, with a pool, of the pool
    int unit_share, unit_extra;     // units of a CTA; the first unit_extra CTAs have one more
    int rows, cbs, cw;              // rows per image, column blocks, output columns per block
    FastDiv d_rows, d_cbs;
    int C, H, W, k, stride, pad, lead;      // lead: a piece starts lead elements before the window (alignment of the loads)
    int P, Q, N, tile_n, npairs;
    int R, D, spr;                  // row slots, steps in flight, convolution rows of a step
    int nsets, nsm, acc_stride;     // accumulator sets (one of a step), accumulators of a row in a set, columns of an accumulator
    int qp;                         // pieces per (slot, channel)
    int pk, ps, pp, PQ;             // max pool
    int pc_log2;                    // staged pixel: 1 << pc_log2 chunks of 16 bytes
    int act, out_ctot, out_coff;
    uint32_t idesc;
    int off_w, off_bias, off_stage, stage_bytes, stage_bufs, off_bar;
    int nprod, rstep;               // producer warps (where they are six, the seventh warp issues every second step's products), of a channel
    int raw_groups, raw_rows, raw_stride, raw_lead, off_raw;      // image rows on their way: groups per producer warp, rows of a group, bytes of a row and of the zeros in front
    int launch_id;
};
constexpr int kStMaxRaw = 4;
// barriers: operand rows of a step full / free, accumulator set full / free, staged pool row full / free, weights, (tensor memory's
// address,) groups of image rows of the producer warps
constexpr int kStAccBar = 2 * kStMaxSteps, kStStageBar = kStAccBar + 2 * kStMaxSets, kStWeightBar = kStStageBar + 4, kStRawBar = kStWeightBar + 2;
static_assert(8 * (kStRawBar + kStMaxRaw * kStMaxProd) <= 768, "barriers exceed their place");

constexpr int kStNoRow = 1 << 16;      // index of the first row of a warp that has none

struct StemRun { int n, out0, out1, row, len, p0, p1, base, width; };

// The rows of one column block of one image that start at unit u.
template <bool kPool>
__device__ __forceinline__ StemRun stem_run(const StemParams &g, int u, int u1) {
    StemRun r;
    const int blk = (int)g.d_rows.div((uint32_t)u);
    r.row = u - blk * g.rows;
    r.n = (int)g.d_cbs.div((uint32_t)blk);
    r.len = min(u1 - u, g.rows - r.row);
    r.out0 = (blk - r.n * g.cbs) * g.cw;
    r.out1 = min(r.out0 + g.cw, kPool ? g.PQ : g.Q);
    if (kPool) {
        r.p0 = max(0, r.row * g.ps - g.pp);
        r.p1 = min(g.P, (r.row + r.len - 1) * g.ps - g.pp + g.pk);
        r.base = max(0, r.out0 * g.ps - g.pp) & ~1;
        r.width = min(g.Q, (r.out1 - 1) * g.ps - g.pp + g.pk) - r.base;
    } else {
        r.p0 = r.row; r.p1 = r.row + r.len;
        r.base = r.out0; r.width = r.out1 - r.out0;
    }
    return r;
}

// ---- image rows -> operand pieces ----------------------------------------------------------------------------------
// A lane makes the pieces of `run` adjacent columns from the elements they share; a warp makes a whole row of one channel in up
// to four passes of 32 lanes.  The loads of a warp's next row are on the way while it signals this one and waits for room.
// SM_ANY: any stride, one column; SM_S1: stride 1; SM_S2: stride 2, rows and pieces on whole groups of 4 elements; SM_S2X:
// stride 2 otherwise (row lengths that are no multiple of 4).  All but SM_S2 load element by element.
enum { SM_ANY = 0, SM_S1 = 1, SM_S2 = 2, SM_S2X = 3 };
template <int kMode, bool kF32>
struct StemForm {
    static constexpr bool vec = kMode == SM_S2;
    static constexpr int S = kMode == SM_ANY ? 0 : kMode == SM_S1 ? 1 : 2;
    static constexpr int run = kMode == SM_ANY ? 1 : 2;
    static constexpr int words = vec && !kF32 ? 5 : 10;       // registers of a lane's elements
    static constexpr int elems = kMode == SM_ANY ? 8 : kMode == SM_S1 ? 9 : 10;
};

// Loads of the image, zero where the predicate is false.
__device__ __forceinline__ void stem_ld4(uint32_t *r, const uint8_t *s, bool p) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
                 "@p ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "l"(s), "r"((int)p));
}
__device__ __forceinline__ void stem_ld2(uint32_t *r, const uint8_t *s, bool p) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\t@p ld.global.nc.v2.b32 {%0, %1}, [%2];\n\t}"
                 : "=r"(r[0]), "=r"(r[1]) : "l"(s), "r"((int)p));
}
__device__ __forceinline__ void stem_ld1(uint32_t *r, const uint8_t *s, bool p) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.b32 %0, [%1];\n\t}" : "=r"(r[0]) : "l"(s), "r"((int)p));
}
__device__ __forceinline__ void stem_ldh(uint32_t *r, const uint8_t *s, bool p) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.u16 %0, [%1];\n\t}" : "=r"(r[0]) : "l"(s), "r"((int)p));
}

__device__ __forceinline__ void st_shared16_if(uint32_t dst, const uint4 &v, bool p) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t@p st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((int)p) : "memory");
}
// The states of two barriers' phases, asked for together (bit 0 and bit 1): one answer takes some 250 cycles here, two as long.
__device__ __forceinline__ uint32_t mbar_test2(uint32_t bar0, uint32_t ph0, uint32_t bar1, uint32_t ph1) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b32 x, y;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 q, [%3], %4;\n\t"
        "selp.u32 x, 1, 0, p;\n\tselp.u32 y, 2, 0, q;\n\tor.b32 %0, x, y;\n\t}"
        : "=r"(done) : "r"(bar0), "r"(ph0), "r"(bar1), "r"(ph1) : "memory");
    return done;
}

// A row's elements to registers: s and e are this lane's first element's address and column, W the row length (0 for a row
// outside the image: zeros).
template <int kMode, bool kF32>
__device__ __forceinline__ void stem_load(uint32_t (&raw)[4][StemForm<kMode, kF32>::words], const uint8_t *s, int e, int W, int passes, int stride) {
    using F = StemForm<kMode, kF32>;
    const int S = F::S ? F::S : stride;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i >= passes) break;
        const int de = 32 * F::run * S * i;
        const uint8_t *a = s + de * (kF32 ? 4 : 2);
        auto in = [&](int j) { return (unsigned)(e + de + j) < (unsigned)W; };
        uint32_t *r = raw[i];
        if (kMode == SM_S2 && kF32) {
            stem_ld4(r, a, in(0));
            stem_ld4(r + 4, a + 16, in(4));
            stem_ld2(r + F::words - 2, a + 32, in(8));
        } else if (kMode == SM_S2) {
            stem_ld2(r, a, in(0));
            stem_ld2(r + 2, a + 8, in(4));
            stem_ld1(r + 4, a + 16, in(8));
        } else {
            r[F::words - 1] = 0u;
            r[F::words - 2] = 0u;
#pragma unroll
            for (int j = 0; j < F::elems; ++j) {
                if (kF32) stem_ld1(r + j % F::words, a + 4 * j, in(j));
                else stem_ldh(r + j % F::words, a + 2 * j, in(j));
            }
        }
    }
}

// ... and from there to the ring: dst is this lane's first piece, again the distance of a repetition (0: none), left the lanes'
// worth of the row from this lane on, in_window the elements of a piece that belong to its window.
template <int kMode, bool kF32, int kPasses>
__device__ __forceinline__ void stem_store(const uint32_t (&raw)[kPasses][StemForm<kMode, kF32>::words], uint32_t dst, uint32_t again, int left, int passes, int lane,
                                           const uint4 &in_window) {
    using F = StemForm<kMode, kF32>;
    // eight lanes store 128 bytes apart in pairs: every second group of four lanes stores its second piece first, so that the
    // eight pieces of a store meet eight different groups of banks
    const uint32_t f = (uint32_t)(lane >> 2) & 1u, d0 = dst + f * 16u, d1 = dst + (f ^ 1u) * 16u;
#pragma unroll
    for (int i = 0; i < kPasses; ++i) {
        if (i >= passes) break;
        const uint32_t *r = raw[i];
        uint32_t w[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            if (2 * j >= F::elems) w[j] = 0u;
            else if (F::words == 5) w[j] = r[j];
            else if (kF32) w[j] = pack2(__uint_as_float(r[2 * j % F::words]), __uint_as_float(r[(2 * j + 1) % F::words]));
            else w[j] = r[2 * j % F::words] | (r[(2 * j + 1) % F::words] << 16);
        }
        const uint32_t step = (uint32_t)(32 * F::run * 16 * i);
        auto piece = [&](uint32_t x, uint32_t y, uint32_t z, uint32_t u) {
            return make_uint4(x & in_window.x, y & in_window.y, z & in_window.z, u & in_window.w);
        };
        const uint4 a = piece(w[0], w[1], w[2], w[3]);
        const bool live = 32 * i < left;
        {
            if (F::run == 1) {
                st_shared16_if(dst + step, a, live);
                if (again) st_shared16_if(dst + again + step, a, live);
            } else {
                const uint4 b = F::S == 2 ? piece(w[1], w[2], w[3], w[4])
                                          : piece(__funnelshift_r(w[0], w[1], 16), __funnelshift_r(w[1], w[2], 16),
                                                  __funnelshift_r(w[2], w[3], 16), __funnelshift_r(w[3], w[4], 16));
                const uint4 x = f ? b : a, y = f ? a : b;
                st_shared16_if(d0 + step, x, live);
                st_shared16_if(d1 + step, y, live);
                if (again) { st_shared16_if(d0 + again + step, x, live); st_shared16_if(d1 + again + step, y, live); }
            }
        }
    }
}

// The slots of another run's first rows lie anywhere in the ring: all earlier steps have been multiplied.  Two threads issue them, and a
// commit covers the products of its own thread only: the last step is behind the barrier before this one's, and the step before it,
// the other thread's last, behind the one before that.
__device__ __forceinline__ bool stem_drained(uint32_t bar, int t, int sl, int D, uint32_t ph) {
    const int s1 = sl > 0 ? sl - 1 : D - 1, s2 = sl > 1 ? sl - 2 : sl + D - 2;
    if (!mbar_wait(bar + 8u * (kStMaxSteps + s1), sl > 0 ? ph : ph ^ 1u)) return false;
    return t < 2 || mbar_wait(bar + 8u * (kStMaxSteps + s2), sl > 1 ? ph : ph ^ 1u);
}

// A producer warp: one channel, every rstep-th new row of a step (three channels: two rows each of a step of two convolution rows
// of stride 2).
template <int kMode, bool kF32, bool kPool>
__device__ __forceinline__ bool stem_produce(const StemParams &g, uint32_t sbase, uint32_t bar, int u0, int u1, int w, int lane) {
    using F = StemForm<kMode, kF32>;
    constexpr int es = kF32 ? 4 : 2;
    const int C = in_reg(g.C), k = in_reg(g.k), stride = F::S ? F::S : in_reg(g.stride), R = in_reg(g.R), D = in_reg(g.D), W = in_reg(g.W), H = in_reg(g.H);
    const int pad = in_reg(g.pad), spr = in_reg(g.spr), rstep = in_reg(g.rstep), nr = min(stride, k);
    int j0 = 0, c = w;
    for (; c >= C; c -= C) ++j0;
    if (j0 >= rstep) j0 = kStNoRow;                       // a warp without rows only keeps the steps' counts
    const uint32_t slot_bytes = in_reg((uint32_t)(g.qp * C * 16)), ring = in_reg(sbase + (uint32_t)((c * g.qp + F::run * lane) * 16)), wrap = (uint32_t)R * slot_bytes;
    const uint32_t pitch = in_reg((uint32_t)(W * es));
    auto both = [&](int j) {                              // which of elements j, j + 1 of a piece the window takes
        const uint32_t x = (unsigned)(j - g.lead) < (unsigned)k, y = (unsigned)(j + 1 - g.lead) < (unsigned)k;
        return in_reg(x * 0xffffu | y * 0xffff0000u);
    };
    const uint4 in_window = make_uint4(both(0), both(2), both(4), both(6));
    uint32_t raw[4][F::words];
    int t = 0, sl = 0, slot = 0;                          // step, its barrier, ring slot of its window row 0
    uint32_t ph = 0;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len;
        const int e = (r.base + F::run * lane) * stride - pad - g.lead;
        const uint8_t *col = reinterpret_cast<const uint8_t *>(g.src) + ((long long)(r.n * C + c) * H * W + e) * es;
        const int lanes = (r.width + F::run - 1) / F::run, passes = (lanes + 31) >> 5, left = lanes - lane;
        auto load = [&](int ih) {
            stem_load<kMode, kF32>(raw, col + (long long)ih * (long long)pitch, e, (unsigned)ih < (unsigned)H ? W : 0, passes, stride);
        };
        // (the slots of a step's rows are free when the step D before it has been multiplied)
        uint32_t room = bar + 8u * (kStMaxSteps + sl), room_ph = ph ^ 1u;
        int p = r.p0, d = j0, ih0 = p * stride - pad, nb = min(spr, r.p1 - p), kk = k + (nb - 1) * nr;
        bool start = true, fresh = true, have = false;
#pragma unroll 1
        for (;;) {
            if (!start) {
                if (fresh) {
                    if (!(p == r.p0 && t > 0 ? stem_drained(bar, t, sl, D, ph) : mbar_wait(room, room_ph))) return false;
                    fresh = false;
                }
                if (have) {
                    int s = slot + d;
                    if (s >= R) s -= R;
                    stem_store<kMode, kF32, 4>(raw, ring + (uint32_t)s * slot_bytes, s == 0 ? wrap : 0u, left, passes, lane, in_window);
                    d += rstep;
                }
                if (d >= kk) {
                    fence_proxy_async();
                    warp_arrive(bar + 8u * sl, lane);
                    if (++sl == D) { sl = 0; ph ^= 1u; }
                    ++t;
                    p += nb;
                    slot += p == r.p1 ? kk : nb * nr;
                    if (slot >= R) slot -= R;
                    if (p == r.p1) break;
                    room = bar + 8u * (kStMaxSteps + sl); room_ph = ph ^ 1u;
                    fresh = true;
                    ih0 += nb * stride;
                    nb = min(spr, r.p1 - p); kk = k + (nb - 1) * nr;
                    d = k - nr + j0;
                }
            }
            start = false;
            have = d < kk;
            if (have) load(ih0 + d);
        }
    }
    return true;
}

// The rows of a producer warp in the order it makes them, a group of at most raw_rows (rstep apart, of one step) at a time.
template <bool kPool>
struct StemCursor {
    int u, n, p, p1, nb, d, ih0;
    bool more;
    __device__ __forceinline__ void run(const StemParams &g, int u1, int j0, int stride, int pad, int spr) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len; n = r.n; p = r.p0; p1 = r.p1; nb = min(spr, p1 - p); d = j0; ih0 = p * stride - pad;
    }
    // to the step that holds the next group, if this one has no more
    __device__ __forceinline__ void settle(const StemParams &g, int u1, int j0, int k, int nr, int stride, int pad, int spr) {
        while (d >= k + (nb - 1) * nr) {
            p += nb; ih0 += nb * stride;
            if (p < p1) { nb = min(spr, p1 - p); d = k - nr + j0; }
            else if (u < u1) run(g, u1, j0, stride, pad, spr);
            else { more = false; return; }
        }
    }
};

// The same where rows are whole 16-byte pieces of memory: a warp keeps raw_groups groups of its rows on their way by bulk copies
// and reads them from shared memory, between zeros for the padding (a row outside the image is a slot of zeros).  With the loads of
// one row ahead in registers every step cost the latency of a load from memory, 1000 to 1900 cycles.  A group has one barrier: with
// one per row a step of two rows took 500 cycles more for their answers.
template <int kMode, bool kF32, int kPasses>
__device__ __forceinline__ void stem_read(uint32_t (&raw)[kPasses][StemForm<kMode, kF32>::words], uint32_t s, int stride) {
    using F = StemForm<kMode, kF32>;
    constexpr int es = kF32 ? 4 : 2;
    const int S = F::S ? F::S : stride;
#pragma unroll
    for (int i = 0; i < kPasses; ++i) {
        const uint32_t a = s + (uint32_t)(32 * F::run * S * i * es);
        uint32_t *r = raw[i];
        auto ld2 = [](uint32_t *d, uint32_t at) { asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(d[0]), "=r"(d[1]) : "r"(at)); };
        if (kMode == SM_S2 && kF32) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[4 * j]), "=r"(r[4 * j + 1]), "=r"(r[4 * j + 2]), "=r"(r[4 * j + 3]) : "r"(a + 16u * j));
            ld2(r + F::words - 2, a + 32u);
        } else if (kMode == SM_S2) {
            ld2(r, a);
            ld2(r + 2, a + 8u);
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(r[4]) : "r"(a + 16u));
        } else {
            r[F::words - 1] = 0u;
            r[F::words - 2] = 0u;
#pragma unroll
            for (int j = 0; j < F::elems; ++j) {
                if (kF32) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(r[j % F::words]) : "r"(a + 4u * j));
                else {
                    unsigned short h;
                    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(a + 2u * j));
                    r[j % F::words] = h;
                }
            }
        }
    }
}
template <int kMode, bool kF32, bool kPool>
__device__ __forceinline__ bool stem_produce_rows(const StemParams &g, uint32_t sbase, uint32_t bar, int u0, int u1, int w, int lane) {
    using F = StemForm<kMode, kF32>;
    constexpr int es = kF32 ? 4 : 2;
    const int C = in_reg(g.C), k = in_reg(g.k), stride = F::S ? F::S : in_reg(g.stride), R = in_reg(g.R), D = in_reg(g.D), H = in_reg(g.H);
    const int pad = in_reg(g.pad), spr = in_reg(g.spr), rstep = in_reg(g.rstep), nr = min(stride, k);
    int j0 = 0, c = w;
    for (; c >= C; c -= C) ++j0;
    if (j0 >= rstep) j0 = kStNoRow;                       // a warp without rows only keeps the steps' counts
    const uint32_t slot_bytes = in_reg((uint32_t)(g.qp * C * 16)), ring = in_reg(sbase + (uint32_t)((c * g.qp + F::run * lane) * 16)), wrap = (uint32_t)R * slot_bytes;
    const uint32_t row_bytes = in_reg((uint32_t)(g.W * es)), raw_stride = in_reg((uint32_t)g.raw_stride), lead = (uint32_t)g.raw_lead;
    const uint32_t zeros = sbase + (uint32_t)g.off_raw + lead;                                    // slot 0 of the region: a row of zeros
    const int rows = in_reg(g.raw_rows);
    const uint32_t group_bytes = raw_stride * (uint32_t)rows;
    const uint32_t mine = zeros + raw_stride + group_bytes * (uint32_t)(w * g.raw_groups), mine_end = mine + group_bytes * (uint32_t)g.raw_groups;
    const uint32_t bar0 = bar + 8u * (uint32_t)(kStRawBar + kStMaxRaw * w);
    auto both = [&](int j) {                              // which of elements j, j + 1 of a piece the window takes
        const uint32_t x = (unsigned)(j - g.lead) < (unsigned)k, y = (unsigned)(j + 1 - g.lead) < (unsigned)k;
        return in_reg(x * 0xffffu | y * 0xffff0000u);
    };
    const uint4 in_window = make_uint4(both(0), both(2), both(4), both(6));
    // The groups' barriers and slots are this warp's own: it asks for the first rows while the rest of the CTA is being set up
    // (asks and set-up take some 2000 cycles each).  Zeros for the padding of its slots; rows outside the image are read from the
    // region's first slot.
    if (lane < g.raw_groups) mbar_init(bar0 + 8u * (uint32_t)lane, 1);
    for (uint32_t at = mine - lead; at < mine_end - lead; at += raw_stride)
        for (uint32_t i = 16u * (uint32_t)lane; i < raw_stride - row_bytes; i += 512u) st_shared16(at + i + (i < lead ? 0u : row_bytes), make_uint4(0u, 0u, 0u, 0u));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    __syncwarp();
    pdl_wait();
    StemCursor<kPool> ahead;
    ahead.u = u0; ahead.more = u0 < u1 && j0 < rstep;
    if (ahead.more) {
        ahead.run(g, u1, j0, stride, pad, spr);
        ahead.settle(g, u1, j0, k, nr, stride, pad, spr);
    }
    uint32_t raw_at = mine, raw_bar = bar0, raw_ph = 0u;      // the group that is read next; it is filled again behind the read
    // The next group's rows into its slots.  Behind the first step of a run groups lie a step apart: `again` of them follow without
    // another look at the walk (which made the request 700 cycles).
    const uint32_t step_bytes = (uint32_t)(spr * stride) * row_bytes, apart_bytes = (uint32_t)rstep * row_bytes;
    const uint8_t *src = nullptr;
    int again = 0, count = 0;
    // (lane i asks for row i of the group)
    const uint32_t lane_at = (uint32_t)lane * raw_stride;
    const long long lane_src = (long long)lane * (long long)apart_bytes;
    auto copy = [&](uint32_t at, uint32_t b, bool have) {
        if (have)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(at + lane_at), "l"(src + lane_src), "r"(row_bytes), "r"(b) : "memory");
    };
    auto ask = [&](uint32_t at, uint32_t b) {
        if (again > 0) {
            --again;
            src += step_bytes;
            if (lane == 0) mbar_arrive_expect_tx(b, row_bytes * (uint32_t)count);
            __syncwarp();
            copy(at, b, lane < count);
            return;
        }
        if (!ahead.more) return;
        const int ih = ahead.ih0 + ahead.d;
        src = reinterpret_cast<const uint8_t *>(g.src) + ((long long)(ahead.n * C + c) * H + ih) * (long long)row_bytes;
        const bool row = lane < rows && ahead.d + lane * rstep < k + (ahead.nb - 1) * nr, have = row && (unsigned)(ih + lane * rstep) < (unsigned)H;
        count = __popc(__ballot_sync(0xffffffffu, row));
        const uint32_t n = (uint32_t)__popc(__ballot_sync(0xffffffffu, have));
        if (lane == 0) {
            if (n) mbar_arrive_expect_tx(b, row_bytes * n);
            else mbar_arrive(b);
        }
        __syncwarp();
        copy(at, b, have);
        if (ahead.d == k - nr + j0 && ahead.nb == spr && ih >= 0) {
            // (the whole steps that follow in the run, as far as their rows lie in the image)
            const int two = spr == 2 ? 1 : 0, most = max(0, H - 1 - (ih + (count - 1) * rstep)) >> (two + (F::S == 2 ? 1 : 0));
            again = max(0, min(((ahead.p1 - ahead.p) >> two) - 1, most));
            ahead.p += again * spr; ahead.ih0 += again * spr * stride;
        }
        ahead.d += rows * rstep;
        ahead.settle(g, u1, j0, k, nr, stride, pad, spr);
    };
    for (int i = 0; i < g.raw_groups; ++i) ask(mine + group_bytes * (uint32_t)i, bar0 + 8u * i);
    asm volatile("bar.sync 0;" ::: "memory");             // the CTA is set up
    int t = 0, sl = 0, slot = 0;                          // step, its barrier, ring slot of its window row 0
    uint32_t ph = 0;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len;
        const int e = ((r.base + F::run * lane) * stride - pad - g.lead) * es;
        const int lanes = (r.width + F::run - 1) / F::run, passes = (lanes + 31) >> 5, left = lanes - lane;
        int d = j0, ih0 = r.p0 * stride - pad, nb;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; p += nb, ih0 += nb * stride) {
            nb = min(spr, r.p1 - p);
            const int kk = k + (nb - 1) * nr;
            // (the slots of a step's rows are free when the step D before it has been multiplied)
            const bool first = p == r.p0 && t > 0;
            const uint32_t room = bar + 8u * (kStMaxSteps + sl), room_ph = ph ^ 1u;
            const uint32_t known = mbar_test2(room, room_ph, raw_bar, raw_ph);
            bool here = (known & 2u) != 0;
            if (first ? !stem_drained(bar, t, sl, D, ph) : !(known & 1u) && t >= D && !mbar_wait(room, room_ph)) return false;
#pragma unroll 1
            while (d < kk) {
                if (!here && !mbar_wait(raw_bar, raw_ph)) return false;
                here = false;
                uint32_t at = raw_at + (uint32_t)e;
                const int end = min(d + rows * rstep, kk);
#pragma unroll 1
                for (; d < end; d += rstep, at += raw_stride) {
                    const uint32_t from = (unsigned)(ih0 + d) < (unsigned)H ? at : zeros + (uint32_t)e;
                    int s = slot + d;
                    if (s >= R) s -= R;
                    const uint32_t dst = ring + (uint32_t)s * slot_bytes, twice = s == 0 ? wrap : 0u;
#pragma unroll 1
                    for (int i = 0; i < passes; i += 2) {
                        const uint32_t f = from + (uint32_t)(32 * F::run * stride * es * i), t = dst + (uint32_t)(32 * F::run * 16 * i);
                        if (i + 1 < passes) {
                            uint32_t raw[2][F::words];
                            stem_read<kMode, kF32, 2>(raw, f, stride);
                            stem_store<kMode, kF32, 2>(raw, t, twice, left - 32 * i, 2, lane, in_window);
                        } else {
                            uint32_t raw[1][F::words];
                            stem_read<kMode, kF32, 1>(raw, f, stride);
                            stem_store<kMode, kF32, 1>(raw, t, twice, left - 32 * i, 1, lane, in_window);
                        }
                    }
                }
                d = end;
                __syncwarp();
                ask(raw_at, raw_bar);
                raw_at += group_bytes; raw_bar += 8u;
                if (raw_at == mine_end) { raw_at = mine; raw_bar = bar0; raw_ph ^= 1u; }
            }
            fence_proxy_async();
            warp_arrive(bar + 8u * sl, lane);
            if (++sl == D) { sl = 0; ph ^= 1u; }
            ++t;
            slot += p + nb == r.p1 ? kk : nb * nr;
            if (slot >= R) slot -= R;
            d = k - nr + j0;
        }
    }
    return true;
}

// ---- products --------------------------------------------------------------------------------------------------------
// One to four products (the first always) of operands a_lo, a_lo + a1, + a2, + a3 and of weights `bs` apart.
__device__ __forceinline__ void stem_products(uint32_t d_tmem, uint32_t hi, uint32_t a_lo, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b_lo, uint32_t bs,
                                              uint32_t idesc, uint32_t acc, int n) {
    asm volatile(
        "{\n\t.reg .pred p, s1, s2, s3;\n\t.reg .b64 da, db;\n\t.reg .b32 x, y;\n\t"
        "setp.ne.b32 p, %8, 0;\n\tsetp.gt.s32 s1, %9, 1;\n\tsetp.gt.s32 s2, %9, 2;\n\tsetp.gt.s32 s3, %9, 3;\n\t"
        "mov.b64 da, {%2, %1};\n\tmov.b64 db, {%6, %1};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %10, p;\n\t"
        "setp.eq.u32 p, 0, 0;\n\t"
        "add.u32 x, %2, %3;\n\tadd.u32 y, %6, %7;\n\tmov.b64 da, {x, %1};\n\tmov.b64 db, {y, %1};\n\t"
        "@s1 tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %10, p;\n\t"
        "add.u32 x, %2, %4;\n\tadd.u32 y, y, %7;\n\tmov.b64 da, {x, %1};\n\tmov.b64 db, {y, %1};\n\t"
        "@s2 tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %10, p;\n\t"
        "add.u32 x, %2, %5;\n\tadd.u32 y, y, %7;\n\tmov.b64 da, {x, %1};\n\tmov.b64 db, {y, %1};\n\t"
        "@s3 tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %10, p;\n\t}"
        ::"r"(d_tmem), "r"(hi), "r"(a_lo), "r"(a1), "r"(a2), "r"(a3), "r"(b_lo), "r"(bs), "r"(acc), "r"(n), "r"(idesc) : "memory");
}
// One thread, for every `turn`-th step from step `which` on.  A convolution row of a step is ns accumulators of npairs products each.
template <bool kPool>
__device__ __forceinline__ bool stem_mma(const StemParams &g, uint32_t sbase, uint32_t bar, uint32_t tmem_base, int u0, int u1, int which, int turn) {
    const uint32_t hi = (128u >> 4) | (1u << 14);      // 8-row groups 128 bytes apart, descriptor version, no swizzle
    const uint32_t idesc = in_reg(g.idesc);
    const int C = in_reg(g.C), k = in_reg(g.k), R = in_reg(g.R), D = in_reg(g.D), spr = in_reg(g.spr), nsets = in_reg(g.nsets);
    const uint32_t ring16 = in_reg(sbase >> 4), cp16 = in_reg((uint32_t)g.qp), rp16 = in_reg((uint32_t)(g.qp * g.C));
    const uint32_t w16 = in_reg(((sbase + (uint32_t)g.off_w) >> 4) | ((uint32_t)g.tile_n << 16)), wstep = in_reg(2u * (uint32_t)g.tile_n);
    const uint32_t zeros16 = ring16 + (uint32_t)(R + 1) * rp16, accf = bar + 8u * kStAccBar, acce = accf + 8u * kStMaxSets;
    const uint32_t acc_cols = in_reg((uint32_t)g.acc_stride), row_cols = (uint32_t)g.nsm * acc_cols, set_cols = (uint32_t)spr * row_cols;
    const int nr = min(g.stride, g.k), odd = C >> 1;
    int slot0 = 0, sl = 0, a = 0, mine = which;
    uint32_t ph = 0, pa = 0;
    if (!mbar_wait(bar + 8u * kStWeightBar, 0)) return false;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len;
        const int ns = (r.width + kTileM - 1) / kTileM;
        int nb;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; p += nb) {
            nb = min(spr, r.p1 - p);
            int s0 = slot0;
            slot0 += p + nb == r.p1 ? k + (nb - 1) * nr : nb * nr;
            if (slot0 >= R) slot0 -= R;
            const uint32_t rows = bar + 8u * sl, room = rows + 8u * kStMaxSteps, done = accf + 8u * a, freed = acce + 8u * a, rows_ph = ph, freed_ph = pa ^ 1u;
            uint32_t d = tmem_base + (uint32_t)a * set_cols;
            if (++sl == D) { sl = 0; ph ^= 1u; }
            if (++a == nsets) { a = 0; pa ^= 1u; }
            if (--mine >= 0) continue;
            mine = turn - 1;
            const uint32_t known = mbar_test2(rows, rows_ph, freed, freed_ph);
            if (!(known & 1u) && !mbar_wait(rows, rows_ph)) return false;
            if (!(known & 2u) && !mbar_wait(freed, freed_ph)) return false;
            tc_fence_after();
#pragma unroll 1
            for (int j = 0; j < nb; ++j, d += row_cols) {
#pragma unroll 1
                for (int seg = 0; seg < ns; ++seg) {
                    const uint32_t ds = d + (uint32_t)seg * acc_cols, rows16 = ring16 + (uint32_t)seg * 128u;
                    uint32_t acc = 0, bl = w16;
                    int s = s0;
#pragma unroll 1
                    for (int i = 0; i < (k >> 1); ++i) {
                        uint32_t al = (rows16 + (uint32_t)s * rp16) | (rp16 << 16);
#pragma unroll 1
                        for (int c = 0; c < C; c += 4, al += 4 * cp16) {
                            stem_products(ds, hi, al, cp16, 2 * cp16, 3 * cp16, bl, wstep, idesc, acc, C - c);
                            acc = 1u;
                            bl += (uint32_t)min(4, C - c) * wstep;
                        }
                        s += 2;
                        if (s >= R) s -= R;
                    }
                    if (k & 1) {
                        // pairs of channels; a last single channel's chunk before the zeros behind the ring
                        const uint32_t first = rows16 + (uint32_t)s * rp16, al = first | (cp16 << 16), last = first + (uint32_t)(C - 1) * cp16;
                        const uint32_t single = (last | ((zeros16 - last) << 16)) - al;
                        stem_products(ds, hi, C == 1 ? al + single : al, odd == 1 ? single : 2 * cp16, odd == 2 ? single : 4 * cp16, single, bl, wstep, idesc, acc, odd + (C & 1));
                    }
                }
                s0 += nr;
                if (s0 >= R) s0 -= R;
            }
            umma_commit(done);
            umma_commit(room);
        }
    }
    return true;
}

// 16 columns of an accumulator: bias, bf16 pairs, activation.  (Maximum with zero, not the conversion's own clamp, which keeps
// a NaN: max(x, 0) is 0 there, as in every other kernel.)
__device__ __forceinline__ void stem_pack(const float *v, const float2 (&bias)[8], int act, uint32_t (&o)[8]) {
    float2 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = __fadd2_rn(make_float2(v[2 * i], v[2 * i + 1]), bias[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = pack2(x[i].x, x[i].y);
    if (act == 2) {
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = clamp_bf16x2(o[i], 0u, 0x40c040c0u);
    } else if (act) {
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = max_bf16x2(o[i], 0u);
    }
}
__device__ __forceinline__ void stem_bias(const float *at, float2 (&b)[8]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(at) + i);
        b[2 * i] = make_float2(v.x, v.y); b[2 * i + 1] = make_float2(v.z, v.w);
    }
}
// kCh chunks of an accumulator row (a warp with fewer reads columns that nobody stores: they lie inside the allocation).
template <int kCh>
__device__ __forceinline__ void stem_tmem(uint32_t at, float *v) {
    if constexpr (kCh == 2) tmem_ld32(at, v);
    else tmem_ld16(at, v);
}

// What a warp of the epilogue keeps: a quarter of the accumulator's lanes, chn (kCh at most) 16-column chunks of it from ch0 on.
struct StemEpi {
    int lane, px, ch0, chn, n0, live, nsets, spr, act, a;
    uint32_t accf, acce, taddr, pa, acc_cols, row_cols, set_cols;
    __device__ __forceinline__ void init(const StemParams &g, uint32_t bar, uint32_t tmem_base) {
        const int warp = threadIdx.x >> 5, quarter = warp & 3, half = warp >> 2, nch = g.tile_n >> 4;
        lane = threadIdx.x & 31; px = quarter * 32 + lane;
        ch0 = half ? (nch + 1) >> 1 : 0; chn = half ? nch >> 1 : (nch + 1) >> 1;
        n0 = blockIdx.y * g.tile_n; live = min(g.tile_n, g.N - n0);
        nsets = in_reg(g.nsets); spr = in_reg(g.spr); act = in_reg(g.act);
        acc_cols = in_reg((uint32_t)g.acc_stride); row_cols = (uint32_t)g.nsm * acc_cols; set_cols = (uint32_t)spr * row_cols;
        accf = bar + 8u * kStAccBar; acce = accf + 8u * kStMaxSets;
        taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)ch0 * 16u;
        a = 0; pa = 0;
    }
    __device__ __forceinline__ bool full() const { return mbar_test(accf + 8u * a, pa) || mbar_wait(accf + 8u * a, pa); }
    // Behind the last read of the set.
    __device__ __forceinline__ void read() const {
        tc_fence_before();
        warp_arrive(acce + 8u * a, lane);
    }
    __device__ __forceinline__ void next() {
        if (++a == nsets) { a = 0; pa ^= 1u; }
    }
};

template <int kCh>
__device__ __forceinline__ bool stem_epilogue_store(const StemParams &g, uint32_t bar, uint32_t tmem_base, int u0, int u1) {
    StemEpi s;
    s.init(g, bar, tmem_base);
    float2 bias[kCh][8];
#pragma unroll
    for (int h = 0; h < kCh; ++h)
        if (h < s.chn) stem_bias(g.bias + s.n0 + (s.ch0 + h) * 16, bias[h]);
    // 32-byte stores where every chunk is whole and aligned
    const bool wide = ((g.out_ctot | g.out_coff | s.live) & 15) == 0;
    const int ctot = in_reg(g.out_ctot), Q = in_reg(g.Q);
    __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(g.out) + g.out_coff + s.n0 + s.ch0 * 16;
    const size_t row_step = (size_t)Q * ctot, seg_step = (size_t)kTileM * ctot;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<false>(g, u, u1);
        u += r.len;
        __nv_bfloat16 *row = out + (((size_t)r.n * g.P + r.p0) * Q + r.base + s.px) * ctot;
        int nb;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; p += nb) {
            nb = min(s.spr, r.p1 - p);
            if (!s.full()) return false;
            tc_fence_after();
            uint32_t t_row = s.taddr + (uint32_t)s.a * s.set_cols;
#pragma unroll 1
            for (int j = 0; j < nb; ++j, t_row += s.row_cols, row += row_step) {
                __nv_bfloat16 *d = row;
                uint32_t ta = t_row;
#pragma unroll 1
                for (int q = s.px; q - s.px < r.width; q += kTileM, d += seg_step, ta += s.acc_cols) {
                    float v[16 * kCh];
                    stem_tmem<kCh>(ta, v);
                    if (j + 1 == nb && q - s.px + kTileM >= r.width) s.read();
#pragma unroll
                    for (int h = 0; h < kCh; ++h) {
                        uint32_t o[8];
                        stem_pack(v + 16 * h, bias[h], s.act, o);
                        if (q >= r.width || h >= s.chn) continue;
                        if (wide) {
                            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d + 16 * h), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                                         "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]) : "memory");
                        } else {
                            const int nc = (s.ch0 + h) * 16;
                            if (nc + 8 <= s.live) *reinterpret_cast<uint4 *>(d + 16 * h) = make_uint4(o[0], o[1], o[2], o[3]);
                            if (nc + 16 <= s.live) *reinterpret_cast<uint4 *>(d + 16 * h + 8) = make_uint4(o[4], o[5], o[6], o[7]);
                        }
                    }
                }
            }
            s.next();
        }
    }
    return true;
}

// The pool's maximum over rows stays in registers: a lane keeps its column, or one of either segment.  A finished row is staged;
// other warps take the maximum over columns from there (stem_columns), while the next rows are read here.  (With both in the same
// warps, between barriers of the whole epilogue, a row of ResNet-18's pool took 3700 cycles; products and rows are there in 2000.)
template <int kSegs, int kCh>
__device__ __forceinline__ bool stem_epilogue_pool(const StemParams &g, uint32_t sbase, uint32_t bar, uint32_t tmem_base, int u0, int u1) {
    StemEpi s;
    s.init(g, bar, tmem_base);
    const uint32_t bias_at = sbase + (uint32_t)g.off_bias + 128u * (threadIdx.x >> 5);      // this warp's 32 values
    if (s.lane < 16 * s.chn) asm volatile("st.shared.f32 [%0], %1;" ::"r"(bias_at + 4u * (uint32_t)s.lane), "f"(__ldg(g.bias + s.n0 + s.ch0 * 16 + s.lane)) : "memory");
    __syncwarp();
    // (a maximum that starts at zero is ReLU's, too)
    const uint32_t none = in_reg(s.act ? 0u : 0xff80ff80u);
    const int act = s.act == 1 ? 0 : s.act, pk = in_reg(g.pk), ps = in_reg(g.ps), pp = in_reg(g.pp), P = in_reg(g.P);
    const uint32_t pc = (uint32_t)g.pc_log2, m = (1u << pc) - 1u, staged = bar + 8u * kStStageBar, bytes = in_reg((uint32_t)g.stage_bytes);
    const uint32_t seg_step = in_reg((uint32_t)kTileM << (pc + 4));
    // a lane's pieces of its pixel in the staged row (the second segment's are 128 pixels on, where the swizzle is the same)
    uint32_t piece[2 * kCh];
#pragma unroll
    for (int i = 0; i < 2 * kCh; ++i) piece[i] = ((uint32_t)s.px << (pc + 4)) + ((((uint32_t)(s.ch0 * 2 + i)) ^ ((uint32_t)s.px >> (3 - pc) & m)) << 4);
    uint32_t buf = 0, buf_ph = 0, stage = sbase + (uint32_t)g.off_stage;
    const uint32_t bufs = in_reg((uint32_t)g.stage_bufs);
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<true>(g, u, u1);
        u += r.len;
        int w0 = r.row * ps - pp, left = 0;          // first row of the window whose maximum is being formed; rows of the step still to come
        uint32_t cur[kSegs][kCh][8], t_row = 0;
#pragma unroll
        for (int i = 0; i < kSegs * kCh * 8; ++i) cur[i / (8 * kCh)][(i >> 3) % kCh][i & 7] = none;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; ++p) {
            const bool emit = p == min(w0 + pk, P) - 1, again = p >= w0 + ps, within = p >= w0;
            if (left == 0) {
                left = min(s.spr, r.p1 - p);
                if (!s.full()) return false;
                tc_fence_after();
                t_row = s.taddr + (uint32_t)s.a * s.set_cols;
            }
            // (the staged row before last has been read)
            if (emit && !(mbar_test(staged + 16u + 8u * buf, buf_ph ^ 1u) || mbar_wait(staged + 16u + 8u * buf, buf_ph ^ 1u))) return false;
#pragma unroll
            for (int seg = 0; seg < kSegs; ++seg) {
                if (seg > 0 && r.width <= kTileM) continue;
                const bool last = left == 1 && (seg == kSegs - 1 || r.width <= kTileM), live = s.px + seg * kTileM < r.width;
                const uint32_t ta = t_row + (uint32_t)seg * s.acc_cols, at = stage + (uint32_t)seg * seg_step;
                constexpr int kAtOnce = kSegs == 1 ? kCh : 1;      // (two segments: 16 columns at a time, for the registers)
#pragma unroll
                for (int h0 = 0; h0 < kCh; h0 += kAtOnce) {
                    float v[16 * kAtOnce];
                    stem_tmem<kAtOnce>(ta + (uint32_t)h0 * 16u, v);
                    if (last && h0 + kAtOnce == kCh) s.read();
#pragma unroll
                    for (int h = h0; h < h0 + kAtOnce; ++h) {
                        uint32_t o[8];
                        float2 bias[8];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float4 b = ld_shared_f4(bias_at + (uint32_t)(64 * h + 16 * i));
                            bias[2 * i] = make_float2(b.x, b.y); bias[2 * i + 1] = make_float2(b.z, b.w);
                        }
                        stem_pack(v + 16 * (h - h0), bias, act, o);
                        uint32_t(&c)[8] = cur[seg][h];
                        if (within) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) c[i] = max_bf16x2(c[i], o[i]);
                        }
                        if (emit) {
                            st_shared16_if(at + piece[2 * h], make_uint4(c[0], c[1], c[2], c[3]), live && h < s.chn);
                            st_shared16_if(at + piece[2 * h + 1], make_uint4(c[4], c[5], c[6], c[7]), live && h < s.chn);
                            if (again) {
#pragma unroll
                                for (int i = 0; i < 8; ++i) c[i] = max_bf16x2(o[i], none);
                            } else {
#pragma unroll
                                for (int i = 0; i < 8; ++i) c[i] = none;
                            }
                        }
                    }
                }
            }
            t_row += s.row_cols;
            if (--left == 0) s.next();
            if (emit) {
                warp_arrive(staged + 8u * buf, s.lane);
                w0 += ps;
                if (++buf == bufs) { buf = 0; buf_ph ^= 1u; }
                stage = sbase + (uint32_t)g.off_stage + buf * bytes;
            }
        }
    }
    return true;
}

// The pool's maximum over columns: staged rows to the output, a thread's pixels of a row a sweep apart.  A thread's window columns are
// the same in every row of a run (clamped columns repeat a column of the window, which leaves the maximum as it is).
__device__ __forceinline__ bool stem_columns(const StemParams &g, uint32_t sbase, uint32_t bar, int u0, int u1) {
    const int t = (int)threadIdx.x - kStThreads, lane = t & 31, n0 = blockIdx.y * g.tile_n, live = min(g.tile_n, g.N - n0);
    const uint32_t pc = in_reg((uint32_t)g.pc_log2), m = (1u << pc) - 1u, staged = bar + 8u * kStStageBar;
    const int cc = t & (int)m, pk = in_reg(g.pk), ps = in_reg(g.ps), pp = in_reg(g.pp), qlast = g.Q - 1, sweep = 32 * kStColWarps >> pc;
    const size_t out_row = (size_t)g.PQ * g.out_ctot, out_sweep = (size_t)sweep * g.out_ctot;
    const uint32_t bufs = in_reg((uint32_t)g.stage_bufs);
    uint32_t buf = 0, buf_ph = 0;
    auto keep = [](uint4 &v, const uint4 &o) {
        v.x = max_bf16x2(v.x, o.x); v.y = max_bf16x2(v.y, o.y); v.z = max_bf16x2(v.z, o.z); v.w = max_bf16x2(v.w, o.w);
    };
    constexpr int kPix = 4;      // pixels of a thread whose window columns are kept
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<true>(g, u, u1);
        u += r.len;
        const int oq0 = r.out0 + (t >> pc);
        auto column = [&](int oq, int i) {
            const int q = min(max(oq * ps - pp + min(i, pk - 1), 0), qlast) - r.base;
            return ((uint32_t)q << (pc + 4)) + ((((uint32_t)cc) ^ ((uint32_t)q >> (3 - pc) & m)) << 4);
        };
        uint32_t at01[kPix], at2[kPix];
#pragma unroll
        for (int i = 0; i < kPix; ++i) {
            const int oq = min(oq0 + i * sweep, r.out1 - 1);
            at01[i] = column(oq, 0) | (column(oq, 1) << 16); at2[i] = column(oq, 2);
        }
        __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(g.out) + g.out_coff + n0 + cc * 8 + ((size_t)r.n * g.rows + r.row) * out_row + (size_t)oq0 * g.out_ctot;
#pragma unroll 1
        for (int i0 = 0; i0 < r.len; ++i0, out += out_row) {
            if (!(mbar_test(staged + 8u * buf, buf_ph) || mbar_wait(staged + 8u * buf, buf_ph))) return false;
            const uint32_t stage = sbase + (uint32_t)g.off_stage + buf * (uint32_t)g.stage_bytes;
            if (cc * 8 < live) {
                __nv_bfloat16 *d = out;
                int oq = oq0;
                if (pk <= 3) {
#pragma unroll
                    for (int h = 0; h < kPix; h += 2) {
                        uint4 v[2];
#pragma unroll
                        for (int i = h; i < h + 2; ++i) {
                            v[i - h] = ld_shared16(stage + (at01[i] & 0xffffu));
                            keep(v[i - h], ld_shared16(stage + (at01[i] >> 16)));
                            keep(v[i - h], ld_shared16(stage + at2[i]));
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i, oq += sweep, d += out_sweep)
                            if (oq < r.out1) *reinterpret_cast<uint4 *>(d) = v[i];
                    }
                }
#pragma unroll 1
                for (; oq < r.out1; oq += sweep, d += out_sweep) {
                    uint4 v = ld_shared16(stage + column(oq, 0));
#pragma unroll 1
                    for (int i = 1; i < pk; ++i) keep(v, ld_shared16(stage + column(oq, i)));
                    *reinterpret_cast<uint4 *>(d) = v;
                }
            }
            warp_arrive(staged + 16u + 8u * buf, lane);
            if (++buf == bufs) { buf = 0; buf_ph ^= 1u; }
        }
    }
    return true;
}

// kRows: image rows by bulk copies
template <int kMode, bool kF32, bool kPool, bool kRows>
__global__ void __launch_bounds__(kStThreads + (kPool ? 32 * kStColWarps : 0), 1)
stem_tc_kernel(const __grid_constant__ StemParams g) {
    extern __shared__ uint8_t smem_raw[];
    pdl_launch_dependents();
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (sbase - raw);
    const uint32_t bar = sbase + g.off_bar;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + g.off_bar + 8 * (kStWeightBar + 1));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem_cols = (uint32_t)(g.nsets * g.spr * g.nsm * g.acc_stride);
    if (warp == 15) {
        const uint32_t wbar = bar + 8u * kStWeightBar;
        if (lane == 0) {
            // the weights: parameters, which no earlier kernel writes
            mbar_init(wbar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            const uint32_t bytes = (uint32_t)(g.npairs * 2 * g.tile_n * 16);
            mbar_arrive_expect_tx(wbar, bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(sbase + (uint32_t)g.off_w), "l"(reinterpret_cast<const uint8_t *>(g.w) + (size_t)blockIdx.y * bytes), "r"(bytes), "r"(wbar) : "memory");
        }
        // (a lane per barrier)
        if (lane < kStWeightBar) mbar_init(bar + 8u * lane, lane < kStMaxSteps ? g.nprod : lane < kStAccBar + kStMaxSets ? 1 : lane < kStStageBar + 2 ? kStEpiWarps : kStColWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
        // (zeros of one chunk, 128 pieces, behind the ring)
        if (threadIdx.x < 128) st_shared16(sbase + (uint32_t)((g.R + 1) * g.qp * g.C * 16) + threadIdx.x * 16u, make_uint4(0u, 0u, 0u, 0u));
        // (a row of zeros, for rows outside the image)
        if (kRows && warp < kStEpiWarps)
            for (int i = threadIdx.x; i < g.raw_stride / 16; i += 32 * kStEpiWarps) st_shared16(sbase + (uint32_t)g.off_raw + i * 16u, make_uint4(0u, 0u, 0u, 0u));
    }
    // an equal share of the units, to the nearest one
    const int b = (int)blockIdx.x, u0 = b * g.unit_share + min(b, g.unit_extra), u1 = u0 + g.unit_share + (b < g.unit_extra ? 1 : 0);
    const unsigned gave_up = kStatusTimeout | (((unsigned)g.launch_id & 0xfffu) << 12);
    const bool producer = warp >= kStEpiWarps && warp < kStEpiWarps + g.nprod;
    bool ok = true;
    tc_fence_before();
    if (!kRows || !producer) asm volatile("bar.sync 0;" ::: "memory");      // (producers of rows by copies are there later)
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(tmem_slot);
    if (warp < kStEpiWarps) {
        const bool wide = g.tile_n > 32;
        if (kPool) {
            if (g.nsm == 1) ok = wide ? stem_epilogue_pool<1, 2>(g, sbase, bar, tmem_base, u0, u1) : stem_epilogue_pool<1, 1>(g, sbase, bar, tmem_base, u0, u1);
            else ok = wide ? stem_epilogue_pool<2, 2>(g, sbase, bar, tmem_base, u0, u1) : stem_epilogue_pool<2, 1>(g, sbase, bar, tmem_base, u0, u1);
        } else {
            ok = wide ? stem_epilogue_store<2>(g, bar, tmem_base, u0, u1) : stem_epilogue_store<1>(g, bar, tmem_base, u0, u1);
        }
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (5u << 8));
    } else if (warp >= 16) {
        ok = stem_columns(g, sbase, bar, u0, u1);
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (6u << 8));
    } else if (producer) {
        if (!kRows) pdl_wait();
        ok = kRows ? stem_produce_rows<kMode, kF32, kPool>(g, sbase, bar, u0, u1, warp - kStEpiWarps, lane)
                   : stem_produce<kMode, kF32, kPool>(g, sbase, bar, u0, u1, warp - kStEpiWarps, lane);
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (3u << 8));
    } else {
        if (elect_one()) {
            ok = stem_mma<kPool>(g, sbase, bar, tmem_base, u0, u1, 15 - warp, kStMaxProd + 1 - g.nprod);
            if (!ok) atomicCAS(g.status, 0u, gave_up | (2u << 8));
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 15) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
}

}  // namespace xk
