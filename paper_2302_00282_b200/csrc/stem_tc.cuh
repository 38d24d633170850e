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
// of rows is contiguous wherever the ring wraps), one step per convolution row.
//   warps 0..7   : epilogue: bias, activation, bf16; stores, or the running maximum of the pool's rows in registers, the
//                  maximum over columns through a staged row
//   warps 8..14  : image rows -> operand pieces
//   warp 15      : issues the products; a convolution row is one accumulator per 128 columns
// What bounds it: the producers (one row a step and warp: 400 cycles for reading and storing its pieces, the rest for the request
// of the row four ahead and the barriers; 1530 in all while every request walked to its row), then the products' thread, 900 a
// row of 128 columns and 3 x 3 taps; the products themselves read 6 KB of shared memory each for 64 channels (48 cycles), 11 per
// 128 columns for a 7 x 7 window of 3 channels.  With rows loaded through registers one ahead a row of MobileNet's stem at batch
// 32 took 1750 cycles.
#pragma once

#include "conv_tc.cuh"

namespace xk {

constexpr int kStThreads = 512, kStEpiWarps = 8, kStProdWarps = 7;
constexpr int kStMaxSteps = 8, kStMaxAcc = 8;

struct StemParams {
    const void *src;
    const uint4 *w;                 // [pair of chunks][2][tile_n] pieces of 8 weights, per channel tile
    const float *bias;
    void *out;
    unsigned int *status;
    int units;                      // (image, column block, row) triples; rows of the output or, with a pool, of the pool
    int rows, cbs, cw;              // rows per image, column blocks, output columns per block
    FastDiv d_rows, d_cbs;
    int C, H, W, k, stride, pad, lead;      // lead: a piece starts lead elements before the window (alignment of the loads)
    int P, Q, N, tile_n, npairs;
    int R, D, nacc, acc_stride;     // row slots, steps in flight, accumulators
    int qp;                         // pieces per (slot, channel)
    int pk, ps, pp, PQ;             // max pool
    int pc_log2;                    // staged pixel: 1 << pc_log2 chunks of 16 bytes
    int act, out_ctot, out_coff;
    uint32_t idesc;
    int off_w, off_bias, off_stage, stage_bytes, off_bar;
    int raw_slots, raw_stride, raw_lead, off_raw;      // image rows on their way: slots per producer warp, bytes of a slot and of the zeros in front
    int launch_id;
};
constexpr int kStMaxRaw = 6;
constexpr int kStRawBar = 2 * kStMaxSteps + 2 * kStMaxAcc + 2;      // barriers of the row slots, kStMaxRaw per producer warp
static_assert(8 * (kStRawBar + kStMaxRaw * kStProdWarps) <= 768, "barriers exceed their place");

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
template <int kMode, bool kF32>
__device__ __forceinline__ void stem_store(const uint32_t (&raw)[4][StemForm<kMode, kF32>::words], uint32_t dst, uint32_t again, int left, int passes, int lane,
                                           const uint4 &in_window) {
    using F = StemForm<kMode, kF32>;
    // eight lanes store 128 bytes apart in pairs: every second group of four lanes stores its second piece first, so that the
    // eight pieces of a store meet eight different groups of banks
    const uint32_t f = (uint32_t)(lane >> 2) & 1u, d0 = dst + f * 16u, d1 = dst + (f ^ 1u) * 16u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
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
        if (32 * i < left) {
            if (F::run == 1) {
                st_shared16(dst + step, a);
                if (again) st_shared16(dst + again + step, a);
            } else {
                const uint4 b = F::S == 2 ? piece(w[1], w[2], w[3], w[4])
                                          : piece(__funnelshift_r(w[0], w[1], 16), __funnelshift_r(w[1], w[2], 16),
                                                  __funnelshift_r(w[2], w[3], 16), __funnelshift_r(w[3], w[4], 16));
                const uint4 x = f ? b : a, y = f ? a : b;
                st_shared16(d0 + step, x);
                st_shared16(d1 + step, y);
                if (again) { st_shared16(d0 + again + step, x); st_shared16(d1 + again + step, y); }
            }
        }
    }
}

// A producer warp: one channel, every rstep-th new row of a step (three channels: six of the seven warps, a row each per step
// of stride 2).
template <int kMode, bool kF32, bool kPool>
__device__ __forceinline__ bool stem_produce(const StemParams &g, uint32_t sbase, uint32_t bar, int u0, int u1, int w, int lane) {
    using F = StemForm<kMode, kF32>;
    constexpr int es = kF32 ? 4 : 2;
    const int C = in_reg(g.C), k = in_reg(g.k), stride = F::S ? F::S : in_reg(g.stride), R = in_reg(g.R), D = in_reg(g.D), W = in_reg(g.W), H = in_reg(g.H);
    const int pad = in_reg(g.pad), rstep = kStProdWarps / C, nr = min(stride, k);
    int j0 = w / C;
    const int c = w - j0 * C;
    if (j0 >= rstep) j0 = k;                              // a warp without rows only keeps the steps' counts
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
        // (the slots of a step's rows are free when the step D before it has been multiplied; the first rows of another image
        // wait for all of the last one's)
        uint32_t room = bar + 8u * (kStMaxSteps + sl), room_ph = ph ^ 1u;
        if (t > 0) {
            room = bar + 8u * (kStMaxSteps + (sl ? sl - 1 : D - 1));
            room_ph = sl ? ph : ph ^ 1u;
        }
        int p = r.p0, d = j0, ih0 = p * stride - pad;
        bool start = true, fresh = true, have = false;
#pragma unroll 1
        for (;;) {
            if (!start) {
                if (fresh) {
                    if (!mbar_wait(room, room_ph)) return false;
                    fresh = false;
                }
                if (have) {
                    int s = slot + d;
                    if (s >= R) s -= R;
                    stem_store<kMode, kF32>(raw, ring + (uint32_t)s * slot_bytes, s == 0 ? wrap : 0u, left, passes, lane, in_window);
                    d += rstep;
                }
                if (d >= k) {
                    warp_arrive(bar + 8u * sl, lane);
                    if (++sl == D) { sl = 0; ph ^= 1u; }
                    ++t;
                    slot += ++p == r.p1 ? k : nr;
                    if (slot >= R) slot -= R;
                    if (p == r.p1) break;
                    room = bar + 8u * (kStMaxSteps + sl); room_ph = ph ^ 1u;
                    fresh = true;
                    ih0 += stride;
                    d = j0 < nr ? k - nr + j0 : k;
                }
            }
            start = false;
            have = d < k;
            if (have) load(ih0 + d);
        }
    }
    return true;
}

// The rows of a producer warp in the order it makes them.
template <bool kPool>
struct StemCursor {
    int u, n, p, p1, d, ih0;
    bool more;
    __device__ __forceinline__ void run(const StemParams &g, int u1, int j0, int stride, int pad) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len; n = r.n; p = r.p0; p1 = r.p1; d = j0; ih0 = p * stride - pad;
    }
    __device__ __forceinline__ void next(const StemParams &g, int u1, int j0, int rstep, int k, int nr, int stride, int pad) {
        d += rstep;
        while (d >= k) {
            if (++p < p1) { ih0 += stride; d = j0 < nr ? k - nr + j0 : k; }
            else if (u < u1) run(g, u1, j0, stride, pad);
            else { more = false; return; }
        }
    }
};

// The same where rows are whole 16-byte pieces of memory: a warp keeps raw_slots of its rows on their way by bulk copies and
// reads them from shared memory, between zeros for the padding (a row outside the image is a slot of zeros).  With the loads of
// one row ahead in registers every step cost the latency of a load from memory, 1000 to 1900 cycles.
template <int kMode, bool kF32>
__device__ __forceinline__ void stem_read(uint32_t (&raw)[4][StemForm<kMode, kF32>::words], uint32_t s, int passes, int stride) {
    using F = StemForm<kMode, kF32>;
    constexpr int es = kF32 ? 4 : 2;
    const int S = F::S ? F::S : stride;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i >= passes) break;
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
    const int pad = in_reg(g.pad), rstep = kStProdWarps / C, nr = min(stride, k);
    int j0 = w / C;
    const int c = w - j0 * C;
    if (j0 >= rstep) j0 = k;                              // a warp without rows only keeps the steps' counts
    const uint32_t slot_bytes = in_reg((uint32_t)(g.qp * C * 16)), ring = in_reg(sbase + (uint32_t)((c * g.qp + F::run * lane) * 16)), wrap = (uint32_t)R * slot_bytes;
    const uint32_t row_bytes = in_reg((uint32_t)(g.W * es)), raw_stride = in_reg((uint32_t)g.raw_stride), lead = (uint32_t)g.raw_lead;
    const uint32_t zeros = sbase + (uint32_t)g.off_raw + lead;                                    // slot 0 of the region: a row of zeros
    const uint32_t mine = zeros + raw_stride * (uint32_t)(1 + w * g.raw_slots), mine_end = mine + raw_stride * (uint32_t)g.raw_slots;
    const uint32_t bar0 = bar + 8u * (uint32_t)(kStRawBar + kStMaxRaw * w);
    auto both = [&](int j) {                              // which of elements j, j + 1 of a piece the window takes
        const uint32_t x = (unsigned)(j - g.lead) < (unsigned)k, y = (unsigned)(j + 1 - g.lead) < (unsigned)k;
        return in_reg(x * 0xffffu | y * 0xffff0000u);
    };
    const uint4 in_window = make_uint4(both(0), both(2), both(4), both(6));
    StemCursor<kPool> ahead;
    ahead.u = u0; ahead.more = u0 < u1 && j0 < k;
    if (ahead.more) ahead.run(g, u1, j0, stride, pad);
    uint32_t raw_at = mine, raw_bar = bar0, raw_ph = 0u;      // the slot that is read next; it is filled again behind the read
    // A row into a slot.  Behind the first step of a run a warp's rows of it lie a stride apart, one per step: `again` of them
    // follow without another look at the walk (which made the request 700 cycles of a step).
    const uint8_t *src = nullptr;
    int again = 0;
    auto ask = [&](uint32_t at, uint32_t b) {
        if (again > 0) {
            --again;
            src += (uint32_t)stride * row_bytes;
        } else {
            while (ahead.more && (unsigned)(ahead.ih0 + ahead.d) >= (unsigned)H) ahead.next(g, u1, j0, rstep, k, nr, stride, pad);
            if (!ahead.more) return;
            const int ih = ahead.ih0 + ahead.d;
            src = reinterpret_cast<const uint8_t *>(g.src) + ((size_t)(ahead.n * C + c) * H + ih) * row_bytes;
            if (ahead.d == k - nr + j0 && ahead.d + rstep >= k) {
                again = min(ahead.p1 - 1 - ahead.p, (H - 1 - ih) >> (F::S == 2 ? 1 : 0));
                ahead.p += again; ahead.ih0 += again * stride;
            }
            ahead.next(g, u1, j0, rstep, k, nr, stride, pad);
        }
        if (lane == 0) {
            mbar_arrive_expect_tx(b, row_bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(at), "l"(src), "r"(row_bytes), "r"(b) : "memory");
        }
    };
    for (int i = 0; i < g.raw_slots; ++i) ask(mine + raw_stride * (uint32_t)i, bar0 + 8u * i);
    uint32_t raw[4][F::words];
    int t = 0, sl = 0, slot = 0;                          // step, its barrier, ring slot of its window row 0
    uint32_t ph = 0;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len;
        const int e = ((r.base + F::run * lane) * stride - pad - g.lead) * es;
        const int lanes = (r.width + F::run - 1) / F::run, passes = (lanes + 31) >> 5, left = lanes - lane;
        int d = j0, ih0 = r.p0 * stride - pad;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; ++p, ih0 += stride) {
            // (the slots of a step's rows are free when the step D before it has been multiplied; the first rows of another image
            // wait for all of the last one's)
            if (p == r.p0 && t > 0) {
                if (!mbar_wait(bar + 8u * (kStMaxSteps + (sl ? sl - 1 : D - 1)), sl ? ph : ph ^ 1u)) return false;
            } else if (t >= D) {
                if (!mbar_wait(bar + 8u * (kStMaxSteps + sl), ph ^ 1u)) return false;
            }
#pragma unroll 1
            for (; d < k; d += rstep) {
                const bool in = (unsigned)(ih0 + d) < (unsigned)H;
                if (in && !mbar_wait(raw_bar, raw_ph)) return false;
                stem_read<kMode, kF32>(raw, (in ? raw_at : zeros) + (uint32_t)e, passes, stride);
                int s = slot + d;
                if (s >= R) s -= R;
                stem_store<kMode, kF32>(raw, ring + (uint32_t)s * slot_bytes, s == 0 ? wrap : 0u, left, passes, lane, in_window);
                if (in) {
                    __syncwarp();
                    ask(raw_at, raw_bar);
                    raw_at += raw_stride; raw_bar += 8u;
                    if (raw_at == mine_end) { raw_at = mine; raw_bar = bar0; raw_ph ^= 1u; }
                }
            }
            warp_arrive(bar + 8u * sl, lane);
            if (++sl == D) { sl = 0; ph ^= 1u; }
            ++t;
            slot += p + 1 == r.p1 ? k : nr;
            if (slot >= R) slot -= R;
            d = j0 < nr ? k - nr + j0 : k;
        }
    }
    return true;
}

// ---- products --------------------------------------------------------------------------------------------------------
// One thread: a convolution row is ns accumulators of npairs products each.
template <bool kPool>
__device__ __forceinline__ bool stem_mma(const StemParams &g, uint32_t sbase, uint32_t bar, uint32_t tmem_base, int u0, int u1) {
    const uint32_t hi = (128u >> 4) | (1u << 14);      // 8-row groups 128 bytes apart, descriptor version, no swizzle
    const uint32_t idesc = in_reg(g.idesc);
    const int C = in_reg(g.C), k = in_reg(g.k), R = in_reg(g.R), D = in_reg(g.D), nacc = in_reg(g.nacc);
    const uint32_t ring16 = in_reg(sbase >> 4), cp16 = in_reg((uint32_t)g.qp), rp16 = in_reg((uint32_t)(g.qp * g.C));
    const uint32_t w16 = in_reg(((sbase + (uint32_t)g.off_w) >> 4) | ((uint32_t)g.tile_n << 16)), wstep = in_reg(2u * (uint32_t)g.tile_n);
    const uint32_t accf = bar + 8u * 2 * kStMaxSteps, acce = accf + 8u * kStMaxAcc;
    const int new_rows = min(g.stride, g.k);
    int slot0 = 0, sl = 0, a = 0;
    uint32_t ph = 0, pa = 0;
    if (!mbar_wait(bar + 8u * (2 * kStMaxSteps + 2 * kStMaxAcc), 0)) return false;      // the weights
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<kPool>(g, u, u1);
        u += r.len;
        const int ns = (r.width + kTileM - 1) / kTileM;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; ++p) {
            if (!mbar_wait(bar + 8u * sl, ph)) return false;
            fence_proxy_async();
            tc_fence_after();
#pragma unroll 1
            for (int seg = 0; seg < ns; ++seg) {
                if (!mbar_wait(acce + 8u * a, pa ^ 1u)) return false;
                tc_fence_after();
                const uint32_t d = tmem_base + (uint32_t)(a * g.acc_stride);
                uint32_t acc = 0, bl = w16;
                auto mma = [&](uint32_t al) {
                    umma_bf16(d, ((uint64_t)hi << 32) | al, ((uint64_t)hi << 32) | bl, idesc, acc);
                    acc = 1; bl += wstep;
                };
                int s = slot0;
#pragma unroll 1
                for (int i = 0; i < (k >> 1); ++i) {
                    uint32_t al = (ring16 + (uint32_t)s * rp16 + (uint32_t)seg * 128u) | (rp16 << 16);
                    if (C == 3) {
                        mma(al); mma(al + cp16); mma(al + 2 * cp16);
                    } else {
#pragma unroll 1
                        for (int c = 0; c < C; ++c, al += cp16) mma(al);
                    }
                    s += 2;
                    if (s >= R) s -= R;
                }
                if (k & 1) {
                    uint32_t al = (ring16 + (uint32_t)s * rp16 + (uint32_t)seg * 128u) | (cp16 << 16);
#pragma unroll 1
                    for (int c = 1; c < C; c += 2, al += 2 * cp16) mma(al);
                    if (C & 1) {
                        // the last channel's chunk before the zeros behind the ring
                        const uint32_t last = ring16 + (uint32_t)s * rp16 + (uint32_t)(C - 1) * cp16 + (uint32_t)seg * 128u;
                        mma(last | ((ring16 + (uint32_t)(R + 1) * rp16 - last) << 16));
                    }
                }
                umma_commit(accf + 8u * a);
                if (++a == nacc) { a = 0; pa ^= 1u; }
            }
            umma_commit(bar + 8u * (kStMaxSteps + sl));
            if (++sl == D) { sl = 0; ph ^= 1u; }
            slot0 += p + 1 < r.p1 ? new_rows : k;
            if (slot0 >= R) slot0 -= R;
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
__device__ __forceinline__ void stem_bias(uint32_t at, float2 (&b)[8]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 v = ld_shared_f4(at + 16u * i);
        b[2 * i] = make_float2(v.x, v.y); b[2 * i + 1] = make_float2(v.z, v.w);
    }
}

// What a warp of the epilogue keeps: its quarter of the accumulator's lanes, one or two 16-column chunks of it.
struct StemEpi {
    int lane, px, ch0, chn, n0, live, nacc, acc_stride, act, a;
    uint32_t accf, acce, taddr, pa;
    __device__ __forceinline__ void init(const StemParams &g, uint32_t bar, uint32_t tmem_base) {
        const int warp = threadIdx.x >> 5, quarter = warp & 3, half = warp >> 2, nch = g.tile_n >> 4;
        lane = threadIdx.x & 31; px = quarter * 32 + lane;
        ch0 = half ? (nch + 1) >> 1 : 0; chn = half ? nch >> 1 : (nch + 1) >> 1;
        n0 = blockIdx.y * g.tile_n; live = min(g.tile_n, g.N - n0);
        nacc = in_reg(g.nacc); acc_stride = in_reg(g.acc_stride); act = in_reg(g.act);
        accf = bar + 8u * 2 * kStMaxSteps; acce = accf + 8u * kStMaxAcc;
        taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)ch0 * 16u;
        a = 0; pa = 0;
    }
};

__device__ __forceinline__ bool stem_epilogue_store(const StemParams &g, uint32_t sbase, uint32_t bar, uint32_t tmem_base, int u0, int u1) {
    StemEpi s;
    s.init(g, bar, tmem_base);
    float2 bias[2][8];
    stem_bias(sbase + (uint32_t)g.off_bias + (uint32_t)s.ch0 * 64u, bias[0]);
    stem_bias(sbase + (uint32_t)g.off_bias + (uint32_t)(s.ch0 + 1) * 64u, bias[1]);
    // 32-byte stores where every chunk is whole and aligned
    const bool wide = ((g.out_ctot | g.out_coff | s.live) & 15) == 0;
    const int ctot = in_reg(g.out_ctot), Q = in_reg(g.Q);
    __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(g.out) + g.out_coff + s.n0 + s.ch0 * 16;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<false>(g, u, u1);
        u += r.len;
        __nv_bfloat16 *row = out + (((size_t)r.n * g.P + r.p0) * Q + r.base + s.px) * ctot;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; ++p, row += (size_t)Q * ctot) {
            __nv_bfloat16 *d = row;
#pragma unroll 1
            for (int q = s.px; q - s.px < r.width; q += kTileM, d += (size_t)kTileM * ctot) {
                if (!mbar_wait(s.accf + 8u * s.a, s.pa)) return false;
                tc_fence_after();
                float v[32];
                const uint32_t ta = s.taddr + (uint32_t)(s.a * s.acc_stride);
                if (s.chn == 2) tmem_ld32(ta, v);
                else if (s.chn == 1) tmem_ld16(ta, v);
                tc_fence_before();
                warp_arrive(s.acce + 8u * s.a, s.lane);
                if (++s.a == s.nacc) { s.a = 0; s.pa ^= 1u; }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (j >= s.chn) continue;
                    uint32_t o[8];
                    stem_pack(v + 16 * j, bias[j], s.act, o);
                    if (q >= r.width) continue;
                    if (wide) {
                        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d + 16 * j), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                                     "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]) : "memory");
                    } else {
                        const int nc = (s.ch0 + j) * 16;
                        if (nc + 8 <= s.live) *reinterpret_cast<uint4 *>(d + 16 * j) = make_uint4(o[0], o[1], o[2], o[3]);
                        if (nc + 16 <= s.live) *reinterpret_cast<uint4 *>(d + 16 * j + 8) = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                }
            }
        }
    }
    return true;
}

// The pool's maximum over rows stays in registers: a lane keeps its column.  A finished row is staged and the maximum over
// columns read from there.
__device__ __forceinline__ bool stem_epilogue_pool(const StemParams &g, uint32_t sbase, uint32_t bar, uint32_t tmem_base, int u0, int u1) {
    StemEpi s;
    s.init(g, bar, tmem_base);
    const uint32_t bias_at = sbase + (uint32_t)g.off_bias + (uint32_t)s.ch0 * 64u;
    // (a maximum that starts at zero is ReLU's, too)
    const uint32_t none = in_reg(s.act ? 0u : 0xff80ff80u);
    const int act = s.act == 1 ? 0 : s.act;
    const uint32_t pc = in_reg((uint32_t)g.pc_log2), m = (1u << pc) - 1u;
    const int cc = (int)(threadIdx.x & m), pk = in_reg(g.pk), ps = in_reg(g.ps), pp = in_reg(g.pp), qlast = g.Q - 1;
    __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(g.out) + g.out_coff + s.n0 + cc * 8;
    bool ok = true;
    int buf = 0;
#pragma unroll 1
    for (int u = u0; u < u1;) {
        const StemRun r = stem_run<true>(g, u, u1);
        u += r.len;
        int prow = r.row;                            // the row whose maximum is being formed
        uint32_t cur[2][2][8];
#pragma unroll
        for (int i = 0; i < 32; ++i) cur[i >> 4][(i >> 3) & 1][i & 7] = none;
#pragma unroll 1
        for (int p = r.p0; p < r.p1; ++p) {
            const int w0 = prow * ps - pp;
            const bool emit = p == min(w0 + pk, g.P) - 1, again = p >= w0 + ps, within = p >= w0;
            const uint32_t stage = sbase + (uint32_t)(g.off_stage + buf * g.stage_bytes);
            auto segment = [&](int q, uint32_t (&cur)[2][8]) {
                // (after a give-up the warp goes on without waiting, so that the barriers below keep their counts)
                if (ok) ok = mbar_wait(s.accf + 8u * s.a, s.pa);
                tc_fence_after();
                const uint32_t ta = s.taddr + (uint32_t)(s.a * s.acc_stride), freed = s.acce + 8u * s.a;
                if (++s.a == s.nacc) { s.a = 0; s.pa ^= 1u; }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float v[16];
                    if (j < s.chn) tmem_ld16(ta + (uint32_t)j * 16u, v);
                    if (j == 1) {
                        tc_fence_before();
                        warp_arrive(freed, s.lane);
                    }
                    if (j >= s.chn) continue;
                    float2 bias[8];
                    uint32_t o[8];
                    stem_bias(bias_at + (uint32_t)j * 64u, bias);
                    stem_pack(v, bias, act, o);
                    uint32_t(&c)[8] = cur[j];
                    if (within) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) c[i] = max_bf16x2(c[i], o[i]);
                    }
                    if (emit) {
                        if (q < r.width) {
                            const uint32_t x = (uint32_t)q >> (3 - pc) & m, at = stage + ((uint32_t)q << (pc + 4)), c2 = (uint32_t)(s.ch0 + j) * 2u;
                            st_shared16(at + ((c2 ^ x) << 4), make_uint4(c[0], c[1], c[2], c[3]));
                            st_shared16(at + (((c2 + 1) ^ x) << 4), make_uint4(c[4], c[5], c[6], c[7]));
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) c[i] = again ? max_bf16x2(o[i], none) : none;
                    }
                }
            };
            segment(s.px, cur[0]);
            if (r.width > kTileM) segment(s.px + kTileM, cur[1]);
            if (emit) {
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (cc * 8 < s.live && ok) {
                    __nv_bfloat16 *d = out + ((size_t)r.n * g.rows + prow) * g.PQ * g.out_ctot;
                    // (clamped columns repeat a column of the window, which leaves the maximum as it is)
                    auto column = [&](int w, int i) {
                        const int q = min(max(w + min(i, pk - 1), 0), qlast) - r.base;
                        const uint32_t x = (uint32_t)q >> (3 - pc) & m;
                        return ld_shared16(stage + ((uint32_t)q << (pc + 4)) + (((uint32_t)cc ^ x) << 4));
                    };
                    auto keep = [](uint4 &v, const uint4 &o) {
                        v.x = max_bf16x2(v.x, o.x); v.y = max_bf16x2(v.y, o.y); v.z = max_bf16x2(v.z, o.z); v.w = max_bf16x2(v.w, o.w);
                    };
#pragma unroll 2
                    for (int oq = r.out0 + (int)(threadIdx.x >> pc); oq < r.out1; oq += 256 >> pc) {
                        const int w = oq * ps - pp;
                        uint4 v = column(w, 0);
                        keep(v, column(w, 1));
                        keep(v, column(w, 2));
#pragma unroll 1
                        for (int i = 3; i < pk; ++i) keep(v, column(w, i));
                        *reinterpret_cast<uint4 *>(d + (size_t)oq * g.out_ctot) = v;
                    }
                }
                ++prow; buf ^= 1;
            }
        }
    }
    return ok;
}

// kRows: image rows by bulk copies
template <int kMode, bool kF32, bool kPool, bool kRows>
__global__ void __launch_bounds__(kStThreads, 1)
stem_tc_kernel(const __grid_constant__ StemParams g) {
    extern __shared__ uint8_t smem_raw[];
    pdl_launch_dependents();
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (sbase - raw);
    const uint32_t bar = sbase + g.off_bar;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + g.off_bar + 8 * (2 * kStMaxSteps + 2 * kStMaxAcc + 1));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem_cols = (uint32_t)(g.nacc * g.acc_stride);
    if (warp == 15) {
        if (lane == 0) {
            for (int s = 0; s < g.D; ++s) { mbar_init(bar + 8u * s, kStProdWarps); mbar_init(bar + 8u * (kStMaxSteps + s), 1); }
            mbar_init(bar + 8u * (2 * kStMaxSteps + 2 * kStMaxAcc), 1);
            for (int b = 0; b < g.nacc; ++b) { mbar_init(bar + 8u * (2 * kStMaxSteps + b), 1); mbar_init(bar + 8u * (2 * kStMaxSteps + kStMaxAcc + b), kStEpiWarps); }
            if (kRows) for (int b = 0; b < kStMaxRaw * kStProdWarps; ++b) mbar_init(bar + 8u * (kStRawBar + b), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            // the weights: parameters, which no earlier kernel writes
            const uint32_t bytes = (uint32_t)(g.npairs * 2 * g.tile_n * 16), wbar = bar + 8u * (2 * kStMaxSteps + 2 * kStMaxAcc);
            mbar_arrive_expect_tx(wbar, bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(sbase + (uint32_t)g.off_w), "l"(reinterpret_cast<const uint8_t *>(g.w) + (size_t)blockIdx.y * bytes), "r"(bytes), "r"(wbar) : "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
        // (zeros of one chunk, 128 pieces, behind the ring)
        if (threadIdx.x < 128) st_shared16(sbase + (uint32_t)((g.R + 1) * g.qp * g.C * 16) + threadIdx.x * 16u, make_uint4(0u, 0u, 0u, 0u));
        // (the row slots' zeros, before any copy into them)
        if (kRows) {
            for (int i = threadIdx.x; i < (1 + g.raw_slots * kStProdWarps) * g.raw_stride / 16; i += 32 * 15) st_shared16(sbase + (uint32_t)g.off_raw + i * 16u, make_uint4(0u, 0u, 0u, 0u));
            fence_proxy_async();
        }
        if ((int)threadIdx.x < g.tile_n) reinterpret_cast<float *>(sm + g.off_bias)[threadIdx.x] = __ldg(g.bias + blockIdx.y * g.tile_n + threadIdx.x);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // an equal share of the units, to the nearest one
    const int per = g.units / (int)gridDim.x, extra = g.units - per * (int)gridDim.x, b = (int)blockIdx.x;
    const int u0 = b * per + min(b, extra), u1 = u0 + per + (b < extra ? 1 : 0);
    const unsigned gave_up = kStatusTimeout | (((unsigned)g.launch_id & 0xfffu) << 12);
    bool ok = true;
    if (warp < kStEpiWarps) {
        ok = kPool ? stem_epilogue_pool(g, sbase, bar, tmem_base, u0, u1) : stem_epilogue_store(g, sbase, bar, tmem_base, u0, u1);
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (5u << 8));
    } else if (warp < 15) {
        pdl_wait();
        ok = kRows ? stem_produce_rows<kMode, kF32, kPool>(g, sbase, bar, u0, u1, warp - kStEpiWarps, lane)
                   : stem_produce<kMode, kF32, kPool>(g, sbase, bar, u0, u1, warp - kStEpiWarps, lane);
        if (!ok && lane == 0) atomicCAS(g.status, 0u, gave_up | (3u << 8));
    } else {
        if (elect_one()) {
            ok = stem_mma<kPool>(g, sbase, bar, tmem_base, u0, u1);
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
