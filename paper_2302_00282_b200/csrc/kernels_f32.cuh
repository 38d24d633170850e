// fp32 CUDA-core kernels, NCHW.  Used by graphs compiled with XENOS_PRECISION_FP32_CUDA_CORE:
// one kernel per fused operator (unlinked execution) and one kernel for the linked chain
// ConvX -> Conv1x1 -> ZPooling (Table 1 of the Xenos paper), where the intermediate feature
// maps of a tile stay in shared memory in the order the next stage reads them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace xk {

// Programmatic dependent launch: let the next kernel of the stream be scheduled early / wait until
// the previous kernel's memory is complete and visible (no-ops without the launch attribute).
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float apply_act(float v, int act) {
    if (act >= 1) v = fmaxf(v, 0.0f);
    if (act == 2) v = fminf(v, 6.0f);
    return v;
}

// Direct convolution: y[n][k][p][q] = b[k] + sum_{c,r,s} x[n][g*Cg + c][p*st - pad + r][q*st - pad + s] * w[k][c][r][s],
// one output element per thread, then the fused activation.
__global__ void f32_conv_kernel(const float *__restrict__ x, const float *__restrict__ w,
                                const float *__restrict__ b, float *__restrict__ y, int N, int C, int H,
                                int W, int K, int P, int Q, int k, int stride, int pad, int groups, int act) {
    long long total = (long long)N * K * P * Q;
    int Cg = C / groups, Kg = K / groups;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        int q = (int)(i % Q);
        long long t = i / Q;
        int p = (int)(t % P); t /= P;
        int kk = (int)(t % K);
        int n = (int)(t / K);
        int g = kk / Kg;
        float acc = 0.0f;
        for (int c = 0; c < Cg; ++c) {
            const float *xc = x + ((size_t)n * C + (size_t)g * Cg + c) * H * W;
            const float *wc = w + ((size_t)kk * Cg + c) * k * k;
            for (int r = 0; r < k; ++r) {
                int ih = p * stride - pad + r;
                if (ih < 0 || ih >= H) continue;
                for (int s = 0; s < k; ++s) {
                    int iw = q * stride - pad + s;
                    if (iw < 0 || iw >= W) continue;
                    acc = fmaf(xc[(size_t)ih * W + iw], wc[r * k + s], acc);
                }
            }
        }
        y[i] = apply_act(acc + b[kk], act);
    }
}

// Max (kind 0) or average (kind 1, divisor = in-range elements) pooling.
__global__ void f32_pool_kernel(const float *__restrict__ x, float *__restrict__ y, int N, int C, int H, int W,
                                int P, int Q, int k, int stride, int pad, int kind) {
    long long total = (long long)N * C * P * Q;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        int q = (int)(i % Q);
        long long t = i / Q;
        int p = (int)(t % P); t /= P;
        const float *xc = x + (size_t)t * H * W;
        float m = -INFINITY, acc = 0.0f;
        int cnt = 0;
        for (int r = 0; r < k; ++r) {
            int ih = p * stride - pad + r;
            if (ih < 0 || ih >= H) continue;
            for (int s = 0; s < k; ++s) {
                int iw = q * stride - pad + s;
                if (iw < 0 || iw >= W) continue;
                float v = xc[(size_t)ih * W + iw];
                m = fmaxf(m, v);
                acc += v;
                ++cnt;
            }
        }
        y[i] = kind == 0 ? m : (cnt ? acc / (float)cnt : 0.0f);
    }
}

// Global average: one warp per (image, channel), fixed-order lane sums then a shuffle tree.
__global__ void f32_gap_kernel(const float *__restrict__ x, float *__restrict__ y, int NC, int HW) {
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= NC) return;
    const float *xi = x + (size_t)warp * HW;
    float acc = 0.0f;
    for (int i = lane; i < HW; i += 32) acc += xi[i];
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) y[warp] = acc / (float)HW;
}

__global__ void f32_add_kernel(const float *__restrict__ a, const float *__restrict__ b, float *__restrict__ y,
                               long long n, int act) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = apply_act(a[i] + b[i], act);
}

// x.mul (c == nullptr) / x.mac: the product is rounded before the sum (no fused multiply-add).
__global__ void f32_mulmac_kernel(const float *__restrict__ a, const float *__restrict__ b, const float *__restrict__ c,
                                  float *__restrict__ y, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float p = __fmul_rn(a[i], b[i]);
        y[i] = c ? __fadd_rn(p, c[i]) : p;
    }
}

// x.split, one part: y [N][Ci][HW] = x [N][Ctot][HW] at channel offset coff.
__global__ void f32_slice_kernel(const float *__restrict__ x, float *__restrict__ y, int N, int Ci, int HW,
                                 int Ctot, int coff) {
    long long per = (long long)Ci * HW, total = (long long)N * per;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        long long n = i / per, r = i % per;
        y[i] = x[(n * Ctot + coff) * HW + r];
    }
}

// One concat input: x [N][Ci][HW] -> y [N][Ctot][HW] at channel offset coff.
__global__ void f32_concat_part_kernel(const float *__restrict__ x, float *__restrict__ y, int N, int Ci, int HW,
                                       int Ctot, int coff) {
    long long per = (long long)Ci * HW, total = (long long)N * per;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        long long n = i / per, r = i % per;
        y[(n * Ctot + coff) * HW + r] = x[i];
    }
}

// y = W x + B (Eq. 1), one output per thread.
__global__ void f32_fc_kernel(const float *__restrict__ x, const float *__restrict__ w, const float *__restrict__ b,
                              float *__restrict__ y, int N, int C, int K, int act) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * K) return;
    int n = i / K, k = i % K;
    float acc = 0.0f;
    for (int c = 0; c < C; ++c) acc = fmaf(w[(size_t)k * C + c], x[(size_t)n * C + c], acc);
    y[i] = apply_act(acc + b[k], act);
}

// ------------------------------------------------------------------------------------------------
// Linked chain ConvX(+act) -> Conv1x1(+act) -> pool (Table 1), a CTA per (image, outC part, pool tile), walking over
// them when there are more than fit.
//   stage 0: the input patch the tile needs goes to shared memory (zeros outside the image and in the padding of the row pitch)
//   stage 1: ConvX on the patch -> shared memory [Cmid][row][column % pool_stride][column / pool_stride], so that the
//            outputs of one pool tap are adjacent: the order stage 2 reads
//   stage 2: Conv1x1 over the CTA's slice of output channels, pooled in registers
// Both stages are register-tiled: a thread owns TM channels x TP adjacent pixels (pool outputs), lanes of a warp take
// neighbouring pixels of the same channels (weights are broadcast reads), products are packed fp32 pairs over channels.
// Every sum runs over (channel, row, column) in ascending order whatever the tile: a split changes no value.
// Bound by the FMA pipes (8 x 4 tiles: 6 shared-memory reads for 32 multiply-adds); 2 x 1 tiles spread a small map over
// many threads, where latency decides.  Weights sit in shared memory when they fit (kWS), else they are read through L1.
// Measured: 32 -> 64 -> 64 channels, 75 x 75, batch 32: 0.229 ms (35 TFLOP/s; FMA pipes 59 % busy: 49 of a tile's 76 thousand
// cycles are the first stage at three quarters of their rate, 17 the second at half); 16 -> 32 -> 32 channels, 32 x 32, one
// image: 8.6 us.
// ------------------------------------------------------------------------------------------------
struct F32ChainParams {
    const float *x, *w1, *b1, *w2, *b2;      // w1 [C][k][k][mpad], w2 [part][Cmid][kperp]: output channels padded to 8 with zeros
    float *y;
    int N, C, H, W;          // input
    int Cmid, mpad, P, Q;    // stage-1 output
    int k, stride, pad, act1;
    int K2, act2;
    int pool_kind, pool_k, pool_stride, PP, PQ;
    int parts_outc, tile_h, tile_w, tiles_h, tiles_w, halo_h, halo_w;
    int iwp, hp;             // row pitch of the patch; pitch of one column residue of the middle map
    unsigned int *status;
};

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool live) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(live ? 4u : 0u) : "memory");
}

__device__ __forceinline__ void cp_async16_f32(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

template <int TM>
__device__ __forceinline__ void f32_load_w(float2 (&w)[TM / 2], const float *src) {
    if (TM % 4 == 0) {
#pragma unroll
        for (int i = 0; i < TM / 4; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(src + 4 * i);
            w[2 * i] = make_float2(v.x, v.y); w[2 * i + 1] = make_float2(v.z, v.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < TM / 2; ++i) w[i] = *reinterpret_cast<const float2 *>(src + 2 * i);
    }
}

template <int TM, int TP>
__device__ __forceinline__ void f32_fma(float2 (&acc)[TM / 2][TP], const float2 (&w)[TM / 2], const float *x) {
#pragma unroll
    for (int j = 0; j < TP; ++j) {
        const float2 xx = make_float2(x[j], x[j]);
#pragma unroll
        for (int i = 0; i < TM / 2; ++i) acc[i][j] = __ffma2_rn(xx, w[i], acc[i][j]);
    }
}

template <int TM, int TP, bool kWS>
__global__ void __launch_bounds__(TP == 4 ? 512 : 256)
f32_chain_kernel(const F32ChainParams p) {
    extern __shared__ __align__(16) float f32_smem[];
    const int T = blockDim.x;
    const int max_ih = (p.halo_h - 1) * p.stride + p.k;
    const int rp = p.pool_stride * p.hp, mp = p.halo_h * rp;      // pitches of a middle row and of a middle channel
    float *s_in = f32_smem;                                       // [C][max_ih][iwp]
    float *s_mid = s_in + p.C * max_ih * p.iwp;                   // [mpad][halo_h][pool_stride][hp]
    const int kper = p.K2 / p.parts_outc, kperp = (kper + 7) & ~7;
    float *s_b1 = s_mid + p.mpad * mp;                            // [mpad]
    float *s_b2 = s_b1 + p.mpad;                                  // [kperp], the part's slice
    float *s_w1 = s_b2 + kperp;                                   // [C][k][k][mpad]
    float *s_w2 = s_w1 + p.C * p.k * p.k * p.mpad;               // [Cmid][kperp], the part's slice
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (kWS) {
        const int n4 = p.C * p.k * p.k * p.mpad / 4;
        for (int i = threadIdx.x; i < n4; i += T) cp_async16_f32(s_w1 + 4 * i, p.w1 + 4 * i);
    }
    for (int i = threadIdx.x; i < p.mpad; i += T) s_b1[i] = i < p.Cmid ? __ldg(p.b1 + i) : 0.0f;
    const int total = p.N * p.parts_outc * p.tiles_h * p.tiles_w;
    struct Tile { int n, part, py0, px0, th, tw, rh, rw, ih; };
    auto tile_of = [&](int cta) {
        Tile t;
        const int tx = cta % p.tiles_w; cta /= p.tiles_w;
        const int ty = cta % p.tiles_h; cta /= p.tiles_h;
        t.part = cta % p.parts_outc; t.n = cta / p.parts_outc;
        // pool tile -> stage-1 patch -> input patch
        t.py0 = ty * p.tile_h; t.px0 = tx * p.tile_w;
        t.th = min(p.tile_h, p.PP - t.py0); t.tw = min(p.tile_w, p.PQ - t.px0);
        t.rh = (t.th - 1) * p.pool_stride + p.pool_k; t.rw = (t.tw - 1) * p.pool_stride + p.pool_k;
        t.ih = (t.rh - 1) * p.stride + p.k;
        return t;
    };
    // A tile's input patch: 8, 16 or 32 lanes along a row, as many rows of a (channel, row) walk at once as that leaves.  (With a
    // warp and two divisions per row the requests of a 32-channel patch of 8 x 40 took 11 thousand cycles, of a 16-channel one of
    // 4 x 8 4200.)  Small tiles ask for theirs as asynchronous copies, which travel with the weights (one 32 x 32 map 9.1 us when
    // this was chosen, by way of registers 9.9); a warp's 4-byte copies cost some 20 cycles each, 9200 for the larger patch, which large tiles
    // therefore load through registers, up to eight loads of a thread under way (75 x 75, batch 32: then 232 us, as copies 237).
    auto load_patch = [&](const Tile &t) {
        const int lr = p.iwp <= 8 ? 3 : p.iwp <= 16 ? 4 : 5, lanes = 1 << lr, rows = T >> lr;
        const int i0 = t.py0 * p.pool_stride * p.stride - p.pad, j0 = t.px0 * p.pool_stride * p.stride - p.pad;      // may be negative
        const float *img = p.x + (size_t)t.n * p.C * p.H * p.W;
        for (int b = threadIdx.x & (lanes - 1); b < p.iwp; b += 2 * lanes) {
            int a = threadIdx.x >> lr, c = 0;
            while (a >= t.ih) { a -= t.ih; ++c; }
            const bool in0 = (unsigned)(j0 + b) < (unsigned)p.W, in1 = (unsigned)(j0 + b + lanes) < (unsigned)p.W, two = b + lanes < p.iwp;
            while (TP == 1 && c < p.C) {
                const int gy = i0 + a;
                const bool row_in = (unsigned)gy < (unsigned)p.H;
                const float *src = img + ((size_t)c * p.H + (row_in ? gy : 0)) * p.W + j0 + b;
                float *dst = s_in + (c * max_ih + a) * p.iwp + b;
                cp_async4(dst, row_in && in0 ? src : p.x, row_in && in0);
                if (two) cp_async4(dst + lanes, row_in && in1 ? src + lanes : p.x, row_in && in1);
                a += rows;
                while (a >= t.ih) { a -= t.ih; ++c; }
            }
            while (TP != 1 && c < p.C) {
                float v[4][2];
                int d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int gy = i0 + a;
                    const bool row_in = c < p.C && (unsigned)gy < (unsigned)p.H;
                    const float *src = img + ((size_t)c * p.H + gy) * p.W + j0 + b;
                    v[i][0] = row_in && in0 ? __ldg(src) : 0.0f;
                    v[i][1] = row_in && in1 && two ? __ldg(src + lanes) : 0.0f;
                    d[i] = c < p.C ? (c * max_ih + a) * p.iwp + b : -1;
                    a += rows;
                    while (a >= t.ih) { a -= t.ih; ++c; }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (d[i] >= 0) {
                        s_in[d[i]] = v[i][0];
                        if (two) s_in[d[i] + lanes] = v[i][1];
                    }
            }
        }
    };
    int cur_part = -1;
    asm volatile("griddepcontrol.wait;" ::: "memory");      // (the image may be the predecessor's result)
    if ((int)blockIdx.x < total) load_patch(tile_of(blockIdx.x));
    for (int cta = blockIdx.x; cta < total; cta += gridDim.x) {
        const Tile tile = tile_of(cta);
        const int n = tile.n, part = tile.part, py0 = tile.py0, px0 = tile.px0, th = tile.th, tw = tile.tw, rh = tile.rh, rw = tile.rw;
        // (patches are filled ahead of this: binding refuses a plan whose largest tile does not fit)
        if (rh > p.halo_h || rw > p.halo_w || tile.ih > max_ih) {
            if (threadIdx.x == 0) atomicCAS(p.status, 0u, 0x80000000u | 10u);
            asm volatile("cp.async.wait_all;" ::: "memory");
            return;
        }
        const float *w2 = p.w2 + (size_t)part * p.Cmid * kperp;
        if (part != cur_part) {
            cur_part = part;
            if (kWS) for (int i = threadIdx.x; i < p.Cmid * kperp / 4; i += T) cp_async16_f32(s_w2 + 4 * i, w2 + 4 * i);
            for (int i = threadIdx.x; i < kperp; i += T) s_b2[i] = i < kper ? __ldg(p.b2 + part * kper + i) : 0.0f;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // stage 1
        {
            const int gpr = (rw + TP - 1) / TP, npg = rh * gpr, units = npg * (p.mpad / TM);
            for (int u = threadIdx.x; u < units; u += T) {
                const int mg = u / npg, pg = u - mg * npg, a = pg / gpr, b = (pg - a * gpr) * TP;
                float2 acc[TM / 2][TP];
#pragma unroll
                for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                    for (int j = 0; j < TP; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
                const float *in0 = s_in + a * p.stride * p.iwp + b * p.stride;
                const float *wp = (kWS ? s_w1 : p.w1) + mg * TM;
                if (TP == 4 && p.k == 3 && p.stride == 1) {
                    for (int c = 0; c < p.C; ++c)
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            const float *row = in0 + (c * max_ih + r) * p.iwp;
                            const float4 x0 = *reinterpret_cast<const float4 *>(row);
                            const float2 x1 = *reinterpret_cast<const float2 *>(row + 4);
                            const float xs[6] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y};
#pragma unroll
                            for (int s = 0; s < 3; ++s) {
                                float2 w[TM / 2];
                                f32_load_w<TM>(w, wp);
                                wp += p.mpad;
                                f32_fma<TM, TP>(acc, w, xs + s);
                            }
                        }
                } else if (TP == 1 && p.k == 3) {
                    for (int c = 0; c < p.C; ++c) {
                        // (all of a channel's reads before its products: one warp per scheduler has nothing else to hide them)
                        float xs[9];
                        float2 w[9][TM / 2];
#pragma unroll
                        for (int t = 0; t < 9; ++t) {
                            xs[t] = in0[(c * max_ih + t / 3) * p.iwp + t % 3];
                            f32_load_w<TM>(w[t], wp + t * p.mpad);
                        }
#pragma unroll
                        for (int t = 0; t < 9; ++t) f32_fma<TM, TP>(acc, w[t], xs + t);
                        wp += 9 * p.mpad;
                    }
                } else {
                    for (int c = 0; c < p.C; ++c)
                        for (int r = 0; r < p.k; ++r) {
                            const float *row = in0 + (c * max_ih + r) * p.iwp;
#pragma unroll 3
                            for (int s = 0; s < p.k; ++s) {
                                float2 w[TM / 2];
                                float xs[TP];
                                f32_load_w<TM>(w, wp);
                                wp += p.mpad;
#pragma unroll
                                for (int j = 0; j < TP; ++j) xs[j] = row[s + j * p.stride];
                                f32_fma<TM, TP>(acc, w, xs);
                            }
                        }
                }
#pragma unroll
                for (int i = 0; i < TM / 2; ++i) {
                    const int m = mg * TM + 2 * i;
                    const float b0 = s_b1[m], b1 = s_b1[m + 1];
                    float *o = s_mid + m * mp + a * rp;
#pragma unroll
                    for (int j = 0; j < TP; ++j) {
                        const int x = b + j;
                        if (x >= rw) break;
                        const int q = p.pool_stride == 2 ? (x & 1) * p.hp + (x >> 1) : (x % p.pool_stride) * p.hp + x / p.pool_stride;
                        o[q] = apply_act(acc[i][j].x + b0, p.act1);
                        o[mp + q] = apply_act(acc[i][j].y + b1, p.act1);
                    }
                }
            }
        }
        __syncthreads();
        // (the patch is free from here on)
        if (cta + (int)gridDim.x < total) load_patch(tile_of(cta + gridDim.x));
        // stage 2 + pool
        if (p.pool_k == 2) {
            // a thread takes TM channels of one pool output: the window's four pixels are its pixel tile
            const int npg = th * tw, units = npg * (kperp / TM);
            for (int u = threadIdx.x; u < units; u += T) {
                const int kg = u / npg, pg = u - kg * npg, oy = pg / tw, ox = pg - oy * tw, kk0 = part * kper + kg * TM;
                const float *src[4];
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    const int dx = d & 1, sh = dx / p.pool_stride;
                    src[d] = s_mid + (oy * p.pool_stride + (d >> 1)) * rp + (dx - sh * p.pool_stride) * p.hp + sh + ox;
                }
                const float *wp = (kWS ? s_w2 : w2) + kg * TM;
                float2 acc[TM / 2][4];
#pragma unroll
                for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                    for (int d = 0; d < 4; ++d) acc[i][d] = make_float2(0.0f, 0.0f);
                int m = 0;
                // (the reads of several channels before their products, as in stage 1)
                constexpr int kAhead = TP == 1 ? 8 : 2;
                for (; m + kAhead <= p.Cmid; m += kAhead) {
                    float2 w[kAhead][TM / 2];
                    float xs[kAhead][4];
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) {
                        f32_load_w<TM>(w[i], wp + i * kperp);
#pragma unroll
                        for (int d = 0; d < 4; ++d) { xs[i][d] = *src[d]; src[d] += mp; }
                    }
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) f32_fma<TM, 4>(acc, w[i], xs[i]);
                    wp += kAhead * kperp;
                }
#pragma unroll 1
                for (; m < p.Cmid; ++m) {
                    float2 w[TM / 2];
                    float xs[4];
                    f32_load_w<TM>(w, wp);
                    wp += kperp;
#pragma unroll
                    for (int d = 0; d < 4; ++d) { xs[d] = *src[d]; src[d] += mp; }
                    f32_fma<TM, 4>(acc, w, xs);
                }
#pragma unroll
                for (int i = 0; i < TM / 2; ++i) {
                    const int kl = kg * TM + 2 * i;
                    const float bx = s_b2[kl], by = s_b2[kl + 1];
                    const float pool0 = p.pool_kind == 0 ? -INFINITY : 0.0f;
                    float2 res = make_float2(pool0, pool0);
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const float vx = apply_act(acc[i][d].x + bx, p.act2), vy = apply_act(acc[i][d].y + by, p.act2);
                        res.x = p.pool_kind == 0 ? fmaxf(res.x, vx) : res.x + vx;
                        res.y = p.pool_kind == 0 ? fmaxf(res.y, vy) : res.y + vy;
                    }
                    if (p.pool_kind != 0) { res.x /= 4.0f; res.y /= 4.0f; }
                    const size_t oi = (((size_t)n * p.K2 + kk0 + 2 * i) * p.PP + (py0 + oy)) * p.PQ + (px0 + ox);
                    if (kl < kper) p.y[oi] = res.x;
                    if (kl + 1 < kper) p.y[oi + (size_t)p.PP * p.PQ] = res.y;
                }
            }
        } else {
            const int gpr = (tw + TP - 1) / TP, npg = th * gpr, units = npg * (kperp / TM);
            for (int u = threadIdx.x; u < units; u += T) {
                const int kg = u / npg, pg = u - kg * npg, oy = pg / gpr, ox = (pg - oy * gpr) * TP;
                const int kk0 = part * kper + kg * TM;
                const bool is_max = p.pool_kind == 0;
                const float pool0 = is_max ? -INFINITY : 0.0f;
                float2 res[TM / 2][TP], bias[TM / 2];
#pragma unroll
                for (int i = 0; i < TM / 2; ++i) {
                    bias[i] = make_float2(s_b2[kg * TM + 2 * i], s_b2[kg * TM + 2 * i + 1]);
#pragma unroll
                    for (int j = 0; j < TP; ++j) res[i][j] = make_float2(pool0, pool0);
                }
                for (int dy = 0; dy < p.pool_k; ++dy)
                    for (int dx = 0; dx < p.pool_k; ++dx) {
                        const int sh = dx / p.pool_stride;
                        const float *src = s_mid + (oy * p.pool_stride + dy) * rp + (dx - sh * p.pool_stride) * p.hp + sh + ox;
                        const float *wp = (kWS ? s_w2 : w2) + kg * TM;
                        float2 acc[TM / 2][TP];
#pragma unroll
                        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                            for (int j = 0; j < TP; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
                        if (TP == 4 && sh == 0) {
#pragma unroll 4
                            for (int m = 0; m < p.Cmid; ++m) {
                                float2 w[TM / 2];
                                f32_load_w<TM>(w, wp);
                                wp += kperp;
                                const float4 x4 = *reinterpret_cast<const float4 *>(src + m * mp);
                                const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
                                f32_fma<TM, TP>(acc, w, xs);
                            }
                        } else {
#pragma unroll 4
                            for (int m = 0; m < p.Cmid; ++m) {
                                float2 w[TM / 2];
                                float xs[TP];
                                f32_load_w<TM>(w, wp);
                                wp += kperp;
#pragma unroll
                                for (int j = 0; j < TP; ++j) xs[j] = src[m * mp + j];
                                f32_fma<TM, TP>(acc, w, xs);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                            for (int j = 0; j < TP; ++j) {
                                const float vx = apply_act(acc[i][j].x + bias[i].x, p.act2), vy = apply_act(acc[i][j].y + bias[i].y, p.act2);
                                res[i][j].x = is_max ? fmaxf(res[i][j].x, vx) : res[i][j].x + vx;
                                res[i][j].y = is_max ? fmaxf(res[i][j].y, vy) : res[i][j].y + vy;
                            }
                    }
                const float area = (float)(p.pool_k * p.pool_k);
#pragma unroll
                for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                    for (int j = 0; j < TP; ++j) {
                        if (ox + j >= tw) break;
                        const int kl = kg * TM + 2 * i;
                        const size_t oi = (((size_t)n * p.K2 + kk0 + 2 * i) * p.PP + (py0 + oy)) * p.PQ + (px0 + ox + j);
                        if (kl < kper) p.y[oi] = is_max ? res[i][j].x : res[i][j].x / area;
                        if (kl + 1 < kper) p.y[oi + (size_t)p.PP * p.PQ] = is_max ? res[i][j].y : res[i][j].y / area;
                    }
            }
        }
        __syncthreads();      // the patch and the middle map are rewritten for the next tile
    }
}

}  // namespace xk
