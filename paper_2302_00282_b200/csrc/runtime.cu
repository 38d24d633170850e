// CUDA runtime of the library: uploads the packed parameters into the caller's workspace,
// encodes the TMA descriptors, and enqueues one kernel per launch record on the caller's stream.
// Allocates no device memory of its own (the driver keeps some for the pass that a binding records).  (Section 3 of the Xenos paper: the runtime executes the optimised
// model on the parallel units on top of the operator library.)
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "chain2_tc.cuh"
#include "conv_tc.cuh"
#include "stem_tc.cuh"
#include "dw_tc.cuh"
#include "gemm_tc.cuh"
#include "graph.hpp"
#include "kernels_bf16.cuh"
#include "kernels_f32.cuh"
#include "pair_tc.cuh"

namespace xenos {

struct ConvMaps { CUtensorMap a0, a1, o, s; };      // operand segments, result, shortcut of a conv_tc_kernel launch

struct Runtime {
    // The pass as a CUDA graph (null: launches go to the stream one by one), its kernel nodes in launch order, the batch whose
    // grids they hold and the batch of the last call.
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;        // what exec was made of: its nodes name those of exec
    std::vector<cudaGraphNode_t> nodes;
    int exec_batch = 0, last_batch = 0;
    std::mutex exec_mutex;              // a call points the nodes at its buffers and launches them
    ~Runtime() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
    int device = -1;
    int sm_count = 0;
    int optin = 0;                      // shared memory a block may ask for
    std::vector<CUtensorMap> tmaps;     // one per launch record (used by gemm launches only)
    std::vector<CUtensorMap> hmaps;     // halo maps of linked depthwise stages / activation operand maps
    std::vector<CUtensorMap> tmaps2;    // second weight matrix of two linked convolutions
    std::vector<ConvMaps> conv;
    PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    PFN_cuTensorMapEncodeIm2col_v12000 encode_im2col = nullptr;
};

static xenos_status_t cuda_fail(const Graph &g, const char *what, cudaError_t e) {
    return fail(g, XENOS_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

static uint32_t make_idesc(int tile_n) {
    // kind::f16 instruction descriptor: fp32 accumulator, bf16 A and B, both K-major, M = 128
    uint32_t d = 0;
    d |= 1u << 4;                       // D format f32
    d |= 1u << 7;                       // A format bf16
    d |= 1u << 10;                      // B format bf16
    d |= (uint32_t)(tile_n >> 3) << 17; // N / 8
    d |= (uint32_t)(128 >> 4) << 24;    // M / 16
    return d;
}

// 4-D map (C, W, H, N) over the NHWC bf16 input of a linked depthwise stage; box = one halo tile.
// Out-of-range coordinates read zeros, which is the convolution's zero padding.
// `images` is the extent of the outermost dimension: boxes that reach past it (the last image group of
// an odd batch) read zeros there and never touch memory behind the buffer.
static xenos_status_t encode_halo_map(const Graph &g, Runtime *rt, const Launch &L, void *base, int images, CUtensorMap *out) {
    const ASeg &a = L.seg[0];
    cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)images};
    cuuint64_t strides[3] = {(cuuint64_t)a.C * 2, (cuuint64_t)a.W * a.C * 2, (cuuint64_t)a.H * a.W * a.C * 2};
    cuuint32_t box[4] = {(cuuint32_t)L.halo_cb, (cuuint32_t)L.halo_w, (cuuint32_t)L.halo_h, (cuuint32_t)L.ni};
    cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
    if (((uintptr_t)base & 15u) || (strides[0] & 15u) || (box[0] * 2u) % 16u || box[1] > 256u || box[2] > 256u || box[3] > 256u)
        return fail(g, XENOS_E_CUDA, "depthwise input is not 16-byte aligned or its halo tile exceeds the TMA box limits");
    CUresult r = rt->encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled (halo) failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

// ---- maps of conv_tc_kernel ------------------------------------------------------------------------------------------
static CUtensorMapSwizzle swizzle_of(int cols) {
    return cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}
static bool conv_seg_im2col(const ASeg &a) { return !(a.k == 1 && a.stride == 1 && a.pad == 0); }

// Rows of a dense [rows][C] bf16 matrix in boxes of `rows_box` x `cols`, swizzled by the box's width.
static xenos_status_t encode_rows_map(const Graph &g, Runtime *rt, void *base, int C, long long rows, int cols, int rows_box, CUtensorMap *out) {
    cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)C * 2};
    cuuint32_t box[2] = {(cuuint32_t)cols, (cuuint32_t)rows_box};
    cuuint32_t estr[2] = {1u, 1u};
    if (((uintptr_t)base & 15u) || C % 8 || rows_box > 256) return fail(g, XENOS_E_CUDA, "internal: a matrix is not addressable by TMA");
    CUresult r = rt->encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            swizzle_of(cols), CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled (rows) failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

// One segment of the activation operand: matrix rows, or the im2col walk over the window origins of an NHWC tensor
// (bounding box from -pad to the last window origin, traversed with the convolution's stride; padding reads zeros).
static xenos_status_t encode_conv_a(const Graph &g, Runtime *rt, const Launch &L, const ASeg &a, void *base, int images, CUtensorMap *out) {
    if (!conv_seg_im2col(a)) return encode_rows_map(g, rt, base, a.C, (long long)images * a.H * a.W, a.cbox, L.a_rows, out);
    const int hi = a.pad - (a.k - 1);
    cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)images};
    cuuint64_t strides[3] = {(cuuint64_t)a.C * 2, (cuuint64_t)a.W * a.C * 2, (cuuint64_t)a.H * a.W * a.C * 2};
    int lower[2] = {-a.pad, -a.pad}, upper[2] = {hi, hi};
    cuuint32_t estr[4] = {1u, (cuuint32_t)a.stride, (cuuint32_t)a.stride, 1u};
    if (((uintptr_t)base & 15u) || a.C % 8 || a.pad > 127 || hi < -127 || a.stride > 8)
        return fail(g, XENOS_E_UNSUPPORTED, "a convolution window, stride or padding exceeds the copy engine's im2col limits");
    CUresult r = rt->encode_im2col(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, lower, upper, (cuuint32_t)a.cbox,
                                   (cuuint32_t)L.a_rows, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(a.cbox),
                                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeIm2col failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

// The maps of a launch whose tensors sit where `ptr` says; `want_external` selects those on caller buffers (run time, for
// the batch at hand) or those on the workspace (bind time, for max_batch images).
template <class Ptr>
static xenos_status_t encode_conv_maps(const Graph &g, Runtime *rt, const Launch &L, Ptr ptr, int images, bool want_external, ConvMaps *m) {
    auto external = [&](int t) { return g.tensors[t].input_slot >= 0 || g.tensors[t].output_slot >= 0; };
    const ASeg &a0 = L.seg[0], &a1 = L.seg[1];
    xenos_status_t st = XENOS_OK;
    if (external(a0.tensor) == want_external) st = encode_conv_a(g, rt, L, a0, ptr(a0.tensor), images, &m->a0);
    if (st == XENOS_OK && a1.mode != AM_NONE && external(a1.tensor) == want_external) st = encode_conv_a(g, rt, L, a1, ptr(a1.tensor), images, &m->a1);
    const long long rows = (long long)images * L.rows_per_image;
    if (st == XENOS_OK && (L.pair || L.cv_epi == xk::CE_STORE || L.cv_epi == xk::CE_SKIP) && external(L.out) == want_external)
        st = encode_rows_map(g, rt, ptr(L.out), L.out_ctot, rows, L.pair ? 32 : L.chunk, 32, &m->o);
    if (st == XENOS_OK && L.skip >= 0 && (L.pair || L.cv_epi == xk::CE_SKIP) && external(L.skip) == want_external)
        st = encode_rows_map(g, rt, ptr(L.skip), g.tensors[L.skip].c, rows, L.pair ? 32 : L.chunk, 32, &m->s);
    return st;
}
// Depthwise chains: input windows (a0) and result boxes (o: (channel, column, row, image) with a box of one tile).
template <class Ptr>
static xenos_status_t encode_dw_maps(const Graph &g, Runtime *rt, const Launch &L, Ptr ptr, int images, bool want_external, ConvMaps *m) {
    auto external = [&](int t) { return g.tensors[t].input_slot >= 0 || g.tensors[t].output_slot >= 0; };
    xenos_status_t st = XENOS_OK;
    if (external(L.seg[0].tensor) == want_external) st = encode_halo_map(g, rt, L, ptr(L.seg[0].tensor), images, &m->a0);
    if (st != XENOS_OK || L.cv_epi != xk::DE_STORE || external(L.out) != want_external) return st;
    void *base = ptr(L.out);
    const cuuint64_t C = (cuuint64_t)L.out_ctot, W = (cuuint64_t)L.Q, H = (cuuint64_t)L.P;
    cuuint64_t dims[4] = {C, W, H, (cuuint64_t)images}, strides[3] = {C * 2, W * C * 2, H * W * C * 2};
    cuuint32_t box[4] = {(cuuint32_t)L.chunk, (cuuint32_t)L.patch_rw, (cuuint32_t)L.patch_rh, (cuuint32_t)L.ni}, estr[4] = {1u, 1u, 1u, 1u};
    if (((uintptr_t)base & 15u) || (C & 7) || L.patch_rw * L.patch_rh * L.ni > 128) return fail(g, XENOS_E_CUDA, "internal: depthwise result tile violates the TMA limits");
    CUresult r = rt->encode(&m->o, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            swizzle_of(L.chunk), CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled (depthwise result) failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

static bool conv_has_external(const Graph &g, const Launch &L) {
    auto external = [&](int t) { return t >= 0 && (g.tensors[t].input_slot >= 0 || g.tensors[t].output_slot >= 0); };
    return external(L.seg[0].tensor) || (L.seg[1].mode != AM_NONE && external(L.seg[1].tensor)) || external(L.out) || external(L.skip);
}

// Whether a launch reads or writes a buffer that the caller names at run time.
static bool touches_caller(const Graph &g, const Launch &L) {
    auto external = [&](int t) { return t >= 0 && (g.tensors[t].input_slot >= 0 || g.tensors[t].output_slot >= 0); };
    return external(L.in0) || external(L.in1) || external(L.in2) || external(L.out) || external(L.skip) ||
           (L.seg[0].mode != AM_NONE && external(L.seg[0].tensor)) || (L.seg[1].mode != AM_NONE && external(L.seg[1].tensor));
}

static xk::ConvSegment conv_segment(const Launch &L, const ASeg &a) {
    xk::ConvSegment s;
    std::memset(&s, 0, sizeof s);
    if (a.mode == AM_NONE) { s.per_stage = 1; s.k = 1; s.cblocks = 1; s.spb = 4; return s; }
    s.im2col = conv_seg_im2col(a);
    s.k = a.k; s.stride = a.stride; s.low = -a.pad;
    s.taps = a.k * a.k;
    s.kblocks = a.kblocks;
    s.cblocks = a.cbox == 64 ? a.cpad / 64 : 1;
    s.last_steps = a.cbox == 64 ? (a.C - 64 * (s.cblocks - 1) + 15) / 16 : 4;
    s.per_stage = 64 / a.cbox;
    s.spb = a.cbox / 16;
    s.box_bytes = (uint32_t)(L.a_rows * a.cbox * 2);
    s.box_stride = (uint32_t)(128 * a.cbox * 2);
    // version bit, group stride (8 rows of the box), swizzle mode
    const uint32_t mode = a.cbox == 64 ? 2u : a.cbox == 32 ? 4u : 6u;
    s.desc_hi = (uint32_t)((8 * a.cbox * 2) >> 4) | (1u << 14) | (mode << 29);
    return s;
}

// Maps of two linked convolutions: the first one's input (C, W, H, N) with a box of the producer tile, and the two
// packed weight matrices.
static xenos_status_t encode_chain2_input(const Graph &g, Runtime *rt, const Launch &L, void *base, int images, CUtensorMap *out) {
    const ASeg &a = L.seg[0];
    if (((uintptr_t)base & 15u) || (a.C % 64)) return fail(g, XENOS_E_CUDA, "internal: activation operand is not addressable by TMA");
    cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)images};
    cuuint64_t strides[3] = {(cuuint64_t)a.C * 2, (cuuint64_t)a.W * a.C * 2, (cuuint64_t)a.H * a.W * a.C * 2};
    cuuint32_t box[4] = {64u, (cuuint32_t)L.patch_rw, (cuuint32_t)L.patch_rh, 1u};
    cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
    if (box[1] > 256u || box[2] > 256u || box[1] * box[2] > 128u) return fail(g, XENOS_E_CUDA, "internal: producer tile exceeds the TMA box limits");
    CUresult r = rt->encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled (linked convolutions) failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

static xenos_status_t encode_weight_map(const Graph &g, Runtime *rt, void *gaddr, int kpad, int rows, int box_rows, CUtensorMap *out) {
    cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)kpad * 2};
    cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1u, 1u};
    if (((uintptr_t)gaddr & 15u) || (strides[0] & 15u) || box[1] > 256u || box[1] == 0u || box_rows % 16)
        return fail(g, XENOS_E_CUDA, "internal: weight tensor map fields are misaligned");
    CUresult r = rt->encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, gaddr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

// 4-D map (W, H, C, N) over a small-channel NCHW image; box = one tile's input patch, all channels.
static xenos_status_t encode_stem_map(const Graph &g, Runtime *rt, const Launch &L, void *base, int images, CUtensorMap *out) {
    const ASeg &a = L.seg[0];
    const bool f32 = a.src_dtype == XENOS_DTYPE_F32;
    const cuuint64_t es = f32 ? 4 : 2;
    cuuint64_t dims[4] = {(cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.C, (cuuint64_t)images};
    cuuint64_t strides[3] = {(cuuint64_t)a.W * es, (cuuint64_t)a.H * a.W * es, (cuuint64_t)a.C * a.H * a.W * es};
    cuuint32_t box[4] = {(cuuint32_t)L.halo_w, (cuuint32_t)L.halo_h, (cuuint32_t)a.C, 1u};
    cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
    if ((strides[0] & 15u) || (strides[1] & 15u) || (strides[2] & 15u) || (box[0] * es) % 16u || box[0] > 256u || box[1] > 256u || box[2] > 256u)
        return fail(g, XENOS_E_CUDA, "internal: stem image patch violates the TMA limits");
    CUresult r = rt->encode(out, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled (stem) failed with code " + std::to_string((int)r));
    return XENOS_OK;
}

typedef void (*DwKernel)(CUtensorMap, CUtensorMap, CUtensorMap, xk::DwParams);
template <int kEpi, int kCB>
static DwKernel dw_kernel_of(int stride, int br) {
    if (stride == 1) return br == 4 ? xk::dw_tc_kernel<kEpi, 1, 4, kCB> : br == 2 ? xk::dw_tc_kernel<kEpi, 1, 2, kCB> : xk::dw_tc_kernel<kEpi, 1, 1, kCB>;
    return br == 4 ? xk::dw_tc_kernel<kEpi, 2, 4, kCB> : br == 2 ? xk::dw_tc_kernel<kEpi, 2, 2, kCB> : xk::dw_tc_kernel<kEpi, 2, 1, kCB>;
}
// Convolution of an image: how its rows are loaded, the image's type, with or without a pool.
using StemKernel = void (*)(xk::StemParams);
template <int kMode, bool kRows>
static StemKernel stem_kernel_of(bool f32, bool pool) {
    return f32 ? (pool ? xk::stem_tc_kernel<kMode, true, true, kRows> : xk::stem_tc_kernel<kMode, true, false, kRows>)
               : (pool ? xk::stem_tc_kernel<kMode, false, true, kRows> : xk::stem_tc_kernel<kMode, false, false, kRows>);
}
static StemKernel stem_kernel(int mode, bool f32, bool pool, bool rows) {
    if (rows) return mode == xk::SM_S1 ? stem_kernel_of<xk::SM_S1, true>(f32, pool) : stem_kernel_of<xk::SM_S2, true>(f32, pool);
    return mode == xk::SM_S1 ? stem_kernel_of<xk::SM_S1, false>(f32, pool) : mode == xk::SM_S2 ? stem_kernel_of<xk::SM_S2, false>(f32, pool)
         : mode == xk::SM_S2X ? stem_kernel_of<xk::SM_S2X, false>(f32, pool) : stem_kernel_of<xk::SM_ANY, false>(f32, pool);
}

// Whole groups of elements where rows are made of them (images are 16-byte aligned); else element by element.
static StemKernel stem_kernel(const Launch &L) {
    const int mode = L.stride == 2 ? (L.st_vec ? xk::SM_S2 : xk::SM_S2X) : L.stride == 1 ? xk::SM_S1 : xk::SM_ANY;
    return stem_kernel(mode, L.seg[0].src_dtype == XENOS_DTYPE_F32, L.epi == EPI_POOL, L.st_raw > 0);
}

static auto *conv_kernel(const Launch &L) {
    return L.cv_epi == xk::CE_STORE ? xk::conv_tc_kernel<xk::CE_STORE> : L.cv_epi == xk::CE_SKIP ? xk::conv_tc_kernel<xk::CE_SKIP>
         : L.cv_epi == xk::CE_VEC ? xk::conv_tc_kernel<xk::CE_VEC> : L.cv_epi == xk::CE_GAP ? xk::conv_tc_kernel<xk::CE_GAP>
         : L.cv_epi == xk::CE_CLUSTER ? xk::conv_tc_kernel<xk::CE_CLUSTER> : xk::conv_tc_kernel<xk::CE_SPLIT>;
}

static auto *f32_chain_kernel(const Launch &L) {
    return L.f32_big ? (L.f32_ws ? xk::f32_chain_kernel<8, 4, true> : xk::f32_chain_kernel<8, 4, false>)
                     : (L.f32_ws ? xk::f32_chain_kernel<2, 1, true> : xk::f32_chain_kernel<2, 1, false>);
}

static DwKernel dw_kernel(int epi, int stride, int br, int cb) {
    if (epi == xk::DE_STORE)
        return cb == 64 ? dw_kernel_of<xk::DE_STORE, 64>(stride, br) : cb == 32 ? dw_kernel_of<xk::DE_STORE, 32>(stride, br) : dw_kernel_of<xk::DE_STORE, 0>(stride, br);
    return epi == xk::DE_GAP ? dw_kernel_of<xk::DE_GAP, 0>(stride, br) : dw_kernel_of<xk::DE_SPLIT, 0>(stride, br);
}

// Where launch_pass hands its kernels: to a stream, to the node of a recorded pass that holds the launch, or nowhere (the
// kernels of a graph are only made ready to run).
struct Issue {
    enum Mode { LAUNCH, POINT, READY } mode = LAUNCH;
    cudaStream_t stream = nullptr;
    Runtime *rt = nullptr;
    bool external_only = false;         // POINT: only launches that read or write the caller's buffers
    int optin = 0;                      // READY: shared memory a block may ask for
    size_t li = 0;                      // the launch at hand

    // Programmatic dependent launch: the kernel may be scheduled while its predecessor in the stream drains, runs its set-up
    // and then waits (griddepcontrol.wait) before it touches the predecessor's results.
    template <class... P, class... A>
    cudaError_t pdl(void (*kernel)(P...), dim3 grid, int block, int smem, A &&...args) const {
        return put(kernel, grid, dim3((unsigned)block), smem, 1, true, std::forward<A>(args)...);
    }
    template <class... P, class... A>
    cudaError_t pdl_cluster(void (*kernel)(P...), dim3 grid, int block, int smem, int cluster, A &&...args) const {
        return put(kernel, grid, dim3((unsigned)block), smem, cluster, true, std::forward<A>(args)...);
    }
    template <class... P, class... A>
    cudaError_t plain(void (*kernel)(P...), dim3 grid, dim3 block, int smem, A &&...args) const {
        return put(kernel, grid, block, smem, 1, false, std::forward<A>(args)...);
    }

private:
    template <class... P, class... A>
    cudaError_t put(void (*kernel)(P...), dim3 grid, dim3 block, int smem, int cluster, bool programmatic, A &&...args) const {
        return [&](P... exact) {
            void *argv[] = {&exact...};
            return issue(reinterpret_cast<const void *>(kernel), grid, block, smem, cluster, programmatic, argv);
        }(std::forward<A>(args)...);
    }
    cudaError_t issue(const void *kernel, dim3 grid, dim3 block, int smem, int cluster, bool programmatic, void **argv) const {
        if (mode == READY) {
            // the first mention of a kernel loads its code.  The opt-in limit is a per-function, per-device setting shared by
            // every graph in the process: always the device's maximum, so that binding one graph never lowers it for another.
            cudaFuncAttributes at;
            return smem > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) : cudaFuncGetAttributes(&at, kernel);
        }
        if (mode == POINT) {
            cudaKernelNodeParams p = {};
            p.func = const_cast<void *>(kernel); p.gridDim = grid; p.blockDim = block; p.sharedMemBytes = (unsigned)smem; p.kernelParams = argv;
            return cudaGraphExecKernelNodeSetParams(rt->exec, rt->nodes[li], &p);
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid; cfg.blockDim = block;
        cfg.dynamicSmemBytes = (size_t)smem; cfg.stream = stream;
        cudaLaunchAttribute at[2];
        unsigned n = 0;
        if (programmatic) {
            at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[n++].val.programmaticStreamSerializationAllowed = 1;
        }
        if (cluster > 1) {
            at[n].id = cudaLaunchAttributeClusterDimension;
            at[n].val.clusterDim.x = (unsigned)cluster; at[n].val.clusterDim.y = 1; at[n++].val.clusterDim.z = 1;
        }
        cfg.attrs = at; cfg.numAttrs = n;
        return cudaLaunchKernelExC(&cfg, kernel, argv);
    }
};

void runtime_free(Graph &g) {
    delete static_cast<Runtime *>(g.rt);
    g.rt = nullptr;
}

// Uploads the parameters and encodes the maps of what lies in the workspace.
static xenos_status_t attach(Graph &g, void *ws, void *stream_v) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(g, "no CUDA device (this library has no CPU fallback)", e);
    // (single attributes: the whole property record takes 2.8 ms, several times the rest of a binding)
    int major = 0, sms = 0, optin = 0;
    if ((e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess)
        return cuda_fail(g, "cudaDeviceGetAttribute", e);
    if (major != 10) return fail(g, XENOS_E_CUDA, "device is not sm_100 (B200); the kernels are built for sm_100a only");
    runtime_free(g);
    Runtime *rt = new Runtime();
    g.rt = rt;
    rt->device = dev;
    rt->sm_count = sms;
    rt->optin = optin;
    // parameters -> workspace, status words cleared
    if (!g.param_blob.empty())
        if ((e = cudaMemcpyAsync(ws, g.param_blob.data(), g.param_blob.size(), cudaMemcpyHostToDevice, stream)) != cudaSuccess)
            return cuda_fail(g, "parameter upload", e);
    if ((e = cudaMemsetAsync(static_cast<uint8_t *>(ws) + g.status_off, 0, 256 + g.cnt_bytes, stream)) != cudaSuccess)
        return cuda_fail(g, "status clear", e);
    if ((e = cudaStreamSynchronize(stream)) != cudaSuccess) return cuda_fail(g, "parameter upload sync", e);
    g.ws = ws;
    // TMA descriptors of the packed weight matrices
    bool any_gemm = false;
    int max_gemm_smem = 0, max_chain_smem = 0;
    for (const Launch &L : g.launches) {
        if (L.kind == LK_GEMM2) { any_gemm = true; max_gemm_smem = std::max(max_gemm_smem, L.smem_bytes); }
        if (L.kind == LK_GEMM) { any_gemm = true; max_gemm_smem = std::max(max_gemm_smem, L.smem_bytes); }
        if (L.kind == LK_F32_CONV_CONV_POOL) {
            max_chain_smem = std::max(max_chain_smem, L.smem_bytes);
            // (the kernel fills a tile's patch before it looks at the tile's extents)
            if ((L.tile_h - 1) * L.pool_stride + L.pool_k > L.halo_h || (L.tile_w - 1) * L.pool_stride + L.pool_k > L.halo_w)
                return fail(g, XENOS_E_BAD_SPLIT, "internal: a tile's patch exceeds its place in shared memory");
        }
    }
    rt->tmaps.resize(g.launches.size());
    rt->hmaps.resize(g.launches.size());
    rt->tmaps2.resize(g.launches.size());
    rt->conv.resize(g.launches.size());
    std::memset(rt->conv.data(), 0, rt->conv.size() * sizeof(ConvMaps));
    if (any_gemm) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
        if (e != cudaSuccess || !fn || qres != cudaDriverEntryPointSuccess)
            return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
        rt->encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
        e = cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &fn, cudaEnableDefault, &qres);
        if (e != cudaSuccess || !fn || qres != cudaDriverEntryPointSuccess)
            return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeIm2col is not available from the driver");
        rt->encode_im2col = reinterpret_cast<PFN_cuTensorMapEncodeIm2col_v12000>(fn);
        for (size_t i = 0; i < g.launches.size(); ++i) {
            const Launch &L = g.launches[i];
            if (L.kind == LK_GEMM2 && L.pair) {
                xenos_status_t st = encode_weight_map(g, rt, static_cast<uint8_t *>(ws) + L.w_off, L.kblocks * 64, L.n1pad, std::min(128, L.n1pad), &rt->tmaps[i]);
                if (st == XENOS_OK) st = encode_weight_map(g, rt, static_cast<uint8_t *>(ws) + L.w2_off, L.kblocks2 * 64, L.npad, 128, &rt->tmaps2[i]);
                if (st == XENOS_OK) st = encode_conv_maps(g, rt, L, [&](int t) -> void * { return static_cast<uint8_t *>(ws) + g.place[t].off; }, g.max_batch, false, &rt->conv[i]);
                if (st != XENOS_OK) return st;
                continue;
            }
            if (L.kind == LK_GEMM2) {
                xenos_status_t st = encode_weight_map(g, rt, static_cast<uint8_t *>(ws) + L.w_off, L.kblocks * 64, L.n1pad, L.n1pad, &rt->tmaps[i]);
                if (st == XENOS_OK) st = encode_weight_map(g, rt, static_cast<uint8_t *>(ws) + L.w2_off, L.kblocks2 * 64, L.npad, L.tile_n, &rt->tmaps2[i]);
                if (st == XENOS_OK && g.tensors[L.in0].input_slot < 0)
                    st = encode_chain2_input(g, rt, L, static_cast<uint8_t *>(ws) + g.place[L.in0].off, g.max_batch, &rt->hmaps[i]);
                if (st != XENOS_OK) return st;
                continue;
            }
            if (L.kind != LK_GEMM || L.stem_tc) continue;
            cuuint64_t dims[2] = {(cuuint64_t)L.kpad, (cuuint64_t)L.npad};
            cuuint64_t strides[1] = {(cuuint64_t)L.kpad * 2};
            cuuint32_t box[2] = {64u, (cuuint32_t)L.tile_n};
            cuuint32_t estr[2] = {1u, 1u};
            void *gaddr = static_cast<uint8_t *>(ws) + L.w_off;
            // host-side validation of every field the encoder or the copy engine would reject
            if (((uintptr_t)gaddr & 15u) || (strides[0] & 15u) || box[1] > 256u || box[1] == 0u || L.tile_n % 16)
                return fail(g, XENOS_E_CUDA, "internal: weight tensor map fields are misaligned");
            CUresult r = rt->encode(&rt->tmaps[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, gaddr, dims, strides, box, estr,
                                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return fail(g, XENOS_E_CUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
            if (L.conv_tc) {
                if (L.fc_small) continue;
                xenos_status_t st = encode_conv_maps(g, rt, L, [&](int t) -> void * { return static_cast<uint8_t *>(ws) + g.place[t].off; }, g.max_batch, false, &rt->conv[i]);
                if (st != XENOS_OK) return st;
                continue;
            }
            if (L.seg[0].mode == AM_DW) {
                xenos_status_t st = encode_dw_maps(g, rt, L, [&](int t) -> void * { return static_cast<uint8_t *>(ws) + g.place[t].off; }, g.max_batch, false, &rt->conv[i]);
                if (st != XENOS_OK) return st;
            }
        }
    }
    if (max_gemm_smem > optin || max_chain_smem > optin)
        return fail(g, XENOS_E_CUDA, "a kernel of this plan needs more shared memory than the device offers");
    return XENOS_OK;
}

static int ew_grid(long long total, int block, int sms) {
    long long b = (total + block - 1) / block;
    long long cap = (long long)sms * 16;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

// The kernels of one pass, in order; each(li) is called behind launch li.
template <class Each>
static xenos_status_t issue_pass(Graph &g, int batch, const void *const *in, void *const *out, Issue to, Each each) {
    Runtime *rt = static_cast<Runtime *>(g.rt);
    uint8_t *ws = static_cast<uint8_t *>(g.ws);
    unsigned int *status = reinterpret_cast<unsigned int *>(ws + g.status_off);
    auto ptr = [&](int t) -> void * {
        if (t < 0) return nullptr;
        const Tensor &x = g.tensors[t];
        if (x.input_slot >= 0) return const_cast<void *>(in[x.input_slot]);
        if (x.output_slot >= 0) return out[x.output_slot];
        return ws + g.place[t].off;
    };
    const int sms = rt->sm_count;
    for (size_t li = 0; li < g.launches.size(); ++li) {
        const Launch &L = g.launches[li];
        const int N = batch;
        if (to.external_only && !touches_caller(g, L)) continue;
        to.li = li;
        cudaError_t le = cudaSuccess;
        switch (L.kind) {
        case LK_F32_CONV: {
            long long total = (long long)N * L.K * L.P * L.Q;
            le = to.plain(xk::f32_conv_kernel, ew_grid(total, 256, sms), 256, 0,
                (const float *)ptr(L.in0), (const float *)(ws + L.w_off), (const float *)(ws + L.b_off), (float *)ptr(L.out),
                N, L.C, L.H, L.W, L.K, L.P, L.Q, L.k, L.stride, L.pad, L.groups, L.act);
            break;
        }
        case LK_F32_POOL: {
            long long total = (long long)N * L.C * L.P * L.Q;
            le = to.plain(xk::f32_pool_kernel, ew_grid(total, 256, sms), 256, 0,
                (const float *)ptr(L.in0), (float *)ptr(L.out), N, L.C, L.H, L.W, L.P, L.Q, L.pool_k, L.pool_stride, L.pool_pad, L.pool_kind);
            break;
        }
        case LK_F32_GAP: {
            long long warps = (long long)N * L.C;
            le = to.plain(xk::f32_gap_kernel, (int)((warps * 32 + 255) / 256), 256, 0, (const float *)ptr(L.in0), (float *)ptr(L.out), N * L.C, L.H * L.W);
            break;
        }
        case LK_F32_ADD: {
            const Tensor &t = g.tensors[L.out];
            long long total = (long long)N * (t.is_vec ? t.c : t.c * t.h * t.w);
            le = to.plain(xk::f32_add_kernel, ew_grid(total, 256, sms), 256, 0, (const float *)ptr(L.in0), (const float *)ptr(L.in1), (float *)ptr(L.out), total, L.act);
            break;
        }
        case LK_F32_CONCAT_PART: {
            long long total = (long long)N * L.C * L.H * L.W;
            le = to.plain(xk::f32_concat_part_kernel, ew_grid(total, 256, sms), 256, 0, (const float *)ptr(L.in0), (float *)ptr(L.out), N, L.C, L.H * L.W, L.out_ctot, L.out_coff);
            break;
        }
        case LK_F32_FC:
            le = to.plain(xk::f32_fc_kernel, (N * L.K + 255) / 256, 256, 0, (const float *)ptr(L.in0), (const float *)(ws + L.w_off), (const float *)(ws + L.b_off), (float *)ptr(L.out), N, L.C, L.K, L.act);
            break;
        case LK_F32_CONV_CONV_POOL: {
            xk::F32ChainParams p;
            p.x = (const float *)ptr(L.in0); p.y = (float *)ptr(L.out);
            p.w1 = (const float *)(ws + L.w_off); p.b1 = (const float *)(ws + L.b_off);
            p.w2 = (const float *)(ws + L.w2_off); p.b2 = (const float *)(ws + L.b2_off);
            p.N = N; p.C = L.C; p.H = L.H; p.W = L.W; p.Cmid = L.Cmid; p.mpad = L.npad; p.P = L.P; p.Q = L.Q;
            p.k = L.k; p.stride = L.stride; p.pad = L.pad; p.act1 = L.act; p.K2 = L.K2; p.act2 = L.act2;
            p.pool_kind = L.pool_kind; p.pool_k = L.pool_k; p.pool_stride = L.pool_stride; p.PP = L.PP; p.PQ = L.PQ;
            p.parts_outc = L.parts_outc; p.tile_h = L.tile_h; p.tile_w = L.tile_w; p.tiles_h = L.tiles_h; p.tiles_w = L.tiles_w;
            p.halo_h = L.halo_h; p.halo_w = L.halo_w; p.iwp = L.f32_iwp; p.hp = L.f32_hp; p.status = status;
            // a CTA keeps its weights and walks over tiles when there are more tiles than resident CTAs
            const int occ = std::max(1, std::min(2048 / L.block, (228 * 1024) / (L.smem_bytes + 1024)));
            const int grid = (int)std::min<long long>((long long)N * L.grid, (long long)sms * occ);
            le = to.pdl(f32_chain_kernel(L), grid, L.block, L.smem_bytes, p);
            break;
        }
        case LK_STEM3X3: {
            const int grid = N * L.grid;
            if (L.seg[0].src_dtype == XENOS_DTYPE_F32)
                le = to.plain(xk::stem3x3_kernel<float>, grid, 256, L.smem_bytes, (const float *)ptr(L.in0), (const float *)(ws + L.w_off), (const float *)(ws + L.b_off),
                    (__nv_bfloat16 *)ptr(L.out), N, L.C, L.H, L.W, L.K, L.P, L.Q, L.stride, L.pad, L.act);
            else
                le = to.plain(xk::stem3x3_kernel<__nv_bfloat16>, grid, 256, L.smem_bytes, (const __nv_bfloat16 *)ptr(L.in0), (const float *)(ws + L.w_off), (const float *)(ws + L.b_off),
                    (__nv_bfloat16 *)ptr(L.out), N, L.C, L.H, L.W, L.K, L.P, L.Q, L.stride, L.pad, L.act);
            break;
        }
        case LK_DW: {
            long long total = (long long)N * L.P * L.Q * (L.C / 8);
            le = to.plain(xk::dw3x3_kernel, ew_grid(total, 256, sms), 256, 0,
                (const __nv_bfloat16 *)ptr(L.in0), (const float *)(ws + L.w_off), (const float *)(ws + L.b_off),
                (__nv_bfloat16 *)ptr(L.out), N, L.C, L.H, L.W, L.P, L.Q, L.stride, L.pad, L.act);
            break;
        }
        case LK_POOL: {
            long long total = (long long)N * L.P * L.Q * (L.C / 8);
            const bool small = L.pool_kind == 0 && L.pool_k <= 3 && total < (1ll << 31);
            // four outputs a thread where that still fills the device
            const int rows = total >= 4ll * 1024 * sms ? 4 : 1, bands = (L.P + rows - 1) / rows;
            const int items = (int)(small ? (long long)N * bands * L.Q * (L.C / 8) : 0);
            const __nv_bfloat16 *x = (const __nv_bfloat16 *)ptr(L.in0);
            __nv_bfloat16 *y = (__nv_bfloat16 *)ptr(L.out);
            le = small ? to.pdl(rows == 4 ? xk::maxpool_kernel<4> : xk::maxpool_kernel<1>, (items + 255) / 256, 256, 0, x, y, items, L.C / 8,
                                                L.H, L.W, L.P, L.Q, bands, L.pool_k, L.pool_stride, L.pool_pad)
                                   : to.pdl(xk::pool_kernel, ew_grid(total, 256, sms), 256, 0, x, y, N, L.C, L.H, L.W, L.P, L.Q, L.pool_k,
                                                L.pool_stride, L.pool_pad, L.pool_kind);
            break;
        }
        case LK_GAP: {
            le = to.pdl(xk::gap_kernel, dim3((L.C + 63) / 64, N), 256, 0, (const __nv_bfloat16 *)ptr(L.in0), ptr(L.out), L.C, L.H * L.W,
                                        L.out_dtype == XENOS_DTYPE_F32);
            break;
        }
        case LK_ADD: {
            const Tensor &t = g.tensors[L.out];
            long long n8 = (long long)N * (t.is_vec ? t.c : t.c * t.h * t.w) / 8;
            le = to.plain(xk::add_kernel, ew_grid(n8, 256, sms), 256, 0, (const __nv_bfloat16 *)ptr(L.in0), (const __nv_bfloat16 *)ptr(L.in1), (__nv_bfloat16 *)ptr(L.out), n8, L.act);
            break;
        }
        case LK_CONCAT_PART: {
            long long pixels = (long long)N * L.H * L.W;
            le = to.plain(xk::concat_part_kernel, ew_grid(pixels * (L.C / 8), 256, sms), 256, 0, (const __nv_bfloat16 *)ptr(L.in0), (__nv_bfloat16 *)ptr(L.out), pixels, L.C, L.out_ctot, L.out_coff);
            break;
        }
        case LK_MULMAC: {
            const Tensor &t = g.tensors[L.out];
            long long n8 = (long long)N * (t.is_vec ? t.c : t.c * t.h * t.w) / 8;
            le = to.plain(xk::mulmac_kernel, ew_grid(n8, 256, sms), 256, 0, (const __nv_bfloat16 *)ptr(L.in0), (const __nv_bfloat16 *)ptr(L.in1),
                                                                         (const __nv_bfloat16 *)ptr(L.in2), (__nv_bfloat16 *)ptr(L.out), n8);
            break;
        }
        case LK_F32_MULMAC: {
            const Tensor &t = g.tensors[L.out];
            long long total = (long long)N * (t.is_vec ? t.c : t.c * t.h * t.w);
            le = to.plain(xk::f32_mulmac_kernel, ew_grid(total, 256, sms), 256, 0, (const float *)ptr(L.in0), (const float *)ptr(L.in1),
                                                                                (const float *)ptr(L.in2), (float *)ptr(L.out), total);
            break;
        }
        case LK_TRANSPOSE:      // NHWC: per image [H rows][C columns] -> [C][H]
            le = to.plain(xk::transpose_kernel<__nv_bfloat16>, dim3((L.C + 31) / 32, (L.H + 31) / 32, N), dim3(32, 8), 0,
                (const __nv_bfloat16 *)ptr(L.in0), (__nv_bfloat16 *)ptr(L.out), L.H, L.C);
            break;
        case LK_F32_TRANSPOSE:  // NCHW: per image [C][H] -> [H][C]
            le = to.plain(xk::transpose_kernel<float>, dim3((L.H + 31) / 32, (L.C + 31) / 32, N), dim3(32, 8), 0,
                (const float *)ptr(L.in0), (float *)ptr(L.out), L.C, L.H);
            break;
        case LK_SLICE: {
            long long pixels = (long long)N * L.H * L.W;
            le = to.plain(xk::slice_kernel, ew_grid(pixels * (L.K / 8), 256, sms), 256, 0, (const __nv_bfloat16 *)ptr(L.in0), (__nv_bfloat16 *)ptr(L.out), pixels, L.K, L.C, L.out_coff);
            break;
        }
        case LK_F32_SLICE: {
            long long total = (long long)N * L.K * L.H * L.W;
            le = to.plain(xk::f32_slice_kernel, ew_grid(total, 256, sms), 256, 0, (const float *)ptr(L.in0), (float *)ptr(L.out), N, L.K, L.H * L.W, L.C, L.out_coff);
            break;
        }
        case LK_GEMM2: {
            if (L.pair) {
                xk::PairParams p;
                std::memset(&p, 0, sizeof p);
                p.seg = conv_segment(L, L.seg[0]);
                p.bias1 = (const float *)(ws + L.b_off); p.bias2 = (const float *)(ws + L.b2_off); p.status = status;
                p.rows = N * L.rows_per_image; p.tiles = (p.rows + 127) / 128;
                p.d_rpi = xk::make_fastdiv((uint32_t)L.rows_per_image); p.d_q = xk::make_fastdiv((uint32_t)L.Q);
                p.n1pad = L.n1pad; p.n1_slots = (L.n1pad + 127) / 128; p.kblocks2 = L.kblocks2; p.n2_blocks = L.n_tiles; p.npad2 = L.npad;
                p.a_slots = L.a_slots; p.b_slots = L.b_slots; p.s_slots = L.s_slots; p.resident = L.b_resident; p.dbl = L.n1pad <= 128;
                // (without a shortcut the two last clamps are one)
                p.act1 = L.act; p.act2 = L.skip >= 0 ? L.act2 : std::max(L.act2, L.act3); p.act3 = L.act3;
                p.idesc1 = make_idesc(std::min(128, L.n1pad)); p.idesc2 = make_idesc(128);
                p.off_b = L.off_b2; p.off_mid = L.off_mid; p.off_stage = L.off_stg; p.off_bias = L.off_bias; p.off_bar = L.off_bar;
                p.launch_id = (int)li;
                const ConvMaps *maps = &rt->conv[li];
                ConvMaps now;
                if (conv_has_external(g, L)) {
                    now = *maps;
                    xenos_status_t st = encode_conv_maps(g, rt, L, ptr, N, true, &now);
                    if (st != XENOS_OK) return st;
                    maps = &now;
                }
                const int lgrid = (int)std::min(p.tiles, sms), lblock = (int)xk::kCvThreads;
                le = to.pdl(L.skip >= 0 ? xk::pair_tc_kernel<true> : xk::pair_tc_kernel<false>, lgrid, lblock, L.smem_bytes, maps->a0, rt->tmaps[li], rt->tmaps2[li], maps->o, maps->s, p);
                break;
            }
            xk::Chain2Params p;
            std::memset(&p, 0, sizeof p);
            p.bias1 = (const float *)(ws + L.b_off); p.bias2 = (const float *)(ws + L.b2_off);
            p.skip = (const __nv_bfloat16 *)ptr(L.skip); p.skip_ctot = L.skip >= 0 ? g.tensors[L.skip].c : 0;
            p.out = (__nv_bfloat16 *)ptr(L.out); p.status = status;
            p.batch = N; p.P = L.P; p.Q = L.Q;
            p.k1 = L.k; p.pad1 = L.pad; p.cpb1 = L.C / 64; p.kblocks1 = L.kblocks;
            p.k2 = L.k2; p.cpb2 = L.n1pad / 64; p.kblocks2 = L.kblocks2;
            p.n1pad = L.n1pad; p.N2 = L.K; p.tile_n2 = L.tile_n; p.n2_tiles = L.n_tiles;
            p.rh1 = L.patch_rh; p.rw1 = L.patch_rw; p.halo = L.halo2; p.rh2 = L.rh2; p.rw2 = L.rw2;
            p.tiles_y = L.tiles_y; p.tiles_x = L.tiles_x; p.m_tiles = N * L.tiles_y * L.tiles_x;
            p.stages = L.stages; p.stage_bytes = L.stage_bytes; p.a_box_bytes = L.a_box_bytes;
            p.off_mid = L.off_mid; p.off_bar = L.off_bar;
            p.act1 = L.act; p.act2 = L.act2; p.act3 = L.act3; p.out_ctot = L.out_ctot; p.out_coff = L.out_coff;
            p.idesc1 = make_idesc(L.n1pad); p.idesc2 = make_idesc(L.tile_n);
            p.launch_id = (int)li;
            const CUtensorMap *tma = &rt->hmaps[li];
            CUtensorMap tma_now;
            if (g.tensors[L.in0].input_slot >= 0) {
                xenos_status_t st = encode_chain2_input(g, rt, L, ptr(L.in0), N, &tma_now);
                if (st != XENOS_OK) return st;
                tma = &tma_now;
            }
            const int lgrid = (int)std::min(p.m_tiles, sms), lblock = (int)xk::kC2Threads;
            le = to.pdl(xk::chain2_kernel, lgrid, lblock, L.smem_bytes, *tma, rt->tmaps[li], rt->tmaps2[li], p);
            break;
        }
        case LK_GEMM: {
            if (L.fc_small) {
                const int grid = std::min(sms, (L.K + 7) / 8);
                le = to.pdl(N == 1 ? xk::fc_small_kernel<1> : xk::fc_small_kernel<8>, grid, 256, N * L.C * 2,
                    (const __nv_bfloat16 *)ptr(L.seg[0].tensor), (const __nv_bfloat16 *)(ws + L.w_off), (const float *)(ws + L.b_off), ptr(L.out), N, L.C,
                    L.kpad, L.K, L.act, L.out_dtype == XENOS_DTYPE_F32, L.out_ctot, L.out_coff);
                break;
            }
            if (L.stem_tc) {
                xk::StemParams p;
                std::memset(&p, 0, sizeof p);
                const bool pool = L.epi == EPI_POOL;
                p.src = ptr(L.in0); p.w = (const uint4 *)(ws + L.w_off); p.bias = (const float *)(ws + L.b_off); p.out = ptr(L.out); p.status = status;
                p.rows = pool ? L.PP : L.P; p.cbs = L.st_cbs; p.cw = L.st_cw; p.units = N * p.cbs * p.rows;
                p.d_rows = xk::make_fastdiv((uint32_t)p.rows); p.d_cbs = xk::make_fastdiv((uint32_t)p.cbs);
                p.C = L.C; p.H = L.H; p.W = L.W; p.k = L.k; p.stride = L.stride; p.pad = L.pad; p.lead = L.st_lead;
                p.P = L.P; p.Q = L.Q; p.N = L.K; p.tile_n = L.tile_n; p.npairs = L.st_pairs;
                p.R = L.st_slots; p.D = L.hstages; p.nacc = 4; p.acc_stride = L.acc_stride; p.qp = L.st_qp;
                p.pk = L.pool_k; p.ps = L.pool_stride; p.pp = L.pool_pad; p.PQ = L.PQ; p.pc_log2 = L.st_pc;
                p.act = L.act; p.out_ctot = L.out_ctot; p.out_coff = L.out_coff;
                p.idesc = make_idesc(L.tile_n);
                p.off_w = L.off_b; p.off_bias = L.off_bias; p.off_stage = L.off_stg; p.stage_bytes = (L.off_bar - L.off_stg) / 2 & ~15; p.off_bar = L.off_bar;
                p.raw_slots = L.st_raw; p.raw_stride = L.st_raw_stride; p.raw_lead = L.st_raw_lead; p.off_raw = L.off_raw;
                p.launch_id = (int)li;
                const int gx = std::min(p.units, std::max(1, sms / L.n_tiles));
                le = to.pdl(stem_kernel(L), dim3(gx, L.n_tiles), L.block, L.smem_bytes, p);
                break;
            }
            if (L.conv_tc) {
                xk::ConvParams p;
                std::memset(&p, 0, sizeof p);
                p.seg[0] = conv_segment(L, L.seg[0]); p.seg[1] = conv_segment(L, L.seg[1]);
                p.bias = (const float *)(ws + L.b_off); p.out = ptr(L.out); p.status = status;
                p.rows = N * L.rows_per_image;
                p.tile_rows = L.epi == EPI_GAP ? L.tile_rows : 128;
                const int mt = L.gap_parts > 1 ? N * L.gap_parts : (p.rows + p.tile_rows - 1) / p.tile_rows;
                p.d_rpi = xk::make_fastdiv((uint32_t)L.rows_per_image); p.d_q = xk::make_fastdiv((uint32_t)L.Q);
                p.d_nt = xk::make_fastdiv((uint32_t)L.n_tiles); p.d_ks = xk::make_fastdiv((uint32_t)L.ksplit);
                p.total = mt * L.n_tiles * L.ksplit; p.tile_n = L.tile_n; p.npad = L.npad; p.N = L.K;
                p.kblocks = L.kblocks; p.stages = L.stages; p.stage_bytes = L.stage_bytes; p.b_resident = L.b_resident; p.b_group = L.b_group;
                p.acc_stride = L.acc_stride; p.tmem_cols = L.tmem_cols;
                p.chunk = L.chunk; p.nchunks = L.nchunks; p.box_bytes = L.chunk * 64; p.s_slots = L.s_slots;
                // (two clamps in a row with no shortcut between them are one: none < ReLU < ReLU6)
                p.act = L.skip >= 0 ? L.act : std::max(L.act, L.act2); p.act2 = L.skip >= 0 ? L.act2 : 0; p.out_ctot = L.out_ctot; p.out_f32 = L.out_dtype == XENOS_DTYPE_F32;
                p.idesc = make_idesc(L.tile_n);
                p.off_b = L.off_b; p.off_stage = L.off_stg; p.off_bias = L.off_bias; p.off_bar = L.off_bar;
                p.launch_id = (int)li;
                p.gap_imgs = L.gap_imgs; p.gap_rpi = L.gap_rpi; p.gap_parts = L.gap_parts; p.batch = N;
                p.ksplit = L.ksplit; p.kb_per = L.ksplit > 1 ? L.kb_per : L.kblocks; p.split_ld = L.npad;
                p.split_stride = (long long)p.rows * L.npad;
                p.split_part = reinterpret_cast<float *>(ws + g.split_off);
                p.split_cnt = reinterpret_cast<unsigned int *>(ws + L.split_cnt_off);
                p.skip = (const __nv_bfloat16 *)ptr(L.skip); p.skip_ctot = L.skip >= 0 ? g.tensors[L.skip].c : 0;
                const ConvMaps *maps = &rt->conv[li];
                ConvMaps now;
                if (conv_has_external(g, L)) {
                    now = *maps;
                    xenos_status_t st = encode_conv_maps(g, rt, L, ptr, N, true, &now);
                    if (st != XENOS_OK) return st;
                    maps = &now;
                }
                int limit = sms;
                if (L.b_resident) limit = std::max(1, sms / L.n_tiles) * L.n_tiles;
                const int lgrid = (int)std::min(p.total, limit), lblock = (int)xk::kCvThreads;
                le = to.pdl_cluster(conv_kernel(L), L.cv_epi == xk::CE_CLUSTER ? p.total : lgrid, lblock, L.smem_bytes, L.cv_epi == xk::CE_CLUSTER ? L.ksplit : 1, maps->a0, maps->a1, rt->tmaps[li], maps->o, maps->s, p);
                break;
            }
            if (L.seg[0].mode == AM_DW) {
                const ASeg &a = L.seg[0];
                xk::DwParams p;
                std::memset(&p, 0, sizeof p);
                p.dw_w = (const float *)(ws + a.dw_w_off); p.dw_b = (const float *)(ws + a.dw_b_off); p.bias = (const float *)(ws + L.b_off);
                p.out = ptr(L.out); p.status = status;
                p.d_nt = xk::make_fastdiv((uint32_t)L.n_tiles); p.d_ks = xk::make_fastdiv((uint32_t)L.ksplit);
                p.d_tx = xk::make_fastdiv((uint32_t)L.tiles_x); p.d_ty = xk::make_fastdiv((uint32_t)L.tiles_y);
                p.batch = N; p.P = L.P; p.Q = L.Q; p.C = a.C; p.stride = a.stride; p.pad = a.pad; p.dw_act = a.dw_act;
                p.ni = L.ni; p.rh = L.patch_rh; p.rw = L.patch_rw; p.tile_rows = L.tile_rows;
                p.total = (N + L.ni - 1) / L.ni * L.tiles_y * L.tiles_x * L.n_tiles * L.ksplit;
                p.kblocks = L.kblocks; p.last_steps = (a.C - 64 * (L.kblocks - 1) + 15) / 16; p.tile_n = L.tile_n; p.n_acc = L.n_acc; p.N = L.K;
                p.kb_per = L.ksplit > 1 ? L.kb_per : L.kblocks;
                p.groups = L.dw_groups; p.wpg_log2 = L.dw_wpg_log2; p.pairs = L.halo_cb > 32 ? 32 : 16;
                p.batch_tiles = L.dw_batch; p.n_bufs = L.n_acc == 2 ? 1 : 2 * L.dw_batch;
                p.a_stride = L.a_stride; p.a_slots = L.a_slots; p.b_slots = L.b_slots; p.h_slots = L.h_slots; p.b_resident = L.b_resident;
                p.halo_bytes = L.halo_bytes; p.halo_stride = L.halo_stride; p.halo_h = L.halo_h; p.halo_w = L.halo_w; p.halo_cb = L.halo_cb;
                p.acc_stride = L.acc_stride; p.tmem_cols = L.tmem_cols;
                p.chunk = L.chunk; p.nchunks = L.nchunks; p.box_bytes = 128 * L.chunk * 2; p.out_bufs = L.out_bufs;
                p.act = L.act; p.out_ctot = L.out_ctot; p.out_f32 = L.out_dtype == XENOS_DTYPE_F32;
                p.idesc = make_idesc(L.tile_n);
                p.off_b = L.off_b; p.off_halo = L.off_halo; p.off_dww = L.off_dww; p.off_stage = L.off_stg; p.off_bias = L.off_bias; p.off_bar = L.off_bar;
                p.gap_imgs = L.gap_imgs; p.gap_area = L.gap_area; p.gap_rpi = L.gap_rpi;
                p.ksplit = L.ksplit; p.split_ld = L.npad; p.split_stride = (long long)N * L.rows_per_image * L.npad;
                p.split_part = reinterpret_cast<float *>(ws + g.split_off); p.split_cnt = reinterpret_cast<unsigned int *>(ws + L.split_cnt_off);
                p.launch_id = (int)li;
                const ConvMaps *maps = &rt->conv[li];
                ConvMaps now;
                if (conv_has_external(g, L)) {
                    now = *maps;
                    xenos_status_t st = encode_dw_maps(g, rt, L, ptr, N, true, &now);
                    if (st != XENOS_OK) return st;
                    maps = &now;
                }
                // A plan with a tile for every unit of its description lets a tile's results leave through the operand ring: its tiles
                // are a CTA's only ones, also on a device with fewer units.
                const int limit = L.off_stg == 0 && L.cv_epi != xk::DE_SPLIT ? p.total : L.b_resident ? std::max(1, sms / L.n_tiles) * L.n_tiles : sms;
                auto *k = dw_kernel(L.cv_epi, a.stride, L.dw_br, L.halo_cb);
                le = to.pdl(k, std::min(p.total, limit), L.block, L.smem_bytes, maps->a0, rt->tmaps[li], maps->o, p);
                break;
            }
            xk::GemmParams p;
            std::memset(&p, 0, sizeof p);
            for (int s = 0; s < 2; ++s) {
                const ASeg &a = L.seg[s];
                xk::GemmSeg &d = p.seg[s];
                d.mode = a.mode; d.src = ptr(a.tensor); d.C = a.C; d.H = a.H; d.W = a.W; d.k = a.k; d.stride = a.stride; d.pad = a.pad;
                d.kelems = a.kelems; d.kblocks = a.kblocks; d.src_f32 = a.src_dtype == XENOS_DTYPE_F32;
            }
            p.bias = (const float *)(ws + L.b_off);
            p.skip = (const __nv_bfloat16 *)ptr(L.skip);
            p.skip_ctot = L.skip >= 0 ? g.tensors[L.skip].c : 0;
            p.out = ptr(L.out); p.status = status;
            p.batch = N; p.P = L.P; p.Q = L.Q;
            p.ni = L.ni; p.rh = L.patch_rh; p.rw = L.patch_rw; p.tiles_y = L.tiles_y; p.tiles_x = L.tiles_x;
            p.step_y = L.step_y; p.step_x = L.step_x; p.off_y = L.off_y; p.off_x = L.off_x;
            p.pool_k = L.pool_k; p.pool_stride = L.pool_stride; p.PP = L.PP; p.PQ = L.PQ; p.pth = L.patch_th; p.ptw = L.patch_tw;
            p.kblocks = L.kblocks; p.stages = L.stages; p.tile_n = L.tile_n; p.n_tiles = L.n_tiles; p.N = L.K;
            p.acc_stride = L.acc_stride; p.tmem_cols = L.tmem_cols;
            p.hstages = L.hstages; p.halo_bytes = L.halo_bytes; p.halo_stride = L.halo_stride;
            p.halo_h = L.halo_h; p.halo_w = L.halo_w;
            p.stem_tma = L.stem_tma; p.stem_align = L.stem_align;
            p.off_halo = L.off_halo; p.off_stg = L.off_stg; p.off_dww = L.off_dww; p.off_bias = L.off_bias; p.off_bar = L.off_bar;
            p.act = L.act; p.act2 = L.act2; p.epi = L.epi; p.out_ctot = L.out_ctot; p.out_coff = L.out_coff;
            p.out_f32 = L.out_dtype == XENOS_DTYPE_F32;
            p.idesc = make_idesc(L.tile_n);
            p.launch_id = (int)li;
            p.m_tiles = ((N + L.ni - 1) / L.ni) * L.tiles_y * L.tiles_x;
            const CUtensorMap *tmh = &rt->tmaps[li];
            CUtensorMap tmh_now;
            if (L.stem_tma) {
                // the image is a caller buffer: encode its patch map now
                xenos_status_t st = encode_stem_map(g, rt, L, ptr(L.seg[0].tensor), N, &tmh_now);
                if (st != XENOS_OK) return st;
                tmh = &tmh_now;
            }
            const int lgrid = std::min(p.m_tiles * p.n_tiles, sms), lblock = L.block;
            le = to.pdl(xk::gemm_chain_kernel, lgrid, lblock, L.smem_bytes, rt->tmaps[li], *tmh, p);
            break;
        }
        default:
            return fail(g, XENOS_E_UNSUPPORTED, "internal: launch record without a kernel");
        }
        if (le != cudaSuccess) {
            cudaGetLastError();
            return cuda_fail(g, "kernel launch", le);
        }
        const xenos_status_t st = each(li);
        if (st != XENOS_OK) return st;
    }
    return XENOS_OK;
}

static xenos_status_t launch_pass(Graph &g, int batch, const void *const *in, void *const *out, void *stream_v) {
    Issue to;
    to.stream = static_cast<cudaStream_t>(stream_v);
    return issue_pass(g, batch, in, out, to, [](size_t) -> xenos_status_t { return XENOS_OK; });
}

xenos_status_t runtime_profile(Graph &g, int batch, const void *const *in, void *const *out, void *stream_v, float *ms_per_launch) {
    struct Events {
        std::vector<cudaEvent_t> v;
        ~Events() { for (cudaEvent_t e : v) cudaEventDestroy(e); }
    } ev;
    Issue to;
    to.stream = static_cast<cudaStream_t>(stream_v);
    for (size_t i = 0; i <= g.launches.size(); ++i) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return fail(g, XENOS_E_CUDA, "cudaEventCreate failed");
        ev.v.push_back(e);
    }
    cudaEventRecord(ev.v[0], to.stream);
    const xenos_status_t st = issue_pass(g, batch, in, out, to, [&](size_t li) -> xenos_status_t {
        cudaEventRecord(ev.v[li + 1], to.stream);
        return XENOS_OK;
    });
    if (st != XENOS_OK) return st;
    const cudaError_t e = cudaStreamSynchronize(to.stream);
    if (e != cudaSuccess) return cuda_fail(g, "profile synchronize", e);
    for (size_t li = 0; li < g.launches.size(); ++li) {
        ms_per_launch[li] = 0.0f;
        cudaEventElapsedTime(&ms_per_launch[li], ev.v[li], ev.v[li + 1]);
    }
    return XENOS_OK;
}

// Records the pass: a graph's launches for max_batch images, as they follow one another in a stream (programmatic dependencies
// included), with the workspace in the place of the caller's buffers.  Nothing runs.
static xenos_status_t record_pass(Graph &g, const std::vector<void *> &in, const std::vector<void *> &out, cudaStream_t stream) {
    Runtime *rt = static_cast<Runtime *>(g.rt);
    struct Scope {
        cudaStream_t stream = nullptr;
        cudaGraph_t graph = nullptr;
        ~Scope() {
            if (graph) cudaGraphDestroy(graph);
            if (stream) cudaStreamDestroy(stream);
        }
    } sc;
    std::vector<cudaGraphNode_t> nodes(g.launches.size(), nullptr);
    cudaError_t e = cudaStreamCreateWithFlags(&sc.stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_fail(g, "cudaStreamCreateWithFlags", e);
    if ((e = cudaStreamBeginCapture(sc.stream, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return cuda_fail(g, "cudaStreamBeginCapture", e);
    Issue to;
    to.stream = sc.stream;
    const xenos_status_t st = issue_pass(g, g.max_batch, in.data(), out.data(), to, [&](size_t li) -> xenos_status_t {
        // the launch's node is what a next one would depend on
        cudaStreamCaptureStatus cap;
        const cudaGraphNode_t *last = nullptr;
        const cudaGraphEdgeData *edges = nullptr;
        size_t n = 0;
        const cudaError_t e = cudaStreamGetCaptureInfo_v3(sc.stream, &cap, nullptr, nullptr, &last, &edges, &n);
        if (e != cudaSuccess || cap != cudaStreamCaptureStatusActive || n != 1) return cuda_fail(g, "cudaStreamGetCaptureInfo", e);
        nodes[li] = last[0];
        return XENOS_OK;
    });
    e = cudaStreamEndCapture(sc.stream, &sc.graph);
    if (st != XENOS_OK) return st;
    if (e != cudaSuccess) return cuda_fail(g, "cudaStreamEndCapture", e);
    cudaGraphExec_t exec = nullptr;
    if ((e = cudaGraphInstantiate(&exec, sc.graph, 0)) != cudaSuccess) return cuda_fail(g, "cudaGraphInstantiate", e);
    // (else the first pass would wait for it: 147 us instead of 109 for the first pass of SqueezeNet at batch 1)
    // (a run in another stream need not be ordered behind it: it is waited for here)
    if ((e = cudaGraphUpload(exec, stream)) != cudaSuccess || (e = cudaStreamSynchronize(stream)) != cudaSuccess) {
        cudaGraphExecDestroy(exec);
        return cuda_fail(g, "cudaGraphUpload", e);
    }
    rt->exec = exec;
    std::swap(rt->graph, sc.graph);
    rt->nodes.swap(nodes);
    rt->exec_batch = g.max_batch;
    return XENOS_OK;
}

xenos_status_t runtime_bind(Graph &g, void *ws, void *stream_v, bool record) {
    xenos_status_t st = attach(g, ws, stream_v);
    if (st != XENOS_OK) return st;
    Issue to;
    to.mode = Issue::READY;
    to.optin = static_cast<Runtime *>(g.rt)->optin;
    // (any aligned address does for buffers that only a run names; some kernels have a form of their own for one image)
    const std::vector<void *> in(g.inputs.size(), ws), out(g.outputs.size(), ws);
    for (int batch : {g.max_batch, 1}) {
        st = issue_pass(g, batch, in.data(), out.data(), to, [](size_t) -> xenos_status_t { return XENOS_OK; });
        if (st != XENOS_OK) return st;
    }
    if (record && g.launches.size() > 1 && record_pass(g, in, out, static_cast<cudaStream_t>(stream_v)) != XENOS_OK) {
        cudaGetLastError();             // (not a reason to refuse the binding: the kernels are launched one by one then)
        g.err = "bind: passes run kernel by kernel, recording them failed: " + g.err;
    }
    return XENOS_OK;
}

// A pass of several launches runs as the CUDA graph that the binding recorded, the nodes that meet the caller's buffers pointed
// at them on every call (1 us): single launches cost the host 2.3 to 4.5 us each, more than many of these kernels run on a small
// batch, and leave gaps between kernels that follow at once in the graph.  MobileNet at batch 1, other buffers on every call:
// 98.3 us a pass and 4.4 us of the host, 104.1 and 86.6 in single launches.
// Another batch than the recorded one is launched one by one; when it comes a second time in a row, all nodes are set to it
// behind that launch (1.7 us each: before the launch a pass alone would wait 25 us for them).  Passes inside a caller's own
// stream capture and single launches go to the stream directly (a graph of one kernel takes 2.5 us longer than the kernel).
xenos_status_t runtime_run(Graph &g, int batch, const void *const *in, void *const *out, void *stream_v) {
    Runtime *rt = static_cast<Runtime *>(g.rt);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    if (!rt->exec) return launch_pass(g, batch, in, out, stream_v);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return launch_pass(g, batch, in, out, stream_v);
    }
    std::lock_guard<std::mutex> lock(rt->exec_mutex);
    auto point = [&](bool external_only) {
        Issue to;
        to.mode = Issue::POINT; to.rt = rt; to.external_only = external_only;
        rt->exec_batch = 0;             // (until every node has been set)
        const xenos_status_t st = issue_pass(g, batch, in, out, to, [](size_t) -> xenos_status_t { return XENOS_OK; });
        if (st == XENOS_OK) rt->exec_batch = batch;
        return st;
    };
    const bool again = batch == rt->last_batch;
    rt->last_batch = batch;
    if (batch != rt->exec_batch) {
        const xenos_status_t st = launch_pass(g, batch, in, out, stream_v);
        return st == XENOS_OK && again ? point(false) : st;
    }
    if (xenos_status_t st = point(true)) return st;
    const cudaError_t e = cudaGraphLaunch(rt->exec, stream);
    if (e != cudaSuccess) return cuda_fail(g, "kernel launch", e);
    return XENOS_OK;
}

xenos_status_t runtime_status(Graph &g, void *stream_v) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    cudaError_t e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_fail(g, "stream synchronize", e);
    unsigned int word = 0;
    uint8_t *ws = static_cast<uint8_t *>(g.ws);
    if ((e = cudaMemcpy(&word, ws + g.status_off, 4, cudaMemcpyDeviceToHost)) != cudaSuccess) return cuda_fail(g, "status read", e);
    if (word == 0) return XENOS_OK;
    cudaMemset(ws + g.status_off, 0, 256 + g.cnt_bytes);      // (the arrival counters of a run that gave up are stale too)
    int code = -(int)(word & 0xffu);
    if (code == XENOS_E_TIMEOUT) {
        static const char *role[] = {"a wait", "the TMA warp", "the MMA warp", "a producer warp", "a producer warp at the last tile", "an epilogue warp"};
        const unsigned r = (word >> 8) & 0xfu;
        return fail(g, code, std::string("a kernel gave up a bounded wait (") + role[r < 6 ? r : 0] + ", launch " + std::to_string((word >> 12) & 0xfffu) + ")");
    }
    return fail(g, code, "a kernel failed an index check");
}

xenos_status_t runtime_selftest_wait_expiry(Graph &g, void *stream_v) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    unsigned int *status = reinterpret_cast<unsigned int *>(static_cast<uint8_t *>(g.ws) + g.status_off);
    xk::wait_expiry_probe_kernel<<<1, 32, 0, stream>>>(status, 4);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(g, "kernel launch", e);
    return XENOS_OK;
}

// ------------------------------------------------------------------------------------------------
// Built-in scratch: a workspace that lives inside the library image, for callers that must not
// allocate device memory themselves.
// ------------------------------------------------------------------------------------------------
constexpr size_t kBuiltinScratchBytes = 16u << 20;    // 16 MiB, held by every device that loads the library
constexpr int kMaxDevices = 64;
static __device__ __align__(256) unsigned char g_builtin_scratch[kBuiltinScratchBytes];
// In host code the name g_builtin_scratch is only a handle for the symbol, not a device address;
// the address is looked up once per device and cached here.
static void *g_builtin_ptr[kMaxDevices] = {};
static uint64_t g_builtin_owner[kMaxDevices] = {};    // serial of the graph whose parameters the array holds
static std::mutex g_builtin_mutex;                    // guards the two host tables above (not the device array)

size_t runtime_builtin_scratch_bytes() { return kBuiltinScratchBytes; }

void runtime_free_builtin(Graph &g) {
    std::lock_guard<std::mutex> lock(g_builtin_mutex);
    delete static_cast<Runtime *>(g.rt_builtin);
    g.rt_builtin = nullptr;
    for (int d = 0; d < kMaxDevices; ++d)
        if (g_builtin_owner[d] == g.serial) g_builtin_owner[d] = 0;
}

xenos_status_t runtime_run_builtin(Graph &g, int batch, const void *const *in, void *const *out, void *stream_v) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(g, "no CUDA device (this library has no CPU fallback)", e);
    if (dev < 0 || dev >= kMaxDevices) return fail(g, XENOS_E_CUDA, "run_builtin_scratch: device index out of range");
    std::lock_guard<std::mutex> lock(g_builtin_mutex);
    if (!g_builtin_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_builtin_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(g, "cudaGetSymbolAddress(built-in scratch)", e);
        g_builtin_ptr[dev] = p;
    }
    void *scratch = g_builtin_ptr[dev];
    // run with the graph temporarily bound to the built-in scratch; the caller's own binding
    // (xenos_graph_bind) is put back afterwards
    // (put back on every way out of this function, an exception from the bind included)
    struct Restore {
        Graph &g; void *ws, *rt;
        ~Restore() { g.rt_builtin = g.rt; g.ws = ws; g.rt = rt; }
    } restore{g, g.ws, g.rt};
    g.rt = g.rt_builtin;
    g.rt_builtin = nullptr;               // g.rt owns the built-in binding until Restore hands it back
    xenos_status_t st = XENOS_OK;
    Runtime *rb = static_cast<Runtime *>(g.rt);
    if (!rb || rb->device != dev || g_builtin_owner[dev] != g.serial) {
        // the array holds nothing or another graph's data: upload parameters, clear status, encode maps
        g_builtin_owner[dev] = 0;
        st = runtime_bind(g, scratch, stream, false);      // (never recorded: that would allocate)
        g_builtin_owner[dev] = st == XENOS_OK ? g.serial : 0;
    } else {
        g.ws = scratch;
        // the status word keeps the last call's contents: start from zero
        if ((e = cudaMemsetAsync(static_cast<uint8_t *>(scratch) + g.status_off, 0, 256 + g.cnt_bytes, stream)) != cudaSuccess)
            st = cuda_fail(g, "status clear", e);
    }
    if (st == XENOS_OK) st = launch_pass(g, batch, in, out, stream);
    if (st == XENOS_OK) st = runtime_status(g, stream);
    return st;
}

}  // namespace xenos
