// Host passes: Conv-Bn-Relu pre-fusion (Section 4.3), operator linking (Section 4.1, Table 1),
// operator split and lowering to launch records (Section 4.2, Eq. 1), parameter packing.
// Everything here is integer / host fp work and is deterministic: equal graphs give equal plans.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <set>

#include "graph.hpp"

namespace xenos {

uint16_t f32_to_bf16_rne(float f) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    if ((u & 0x7f800000u) == 0x7f800000u) return (uint16_t)(u >> 16);   // inf / nan: truncate
    u += 0x7fffu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}

static size_t blob_reserve(Graph &g, size_t bytes) {
    size_t off = align_up(g.param_blob.size(), 256);
    g.param_blob.resize(off + bytes, 0);
    return off;
}

// ------------------------------------------------------------------------------------------------
// Pre-fusion: Conv + Bn + Bias + Relu -> one CBR operator (Section 4.3).  BatchNorm is folded
// into the convolution: w' = w * gamma / sqrt(var + eps), b' = beta + (b - mean) * gamma / sqrt(var + eps).
// ------------------------------------------------------------------------------------------------
static void fold_bn(Node &n, const Op &bn, int per_out) {
    for (int k = 0; k < n.cout; ++k) {
        double s = (double)bn.gamma[k] / std::sqrt((double)bn.var[k] + (double)bn.eps);
        for (int i = 0; i < per_out; ++i) n.w[(size_t)k * per_out + i] = (float)((double)n.w[(size_t)k * per_out + i] * s);
        n.b[k] = (float)((double)bn.beta[k] + ((double)n.b[k] - (double)bn.mean[k]) * s);
    }
}

xenos_status_t prefuse(Graph &g) {
    g.nodes.clear();
    g.node_of_tensor.assign(g.tensors.size(), -1);
    auto sole_consumer_ok = [&](int t) {
        return g.tensors[t].consumers.size() == 1 && g.tensors[t].output_slot < 0;
    };
    for (int oi = 0; oi < (int)g.ops.size(); ++oi) {
        const Op &op = g.ops[oi];
        const Tensor &x = g.tensors[op.in[0]];
        int src = g.node_of_tensor[op.in[0]];
        switch (op.kind) {
        case XENOS_OP_CONV:
        case XENOS_OP_FC:
        case XENOS_OP_MATMUL: {
            Node n;
            n.kind = op.kind == XENOS_OP_FC ? NK_FC : (op.groups == 1 ? NK_CONV : NK_DW);
            if (op.kind == XENOS_OP_MATMUL) { n.kind = x.is_vec ? NK_FC : NK_CONV; n.from_matmul = true; }
            n.in = op.in; n.out = op.out;
            n.cin = x.c; n.cout = op.cout; n.k = op.k; n.stride = op.stride; n.pad = op.pad; n.act = op.act;
            n.w = op.w;
            n.b.assign(op.cout, 0.0f);
            if (op.has_bias) n.b = op.bias;
            if (op.has_bn) fold_bn(n, op, (int)(n.w.size() / op.cout));
            n.user_ops.push_back(oi);
            g.nodes.push_back(std::move(n));
            g.node_of_tensor[op.out] = (int)g.nodes.size() - 1;
            break;
        }
        case XENOS_OP_BATCHNORM: {
            if (src < 0 || !sole_consumer_ok(op.in[0]) || g.nodes[src].act != XENOS_ACT_NONE ||
                !(g.nodes[src].kind == NK_CONV || g.nodes[src].kind == NK_DW || g.nodes[src].kind == NK_FC))
                return fail(g, XENOS_E_UNSUPPORTED,
                            "BatchNorm that does not directly follow a convolution / fc (single consumer, no activation between) has no kernel");
            Node &n = g.nodes[src];
            fold_bn(n, op, (int)(n.w.size() / n.cout));
            g.node_of_tensor[n.out] = -1;
            n.out = op.out;
            n.user_ops.push_back(oi);
            g.node_of_tensor[op.out] = src;
            break;
        }
        case XENOS_OP_RELU:
        case XENOS_OP_RELU6: {
            if (src < 0 || !sole_consumer_ok(op.in[0]) || g.nodes[src].act != XENOS_ACT_NONE ||
                !(g.nodes[src].kind == NK_CONV || g.nodes[src].kind == NK_DW || g.nodes[src].kind == NK_FC ||
                  g.nodes[src].kind == NK_ADD))
                return fail(g, XENOS_E_UNSUPPORTED,
                            "activation that does not directly follow a convolution, fc or add (single consumer) has no kernel");
            Node &n = g.nodes[src];
            n.act = op.kind == XENOS_OP_RELU ? XENOS_ACT_RELU : XENOS_ACT_RELU6;
            g.node_of_tensor[n.out] = -1;
            n.out = op.out;
            n.user_ops.push_back(oi);
            g.node_of_tensor[op.out] = src;
            break;
        }
        default: {
            Node n;
            n.kind = op.kind == XENOS_OP_POOL_MAX ? NK_MAXPOOL : op.kind == XENOS_OP_POOL_AVG ? NK_AVGPOOL
                   : op.kind == XENOS_OP_POOL_GLOBAL_AVG ? NK_GAP : op.kind == XENOS_OP_ADD ? NK_ADD
                   : op.kind == XENOS_OP_MUL ? NK_MUL : op.kind == XENOS_OP_MAC ? NK_MAC
                   : op.kind == XENOS_OP_TRANSPOSE ? NK_TRANSPOSE : op.kind == XENOS_OP_SPLIT ? NK_SLICE : NK_CONCAT;
            n.in = op.in; n.out = op.out;
            n.cin = x.c; n.cout = g.tensors[op.out].c; n.k = op.k; n.stride = op.stride; n.pad = op.pad; n.act = op.act;
            n.user_ops.push_back(oi);
            g.nodes.push_back(std::move(n));
            g.node_of_tensor[op.out] = (int)g.nodes.size() - 1;
        }
        }
    }
    // every node input must be a graph input or another node's final output
    for (const Node &n : g.nodes)
        for (int t : n.in)
            if (g.tensors[t].input_slot < 0 && g.node_of_tensor[t] < 0)
                return fail(g, XENOS_E_UNSUPPORTED, "a tensor inside a fused Conv-Bn-Relu group is read by another operator");
    for (int t : g.outputs)
        if (g.node_of_tensor[t] < 0) return fail(g, XENOS_E_UNSUPPORTED, "a graph output lies inside a fused Conv-Bn-Relu group");
    return XENOS_OK;
}

// ------------------------------------------------------------------------------------------------
// Linking
// ------------------------------------------------------------------------------------------------
struct LinkCtx {
    Graph &g;
    std::vector<std::vector<int>> cons;   // tensor -> consumer node indices
    explicit LinkCtx(Graph &gg) : g(gg), cons(gg.tensors.size()) {
        for (int i = 0; i < (int)g.nodes.size(); ++i)
            for (int t : g.nodes[i].in) cons[t].push_back(i);
    }
    // the only consumer of node n's output, or -1 (graph outputs have an outside consumer)
    int sole(int n) const {
        int t = g.nodes[n].out;
        if (g.tensors[t].output_slot >= 0 || cons[t].size() != 1) return -1;
        return cons[t][0];
    }
    int rows(int n) const { const Tensor &t = g.tensors[g.nodes[n].out]; return t.h * t.w; }
};

// Max pools that stem_tc_kernel forms row by row, over a map of `rows` rows: windows overlap by one row at most, and no two end with
// the same row (the padding below the map can hold the ends of the last two where it is a whole stride).
static bool pool_in_registers(const Node &p, int rows) {
    const int count = (rows + 2 * p.pad - p.k) / p.stride + 1, below = (count - 1) * p.stride - p.pad + p.k - rows;
    return p.k - p.stride <= 1 && p.pad < p.k && below < p.stride;
}

// largest pool-output tile whose conv-output patch fits the 128-row M tile
static bool pool_patch(int k, int s, int PP, int PQ, int &th, int &tw, int &rh, int &rw) {
    int best = 0;
    for (int a = 1; a <= PP && (a - 1) * s + k <= 128; ++a)
        for (int b = 1; b <= PQ && (b - 1) * s + k <= 128; ++b) {
            int h = (a - 1) * s + k, w = (b - 1) * s + k;
            if (h * w > 128) break;
            int score = a * b;
            if (score > best || (score == best && b > tw)) { best = score; th = a; tw = b; rh = h; rw = w; }
        }
    return best > 0;
}

typedef bool (*AllowFn)(const void *, int);

// Try to grow a chain anchored at node a.  allowed(n) says whether n may join.
// Tile geometry of two linked convolutions: the producer tile rh1 x rw1 (<= 128 pixels, rw1 <= 30 so that every tap
// offset stays inside the middle buffer's spare rows) that needs the fewest tiles for a P x Q map, given the
// consumer's frame h = (k2 - 1) / 2.
static bool chain2_tile(int P, int Q, int h, int &rh1, int &rw1) {
    long best = -1;
    for (int w = 2 * h + 1; w <= std::min(Q + 2 * h, 30); ++w) {
        int hh = std::min(P + 2 * h, 128 / w);
        if (hh < 2 * h + 1) continue;
        long tiles = (long)((P + hh - 2 * h - 1) / (hh - 2 * h)) * ((Q + w - 2 * h - 1) / (w - 2 * h));
        if (best < 0 || tiles < best || (tiles == best && w > rw1)) { best = tiles; rh1 = hh; rw1 = w; }
    }
    return best > 0;
}

// Modelled time of linking two convolutions against running them one after the other (per image, arbitrary
// units): the linked form issues whole 128-row tiles for both products, frame rows included, and moves no
// intermediate; rates are what this library's kernels reach, not the device's peaks.
static bool chain2_pays(const Graph &g, const Node &A, const Node &B, bool skip) {
    const Tensor &o = g.tensors[B.out];
    const int h = (B.k - 1) / 2;
    int rh1 = 0, rw1 = 0;
    if (!chain2_tile(o.h, o.w, h, rh1, rw1)) return false;
    const double tiles = (double)((o.h + rh1 - 2 * h - 1) / (rh1 - 2 * h)) * ((o.w + rw1 - 2 * h - 1) / (rw1 - 2 * h));
    const double tc = 0.5e15, hbm = 4.0e12, px = (double)o.h * o.w;
    const double k1 = (double)A.cin * A.k * A.k, k2 = (double)A.cout * B.k * B.k;
    const double in = px * A.cin * 2, midb = px * A.cout * 2, outb = px * B.cout * 2 * (skip ? 2 : 1);
    const double lin = std::max(2.0 * tiles * 128 * (k1 * A.cout + k2 * B.cout) / tc, (in + outb) / hbm);
    const double unl = std::max(2.0 * px * k1 * A.cout / tc, (in + midb) / hbm) + std::max(2.0 * px * k2 * B.cout / tc, (midb + outb) / hbm);
    return lin <= 1.02 * unl;      // (when the model sees no difference the link still saves a launch and the bytes)
}

template <class Allowed>
static bool try_match(const LinkCtx &cx, int a, Allowed allowed, Chain &out, bool by_model = true) {
    Graph &g = cx.g;
    const Node &A = g.nodes[a];
    out = Chain();
    if (!allowed(a)) return false;
    if (g.precision == XENOS_PRECISION_FP32_CUDA_CORE) {
        // Table 1: ConvX -> ConvY -> ZPooling, with ConvY 1x1
        if (A.kind != NK_CONV) return false;
        int b = cx.sole(a);
        if (b < 0 || !allowed(b) || g.nodes[b].kind != NK_CONV) return false;
        const Node &B = g.nodes[b];
        if (B.k != 1 || B.stride != 1 || B.pad != 0) return false;
        int c = cx.sole(b);
        if (c < 0 || !allowed(c)) return false;
        const Node &C = g.nodes[c];
        if (!(C.kind == NK_MAXPOOL || C.kind == NK_AVGPOOL) || C.pad != 0) return false;
        out.kind = CK_CONV_CONV_POOL;
        out.nodes = {a, b, c};
        out.pattern = "ConvX -> ConvY -> ZPooling";
        return true;
    }
    // ---- bf16 tensor-core chains -----------------------------------------------------------
    if (A.from_matmul) {
        // MatmulX -> MatmulY (last row of Table 1) with constant right operands and nothing but a bias between
        // them: (X B1 + b1) B2 + b2 = X (B1 B2) + (b1 B2 + b2).  The constants are multiplied once at compile time
        // and the intermediate matrix never exists.  Taken only when it does not add multiplications per row.
        int b = A.act == XENOS_ACT_NONE ? cx.sole(a) : -1;
        if (b >= 0 && allowed(b) && g.nodes[b].from_matmul && g.nodes[b].kind == A.kind && A.cin % 8 == 0 &&
            (long)A.cin * g.nodes[b].cout <= (long)A.cin * A.cout + (long)A.cout * g.nodes[b].cout) {
            out.kind = CK_MATMUL_MATMUL;
            out.nodes = {a, b};
            out.pattern = "MatmulX -> MatmulY (MatA * MatB -> MatC * MatD, constants multiplied)";
            return true;
        }
    }
    if (A.kind == NK_DW) {
        // depthwise -> pointwise: the motivating mismatch of Section 2.2 (ConvX -> ConvY row)
        if (A.k != 3 || A.cin % 8 || A.stride > 2) return false;
        int b = cx.sole(a);
        if (b < 0 || !allowed(b)) return false;
        const Node &B = g.nodes[b];
        if (B.kind != NK_CONV || B.k != 1 || B.stride != 1 || B.pad != 0) return false;
        out.kind = CK_DW_PW;
        out.nodes = {a, b};
        out.pattern = "ConvX -> ConvY (depthwise 3x3 -> pointwise 1x1)";
        int c = cx.sole(b);
        const Tensor &bo = g.tensors[B.out];
        if (c >= 0 && allowed(c) && g.nodes[c].kind == NK_GAP && bo.h * ((bo.w + 3) / 4 * 4) <= 128 &&
            ((bo.h + 1) / 2) * ((bo.w + 3) / 4) <= 16) {     // whole images per tile, in 2 x 4 pixel blocks
            out.nodes.push_back(c);
            out.pattern = "ConvX -> ConvY -> ZPooling (depthwise -> pointwise -> global average)";
        }
        return true;
    }
    if (A.kind == NK_CONCAT) {
        // fire expand: {conv1x1, conv3x3} on one input, joined by channel-offset stores
        if (A.in.size() != 2) return false;
        int e0 = g.node_of_tensor[A.in[0]], e1 = g.node_of_tensor[A.in[1]];
        if (e0 < 0 || e1 < 0 || e0 == e1 || !allowed(e0) || !allowed(e1)) return false;
        const Node &E0 = g.nodes[e0], &E1 = g.nodes[e1];
        if (E0.kind != NK_CONV || E1.kind != NK_CONV || E0.in[0] != E1.in[0]) return false;
        if (cx.sole(e0) != a || cx.sole(e1) != a) return false;
        if (E0.act != E1.act || E0.stride != 1 || E1.stride != 1 || E0.cin % 8) return false;
        auto shape_ok = [](const Node &n) { return (n.k == 1 && n.pad == 0) || (n.k == 3 && n.pad == 1); };
        if (!shape_ok(E0) || !shape_ok(E1) || (E0.k == 1 && E1.k == 1)) return false;
        if (E0.cout % 8 || E1.cout % 8) return false;
        out.kind = CK_EXPAND_CONCAT;
        out.nodes = {e0, e1, a};
        out.pattern = "ConvX -> {ConvY ; ConvZ} -> concat (joined without a layout transformation)";
        {
            // the squeeze convolution in front of the two expands: its result stays in shared memory
            int sq = g.node_of_tensor[E0.in[0]];
            const std::vector<int> &sc = cx.cons[E0.in[0]];
            if (sq >= 0 && allowed(sq) && g.nodes[sq].kind == NK_CONV && !g.nodes[sq].from_matmul && g.nodes[sq].stride == 1 &&
                g.nodes[sq].cin % 64 == 0 && (g.nodes[sq].cout <= 64 || g.nodes[sq].cout % 64 == 0) && g.nodes[sq].cout <= 256 &&
                g.tensors[E0.in[0]].output_slot < 0 && sc.size() == 2 && cx.sole(a) >= -1 &&
                !(g.tensors[g.nodes[sq].in[0]].input_slot >= 0 && g.tensors[g.nodes[sq].in[0]].io_layout == XENOS_LAYOUT_NCHW)) {
                int p2 = cx.sole(a);
                const bool pooled = p2 >= 0 && g.nodes[p2].kind == NK_MAXPOOL;      // (no kernel takes the squeeze and the pool)
                // (on request only: SqueezeNet with the squeezes of the six fire modules without a pool on chip takes 148 us
                // against 76 at batch 1, 164 against 86 at batch 4 and 293 against 168 at batch 32, and each of the six alone
                // makes it slower at every batch)
                if (!pooled && !by_model) {
                    out.kind = CK_CONV_CONV;
                    out.nodes = {sq, e0, e1, a};
                    out.pattern = "ConvX -> {ConvY ; ConvZ} -> concat, ConvX's result kept on chip (fire module)";
                    return true;
                }
            }
        }
        int p = cx.sole(a);
        // The pool is attached to small maps only, where it keeps the concatenation off memory: its tiles overlap (27 % more rows
        // of the expands for a 3x3 stride-2 pool) and gather their operand through the cores.  Measured, 32 -> 256 channels with
        // the squeeze before them: on maps of 64 to 484 pixels 12.3 us linked and 10.3 as two kernels (the link never wins
        // time), on 27 x 27 at batches 1, 2 and 4 12.3, 13.1 and 16.4 against 10.3, 10.7 and 12.3.  SqueezeNet with both pools
        // linked: 82 us against 76 at batch 1, 122 against 111 at batch 8.
        const bool small_map = (long)g.max_batch * g.tensors[A.out].h * g.tensors[A.out].w <= 512;
        if (p >= 0 && allowed(p) && g.nodes[p].kind == NK_MAXPOOL && (small_map || !by_model)) {
            int th, tw, rh, rw;
            const Tensor &po = g.tensors[g.nodes[p].out];
            if (pool_patch(g.nodes[p].k, g.nodes[p].stride, po.h, po.w, th, tw, rh, rw)) {
                out.nodes.push_back(p);
                out.pattern += " -> ZPooling";
            }
        }
        return true;
    }
    if (A.kind == NK_CONV) {
        // a convolution that reads the caller's NCHW image stages patches of it: it links with a pool only
        const bool nchw_in = g.tensors[A.in[0]].input_slot >= 0 && g.tensors[A.in[0]].io_layout == XENOS_LAYOUT_NCHW;
        if (!nchw_in && A.cin % 8) return false;
        int b = cx.sole(a);
        if (b < 0 || !allowed(b)) return false;
        const Node &B = g.nodes[b];
        if (B.kind == NK_CONV && !nchw_in && !A.from_matmul && !B.from_matmul && A.stride == 1 && A.cin % 64 == 0 &&
            (A.cout <= 64 || A.cout % 64 == 0) && A.cout <= 256 && A.cout % 8 == 0 && B.stride == 1 &&
            ((B.k == 1 && B.pad == 0) || (B.k == 3 && B.pad == 1)) && B.cout % 8 == 0) {
            // ConvX -> ConvY (rows 1-4 of Table 1) [-> add with an identity branch]: the intermediate tile stays on chip
            int c = cx.sole(b);
            bool with_add = false;
            if (c >= 0 && allowed(c) && g.nodes[c].kind == NK_ADD && B.act == XENOS_ACT_NONE) {
                int other = g.nodes[c].in[0] == B.out ? g.nodes[c].in[1] : g.nodes[c].in[0];
                with_add = other != B.out;
                // a shortcut with its own 1x1 convolution is better served by the shortcut row's link (that convolution
                // joins ConvY's reduction and its result never exists): leave ConvY to it
                int pj = with_add ? g.node_of_tensor[other] : -1;
                if (by_model && pj >= 0 && pj != a && g.nodes[pj].kind == NK_CONV && g.nodes[pj].k == 1 && g.nodes[pj].pad == 0 &&
                    g.nodes[pj].act == XENOS_ACT_NONE && cx.sole(pj) == c && g.nodes[pj].chain < 0 && B.k == 1)
                    return false;
            }
            // (a 3x3 consumer, like a fire module with its squeeze on chip, is linked on request only: the producer's tile carries
            // the consumer's frame and its rows are multiplied again.  Measured, 1x1 128 -> 32 and 3x3 32 -> 32, batch 16 at 64 x 64
            // and batch 32 at 128 x 128: 41 and 252 us linked, 11 + 14 and 35 + 52 as two kernels; ResNet-18 with the two blocks
            // of its first stage linked: 107.5 us against 103.8 at batch 1, 156 against 139 at batch 4, 236 against 188 at 16)
            if (!by_model || (B.k == 1 && chain2_pays(g, A, B, with_add))) {
                out.kind = CK_CONV_CONV;
                out.nodes = {a, b};
                out.pattern = B.k == 1 ? "ConvX -> ConvY (Conv kxk -> Conv 1x1, intermediate on chip)" : "ConvX -> ConvY (Conv kxk -> Conv 3x3, intermediate with its halo on chip)";
                if (with_add) { out.nodes.push_back(c); out.pattern += " + shortcut connection (identity)"; }
                return true;
            }
        }
        if (B.kind == NK_ADD && !nchw_in) {
            int other = B.in[0] == A.out ? B.in[1] : B.in[0];
            if (other == A.out) return false;
            out.kind = CK_CONV_TAIL;
            out.nodes = {a};
            out.pattern = "shortcut connection (ConvX -> {... -> ConvY ; identity})";
            int p = g.node_of_tensor[other];
            // the shortcut's own 1x1 convolution joins the chain as a second K segment
            if (p >= 0 && p != a && allowed(p) && g.nodes[p].kind == NK_CONV && g.nodes[p].k == 1 &&
                g.nodes[p].pad == 0 && g.nodes[p].act == XENOS_ACT_NONE && A.act == XENOS_ACT_NONE &&
                cx.sole(p) == b && g.nodes[p].cin % 8 == 0 && g.nodes[p].chain < 0) {
                out.nodes.push_back(p);
                out.pattern = "shortcut connection (ConvX -> {... -> ConvY ; ConvZ})";
            }
            out.nodes.push_back(b);
            int c = cx.sole(b);
            // (a global average is not attached to a long reduction that would run on a handful of units: the epilogue
            // with the average cannot take part in a reduction split, and at batch 1 the 72 K blocks of ResNet-18's last
            // convolution then run one after the other on 16 units.  The whole graph with the average attached and apart, 16 tiles
            // (batch 1): 110.9 and 103.6 us, 64 tiles (batch 9): 158.9 and 154.8, 112 (16): 193.8 and 188.5, 128 (20): 206.9 and
            // 204.9; from one tile per unit on the link wins: 160 (24): 223.0 and 223.8, 208 (32): 255.4 and 256.9)
            const long gap_tiles = (long)((g.max_batch * cx.rows(b) + 127) / 128) * ((A.cout + 31) / 32);
            const bool serial_k = by_model && (long)A.k * A.k * A.cin >= 16 * 64 && gap_tiles <= g.hw.sm_count;
            if (c >= 0 && allowed(c) && g.nodes[c].kind == NK_GAP && cx.rows(b) <= 128 && !serial_k) {
                out.nodes.push_back(c);
                out.pattern += " -> ZPooling (global average)";
            }
            return true;
        }
        if (B.kind == NK_MAXPOOL) {
            int th, tw, rh, rw;
            const Tensor &po = g.tensors[B.out];
            if (!pool_patch(B.k, B.stride, po.h, po.w, th, tw, rh, rw)) return false;
            // At batch 8 and above an image convolution and its max pool stay two kernels for images up to 256 pixels wide.  The
            // rule was measured with the kernel before stem_tc_kernel, whose pooling pass cost what a pool kernel costs.  With
            // the pool in registers the link is the faster form there, too: SqueezeNet (3x3 stem) 96 us linked against 110
            // at batch 8, 158 against 168 at 32, 245 against 270 at 64; ResNet-18 (7x7 stem) 160 against 160, 246 against 255
            // and 361 against 386; 3x3, 24 channels, 224 x 224: 21 against 30 us at batch 8, 66 against 81 at 32.  It can be
            // requested.  Below batch 8 and for wider images it is linked (7x7 stem at 512 x 512: 31 against 51 us at batch 8, 201
            // against 366 at batch 64).
            if (by_model && nchw_in && g.max_batch >= 8 && g.tensors[A.in[0]].w <= 256 && g.tensors[A.in[0]].h <= 256) return false;
            out.kind = CK_CONV_TAIL;
            out.nodes = {a, b};
            out.pattern = "ConvX -> ZPooling (CBR-MaxPooling)";
            return true;
        }
        // (an image of more than 128 pixels is averaged over several tiles when the convolution is 1x1 on 64-channel
        // blocks: its rows are then plain rows of the activation matrix)
        if (B.kind == NK_GAP && !nchw_in &&
            (cx.rows(a) <= 128 || (A.k == 1 && A.stride == 1 && A.pad == 0 && A.cin % 64 == 0 && g.precision != XENOS_PRECISION_FP32_CUDA_CORE))) {
            out.kind = CK_CONV_TAIL;
            out.nodes = {a, b};
            out.pattern = "ConvX -> ZPooling (CBR-AvgPooling, global)";
            return true;
        }
    }
    return false;
}

xenos_status_t link_pass(Graph &g) {
    LinkCtx cx(g);
    g.chains.clear();
    for (Node &n : g.nodes) n.chain = -1;
    // tensor -> node for every user tensor, including the ones folded away by the pre-fusion
    std::vector<int> node_of_any(g.tensors.size(), -1);
    for (int i = 0; i < (int)g.nodes.size(); ++i)
        for (int oi : g.nodes[i].user_ops) node_of_any[g.ops[oi].out] = i;

    auto commit = [&](Chain &c) {
        int id = (int)g.chains.size();
        for (int n : c.nodes) g.nodes[n].chain = id;
        g.chains.push_back(c);
    };
    // explicit requests first
    for (const LinkRequest &r : g.link_requests) {
        std::set<int> want;
        for (int t : r.ops) {
            int n = node_of_any[t];
            if (n < 0) return fail(g, XENOS_E_NOT_LINKABLE, "link: id is not an operator of the graph");
            if (g.nodes[n].chain >= 0) return fail(g, XENOS_E_NOT_LINKABLE, "link: operator is already part of another chain");
            want.insert(n);
        }
        bool done = false;
        for (int a : want) {
            Chain c;
            if (try_match(cx, a, [&](int n) { return want.count(n) > 0 && g.nodes[n].chain < 0; }, c, false)) {
                std::set<int> got(c.nodes.begin(), c.nodes.end());
                if (got == want) { commit(c); done = true; break; }
            }
        }
        if (!done)
            return fail(g, XENOS_E_NOT_LINKABLE,
                        "link: the requested operators match no linkable pattern that has a kernel");
    }
    if (g.link_auto) {
        // concat-anchored patterns first (their members precede the concat), then in node order
        for (int pass = 0; pass < 2; ++pass)
            for (int a = 0; a < (int)g.nodes.size(); ++a) {
                if (g.nodes[a].chain >= 0) continue;
                if ((pass == 0) != (g.nodes[a].kind == NK_CONCAT)) continue;
                Chain c;
                if (try_match(cx, a, [&](int n) { return g.nodes[n].chain < 0; }, c)) commit(c);
            }
    }
    for (int a = 0; a < (int)g.nodes.size(); ++a)
        if (g.nodes[a].chain < 0) {
            Chain c;
            c.kind = CK_SINGLE; c.nodes = {a}; c.pattern = "-";
            commit(c);
        }
    // execution order: a chain runs after the chains that produce what it reads
    int nc = (int)g.chains.size();
    std::vector<std::set<int>> deps(nc);
    for (int ci = 0; ci < nc; ++ci)
        for (int n : g.chains[ci].nodes)
            for (int t : g.nodes[n].in) {
                int p = g.node_of_tensor[t];
                if (p >= 0 && g.nodes[p].chain != ci) deps[ci].insert(g.nodes[p].chain);
            }
    std::vector<int> order, done(nc, 0);
    auto key = [&](int ci) { return *std::min_element(g.chains[ci].nodes.begin(), g.chains[ci].nodes.end()); };
    while ((int)order.size() < nc) {
        int pick = -1;
        for (int ci = 0; ci < nc; ++ci) {
            if (done[ci]) continue;
            bool ready = true;
            for (int d : deps[ci]) if (!done[d]) { ready = false; break; }
            if (ready && (pick < 0 || key(ci) < key(pick))) pick = ci;
        }
        if (pick < 0) return fail(g, XENOS_E_NOT_LINKABLE, "link: the requested chains depend on each other in a cycle");
        done[pick] = 1;
        order.push_back(pick);
    }
    std::vector<Chain> sorted;
    for (int ci : order) sorted.push_back(g.chains[ci]);
    g.chains.swap(sorted);
    for (int ci = 0; ci < nc; ++ci)
        for (int n : g.chains[ci].nodes) g.nodes[n].chain = ci;
    // attach split requests
    for (auto &rq : g.split_requests) {
        int n = node_of_any[rq.first];
        if (n < 0) return fail(g, XENOS_E_BAD_SPLIT, "split: id is not an operator of the graph");
        g.chains[g.nodes[n].chain].split = rq.second;
    }
    return XENOS_OK;
}

// ------------------------------------------------------------------------------------------------
// Split + lowering
// ------------------------------------------------------------------------------------------------
static int round_up(int v, int a) { return (v + a - 1) / a * a; }
static int ceil_div(int a, int b) { return (a + b - 1) / b; }

static size_t tensor_elems(const Tensor &t) { return t.is_vec ? (size_t)t.c : (size_t)t.c * t.h * t.w; }

struct Lower {
    Graph &g;
    explicit Lower(Graph &gg) : g(gg) {}
    int esize() const { return g.precision == XENOS_PRECISION_FP32_CUDA_CORE ? 4 : 2; }

    double tbytes(int t) const {
        const Tensor &x = g.tensors[t];
        int es = esize();
        if (g.precision == XENOS_PRECISION_BF16_TENSOR) {
            if (x.input_slot >= 0 && x.io_dtype == XENOS_DTYPE_F32) es = 4;
            if (x.output_slot >= 0 && x.is_vec) es = 4;
        }
        return (double)g.max_batch * tensor_elems(x) * es;
    }
    double node_macs(const Node &n) const {
        const Tensor &o = g.tensors[n.out];
        if (n.kind == NK_CONV) return (double)g.max_batch * o.h * o.w * n.cout * n.cin * n.k * n.k;
        if (n.kind == NK_DW) return (double)g.max_batch * o.h * o.w * n.cout * n.k * n.k;
        if (n.kind == NK_FC) return (double)g.max_batch * n.cout * n.cin;
        return 0;
    }
    double node_param_bytes(const Node &n) const {
        if (n.w.empty()) return 0;
        return (double)n.w.size() * esize() + 4.0 * n.b.size();
    }

    // ---- fp32 (CUDA-core) lowering ---------------------------------------------------------
    size_t put_f32(const std::vector<float> &v) {
        size_t off = blob_reserve(g, v.size() * 4);
        std::memcpy(g.param_blob.data() + off, v.data(), v.size() * 4);
        return off;
    }
    void push(Launch &L, int chain) {
        L.chain = chain;
        g.chains[chain].launches.push_back((int)g.launches.size());
        g.launches.push_back(L);
    }
    void fill_io(Launch &L, const Node &n) {
        const Tensor &x = g.tensors[n.in[0]];
        const Tensor &y = g.tensors[n.out];
        L.in0 = n.in[0]; L.out = n.out;
        L.C = x.c; L.H = x.h; L.W = x.w; L.K = y.c; L.P = y.h; L.Q = y.w;
        L.k = n.k; L.stride = n.stride; L.pad = n.pad; L.act = n.act;
        L.out_coff = 0; L.out_ctot = y.c;
    }
    xenos_status_t lower_single_common(int ci, int ni, bool f32) {
        const Node &n = g.nodes[ni];
        Launch L;
        L.nodes = {ni};
        fill_io(L, n);
        L.flops = 2.0 * node_macs(n);
        L.bytes = tbytes(n.out) + node_param_bytes(n);
        for (int t : n.in) L.bytes += tbytes(t);
        L.block = 256;
        switch (n.kind) {
        case NK_MAXPOOL:
        case NK_AVGPOOL:
            L.kind = f32 ? LK_F32_POOL : LK_POOL;
            L.pool_kind = n.kind == NK_MAXPOOL ? 0 : 1;
            L.pool_k = n.k; L.pool_stride = n.stride; L.pool_pad = n.pad; L.PP = L.P; L.PQ = L.Q;
            break;
        case NK_GAP:
            L.kind = f32 ? LK_F32_GAP : LK_GAP;
            L.out_dtype = (f32 || g.tensors[n.out].output_slot >= 0) ? XENOS_DTYPE_F32 : XENOS_DTYPE_BF16;
            break;
        case NK_ADD:
            L.kind = f32 ? LK_F32_ADD : LK_ADD;
            L.in1 = n.in[1];
            break;
        case NK_MUL:
        case NK_MAC:
            L.kind = f32 ? LK_F32_MULMAC : LK_MULMAC;
            L.in1 = n.in[1];
            if (n.kind == NK_MAC) L.in2 = n.in[2];
            break;
        case NK_TRANSPOSE:
            L.kind = f32 ? LK_F32_TRANSPOSE : LK_TRANSPOSE;
            if (!f32 && (L.C % 8 || L.H % 8)) return fail(g, XENOS_E_UNSUPPORTED, "bf16 transpose needs row and column counts that are multiples of 8");
            break;
        case NK_SLICE:
            L.kind = f32 ? LK_F32_SLICE : LK_SLICE;
            L.out_coff = n.pad;             // first channel of the part
            if (!f32 && (n.pad % 8 || n.cout % 8)) return fail(g, XENOS_E_UNSUPPORTED, "bf16 split needs channel offsets and counts that are multiples of 8");
            break;
        case NK_CONCAT: {
            int off = 0;
            for (int t : n.in) {
                Launch P = L;
                P.kind = f32 ? LK_F32_CONCAT_PART : LK_CONCAT_PART;
                P.in0 = t; P.C = g.tensors[t].c; P.out_coff = off; P.out_ctot = g.tensors[n.out].c;
                P.bytes = 2.0 * tbytes(t);
                off += g.tensors[t].c;
                push(P, ci);
            }
            return XENOS_OK;
        }
        default:
            return fail(g, XENOS_E_UNSUPPORTED, "internal: unexpected operator in lower_single_common");
        }
        push(L, ci);
        return XENOS_OK;
    }

    xenos_status_t lower_f32_single(int ci, int ni) {
        const Node &n = g.nodes[ni];
        if (n.kind == NK_CONV || n.kind == NK_DW || n.kind == NK_FC) {
            Launch L;
            L.nodes = {ni};
            fill_io(L, n);
            L.kind = n.kind == NK_FC ? LK_F32_FC : LK_F32_CONV;
            L.groups = n.kind == NK_DW ? n.cin : 1;
            L.w_off = put_f32(n.w); L.b_off = put_f32(n.b);
            L.flops = 2.0 * node_macs(n);
            L.bytes = tbytes(n.in[0]) + tbytes(n.out) + node_param_bytes(n);
            L.block = 256;
            if (g.chains[ci].split.user && (g.chains[ci].split.outc > 1 || g.chains[ci].split.h > 1 || g.chains[ci].split.w > 1 || g.chains[ci].split.k > 1))
                return fail(g, XENOS_E_BAD_SPLIT, "split: unlinked fp32 operators are split one output element per thread; no explicit split");
            push(L, ci);
            return XENOS_OK;
        }
        return lower_single_common(ci, ni, true);
    }

    // ConvX -> Conv1x1 -> pool as one CUDA-core kernel.  A CTA owns a tile of POOL outputs and a
    // slice of the second conv's output channels; it evaluates stage 1 on the patch the tile
    // needs (no overlap between tiles when the pool windows do not overlap).
    xenos_status_t lower_f32_linked(int ci) {
        Chain &ch = g.chains[ci];
        const Node &A = g.nodes[ch.nodes[0]], &B = g.nodes[ch.nodes[1]], &C = g.nodes[ch.nodes[2]];
        Launch L;
        L.kind = LK_F32_CONV_CONV_POOL;
        L.nodes = ch.nodes;
        fill_io(L, A);
        L.out = C.out;
        const Tensor &po = g.tensors[C.out];
        L.Cmid = A.cout; L.K2 = B.cout; L.act2 = B.act;
        L.pool_kind = C.kind == NK_MAXPOOL ? 0 : 1;
        L.pool_k = C.k; L.pool_stride = C.stride; L.pool_pad = 0; L.PP = po.h; L.PQ = po.w;
        L.out_ctot = B.cout;
        const SplitRequest &rq = ch.split;
        if (rq.user && rq.k > 1)
            return fail(g, XENOS_E_UNSUPPORTED, "split: the fp32 CUDA-core chain keeps every reduction inside one thread; parts_k applies to tensor-core convolutions and fc");
        const int smem_cap = std::min(g.hw.smem_bytes_per_cta, 227 * 1024) - 1024;
        auto region = [&](int t) { return (t - 1) * C.stride + C.k; };        // conv-output rows a tile of t pool rows reads
        const int mpad = round_up(A.cout, 8), taps = A.cin * A.k * A.k;
        auto patch_pitch = [&](int tw) { return round_up((round_up(region(tw), 4) - 1) * A.stride + A.k, 4); };
        auto mid_pitch = [&](int tw) { return round_up(tw, 4) + round_up((C.k - 1) / C.stride, 4); };
        auto smem_need = [&](int th, int tw, int po, bool ws) {
            const int rh = region(th), ih = (rh - 1) * A.stride + A.k;
            size_t f = (size_t)A.cin * ih * patch_pitch(tw) + (size_t)mpad * rh * C.stride * mid_pitch(tw) + mpad + round_up(B.cout / po, 8);
            if (ws) f += (size_t)taps * mpad + (size_t)A.cout * round_up(B.cout / po, 8);
            return 4 * f;
        };
        int best_po = 0, best_th = 0, best_tw = 0, best_var = 0;
        double best_cost = 0;
        std::vector<int> po_cands, th_cands, tw_cands;
        if (rq.user && rq.outc > 0) {
            if (rq.outc > B.cout || B.cout % rq.outc) return fail(g, XENOS_E_BAD_SPLIT, "split: parts_outc must divide the output channels");
            po_cands = {rq.outc};
        } else
            for (int p = 1; p <= B.cout && p <= 16; ++p) if (B.cout % p == 0) po_cands.push_back(p);
        auto dim_cands = [&](int req, int extent, std::vector<int> &out_tiles) -> bool {
            if (rq.user && req > 0) {
                if (req > extent) return false;
                out_tiles = {ceil_div(extent, req)};
                return ceil_div(extent, out_tiles[0]) == req;
            }
            for (int t = 1; t <= extent; ++t) out_tiles.push_back(t);
            return true;
        };
        if (!dim_cands(rq.h, po.h, th_cands)) return fail(g, XENOS_E_BAD_SPLIT, "split: parts_h does not divide the output rows into equal-height tiles");
        if (!dim_cands(rq.w, po.w, tw_cands)) return fail(g, XENOS_E_BAD_SPLIT, "split: parts_w does not divide the output columns into equal-width tiles");
        // Modelled cycles of a plan: waves over the units, per tile the patch's copy and, per stage, the warp-sized groups of
        // register tiles that a scheduler runs in turn (8 x 4 tiles: 32 cycles of the FMA pipe per product step, at least four
        // groups' worth because one warp alone waits for its own results; 2 x 1 tiles: 8 cycles, latency included).
        // bit 0 of a variant: 8 x 4 tiles, bit 1: weights in shared memory.
        for (int p : po_cands)
            for (int th : th_cands)
                for (int tw : tw_cands)
                    for (int var = 0; var < 4; ++var) {
                        const bool big = var & 1, ws = var & 2;
                        const size_t need = smem_need(th, tw, p, ws);
                        if (need > (size_t)smem_cap) continue;
                        const int rh = region(th), rw = region(tw), tm = big ? 8 : 2, tp = big ? 4 : 1;
                        const double step = (big ? 32.0 : 8.0) * (ws ? 1.0 : 1.6), least = big ? 4.0 : 1.0;
                        auto groups = [&](double units) { return std::max(least, std::ceil(std::ceil(units / 32.0) / 4.0)); };
                        const double s1 = taps * step * groups((double)(mpad / tm) * rh * ceil_div(rw, tp));
                        const double wide = round_up(B.cout / p, 8) / tm;
                        const double s2 = C.k == 2 ? A.cout * (big ? step : 3.0 * step) * groups(wide * th * tw)      // (four window pixels at a time)
                                                   : (double)C.k * C.k * A.cout * step * groups(wide * th * ceil_div(tw, tp));
                        const double copy = 800.0 + (double)A.cin * ((rh - 1) * A.stride + A.k) * patch_pitch(tw) / 16.0;
                        const long ctas = (long)p * ceil_div(po.h, th) * ceil_div(po.w, tw) * g.max_batch;
                        const double cost = std::ceil((double)ctas / g.hw.sm_count) * (s1 + s2 + copy) + (ws ? (taps * mpad + A.cout * B.cout / p) * 4.0 / 50.0 : 0.0);
                        if (best_po == 0 || cost < best_cost) { best_cost = cost; best_po = p; best_th = th; best_tw = tw; best_var = var; }
                    }
        if (best_po == 0) return fail(g, XENOS_E_BAD_SPLIT, "split: no tile of the linked chain fits shared memory");
        L.parts_outc = best_po; L.tile_h = best_th; L.tile_w = best_tw;
        L.tiles_h = ceil_div(po.h, best_th); L.tiles_w = ceil_div(po.w, best_tw);
        L.halo_h = region(best_th); L.halo_w = region(best_tw);
        L.f32_big = best_var & 1; L.f32_ws = (best_var >> 1) & 1;
        L.f32_iwp = patch_pitch(best_tw); L.f32_hp = mid_pitch(best_tw); L.npad = mpad;
        L.smem_bytes = (int)smem_need(best_th, best_tw, best_po, L.f32_ws);
        L.grid = L.parts_outc * L.tiles_h * L.tiles_w;   // per image
        L.block = L.f32_big ? 512 : 256;
        {
            // w1 [channel][row][column][Cmid], w2 [part][Cmid][channels of the part]: output channels innermost, padded to 8
            std::vector<float> w1((size_t)taps * mpad, 0.0f);
            for (int m = 0; m < A.cout; ++m)
                for (int t = 0; t < taps; ++t) w1[(size_t)t * mpad + m] = A.w[(size_t)m * taps + t];
            const int kper = B.cout / best_po, kperp = round_up(kper, 8);
            std::vector<float> w2((size_t)best_po * A.cout * kperp, 0.0f);
            for (int k = 0; k < B.cout; ++k)
                for (int m = 0; m < A.cout; ++m) w2[((size_t)(k / kper) * A.cout + m) * kperp + k % kper] = B.w[(size_t)k * A.cout + m];
            L.w_off = put_f32(w1); L.b_off = put_f32(A.b);
            L.w2_off = put_f32(w2); L.b2_off = put_f32(B.b);
        }
        L.flops = 2.0 * (node_macs(A) + node_macs(B));
        L.bytes = tbytes(A.in[0]) + tbytes(C.out) + node_param_bytes(A) + node_param_bytes(B);
        push(L, ci);
        return XENOS_OK;
    }

    // ---- bf16 tensor-core lowering ---------------------------------------------------------
    // ---- tiles of conv_tc_kernel ------------------------------------------------------------------------------------
    // Clusters of ks CTAs that fit the units of the hardware description at once, one CTA or two (half) per unit.  The table is
    // what the 148 SMs of a B200 answer (clusters stay inside a GPC, so the larger ones leave SMs unused); other unit counts get
    // their share of it.
    int cluster_capacity(int ks, bool half) const {
        static const int one[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15}, two[9] = {0, 296, 148, 93, 71, 56, 45, 37, 33};
        return (int)((long)(half ? two[ks] : one[ks]) * g.hw.sm_count / 148);
    }
    int conv_smem_cap(bool half) const { return std::min(g.hw.smem_bytes_per_cta, half ? kClusterSmem : 227 * 1024); }
    static constexpr int kClusterSmem = 112 * 1024;      // what two CTAs of an SM can have each
    // Exchange buffer of a cluster's partial sums.
    static int cluster_bytes(int rows, int tile_n, int ks) { return (int)align_up((size_t)ks * ceil_div(rows, ks) * (tile_n + 4) * 4, 1024); }
    // Modelled cycles of a plan with tile_n columns and ksplit chunks on `units` SMs.  Per 64-wide K block a CTA waits for
    // the slower of the tensor pipe (max(48, tile_n / 2) cycles per K = 16 step) and the operand traffic from L2 (75
    // bytes per cycle and SM); a tile's epilogue overlaps the next tile's product; a split adds the exchange of the partial
    // sums.  The constants are measurements on B200 (see conv_tc.cuh), but a stage of several copy requests is charged like one
    // (four im2col boxes of 16 channels are 300 cycles here and 720 of a filling thread, of which there are two), and the exchange is that
    // of 16-byte stores through distributed shared memory, before the bulk copies.
    double conv_cycles(const Launch &L, int tile_n, int n_tiles, int ksplit, bool half) const {
        const double units = g.hw.sm_count;
        const double tiles = (double)L.m_tiles * n_tiles;
        const int kb = ceil_div(L.kblocks, ksplit);
        const double mma = 4.0 * std::max(48.0, tile_n / 2.0);
        const double load = (L.a_rows * 128.0 + tile_n * 128.0) / 75.0;
        const double main = kb * std::max(mma, std::max(load, 300.0));
        const double epi = 400.0 + 5.0 * tile_n;
        if (ksplit == 1) return std::ceil(tiles / units) * std::max(main, epi) + std::min(main, epi);
        const double shared = std::max(1.0, tiles * ksplit / units);      // CTAs of one SM share its pipes
        return std::ceil(tiles / cluster_capacity(ksplit, half)) * (main * (half ? std::min(2.0, shared) : 1.0) + epi) + 1700.0 + L.a_rows * tile_n / 32.0;
    }
    // Widths are the equal cuts of the output channels (Section 4.2.1) down to 32 columns; the reduction is cut (Section
    // 4.2.2) only where that is modelled to be faster, into chunks of at least two K blocks that run at the same time.
    void choose_conv_tiles(Launch &L, int N16, const SplitRequest &rq, bool fc, int &ksplit) const {
        double best = -1;
        const bool can_split = L.epi == EPI_STORE && !rq.user;
        ksplit = 1;
        for (int nt = ceil_div(N16, 256); nt <= N16 / 16; ++nt) {
            const int tn = round_up(ceil_div(N16, nt), 16);
            if ((nt - 1) * tn >= N16) continue;                    // an empty last tile
            if (tn < 32 && nt > ceil_div(N16, 256)) break;
            for (int ks = 1; ks <= 8; ++ks)
                for (int half = 0; half < 2; ++half) {
                    const int per = ceil_div(L.kblocks, ks);
                    if (ks == 1 && half) continue;
                    if (ks > 1) {
                        if (!can_split || L.kblocks < 2 * ks || ceil_div(L.kblocks, per) != ks) continue;
                        const int ring = conv_smem_cap(half) - 1536 - (int)align_up((size_t)nt * tn * 4, 128) - cluster_bytes(L.a_rows, tn, ks);
                        if (ring < std::min(4, std::max(3, per)) * (16384 + tn * 128)) continue;
                        if ((long)L.m_tiles * nt > cluster_capacity(ks, half) || (fc && (long)L.m_tiles * nt * ks > g.hw.sm_count)) continue;
                    }
                    // (a fully connected layer of few rows is a pass over its weights: it always spreads over the units)
                    const double c = conv_cycles(L, tn, nt, ks, half) + (fc && ks == 1 && L.m_tiles == 1 && L.kblocks >= 4 ? 1e6 : 0);
                    if (best < 0 || c < best) { best = c; L.n_tiles = nt; L.tile_n = tn; ksplit = ks; L.half = half; }
                }
        }
    }
    // Convolution of an NCHW image in stem_tc_kernel: false when the shape is outside it (1 x 1 windows, more than 7 channels, a
    // pool whose windows overlap by more than one row, rows too wide for the ring).
    bool layout_stem(Launch &L, const Node &M, const Tensor &src, const Node *pooln, int N, const SplitRequest &rq) {
        const int C = src.c, k = M.k, S = M.stride;
        if (k < 2 || k > 8 || C > 7 || (rq.user && (rq.h > 1 || rq.w > 1 || rq.k > 1))) return false;
        if (pooln && !pool_in_registers(*pooln, L.P)) return false;
        L.n_tiles = rq.user && rq.outc > 0 ? rq.outc : ceil_div(N, 64);
        L.tile_n = round_up(ceil_div(N, L.n_tiles), 16);
        if (L.tile_n > 64 || (L.n_tiles - 1) * L.tile_n >= N) return false;
        L.npad = L.n_tiles * L.tile_n;
        // A piece may start before its window (the extra elements meet zero weights) where that makes the loads of two
        // adjacent columns of a stride-2 window whole aligned groups of 4 elements; rows must then be multiples of a group, too.
        L.st_lead = 0; L.st_vec = 0;
        if (S == 2) {
            const int lead = (4 - M.pad % 4) % 4;
            if (k + lead <= 8) { L.st_lead = lead; L.st_vec = src.w % 4 == 0 ? 1 : 0; }
        }
        const int rows = pooln ? L.PP : L.P, cols = pooln ? L.PQ : L.Q;
        L.st_pairs = k / 2 * C + (k % 2 ? (C + 1) / 2 : 0);
        // Rows that are whole 16-byte pieces travel by bulk copies, several per producer warp under way (strides 1 and 2): a slot
        // holds a row between zeros for the padding, and the region starts with a row of zeros.
        const int es = src.io_dtype == XENOS_DTYPE_F32 ? 4 : 2;
        const bool by_rows = src.w * es % 16 == 0 && src.w * es <= 4096 && (S == 1 || L.st_vec);
        L.st_raw_lead = round_up((M.pad + L.st_lead) * es, 16);
        L.st_raw_stride = L.st_raw_lead + src.w * es + round_up(M.pad * es, 16);
        const int wbytes = L.st_pairs * 2 * L.tile_n * 16, pc = L.tile_n <= 16 ? 1 : L.tile_n <= 32 ? 2 : 3;
        const int cap = std::min(g.hw.smem_bytes_per_cta, 227 * 1024) - 1024 - 512;
        // (a producer warp makes at most 128 lanes' worth of a row: two columns each, or one for strides above 2)
        const int most = S <= 2 ? 256 : 128;
        auto fit = [&](int cbs) {
            L.st_cbs = cbs;
            L.st_cw = round_up(ceil_div(cols, cbs), 2);
            // (columns of the convolution behind a block of the pool's columns; their first is rounded down to an even one)
            const int width = std::min(L.Q, pooln ? (L.st_cw - 1) * pooln->stride + pooln->k + 1 : L.st_cw);
            if (width > most) return false;
            L.st_qp = round_up(width, 8);
            const int row = C * L.st_qp * 16, stage = pooln ? 2 * width << (4 + pc) : 0;
            const int base = wbytes + 2048 + 256 + 512 + (int)align_up((size_t)stage, 128);
            // four rows of a warp under way before more steps of the ring; two where four do not fit; else loads into registers
            auto deepest = [&](int raw) {
                const int rbytes = raw ? (int)align_up((size_t)(1 + 7 * raw) * L.st_raw_stride, 128) : 0;
                for (int D = 6; D >= 2; --D) {
                    L.st_slots = (D - 1) * std::min(S, k) + k;
                    if ((L.st_slots + 1) * row + rbytes + base <= cap) { L.hstages = D; L.st_raw = raw; return rbytes; }
                }
                return -1;
            };
            int rbytes = -1;
            if (by_rows) { rbytes = deepest(4); if (rbytes < 0) rbytes = deepest(2); }
            if (rbytes < 0) rbytes = deepest(0);
            if (rbytes >= 0) {
                L.off_raw = (int)align_up((size_t)(L.st_slots + 1) * row + 2048, 128);       // (zeros of one chunk; a tile's last rows read past its pieces)
                L.off_b = L.off_raw + rbytes;
                L.off_bias = L.off_b + wbytes;
                L.off_stg = L.off_bias + 256;
                L.off_bar = (int)align_up((size_t)(L.off_stg + stage), 128);
                L.smem_bytes = L.off_bar + 768 + 1024;
                return true;
            }
            return false;
        };
        int cbs = ceil_div(cols, most);
        while (!fit(cbs)) {
            if (ceil_div(cols, cbs) <= 8) return false;
            ++cbs;
        }
        // few images: columns are cut until the rows of all blocks cover the units (a block of at least 32 columns)
        while ((long)g.max_batch * rows * cbs * L.n_tiles * 2 <= g.hw.sm_count && ceil_div(L.Q, cbs * 2) >= 32 && fit(cbs * 2)) cbs *= 2;
        if (!fit(cbs)) return false;
        L.st_cbs = ceil_div(cols, L.st_cw);
        L.stem_tc = 1; L.st_pc = pc;
        L.m_tiles = pooln ? g.max_batch * L.tiles_y * L.tiles_x : g.max_batch * L.P * L.st_cbs * ceil_div(L.st_qp, 128);
        L.stages = L.hstages;
        L.grid = (int)std::min<long>((long)g.max_batch * rows * L.st_cbs, std::max(1, g.hw.sm_count / L.n_tiles)) * L.n_tiles;
        L.block = 512;
        L.acc_stride = L.tile_n <= 32 ? 32 : 64;
        L.tmem_cols = 4 * L.acc_stride;
        return true;
    }
    // Weights in the order of its products: [channel tile][pair][two chunks][output channel][8 elements of a window row].
    void pack_stem(Launch &L, const Node &M, int C) {
        const int k = M.k;
        L.w_off = blob_reserve(g, (size_t)L.n_tiles * L.st_pairs * 2 * L.tile_n * 16);
        L.b_off = blob_reserve(g, (size_t)L.npad * 4);
        uint16_t *wp = reinterpret_cast<uint16_t *>(g.param_blob.data() + L.w_off);
        float *bp = reinterpret_cast<float *>(g.param_blob.data() + L.b_off);
        auto chunk = [&](int pair, int half, int c, int r) {
            for (int o = 0; o < M.cout; ++o) {
                const int nt = o / L.tile_n, n = o - nt * L.tile_n;
                uint16_t *d = wp + ((((size_t)nt * L.st_pairs + pair) * 2 + half) * L.tile_n + n) * 8 + L.st_lead;
                for (int s = 0; s < k; ++s) d[s] = f32_to_bf16_rne(M.w[(((size_t)o * C + c) * k + r) * k + s]);
            }
        };
        int pair = 0;
        for (int r = 0; r + 1 < k; r += 2)
            for (int c = 0; c < C; ++c, ++pair) { chunk(pair, 0, c, r); chunk(pair, 1, c, r + 1); }
        if (k % 2) {
            for (int c = 0; c + 1 < C; c += 2, ++pair) { chunk(pair, 0, c, k - 1); chunk(pair, 1, c + 1, k - 1); }
            if (C % 2) chunk(pair, 0, C - 1, k - 1);      // (its second chunk meets zeros)
        }
        for (int o = 0; o < M.cout; ++o) bp[o] = M.b[o];
    }

    // Shared memory and epilogue shape of conv_tc_kernel.
    xenos_status_t layout_conv(Launch &L, const Tensor &ot) {
        const bool vec = L.out_dtype == XENOS_DTYPE_F32 || ot.c % 8;
        // (up to eight chunks are the CTAs of a cluster while the exchange buffer leaves room for the ring; other splits go
        // through the workspace).  The exchange parks a tile's partial sums, 128 rows of tile_n + 4 words, in the ring: three stages
        // hold them at every width, two do so only below 124 columns.
        const int xbytes = cluster_bytes(std::min(128, g.max_batch * L.rows_per_image), L.tile_n, L.ksplit);
        const bool cluster = L.ksplit > 1 && L.ksplit <= 8 && xbytes + 3 * (16384 + L.tile_n * 128) + L.npad * 4 + 2048 <= conv_smem_cap(L.half);
        L.cv_epi = L.epi == EPI_GAP ? 3 : cluster ? 5 : L.ksplit > 1 ? 4 : vec ? 2 : L.skip >= 0 ? 1 : 0;
        if (L.cv_epi == 2 && L.skip >= 0) return fail(g, XENOS_E_UNSUPPORTED, "internal: shortcut on a vector result");
        int stg = 0;
        L.chunk = 16;
        if (L.cv_epi == 0 || L.cv_epi == 1) {
            // the widest column chunk that gives both warps of a quarter the same number of chunks
            // (at tile_n = 256 the 64-column boxes would take the fourth stage of the ring)
            for (int c : {64, 32, 16})
                if (L.tile_n % c == 0 && (L.tile_n / c) % 2 == 0 && !(c == 64 && L.tile_n > 160)) { L.chunk = c; break; }
            if (L.cv_epi == 1) L.s_slots = 4;
            stg = 8 * L.s_slots * L.chunk * 64;      // 32-row boxes of eight warps
        } else if (L.cv_epi == 5) {
            stg = xbytes;
        } else if (L.cv_epi == 3) {
            L.chunk = 32;
            stg = 2 * 4352 * 4;
        }
        L.nchunks = ceil_div(L.tile_n, L.chunk);
        stg = (int)align_up((size_t)stg, 1024);
        const int bias = (int)align_up((size_t)L.npad * 4, 128);
        // (a CTA with one tile takes half an SM when four stages fit there: the next kernel's CTAs can then set up beside it)
        const bool half = (L.cv_epi == 5 && L.half) || (L.ksplit == 1 && (long)L.m_tiles * L.n_tiles <= g.hw.sm_count &&
                                                        kClusterSmem - 1536 - bias - stg >= std::min(4, std::max(2, L.kblocks)) * (16384 + L.tile_n * 128));
        const int room = conv_smem_cap(half) - 1024 - 512 - bias - stg;
        const int bbytes = L.kblocks * L.tile_n * 128;
        // weights stay in shared memory when a CTA meets more than one tile of its channel tile and four operand stages
        // still fit beside them
        const int rgrid = g.hw.sm_count / L.n_tiles * L.n_tiles;
        L.b_resident = L.ksplit == 1 && rgrid > 0 && (long)L.m_tiles * L.n_tiles > rgrid && room - bbytes >= 4 * 16384;
        const int stage = 16384 + (L.b_resident ? 0 : L.tile_n * 128);
        L.stage_bytes = stage;
        L.stages = std::min(6, (room - (L.b_resident ? bbytes : 0)) / stage);
        if (L.stages < 2) return fail(g, XENOS_E_BAD_SPLIT, "split: pipeline does not fit shared memory");
        L.b_group = ceil_div(L.kblocks, 4);
        L.off_b = L.stages * stage;
        L.off_stg = L.off_b + (L.b_resident ? bbytes : 0);
        L.off_bias = L.off_stg + stg;
        L.off_bar = L.off_bias + bias;
        L.smem_bytes = L.off_bar + 512 + 1024;
        L.grid = std::min(L.m_tiles * L.n_tiles * L.ksplit, L.b_resident ? rgrid : g.hw.sm_count);
        L.block = 384;
        return XENOS_OK;
    }

    // Worker groups, rings and shared memory of dw_tc_kernel for the tile geometry at hand.  A group of 2^w warps covers a
    // tile's units (a lane owns br x 4 pixels of a channel pair); an item takes the slower of the issue slots of its warps
    // (a scheduler runs a quarter of the 16 warps) and its own latency shared by the groups.  The configuration with the least time whose rings fit is taken; what is left goes to deeper rings.
    xenos_status_t layout_dw(Launch &L) {
        const ASeg &s0 = L.seg[0];
        const int C = s0.C, cols = L.n_acc * L.tile_n, pairs = L.halo_cb > 32 ? 32 : 16;
        const long tiles = (long)L.m_tiles * L.n_tiles * L.ksplit;
        const bool one = tiles <= g.hw.sm_count;                  // a CTA's only tile: results leave through the operand ring
        const int dww = (int)align_up((size_t)40 * C, 1024), bias = (int)align_up((size_t)L.npad * 4, 128);
        const int room = std::min(g.hw.smem_bytes_per_cta, 227 * 1024) - 2048 - 512 - dww - bias;
        // A slot of the operand ring holds the tile's rows, in whole groups of eight; a product reads 128 rows from its start and
        // what the rows behind the tile's own give is not stored.  `ops_end`: the reads of the last slot stay inside the allocation.
        L.a_stride = ceil_div(L.tile_rows, 8) * 1024;
        auto ops_end = [&](int a_slots, int b_bytes) { return std::max(a_slots * L.a_stride + b_bytes, (a_slots - 1) * L.a_stride + 16384); };
        const int bslot = L.tile_n * 128, bblk = L.n_acc * bslot;      // a slot of the weight ring; the weights of a K block
        // (the window covers whole blocks of br rows)
        auto window_h = [&](int br) { return (round_up(L.patch_rh, br) - 1) * s0.stride + 3; };
        auto window = [&](int br) { return (int)align_up((size_t)L.ni * window_h(br) * L.halo_w * L.halo_cb * 2, 128); };
        const int rgrid = g.hw.sm_count / L.n_tiles * L.n_tiles;
        L.cv_epi = L.epi == EPI_GAP ? 1 : L.ksplit > 1 ? 2 : 0;
        const bool batched = L.cv_epi == 0 && L.n_acc == 1 && !one;
        auto staging = [&](int chunk, int bufs) {
            if (L.cv_epi == 2) return 0;
            if (L.cv_epi == 1) {
                const int per = 4 * L.gap_imgs * 32, parts = per * 4 <= 512 ? 4 : (per * 2 <= 512 ? 2 : 1);
                return (int)align_up((size_t)4 * 128 * 33 * 4 + (size_t)per * parts * 4, 1024);
            }
            return 4 * bufs * 128 * chunk * 2;
        };
        double best = -1;
        for (int br : {4, 2, 1}) {
            if (br > 1 && L.patch_rh <= br / 2) continue;
            const int units = L.ni * ceil_div(L.patch_rh, br) * (L.patch_rw / 4) * pairs, hstride = window(br);
            const double issue = s0.stride == 1 ? (br == 4 ? 340.0 : br == 2 ? 200.0 : 125.0) : (br == 4 ? 460.0 : br == 2 ? 270.0 : 160.0);
            if (window_h(br) > 256) continue;
            for (int w = 0; w <= 4; ++w) {
                if ((32 << w) < units) continue;
                const int groups = 16 >> w;
                // tiles of a batch: at least one item for every group, an accumulator pair each, no more than a CTA has
                const int nb_most = batched ? std::max(1, std::min({g.hw.tmem_columns / (2 * L.acc_stride), 4, (int)((tiles + g.hw.sm_count - 1) / g.hw.sm_count)})) : 1;
                const int nb_least = std::min(nb_most, batched ? ceil_div(groups, L.kblocks) : 1);
                for (int res = 1; res >= 0; --res)
                    for (int chunk : {64, 32, 16})
                      for (int nb = nb_least; nb <= nb_most; ++nb)
                        for (int bufs = 2; bufs >= 1; --bufs) {
                            if (L.cv_epi == 0 && cols % chunk) continue;
                            if (L.cv_epi != 0 && (chunk != (L.cv_epi == 1 ? 32 : 16) || bufs == 2)) continue;
                            if (res && (L.ksplit > 1 || L.n_acc > 1 || rgrid == 0)) continue;
                            const int a_min = std::max(2, groups), h_min = std::max(2, groups), b_min = res ? 0 : 1 + L.n_acc;
                            const int ops = ops_end(a_min, res ? L.kblocks * bblk : b_min * bslot), st = staging(chunk, bufs);
                            const int need = (one ? std::max(ops, st) : ops + st) + h_min * hstride;
                            if (a_min > 8 || h_min > 8 || need > room) continue;
                            // The workers' time per tile: the stencils, then their group's boxes, which cost some 1100 cycles and
                            // 14 a column (measured, barriers and store hand-over included), so that four groups with one 64-column
                            // box each of four tiles beat four 16-column boxes of every tile.  (A single box buffer is charged 10
                            // cycles per K block, an estimate.)
                            const double t = L.kblocks * (std::max((1 << w) * issue / 4.0, (300.0 + 2.2 * issue) / groups) + (res ? 0.0 : 20.0) + (bufs == 1 ? 10.0 : 0.0)) +
                                             (L.cv_epi == 0 ? (double)ceil_div(nb * ceil_div(cols, chunk), 4) / nb * (1100.0 + 14.0 * chunk) : 0.0);
                            if (best >= 0 && t >= best) continue;
                            best = t;
                            L.chunk = chunk; L.dw_batch = nb;
                            L.dw_br = br; L.dw_wpg_log2 = w; L.dw_groups = groups; L.b_resident = res; L.out_bufs = bufs;
                            L.a_slots = a_min; L.h_slots = h_min; L.b_slots = b_min;
                        }
            }
        }
        if (best < 0) return fail(g, XENOS_E_BAD_SPLIT, "split: pipeline does not fit shared memory");
        const int st = staging(L.chunk, L.out_bufs), groups = L.dw_groups, hstride = window(L.dw_br);
        L.halo_h = window_h(L.dw_br);
        L.halo_bytes = L.ni * L.halo_h * L.halo_w * L.halo_cb * 2;
        L.halo_stride = hstride;
        auto used = [&]() {
            const int ops = ops_end(L.a_slots, L.b_resident ? L.kblocks * bblk : L.b_slots * bslot);
            return (one ? std::max(ops, st) : ops + st) + L.h_slots * hstride;
        };
        // deeper rings with what is left: windows first (they come from the predecessor's tensor), then weights, then operands
        auto grow = [&](int &slots, int by, int most) { while (slots + by <= most) { slots += by; if (used() > room) { slots -= by; break; } } };
        grow(L.h_slots, groups, std::min(8, 2 * std::max(2, groups)));
        // (a CTA with one tile asks for all of its weights while the predecessor drains, where they fit)
        if (!L.b_resident) grow(L.b_slots, 1, std::min(one ? 8 : 4, std::max(2, L.n_acc * L.kblocks)));
        grow(L.a_slots, groups, std::min(8, one ? L.kblocks : 2 * std::max(2, groups)));
        L.nchunks = ceil_div(cols, L.chunk);
        L.off_b = L.a_slots * L.a_stride;
        const int ops = ops_end(L.a_slots, L.b_resident ? L.kblocks * bblk : L.b_slots * bslot);
        L.off_stg = one ? 0 : ops;
        L.off_halo = (int)align_up((size_t)(one ? std::max(ops, st) : ops + st), 1024);
        L.off_dww = (int)align_up((size_t)L.off_halo + (size_t)L.h_slots * hstride, 128);
        L.off_bias = L.off_dww + dww;
        L.off_bar = L.off_bias + bias;
        L.smem_bytes = L.off_bar + 512 + 1024;
        L.stages = std::min(6, L.a_slots); L.hstages = L.h_slots;
        L.dw_workers = 16;
        L.grid = (int)std::min<long>(tiles, L.b_resident ? rgrid : g.hw.sm_count);
        L.block = 96 + 32 * 16;
        L.tmem_cols = 32;
        while (L.tmem_cols < (L.n_acc == 2 ? 2 : 2 * L.dw_batch) * L.acc_stride) L.tmem_cols *= 2;
        return XENOS_OK;
    }

    xenos_status_t make_gemm(int ci, const std::vector<int> &cover, const Node *dw, const Node *mainc,
                             const Node *shortcut, const Node *expand2, const Node *addn, const Node *pooln,
                             const Node *gapn, const Node *catn, bool fc) {
        Chain &ch = g.chains[ci];
        Launch L;
        L.kind = LK_GEMM;
        L.nodes = cover;
        const Node &M = *mainc;
        const Tensor &src = g.tensors[dw ? dw->in[0] : M.in[0]];
        const Tensor &convout = g.tensors[M.out];
        L.in0 = dw ? dw->in[0] : M.in[0];
        L.C = src.c; L.H = fc ? 1 : src.h; L.W = fc ? 1 : src.w;
        L.P = fc ? 1 : convout.h; L.Q = fc ? 1 : convout.w;
        L.rows_per_image = L.P * L.Q;
        L.k = M.k; L.stride = M.stride; L.pad = M.pad;
        int N = M.cout + (expand2 ? expand2->cout : 0);
        L.K = N;
        // --- A segments
        ASeg &s0 = L.seg[0];
        s0.tensor = L.in0; s0.C = src.c; s0.H = L.H; s0.W = L.W;
        int kk = expand2 ? std::max(M.k, expand2->k) : M.k;     // merged expand reads the 3x3 window
        int kpadg = expand2 ? 1 : M.pad;
        if (dw) {
            s0.mode = AM_DW; s0.k = dw->k; s0.stride = dw->stride; s0.pad = dw->pad;
            s0.kelems = src.c; s0.dw_act = dw->act;
            // depthwise taps, tap-major fp32 [9][C], so a thread reads 8 consecutive channels per tap
            std::vector<float> wt((size_t)9 * src.c);
            for (int c = 0; c < src.c; ++c)
                for (int t = 0; t < 9; ++t) wt[(size_t)t * src.c + c] = dw->w[(size_t)c * 9 + t];
            s0.dw_w_off = put_f32(wt);
            s0.dw_b_off = put_f32(dw->b);
        } else if (src.input_slot >= 0 && src.io_layout == XENOS_LAYOUT_NCHW) {
            if (expand2) return fail(g, XENOS_E_UNSUPPORTED, "internal: expand on an NCHW input");
            // K order of a stem with k > 4: (channel, tap row) segments of 8 elements, the taps of one window row,
            // which are adjacent in the image: a producer thread copies a segment instead of gathering elements.
            // Small kernels keep (tap, channel) order without padding inside K.
            if (M.k > 8) return fail(g, XENOS_E_UNSUPPORTED, "a convolution on an NCHW image supports kernels up to 8 x 8");
            s0.mode = AM_STEM; s0.k = M.k; s0.stride = M.stride; s0.pad = M.pad;
            s0.kelems = M.k > 4 ? src.c * M.k * 8 : M.k * M.k * src.c; s0.src_dtype = src.io_dtype;
        } else {
            if (src.c % 8) return fail(g, XENOS_E_UNSUPPORTED, "bf16 NHWC tensors need a channel count that is a multiple of 8");
            s0.mode = AM_GATHER; s0.k = kk; s0.stride = M.stride; s0.pad = expand2 ? kpadg : M.pad;
            s0.kelems = kk * kk * src.c;
        }
        // Everything that gathers an NHWC window and stores rows, vectors or averages runs in conv_tc_kernel: the copy
        // engine brings a tap's channels in boxes of 64, 32 or 16, so the packed K order gives every tap whole boxes.
        const bool tc = s0.mode == AM_GATHER && !pooln;
        auto boxes = [&](ASeg &a) {
            a.cbox = a.C > 32 ? 64 : a.C > 16 ? 32 : 16;
            a.cpad = a.cbox == 64 ? round_up(a.C, 64) : a.cbox;
            a.kelems = a.k * a.k * a.cpad;
        };
        if (tc) boxes(s0);
        s0.kblocks = ceil_div(s0.kelems, 64);
        ASeg &s1 = L.seg[1];
        if (shortcut) {
            const Tensor &ss = g.tensors[shortcut->in[0]];
            s1.mode = AM_GATHER; s1.tensor = shortcut->in[0]; s1.C = ss.c; s1.H = ss.h; s1.W = ss.w;
            s1.k = 1; s1.stride = shortcut->stride; s1.pad = 0; s1.kelems = ss.c;
            if (tc) boxes(s1);
            s1.kblocks = ceil_div(s1.kelems, 64);
        }
        L.kblocks = s0.kblocks + s1.kblocks;
        L.kpad = 64 * L.kblocks;
        // --- epilogue
        L.act = M.act;
        const Node *last = mainc;
        if (catn) last = catn;
        if (addn) {
            last = addn;
            L.act2 = addn->act;
            if (!shortcut) L.skip = addn->in[0] == M.out ? addn->in[1] : addn->in[0];
        }
        if (pooln) {
            last = pooln;
            L.epi = EPI_POOL; L.map_mode = MAP_PATCH;
            L.pool_kind = 0; L.pool_k = pooln->k; L.pool_stride = pooln->stride; L.pool_pad = pooln->pad;
            const Tensor &po = g.tensors[pooln->out];
            L.PP = po.h; L.PQ = po.w;
            if (!pool_patch(pooln->k, pooln->stride, po.h, po.w, L.patch_th, L.patch_tw, L.patch_rh, L.patch_rw))
                return fail(g, XENOS_E_UNSUPPORTED, "internal: pool patch does not fit");
            L.tiles_y = ceil_div(po.h, L.patch_th); L.tiles_x = ceil_div(po.w, L.patch_tw);
            L.ni = 1;
            L.step_y = L.patch_th * pooln->stride; L.step_x = L.patch_tw * pooln->stride;
            L.off_y = L.off_x = pooln->pad;
            L.tile_rows = L.patch_rh * L.patch_rw;
        }
        if (gapn) {
            last = gapn;
            L.epi = EPI_GAP;
            L.imgs_per_tile = 128 / L.rows_per_image;
            L.tile_rows = L.imgs_per_tile * L.rows_per_image;
            L.gap_imgs = L.imgs_per_tile; L.gap_area = L.rows_per_image; L.gap_rpi = L.rows_per_image;
            if (L.rows_per_image > 128) {
                // several tiles per image: 128 rows each, their column sums combined by the tile that finishes last
                if (dw || shortcut || expand2 || M.k != 1 || M.stride != 1 || M.pad != 0 || src.c % 64)
                    return fail(g, XENOS_E_UNSUPPORTED, "internal: global average over more than 128 pixels needs a 1x1 convolution on 64-channel blocks");
                L.gap_parts = ceil_div(L.rows_per_image, 128);
                L.imgs_per_tile = 1; L.tile_rows = 128;
                L.gap_imgs = 1; L.gap_area = 128;
            }
        }
        // (which activation operands are plain boxes of the tensor: 1 rows of the [pixels][C] matrix, 2 a patch per tap;
        // the others need the im2col form, or share a K block between taps)
        if (tc) {
            if (!expand2 && !shortcut && src.c % 64 == 0 && M.stride == 1) L.a_tma = (M.k == 1 && M.pad == 0) ? 1 : (!gapn && !fc) ? 2 : 0;
            L.conv_tc = 1;
            L.a_rows = gapn ? 128 : std::min(128, round_up(g.max_batch * L.rows_per_image, 16));
        }
        if (s0.mode == AM_STEM) {
            // The stem stages the tile's input patch in shared memory, so its tile is a patch too:
            // the pool patch when a pool is linked, else th x tw output pixels with the fewest tiles.
            if (gapn) return fail(g, XENOS_E_UNSUPPORTED, "a convolution on an NCHW image cannot be linked with a global average");
            if (!addn && !catn && last->out >= 0 && !g.tensors[last->out].is_vec && g.tensors[last->out].c % 8 == 0 && layout_stem(L, M, src, pooln, N, ch.split)) {
                L.out = last->out;
                L.out_ctot = g.tensors[L.out].c; L.out_coff = 0;
                pack_stem(L, M, src.c);
                for (int ni : cover) L.flops += 2.0 * node_macs(g.nodes[ni]);
                L.bytes = tbytes(L.in0) + tbytes(L.out) + (double)L.npad * L.st_pairs * 32 + 4.0 * L.npad;
                push(L, ci);
                return XENOS_OK;
            }
            if (!pooln) {
                L.map_mode = MAP_PATCH;
                L.ni = 1;
                long best = -1;
                for (int tw = 1; tw <= std::min(L.Q, 128); ++tw) {
                    int th = std::min(L.P, 128 / tw);
                    // (tiles whose input patch the copy engine can fetch: at most 256 columns and rows)
                    if (tw > 1 && ((tw - 1) * M.stride + (M.k > 4 ? 10 : M.k) + 8 > 256 || (th - 1) * M.stride + M.k > 256)) continue;
                    long tiles = (long)ceil_div(L.P, th) * ceil_div(L.Q, tw);
                    if (best < 0 || tiles < best || (tiles == best && tw > L.patch_rw)) { best = tiles; L.patch_rh = th; L.patch_rw = tw; }
                }
                L.tiles_y = ceil_div(L.P, L.patch_rh); L.tiles_x = ceil_div(L.Q, L.patch_rw);
                L.step_y = L.patch_rh; L.step_x = L.patch_rw; L.off_y = L.off_x = 0;
                L.tile_rows = L.patch_rh * L.patch_rw;
            }
            // TMA fetches the patch when the image rows are 16-byte multiples; the box is widened so
            // that its x origin can be rounded down to a 16-byte boundary
            const int es = src.io_dtype == XENOS_DTYPE_F32 ? 4 : 2;
            L.stem_align = 16 / es;
            L.stem_tma = (src.w * es) % 16 == 0 ? 1 : 0;
            L.halo_h = (L.patch_rh - 1) * M.stride + M.k;
            // (a segment is read whole, kp elements plus up to two for the alignment of 16-bit images)
            L.halo_w = round_up((L.patch_rw - 1) * M.stride + (M.k > 4 ? 8 + 2 : M.k) + L.stem_align - 1, L.stem_align);
            L.halo_cb = src.c;
            // (small kernels keep patch offsets as 16-bit table entries)
            if (L.halo_h > 256 || L.halo_w > 256 || src.c > 256 || (M.k <= 4 && (long)src.c * L.halo_h * L.halo_w >= 65535)) L.stem_tma = 0;
            if (L.stem_tma) {
                L.halo_bytes = src.c * L.halo_h * L.halo_w * es;
                L.halo_stride = (int)align_up((size_t)L.halo_bytes, 128);
            }
        }
        if (dw) {
            // The depthwise stage reads a halo tile that TMA fetches as one 4-D box, so the tile is a
            // patch: ni whole images when an image fits 128 rows, else th x tw output pixels of one image.
            L.map_mode = MAP_PATCH;
            // the tile's row pitch is a multiple of 4: a producer thread owns 4 adjacent pixels of a row
            // ... made of br x 4 pixel blocks, the unit of work of a depthwise producer thread: 16 blocks of
            // 2 x 4 when a K block has 64 channels, 32 blocks of 1 x 4 otherwise
            const int Qp = round_up(L.Q, 4);
            const int br = std::min(64, src.c) > 32 ? 2 : 1, nblk = br == 2 ? 16 : 32;
            auto blocks_of = [&](int th, int tw) { return ceil_div(th, br) * (tw / 4); };
            // keep one halo tile (64 channels of the input window) small enough for a 2-3 deep ring
            auto halo_of = [&](int ni, int th, int tw) {
                return (long)ni * ((round_up(th, br) - 1) * dw->stride + 3) * ((tw - 1) * dw->stride + 3) * std::min(64, src.c) * 2;
            };
            if (L.P * Qp <= 128 && blocks_of(L.P, Qp) <= nblk) {
                L.ni = std::min(128 / (L.P * Qp), nblk / blocks_of(L.P, Qp)); L.patch_rh = L.P; L.patch_rw = Qp;
            } else {
                if (gapn) return fail(g, XENOS_E_UNSUPPORTED, "internal: global average needs whole images per tile");
                L.ni = 1;
                long best = -1;
                // (with few tiles per unit fewer of them gain nothing: the window then trims the rows afterwards)
                const bool many = (long)g.max_batch * L.P * L.Q >= 2l * 128 * g.hw.sm_count;
                for (int tw = 4; tw <= std::min(Qp, 64); tw += 4) {
                    int th = std::min(L.P, br * (nblk / (tw / 4)));
                    while (many && th > 1 && halo_of(1, th, tw) > 44 * 1024) --th;
                    const long tiles = (long)ceil_div(L.P, th) * ceil_div(L.Q, tw);
                    // fewest tiles first (within the window's limit: 8 x 8 instead of 1 x 56 at stride 2, 34.6 -> 30.5 us for 64 -> 128
                    // channels, 112 x 112, batch 32); then the widest tile (longest contiguous rows in memory)
                    if (best < 0 || tiles < best || (tiles == best && tw > L.patch_rw)) { best = tiles; L.patch_rh = th; L.patch_rw = tw; }
                }
            }
            while (L.ni > 1 && halo_of(L.ni, L.patch_rh, L.patch_rw) > 40 * 1024) --L.ni;
            // the depthwise stage is recomputed per channel tile and its time grows with the tile's pixels:
            // while SMs would stay idle, fewer images per tile spread it over more of them
            while (L.ni > 1 && (long)ceil_div(g.max_batch, L.ni) * ceil_div(round_up(N, 16), 256) * 2 <= g.hw.sm_count) --L.ni;
            while (!gapn && L.patch_rh > 1 && halo_of(L.ni, L.patch_rh, L.patch_rw) > 44 * 1024) --L.patch_rh;
            // Small batches leave most units idle while each tile's depthwise stage runs its K blocks one after the
            // other, at a pace set by the pixels per tile: while at least half of the units would stay idle, halve the
            // tile's rows (the MMA tile is then partly empty, which costs nothing there).
            while (!gapn && L.ni == 1 && L.patch_rh > 1 &&
                   (long)g.max_batch * ceil_div(L.P, (L.patch_rh + 1) / 2) * ceil_div(L.Q, L.patch_rw) * ceil_div(round_up(N, 16), 256) * 2 <= g.hw.sm_count)
                L.patch_rh = (L.patch_rh + 1) / 2;
            L.tiles_y = ceil_div(L.P, L.patch_rh); L.tiles_x = ceil_div(L.Q, L.patch_rw);
            L.step_y = L.patch_rh; L.step_x = L.patch_rw; L.off_y = L.off_x = 0;
            L.tile_rows = L.ni * L.patch_rh * L.patch_rw;
            // (the box covers whole blocks: a producer thread reads its block's full window)
            L.halo_h = (round_up(L.patch_rh, br) - 1) * dw->stride + 3; L.halo_w = (L.patch_rw - 1) * dw->stride + 3;
            L.halo_cb = std::min(64, src.c);
            L.halo_bytes = L.ni * L.halo_h * L.halo_w * L.halo_cb * 2;
            L.halo_stride = (int)align_up((size_t)L.halo_bytes, 128);
            if (L.halo_h > 256 || L.halo_w > 256) return fail(g, XENOS_E_UNSUPPORTED, "internal: halo tile exceeds the TMA box limit");
            if (gapn) { L.gap_imgs = L.ni; L.gap_area = L.patch_rh * L.patch_rw; L.gap_rpi = L.rows_per_image; }
        }
        L.out = last->out;
        const Tensor &ot = g.tensors[L.out];
        L.out_ctot = ot.c; L.out_coff = 0;
        L.out_dtype = (ot.is_vec && ot.output_slot >= 0) ? XENOS_DTYPE_F32 : XENOS_DTYPE_BF16;
        if (!ot.is_vec && ot.c % 8) return fail(g, XENOS_E_UNSUPPORTED, "bf16 NHWC tensors need a channel count that is a multiple of 8");
        // --- split (Section 4.2.1: output channels first, then rows / columns of the feature map)
        const SplitRequest &rq = ch.split;
        int N16 = round_up(N, 16);
        if (L.map_mode == MAP_PATCH) L.m_tiles = ceil_div(g.max_batch, L.ni) * L.tiles_y * L.tiles_x;
        else if (L.epi == EPI_GAP) L.m_tiles = L.gap_parts > 1 ? g.max_batch * L.gap_parts : ceil_div(g.max_batch, L.imgs_per_tile);
        else L.m_tiles = ceil_div(g.max_batch * L.rows_per_image, 128);
        if (rq.user && (rq.h > 1 || rq.w > 1))
            return fail(g, XENOS_E_BAD_SPLIT, "split: tensor-core chains cut rows / columns into 128-row tiles themselves; only parts_outc can be set");
        int tc_ksplit = 1;
        if (L.conv_tc && !(rq.user && rq.outc > 0)) {
            choose_conv_tiles(L, N16, rq, fc, tc_ksplit);
        } else if (rq.user && rq.outc > 0) {
            L.n_tiles = rq.outc;
            L.tile_n = round_up(ceil_div(N16, rq.outc), 16);
            if (L.tile_n > 256 || (rq.outc - 1) * L.tile_n >= N)
                return fail(g, XENOS_E_BAD_SPLIT, "split: parts_outc gives an output-channel tile that is empty or wider than 256");
        } else {
            L.n_tiles = ceil_div(N16, 256);
            L.tile_n = round_up(ceil_div(N16, L.n_tiles), 16);
            // kernels are dealt to idle units first: halve the channel tile while units stay idle
            // (a linked depthwise stage is recomputed per channel tile, so it stops halving earlier)
            // (unless most units are idle anyway: then narrower channel tiles shorten every CTA's weight loads and store)
            const int min_tile_n = dw ? ((long)L.m_tiles * L.n_tiles * 4 <= g.hw.sm_count ? 64 : 256) : 32;
            while (L.m_tiles * L.n_tiles < g.hw.sm_count && L.tile_n >= 2 * min_tile_n) {
                int nt = L.n_tiles * 2, tn = round_up(ceil_div(N16, nt), 16);
                if ((nt - 1) * tn >= N) break;
                L.n_tiles = nt; L.tile_n = tn;
            }
        }
        L.npad = L.n_tiles * L.tile_n;
        // --- reduction split (Section 4.2.2: C, R, S after K; it needs an additional reduction).  The K blocks
        // (64 elements of the (tap, channel) order) are cut into chunks of equal size, ascending; a chunk's partial
        // sums are fp32 and the chunks are added in ascending order.  Chosen automatically only when the tiles
        // leave most units idle and K is long (fc, late convolutions at small batch).
        {
            // (a linked depthwise stage can be split on request: a chunk's CTA then produces only its own channels of
            // the depthwise result.  It is not chosen automatically: measured at batch 1, with partial sums through the workspace,
            // the only form these chains have, the reduction costs more than the shorter depthwise loop saves; the split
            // search may still pick it.)
            // (a fully connected layer of at most 8 vectors runs on the CUDA cores: one pass over the weight matrix,
            // no partial sums; its input must be a bf16 vector that fits shared memory.  Measured, 1024 -> 1000:
            // 6.6 against 12 us at batch 1, 16.8 against 15.8 us at batch 32, where the tensor-core tiles win)
            if (fc && !rq.user && g.max_batch <= 8 && L.epi == EPI_STORE && L.skip < 0 && !shortcut && src.c % 8 == 0 &&
                (long)g.max_batch * src.c * 2 <= 160 * 1024 && !(src.input_slot >= 0 && src.io_dtype != XENOS_DTYPE_BF16))
                L.fc_small = 1;
            // (a linked shortcut convolution, the second K segment, is cut with its block: the chunks are blocks of the
            // concatenated K)
            const bool can = ((L.conv_tc && !L.fc_small) || (s0.mode == AM_DW && s1.mode == AM_NONE)) && L.epi == EPI_STORE;
            int want = 1;
            if (rq.user && rq.k > 1) {
                if (!can) return fail(g, XENOS_E_UNSUPPORTED, "split: parts_k applies to a convolution, depthwise -> pointwise chain or fc that stores its tile (no image stem or pooling epilogue)");
                if (rq.k > L.kblocks) return fail(g, XENOS_E_BAD_SPLIT, "split: parts_k exceeds the number of 64-element K blocks");
                want = rq.k;
            } else if (!rq.user && can && L.conv_tc) {
                want = tc_ksplit;
            }
            if (want > 1) {
                L.kb_per = ceil_div(L.kblocks, want);
                L.ksplit = ceil_div(L.kblocks, L.kb_per);
                if (rq.user && rq.k > 1 && L.ksplit != want)
                    return fail(g, XENOS_E_BAD_SPLIT, "split: parts_k does not cut the K blocks into that many non-empty chunks of equal size");
                if (L.ksplit < 2) { L.ksplit = 1; L.kb_per = 0; }
            }
        }
        // A depthwise -> pointwise chain with at most one tile per CTA and two 256-wide channel tiles: one CTA keeps both
        // channel tiles of its pixels (the two accumulators hold one 512-column tile; with a single tile per CTA
        // nothing is double-buffered anyway), so the depthwise stage is computed once per pixel tile instead of once
        // per channel tile, and the tiles get fewer rows until they cover the units again.
        if (dw && L.epi == EPI_STORE && L.ksplit == 1 && s1.mode == AM_NONE && !rq.user && L.ni == 1 && L.tile_n == 256 &&
            L.n_tiles % 2 == 0 && L.halo_cb == 64 && (long)L.m_tiles * L.n_tiles <= g.hw.sm_count) {
            const int nt2 = L.n_tiles / 2;
            int th = L.patch_rh;
            for (int t = 1; t <= L.patch_rh; ++t)
                if ((long)g.max_batch * ceil_div(L.P, t) * L.tiles_x * nt2 <= g.hw.sm_count) { th = t; break; }
            const int hh = (th - 1) * dw->stride + 3;
            const int hstride = (int)align_up((size_t)hh * L.halo_w * 128, 128);
            const int room2 = std::min(g.hw.smem_bytes_per_cta, 227 * 1024) - 1024 - 256 - 2048 - (int)align_up((size_t)40 * src.c, 128);
            if (2 * (16384 + 2 * 256 * 128) + 2 * hstride <= room2) {
                L.n_acc = 2; L.n_tiles = nt2;
                L.patch_rh = th; L.tiles_y = ceil_div(L.P, th); L.step_y = th;
                L.tile_rows = th * L.patch_rw;
                L.halo_h = hh; L.halo_bytes = hh * L.halo_w * 128; L.halo_stride = hstride;
                L.m_tiles = g.max_batch * L.tiles_y * L.tiles_x;
            }
        }
        // two accumulators in tensor memory so the epilogue of one tile overlaps the MMAs of the next
        L.acc_stride = round_up(L.tile_n, 32);
        L.tmem_cols = 32;
        while (L.tmem_cols < 2 * L.acc_stride) L.tmem_cols *= 2;
        if (L.tmem_cols > g.hw.tmem_columns) return fail(g, XENOS_E_BAD_SPLIT, "split: accumulator tiles exceed tensor memory columns");
        if (L.conv_tc) {
            const xenos_status_t lst = layout_conv(L, ot);
            if (lst != XENOS_OK) return lst;
        } else if (dw) {
            const xenos_status_t lst = layout_dw(L);
            if (lst != XENOS_OK) return lst;
        } else {
        // shared memory of the one persistent CTA per SM: [A|B ring][halo ring][epilogue staging][barriers]
        int stage_bytes = 16384 + L.n_acc * L.tile_n * 128;
        int stg_bytes = L.epi == EPI_POOL ? 128 * (L.tile_n * 2 + 16) : (L.epi == EPI_GAP ? 128 * 33 * 4 + 512 : 0);
        stg_bytes = (int)align_up((size_t)stg_bytes, 128);
        // depthwise tap weights + bias of the linked stage (fp32 [10][C]) and two bias slices of the GEMM
        // (a TMA-fed stem keeps its K-index -> patch-offset table there instead)
        int dww_bytes = dw ? (int)align_up((size_t)40 * src.c, 128) : (L.stem_tma ? (int)align_up((size_t)L.kpad * 2, 128) : 0);
        int cap = std::min(g.hw.smem_bytes_per_cta, 227 * 1024) - 1024 - 256 - 2048 - dww_bytes;
        // a linked depthwise stage is bound by its own arithmetic, not by the MMA: give the halo ring
        // (the TMA prefetch distance) up to four stages first, the A|B ring keeps three when it can
        L.hstages = 0;
        if (dw || L.stem_tma) {
            L.hstages = 2;
            while (L.hstages < 4 && cap - stg_bytes - (L.hstages + 1) * L.halo_stride >= 3 * stage_bytes) ++L.hstages;
        }
        int room = cap - stg_bytes - L.hstages * L.halo_stride;
        L.stages = std::min(6, room / stage_bytes);
        if (L.stages < 1) return fail(g, XENOS_E_BAD_SPLIT, "split: pipeline does not fit shared memory");
        L.off_halo = L.stages * stage_bytes;
        L.off_stg = L.off_halo + L.hstages * L.halo_stride;
        L.off_dww = (int)align_up((size_t)(L.off_stg + stg_bytes), 128);
        L.off_bias = L.off_dww + dww_bytes;
        L.off_bar = L.off_bias + 2048;
        L.pipe_bytes = L.off_bar;
        L.smem_bytes = L.off_bar + 256 + 1024;     // + barriers, alignment slack
        L.grid = std::min(L.m_tiles * L.n_tiles * L.ksplit, g.hw.sm_count);
        L.block = 448;
        }
        // --- pack weights + bias
        L.w_off = blob_reserve(g, (size_t)L.npad * L.kpad * 2);
        L.b_off = blob_reserve(g, (size_t)L.npad * 4);
        uint16_t *wp = reinterpret_cast<uint16_t *>(g.param_blob.data() + L.w_off);
        float *bp = reinterpret_cast<float *>(g.param_blob.data() + L.b_off);
        auto pack_conv = [&](const Node &n, int row0, int kbase, int kwin, int C, int Cp) {
            // n.w is [cout][C][n.k][n.k]; it sits centred in a kwin x kwin window
            int shift = (kwin - n.k) / 2;
            for (int o = 0; o < n.cout; ++o)
                for (int c = 0; c < C; ++c)
                    for (int r = 0; r < n.k; ++r)
                        for (int s = 0; s < n.k; ++s) {
                            int tap = (r + shift) * kwin + (s + shift);
                            wp[(size_t)(row0 + o) * L.kpad + kbase + tap * Cp + c] =
                                f32_to_bf16_rne(n.w[(((size_t)o * C + c) * n.k + r) * n.k + s]);
                        }
            for (int o = 0; o < n.cout; ++o) bp[row0 + o] += n.b[o];
        };
        if (fc || dw) {
            for (int o = 0; o < M.cout; ++o) {
                for (int c = 0; c < M.cin; ++c) wp[(size_t)o * L.kpad + c] = f32_to_bf16_rne(M.w[(size_t)o * M.cin + c]);
                bp[o] = M.b[o];
            }
        } else if (expand2) {
            // concat order decides the row offsets; both read the same kk x kk window
            const int cp = tc ? s0.cpad : src.c;
            pack_conv(M, 0, 0, kk, src.c, cp);
            pack_conv(*expand2, M.cout, 0, kk, src.c, cp);
        } else if (s0.mode == AM_STEM && M.k > 4) {
            const int kp = 8;
            for (int o = 0; o < M.cout; ++o) {
                for (int c = 0; c < src.c; ++c)
                    for (int r = 0; r < M.k; ++r)
                        for (int sx = 0; sx < M.k; ++sx)
                            wp[(size_t)o * L.kpad + (c * M.k + r) * kp + sx] =
                                f32_to_bf16_rne(M.w[(((size_t)o * src.c + c) * M.k + r) * M.k + sx]);
                bp[o] += M.b[o];
            }
        } else {
            pack_conv(M, 0, 0, M.k, src.c, tc ? s0.cpad : src.c);
        }
        if (shortcut) pack_conv(*shortcut, 0, 64 * s0.kblocks, 1, s1.C, s1.C);
        // --- modelled work
        for (int ni : cover) L.flops += 2.0 * node_macs(g.nodes[ni]);
        L.bytes = tbytes(L.in0) + tbytes(L.out) + (double)L.npad * L.kpad * 2 + 4.0 * L.npad;
        if (shortcut) L.bytes += tbytes(s1.tensor);
        if (L.skip >= 0) L.bytes += tbytes(L.skip);
        if (dw) L.bytes += node_param_bytes(*dw);
        push(L, ci);
        return XENOS_OK;
    }

    // ---- two linked convolutions, intermediate tile in shared memory (chain2_kernel) ---------------------------
    // A: first convolution (stride 1, input channels a multiple of 64).  Second stage: one convolution B (1x1, or
    // 3x3 with padding 1), or the two expand convolutions of a fire module merged over the 3x3 window in concat order.
    xenos_status_t make_gemm2(int ci, const std::vector<int> &cover, const Node &A, const Node *B, const Node *E0, const Node *E1,
                              const Node *addn, const Node *last) {
        Launch L;
        L.kind = LK_GEMM2;
        L.nodes = cover;
        const Tensor &src = g.tensors[A.in[0]];
        const Tensor &ot = g.tensors[last->out];
        const int k2 = B ? B->k : 3, h = (k2 - 1) / 2;
        const int N2 = B ? B->cout : E0->cout + E1->cout;
        L.in0 = A.in[0]; L.out = last->out;
        L.C = src.c; L.H = src.h; L.W = src.w; L.P = ot.h; L.Q = ot.w; L.K = N2; L.rows_per_image = L.P * L.Q;
        L.k = A.k; L.stride = 1; L.pad = A.pad; L.k2 = k2; L.halo2 = h;
        L.Cmid = A.cout; L.n1pad = round_up(A.cout, 64);
        L.seg[0].tensor = L.in0; L.seg[0].C = src.c; L.seg[0].H = src.h; L.seg[0].W = src.w; L.seg[0].k = A.k; L.seg[0].pad = A.pad;
        L.seg[0].mode = AM_GATHER; L.seg[0].cbox = 64; L.seg[0].cpad = src.c;
        L.kblocks = L.seg[0].kblocks = A.k * A.k * (src.c / 64);
        L.kblocks2 = k2 * k2 * (L.n1pad / 64);
        L.act = A.act; L.act2 = B ? B->act : E0->act;
        if (addn) {
            L.act3 = addn->act;
            const int mine = B->out;
            L.skip = addn->in[0] == mine ? addn->in[1] : addn->in[0];
        }
        if (src.c % 64 || g.tensors[A.out].h != ot.h || g.tensors[A.out].w != ot.w)
            return fail(g, XENOS_E_UNSUPPORTED, "internal: two linked convolutions need 64-channel input blocks and a consumer of equal extent");
        if (!chain2_tile(L.P, L.Q, h, L.patch_rh, L.patch_rw)) return fail(g, XENOS_E_UNSUPPORTED, "internal: no tile for two linked convolutions");
        L.rh2 = L.patch_rh - 2 * h; L.rw2 = L.patch_rw - 2 * h;
        L.tiles_y = ceil_div(L.P, L.rh2); L.tiles_x = ceil_div(L.Q, L.rw2);
        L.m_tiles = g.max_batch * L.tiles_y * L.tiles_x;
        L.a_box_bytes = L.patch_rh * L.patch_rw * 128;
        const int cap = std::min(g.hw.smem_bytes_per_cta, 227 * 1024) - 1024;
        L.out_ctot = ot.c; L.out_coff = 0;
        if (k2 == 1) {
            // pair_tc_kernel: tiles of 128 consecutive pixels, 128 output channels at a time; 16 KB slots for activation and
            // weight blocks share what the middle tile, the staging boxes and the biases leave
            L.pair = 1;
            L.m_tiles = ceil_div(g.max_batch * L.rows_per_image, 128);
            L.tile_n = 128; L.n_tiles = ceil_div(N2, 128); L.npad = L.n_tiles * 128;
            const int mid = (L.n1pad / 64) * 16384, bias = (int)align_up((size_t)(L.n1pad + L.npad) * 4, 128);
            if (L.skip >= 0) L.s_slots = 3;      // (a fourth box each takes operand slots: 256 against 276 us, 64 channels, 128 x 128, batch 64; 295 with two)
            const int stg = 8 * L.s_slots * 2048;
            const int room = cap - 1024 - mid - stg - bias;
            const int weights = L.kblocks * L.n1pad * 128 + L.kblocks2 * L.n_tiles * 16384;
            // (the kernel keeps one 128-row weight block per operand block: wider middle tiles take theirs in two halves, which travel
            // through the ring)
            L.b_resident = L.n1pad <= 128 && room - weights >= 3 * 16384;
            const int slots = (room - (L.b_resident ? weights : 0)) / 16384;
            L.a_slots = L.b_resident ? std::min(8, slots) : slots * 2 / 5;
            L.b_slots = L.b_resident ? 0 : std::min(8, slots - L.a_slots);
            L.a_slots = std::min(8, L.a_slots);
            if (L.a_slots < 2 || (!L.b_resident && L.b_slots < 2)) return fail(g, XENOS_E_BAD_SPLIT, "split: two linked convolutions do not fit shared memory");
            L.off_b2 = L.a_slots * 16384;
            L.off_mid = L.off_b2 + (L.b_resident ? weights : L.b_slots * 16384);
            L.off_stg = L.off_mid + mid;
            L.off_bias = L.off_stg + stg;
            L.off_bar = L.off_bias + bias;
            L.smem_bytes = L.off_bar + 1024 + 1024;
            L.stages = L.a_slots;
            L.a_rows = 128;
            L.block = 384;
        } else {
            const int N216 = round_up(N2, 16);
            L.n_tiles = ceil_div(N216, 256);
            L.tile_n = round_up(ceil_div(N216, L.n_tiles), 16);
            L.npad = L.n_tiles * L.tile_n;
            L.stage_bytes = 16384 + std::max(L.n1pad, L.tile_n) * 128;
            const int mid_bytes = (L.n1pad / 64) * (128 + 64) * 128;
            L.stages = std::min(6, (cap - 256 - mid_bytes) / L.stage_bytes);
            if (L.stages < 2) return fail(g, XENOS_E_BAD_SPLIT, "split: two linked convolutions do not fit shared memory");
            L.off_mid = L.stages * L.stage_bytes;
            L.off_bar = L.off_mid + mid_bytes;
            L.smem_bytes = L.off_bar + 256 + 1024;
            L.block = 320;
        }
        L.tmem_cols = 512;
        L.grid = std::min(L.m_tiles, g.hw.sm_count);
        if (g.chains[ci].split.user && (g.chains[ci].split.outc > 1 || g.chains[ci].split.h > 1 || g.chains[ci].split.w > 1 || g.chains[ci].split.k > 1))
            return fail(g, XENOS_E_BAD_SPLIT, "split: two linked convolutions keep all output channels of a tile in one CTA; no explicit split");
        // --- parameters: W1 [n1pad][K1], bias1 [n1pad]; W2 [npad][k2*k2*n1pad], bias2 [npad]; K order (tap, channel)
        const int K1 = L.kblocks * 64, K2 = L.kblocks2 * 64;
        L.kpad = K1;
        L.w_off = blob_reserve(g, (size_t)L.n1pad * K1 * 2);
        L.b_off = blob_reserve(g, (size_t)L.n1pad * 4);
        L.w2_off = blob_reserve(g, (size_t)L.npad * K2 * 2);
        L.b2_off = blob_reserve(g, (size_t)L.npad * 4);
        uint16_t *w1 = reinterpret_cast<uint16_t *>(g.param_blob.data() + L.w_off);
        float *b1 = reinterpret_cast<float *>(g.param_blob.data() + L.b_off);
        uint16_t *w2 = reinterpret_cast<uint16_t *>(g.param_blob.data() + L.w2_off);
        float *b2 = reinterpret_cast<float *>(g.param_blob.data() + L.b2_off);
        for (int o = 0; o < A.cout; ++o) {
            for (int c = 0; c < src.c; ++c)
                for (int r = 0; r < A.k; ++r)
                    for (int s2 = 0; s2 < A.k; ++s2)
                        w1[(size_t)o * K1 + (r * A.k + s2) * src.c + c] = f32_to_bf16_rne(A.w[(((size_t)o * src.c + c) * A.k + r) * A.k + s2]);
            b1[o] = A.b[o];
        }
        auto pack2 = [&](const Node &n, int row0) {
            const int shift = (k2 - n.k) / 2;
            for (int o = 0; o < n.cout; ++o) {
                for (int c = 0; c < A.cout; ++c)
                    for (int r = 0; r < n.k; ++r)
                        for (int s2 = 0; s2 < n.k; ++s2)
                            w2[(size_t)(row0 + o) * K2 + ((r + shift) * k2 + (s2 + shift)) * L.n1pad + c] =
                                f32_to_bf16_rne(n.w[(((size_t)o * A.cout + c) * n.k + r) * n.k + s2]);
                b2[row0 + o] = n.b[o];
            }
        };
        if (B) pack2(*B, 0);
        else { pack2(*E0, 0); pack2(*E1, E0->cout); }
        for (int ni : cover) L.flops += 2.0 * node_macs(g.nodes[ni]);
        L.bytes = tbytes(L.in0) + tbytes(L.out) + (double)L.n1pad * K1 * 2 + (double)L.npad * K2 * 2 + 4.0 * (L.n1pad + L.npad);
        if (L.skip >= 0) L.bytes += tbytes(L.skip);
        push(L, ci);
        return XENOS_OK;
    }

    xenos_status_t lower_bf16_single(int ci, int ni) {
        const Node &n = g.nodes[ni];
        if (n.kind == NK_CONV) {
            // the first layer at small batch: a 3x3 convolution of an NCHW image runs on the CUDA cores (K = 27 fills
            // less than half of one 64-wide K block of the MMA; a launch of the persistent kernel costs more than this
            // whole layer).  Same-box A/B on MobileNet: batch 1 0.1506 -> 0.1424 ms; at batch 32 the tensor-core stem
            // with its TMA-fetched patches is faster (30 against 35.5 us), so larger batches keep it.
            const Tensor &x = g.tensors[n.in[0]];
            const bool no_request = !g.chains[ci].split.user;
            if (x.input_slot >= 0 && x.io_layout == XENOS_LAYOUT_NCHW && x.c <= 4 && n.k == 3 && (n.stride == 1 || n.stride == 2) &&
                n.cout % 8 == 0 && n.cout <= 64 && n.cin == x.c && no_request && !n.from_matmul && g.max_batch <= 8) {
                Launch L;
                L.kind = LK_STEM3X3;
                L.nodes = {ni};
                fill_io(L, n);
                L.seg[0].src_dtype = x.io_dtype;
                // weights [tap row][tap column][channel][cout], fp32
                std::vector<float> wt((size_t)9 * n.cin * n.cout);
                for (int o = 0; o < n.cout; ++o)
                    for (int c = 0; c < n.cin; ++c)
                        for (int t9 = 0; t9 < 9; ++t9) wt[((size_t)t9 * n.cin + c) * n.cout + o] = n.w[((size_t)o * n.cin + c) * 9 + t9];
                L.w_off = put_f32(wt); L.b_off = put_f32(n.b);
                L.flops = 2.0 * node_macs(n);
                L.bytes = tbytes(n.in[0]) + tbytes(n.out) + node_param_bytes(n);
                const int ih = 7 * n.stride + 3, iw = 31 * n.stride + 3;
                L.smem_bytes = 4 * (((n.cin * ih * (iw | 1) + 3) & ~3) + 9 * n.cin * n.cout + n.cout);
                L.grid = ceil_div(L.P, 8) * ceil_div(L.Q, 32);      // per image
                L.block = 256;
                push(L, ci);
                return XENOS_OK;
            }
        }
        if (n.kind == NK_CONV) return make_gemm(ci, {ni}, nullptr, &n, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, false);
        if (n.kind == NK_FC) {
            if (n.cin % 8) return fail(g, XENOS_E_UNSUPPORTED, "fc input length must be a multiple of 8");
            return make_gemm(ci, {ni}, nullptr, &n, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, true);
        }
        if (g.chains[ci].split.user && (g.chains[ci].split.outc > 1 || g.chains[ci].split.h > 1 || g.chains[ci].split.w > 1 || g.chains[ci].split.k > 1))
            return fail(g, XENOS_E_BAD_SPLIT, "split: element-wise, pooling and depthwise kernels are split one vector per thread; no explicit split");
        const Tensor &x = g.tensors[n.in[0]];
        if (!x.is_vec && x.c % 8) return fail(g, XENOS_E_UNSUPPORTED, "bf16 NHWC tensors need a channel count that is a multiple of 8");
        if (n.kind == NK_DW) {
            if (n.k != 3) return fail(g, XENOS_E_UNSUPPORTED, "depthwise convolution: only 3x3 has a kernel");
            Launch L;
            L.kind = LK_DW;
            L.nodes = {ni};
            fill_io(L, n);
            L.groups = n.cin;
            std::vector<float> wt((size_t)9 * n.cin);
            for (int c = 0; c < n.cin; ++c)
                for (int t = 0; t < 9; ++t) wt[(size_t)t * n.cin + c] = n.w[(size_t)c * 9 + t];
            L.w_off = put_f32(wt); L.b_off = put_f32(n.b);
            L.flops = 2.0 * node_macs(n);
            L.bytes = tbytes(n.in[0]) + tbytes(n.out) + node_param_bytes(n);
            L.block = 256;
            push(L, ci);
            return XENOS_OK;
        }
        return lower_single_common(ci, ni, false);
    }

    xenos_status_t lower_chain(int ci) {
        Chain &ch = g.chains[ci];
        // modelled traffic if every member ran alone (the unlinked baseline of the same chain)
        for (int ni : ch.nodes) {
            const Node &n = g.nodes[ni];
            ch.bytes_unlinked += tbytes(n.out) + node_param_bytes(n);
            for (int t : n.in) ch.bytes_unlinked += tbytes(t);
            ch.flops += 2.0 * node_macs(n);
        }
        xenos_status_t st = XENOS_OK;
        bool f32 = g.precision == XENOS_PRECISION_FP32_CUDA_CORE;
        auto find = [&](int kind, int nth = 0) -> const Node * {
            for (int ni : ch.nodes)
                if (g.nodes[ni].kind == kind && nth-- == 0) return &g.nodes[ni];
            return nullptr;
        };
        switch (ch.kind) {
        case CK_SINGLE:
            st = f32 ? lower_f32_single(ci, ch.nodes[0]) : lower_bf16_single(ci, ch.nodes[0]);
            break;
        case CK_CONV_CONV_POOL:
            st = lower_f32_linked(ci);
            break;
        case CK_DW_PW:
            st = make_gemm(ci, ch.nodes, find(NK_DW), find(NK_CONV), nullptr, nullptr, nullptr, nullptr, find(NK_GAP), nullptr, false);
            break;
        case CK_CONV_TAIL: {
            const Node *addn = find(NK_ADD);
            const Node *mainc = &g.nodes[ch.nodes[0]];
            const Node *sc = (addn && find(NK_CONV, 1)) ? find(NK_CONV, 1) : nullptr;
            st = make_gemm(ci, ch.nodes, nullptr, mainc, sc, nullptr, addn, find(NK_MAXPOOL), find(NK_GAP), nullptr, false);
            break;
        }
        case CK_MATMUL_MATMUL: {
            const Node &A = g.nodes[ch.nodes[0]], &B = g.nodes[ch.nodes[1]];
            Node M;                      // the one product that stands for both
            M.kind = A.kind; M.in = A.in; M.out = B.out; M.cin = A.cin; M.cout = B.cout; M.k = 1; M.stride = 1; M.pad = 0; M.act = B.act;
            M.w.assign((size_t)B.cout * A.cin, 0.0f);
            M.b.assign(B.cout, 0.0f);
            for (int o = 0; o < B.cout; ++o) {
                std::vector<double> row(A.cin, 0.0);
                double bias = B.b[o];
                for (int m = 0; m < A.cout; ++m) {
                    const double w2 = B.w[(size_t)o * A.cout + m];
                    bias += w2 * A.b[m];
                    const float *w1 = &A.w[(size_t)m * A.cin];
                    for (int c = 0; c < A.cin; ++c) row[c] += w2 * w1[c];
                }
                for (int c = 0; c < A.cin; ++c) M.w[(size_t)o * A.cin + c] = (float)row[c];
                M.b[o] = (float)bias;
            }
            st = make_gemm(ci, ch.nodes, nullptr, &M, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, A.kind == NK_FC);
            // (the modelled work of the launch is the merged product's, not the sum of the two it replaces)
            if (st == XENOS_OK) g.launches.back().flops = 2.0 * node_macs(M);
            break;
        }
        case CK_CONV_CONV: {
            const Node *cat = find(NK_CONCAT);
            if (cat) {
                const Node *first = &g.nodes[g.node_of_tensor[cat->in[0]]];
                const Node *second = &g.nodes[g.node_of_tensor[cat->in[1]]];
                st = make_gemm2(ci, ch.nodes, g.nodes[ch.nodes[0]], nullptr, first, second, nullptr, cat);
            } else {
                const Node *addn = find(NK_ADD);
                const Node &B = g.nodes[ch.nodes[1]];
                st = make_gemm2(ci, ch.nodes, g.nodes[ch.nodes[0]], &B, nullptr, nullptr, addn, addn ? addn : &B);
            }
            break;
        }
        case CK_EXPAND_CONCAT: {
            const Node *cat = find(NK_CONCAT);
            const Node *first = &g.nodes[g.node_of_tensor[cat->in[0]]];
            const Node *second = &g.nodes[g.node_of_tensor[cat->in[1]]];
            st = make_gemm(ci, ch.nodes, nullptr, first, nullptr, second, nullptr, find(NK_MAXPOOL), nullptr, cat, false);
            break;
        }
        default:
            st = fail(g, XENOS_E_UNSUPPORTED, "internal: unknown chain kind");
        }
        if (st != XENOS_OK) return st;
        for (int li : ch.launches) ch.bytes_linked += g.launches[li].bytes;
        return XENOS_OK;
    }
};

xenos_status_t split_and_lower(Graph &g) {
    g.launches.clear();
    g.param_blob.clear();
    Lower lw(g);
    for (int ci = 0; ci < (int)g.chains.size(); ++ci) {
        xenos_status_t st = lw.lower_chain(ci);
        if (st != XENOS_OK) return st;
    }
    return XENOS_OK;
}

// ------------------------------------------------------------------------------------------------
// Workspace: parameters, status words, then an arena for the tensors that live between kernels,
// placed first-fit by live interval (the memory-management part of the paper's runtime layer, Section 6).
// ------------------------------------------------------------------------------------------------
xenos_status_t plan_workspace(Graph &g) {
    int nt = (int)g.tensors.size();
    g.place.assign(nt, TensorPlace());
    bool f32 = g.precision == XENOS_PRECISION_FP32_CUDA_CORE;
    auto touch = [&](int t, int li, bool def) {
        if (t < 0) return;
        TensorPlace &p = g.place[t];
        p.materialised = true;
        if (p.first < 0 || (def && li < p.first)) p.first = p.first < 0 ? li : std::min(p.first, li);
        p.last = std::max(p.last, li);
    };
    for (int li = 0; li < (int)g.launches.size(); ++li) {
        const Launch &L = g.launches[li];
        touch(L.out, li, true);
        touch(L.in0, li, false); touch(L.in1, li, false); touch(L.in2, li, false); touch(L.skip, li, false);
        touch(L.seg[0].tensor, li, false); touch(L.seg[1].tensor, li, false);
    }
    size_t off = align_up(g.param_blob.size(), 256);
    g.status_off = off;
    off += 256;
    // arrival counters of the reduction-split launches sit behind the status words and are cleared with them
    g.cnt_bytes = 0; g.split_bytes = 0;
    for (Launch &L : g.launches)
        if (L.kind == LK_GEMM && L.ksplit > 1 && !(L.conv_tc && L.cv_epi == 5)) {
            L.split_cnt_off = off + g.cnt_bytes;
            g.cnt_bytes += align_up((size_t)L.m_tiles * L.n_tiles * 8, 16);      // [arrived, reduced] per tile
            g.split_bytes = std::max(g.split_bytes, (size_t)L.ksplit * g.max_batch * L.rows_per_image * L.npad * 4);
        } else if (L.kind == LK_GEMM && L.gap_parts > 1) {
            L.split_cnt_off = off + g.cnt_bytes;
            g.cnt_bytes += align_up((size_t)g.max_batch * L.n_tiles * 8, 16);   // one counter per (image, channel tile)
            g.split_bytes = std::max(g.split_bytes, (size_t)g.max_batch * L.gap_parts * L.npad * 4);
        }
    g.cnt_bytes = align_up(g.cnt_bytes, 256);
    off += g.cnt_bytes;
    g.act_off = off;
    struct Live { size_t off, bytes; int last; };
    std::vector<Live> live;
    std::vector<int> order;
    for (int t = 0; t < nt; ++t) if (g.place[t].materialised) order.push_back(t);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return g.place[a].first < g.place[b].first; });
    size_t arena = 0;
    for (int t : order) {
        TensorPlace &p = g.place[t];
        const Tensor &x = g.tensors[t];
        if (f32) { p.dtype = XENOS_DTYPE_F32; p.layout = XENOS_LAYOUT_NCHW; }
        else { p.dtype = XENOS_DTYPE_BF16; p.layout = XENOS_LAYOUT_NHWC; }
        if (x.input_slot >= 0 || x.output_slot >= 0) {
            p.external = true;
            p.dtype = x.io_dtype; p.layout = x.io_layout;
            if (x.input_slot >= 0) p.first = 0;
            continue;
        }
        p.bytes = align_up((size_t)g.max_batch * tensor_elems(x) * (p.dtype == XENOS_DTYPE_F32 ? 4 : 2), 256);
        // lowest offset that overlaps no tensor still live when this one is defined
        std::vector<std::pair<size_t, size_t>> busy;
        for (const Live &l : live) if (l.last >= p.first) busy.push_back({l.off, l.off + l.bytes});
        std::sort(busy.begin(), busy.end());
        size_t cand = 0;
        for (auto &b : busy) {
            if (cand + p.bytes <= b.first) break;
            cand = std::max(cand, b.second);
        }
        p.off = g.act_off + cand;
        live.push_back({cand, p.bytes, p.last});
        arena = std::max(arena, cand + p.bytes);
    }
    g.split_off = align_up(g.act_off + arena, 256);
    g.workspace_bytes = g.split_off + g.split_bytes;
    // a graph input that is also read late must outlive everything: external, nothing to do.
    return XENOS_OK;
}

// ------------------------------------------------------------------------------------------------
// Plan as JSON
// ------------------------------------------------------------------------------------------------
static void jstr(std::string &s, const char *k, const std::string &v, bool comma = true) {
    s += "\""; s += k; s += "\":\""; s += v; s += "\""; if (comma) s += ",";
}
static void jint(std::string &s, const char *k, long long v, bool comma = true) {
    s += "\""; s += k; s += "\":"; s += std::to_string(v); if (comma) s += ",";
}
static void jdbl(std::string &s, const char *k, double v, bool comma = true) {
    char buf[64];
    snprintf(buf, sizeof buf, "%.0f", v);
    s += "\""; s += k; s += "\":"; s += buf; if (comma) s += ",";
}
static void jarr(std::string &s, const char *k, const std::vector<int> &v, bool comma = true) {
    s += "\""; s += k; s += "\":[";
    for (size_t i = 0; i < v.size(); ++i) { if (i) s += ","; s += std::to_string(v[i]); }
    s += "]"; if (comma) s += ",";
}

// The kernel a launch runs (a pool of windows up to 3 runs maxpool_kernel when its items fit 31 bits).
static std::string kernel_of(const Launch &L) {
    if (L.kind == LK_GEMM)
        return L.fc_small ? "fc_small_kernel" : L.stem_tc ? "stem_tc_kernel" : L.conv_tc ? "conv_tc_kernel" : L.seg[0].mode == AM_DW ? "dw_tc_kernel" : "gemm_chain_kernel";
    if (L.kind == LK_GEMM2) return L.pair ? "pair_tc_kernel" : "chain2_kernel";
    if (L.kind == LK_POOL) return L.pool_kind == 0 && L.pool_k <= 3 ? "maxpool_kernel" : "pool_kernel";
    static const char *k[] = {"?", "gemm_chain_kernel", "dw3x3_kernel", "pool_kernel", "gap_kernel", "add_kernel", "concat_part_kernel", "mulmac_kernel",
                              "transpose_kernel", "slice_kernel", "f32_conv_kernel", "f32_pool_kernel", "f32_gap_kernel", "f32_add_kernel",
                              "f32_concat_part_kernel", "f32_fc_kernel", "f32_chain_kernel", "f32_mulmac_kernel", "transpose_kernel", "f32_slice_kernel",
                              "chain2_kernel", "stem3x3_kernel"};
    return k[L.kind];
}

void emit_plan_json(Graph &g) {
    static const char *nk[] = {"?", "conv", "dwconv", "fc", "maxpool", "avgpool", "gap", "add", "concat", "mul", "mac", "transpose", "split"};
    static const char *ck[] = {"single", "conv_conv_pool", "dw_pw", "conv_tail", "expand_concat", "matmul_matmul", "conv_conv"};
    static const char *lk[] = {"?", "gemm", "dw", "pool", "gap", "add", "concat_part", "mulmac", "transpose", "slice", "f32_conv", "f32_pool",
                               "f32_gap", "f32_add", "f32_concat_part", "f32_fc", "f32_conv_conv_pool", "f32_mulmac", "f32_transpose", "f32_slice", "gemm2", "stem3x3"};
    static const char *am[] = {"none", "gather", "stem", "dw"};
    std::string s = "{";
    jstr(s, "precision", g.precision == XENOS_PRECISION_FP32_CUDA_CORE ? "fp32_cuda_core" : "bf16_tensor");
    jint(s, "max_batch", g.max_batch);
    s += "\"hw\":{";
    jint(s, "sm_count", g.hw.sm_count); jint(s, "smem_bytes_per_cta", g.hw.smem_bytes_per_cta);
    jint(s, "tmem_columns", g.hw.tmem_columns); jint(s, "l2_bytes", g.hw.l2_bytes, false);
    s += "},";
    jstr(s, "cta_to_tile", "gemm: cta = m_tile * n_tiles + n_tile, tiles dealt to units round-robin in ascending order; "
                            "f32 chain: cta = ((image * parts_outc + outc_part) * tiles_h + tile_y) * tiles_w + tile_x");
    s += "\"nodes\":[";
    for (size_t i = 0; i < g.nodes.size(); ++i) {
        const Node &n = g.nodes[i];
        if (i) s += ",";
        s += "{";
        jint(s, "id", (long long)i); jstr(s, "kind", nk[n.kind]); jarr(s, "in", n.in); jint(s, "out", n.out);
        jint(s, "cin", n.cin); jint(s, "cout", n.cout); jint(s, "k", n.k); jint(s, "stride", n.stride);
        jint(s, "pad", n.pad); jint(s, "act", n.act); jarr(s, "user_ops", n.user_ops); jint(s, "chain", n.chain, false);
        s += "}";
    }
    s += "],\"chains\":[";
    double tf = 0, tb = 0, tu = 0;
    for (size_t i = 0; i < g.chains.size(); ++i) {
        const Chain &c = g.chains[i];
        if (i) s += ",";
        s += "{";
        jint(s, "id", (long long)i); jstr(s, "kind", ck[c.kind]); jstr(s, "pattern", c.pattern);
        jarr(s, "nodes", c.nodes); jarr(s, "launches", c.launches);
        jdbl(s, "flops", c.flops); jdbl(s, "bytes_linked", c.bytes_linked); jdbl(s, "bytes_unlinked", c.bytes_unlinked, false);
        s += "}";
        tf += c.flops; tb += c.bytes_linked; tu += c.bytes_unlinked;
    }
    s += "],\"launches\":[";
    for (size_t i = 0; i < g.launches.size(); ++i) {
        const Launch &L = g.launches[i];
        if (i) s += ",";
        s += "{";
        jint(s, "id", (long long)i); jstr(s, "kind", lk[L.kind]); jstr(s, "kernel", kernel_of(L)); jint(s, "chain", L.chain); jarr(s, "nodes", L.nodes);
        jint(s, "in0", L.in0); jint(s, "in1", L.in1); jint(s, "in2", L.in2); jint(s, "skip", L.skip); jint(s, "out", L.out);
        jint(s, "out_coff", L.out_coff); jint(s, "out_ctot", L.out_ctot);
        jint(s, "C", L.C); jint(s, "H", L.H); jint(s, "W", L.W); jint(s, "K", L.K); jint(s, "P", L.P); jint(s, "Q", L.Q);
        jint(s, "k", L.k); jint(s, "stride", L.stride); jint(s, "pad", L.pad);
        if (L.kind == LK_GEMM) {
            jstr(s, "a0", am[L.seg[0].mode]); jstr(s, "a1", am[L.seg[1].mode]);
            jint(s, "kblocks", L.kblocks); jint(s, "npad", L.npad); jint(s, "tile_m", 128); jint(s, "tile_n", L.tile_n);
            jint(s, "tile_k", 64); jint(s, "n_tiles", L.n_tiles); jint(s, "m_tiles", L.m_tiles);
            jint(s, "tile_rows", L.tile_rows); jint(s, "epi", L.epi); jint(s, "map", L.map_mode);
            jint(s, "imgs_per_tile", L.imgs_per_tile);
            jint(s, "patch_th", L.patch_th); jint(s, "patch_tw", L.patch_tw); jint(s, "patch_rh", L.patch_rh);
            jint(s, "patch_rw", L.patch_rw); jint(s, "tiles_y", L.tiles_y); jint(s, "tiles_x", L.tiles_x);
            jint(s, "stages", L.stages); jint(s, "tmem_cols", L.tmem_cols); jint(s, "acc_stride", L.acc_stride);
            jint(s, "ni", L.ni); jint(s, "step_y", L.step_y); jint(s, "step_x", L.step_x); jint(s, "off_y", L.off_y); jint(s, "off_x", L.off_x);
            jint(s, "hstages", L.hstages); jint(s, "stem_tc", L.stem_tc); jint(s, "halo_h", L.halo_h); jint(s, "halo_w", L.halo_w); jint(s, "halo_cb", L.halo_cb);
            jint(s, "halo_bytes", L.halo_bytes);
            jint(s, "ksplit", L.ksplit); jint(s, "kb_per", L.kb_per); jint(s, "a_tma", L.a_tma); jint(s, "fc_small", L.fc_small); jint(s, "dw_workers", L.dw_workers); jint(s, "dw_groups", L.dw_groups); jint(s, "dw_br", L.dw_br); jint(s, "dw_batch", L.dw_batch); jint(s, "chunk", L.chunk); jint(s, "out_bufs", L.out_bufs); jint(s, "b_slots", L.b_slots); jint(s, "n_acc", L.n_acc); jint(s, "gap_parts", L.gap_parts); jint(s, "conv_tc", L.conv_tc); jint(s, "b_resident", L.b_resident);
        }
        if (L.kind == LK_GEMM2) {
            jint(s, "k2", L.k2); jint(s, "cmid", L.Cmid); jint(s, "n1pad", L.n1pad); jint(s, "kblocks", L.kblocks); jint(s, "kblocks2", L.kblocks2);
            jint(s, "tile_n", L.tile_n); jint(s, "n_tiles", L.n_tiles); jint(s, "m_tiles", L.m_tiles); jint(s, "npad", L.npad);
            jint(s, "patch_rh", L.patch_rh); jint(s, "patch_rw", L.patch_rw); jint(s, "rh2", L.rh2); jint(s, "rw2", L.rw2);
            jint(s, "tiles_y", L.tiles_y); jint(s, "tiles_x", L.tiles_x); jint(s, "stages", L.stages); jint(s, "b_resident", L.b_resident);
        }
        if (L.kind == LK_F32_CONV_CONV_POOL) {
            jint(s, "parts_outc", L.parts_outc); jint(s, "tile_h", L.tile_h); jint(s, "tile_w", L.tile_w);
            jint(s, "tiles_h", L.tiles_h); jint(s, "tiles_w", L.tiles_w); jint(s, "halo_h", L.halo_h); jint(s, "halo_w", L.halo_w);
        }
        jint(s, "w_off", (long long)L.w_off); jint(s, "b_off", (long long)L.b_off);
        jint(s, "smem_bytes", L.smem_bytes); jint(s, "grid", L.grid); jint(s, "block", L.block);
        jdbl(s, "flops", L.flops); jdbl(s, "bytes", L.bytes, false);
        s += "}";
    }
    s += "],\"tensors\":[";
    bool firstt = true;
    for (size_t t = 0; t < g.tensors.size(); ++t) {
        const TensorPlace &p = g.place[t];
        if (!p.materialised) continue;
        if (!firstt) s += ",";
        firstt = false;
        const Tensor &x = g.tensors[t];
        s += "{";
        jint(s, "id", (long long)t); jint(s, "c", x.c); jint(s, "h", x.h); jint(s, "w", x.w);
        jint(s, "external", p.external); jint(s, "off", (long long)p.off); jint(s, "bytes", (long long)p.bytes);
        jint(s, "first", p.first); jint(s, "last", p.last, false);
        s += "}";
    }
    s += "],";
    jint(s, "param_bytes", (long long)g.param_blob.size());
    jint(s, "workspace_bytes", (long long)g.workspace_bytes);
    jdbl(s, "flops", tf); jdbl(s, "bytes_linked", tb); jdbl(s, "bytes_unlinked", tu, false);
    s += "}";
    g.plan_json.swap(s);
}

}  // namespace xenos
