// Host side of the library: the layer list and its shape / operation-count inference (Eq. 1,
// Eq. 2), fusion plans (Algorithm 1's two output arrays) and their validation, the launcher that
// turns a plan into one kernel per group on a persistent grid of `sm_count` CTAs, timing, the
// auto-tuner (Eq. 5 + Algorithm 1) and the reduced brute-force search (Sec. V).
#include <cuda.h>
#include <cuda_runtime.h>
#include <cxxabi.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <limits>
#include <new>
#include <string>
#include <vector>

#include "internal.h"

namespace dlf {

static thread_local int g_last_cuda_error = 0;
int g_use_pdl = 1;
thread_local bool g_stream_order = false;
thread_local const GraphNodeUpdate* g_node_update = nullptr;
thread_local LaunchRecord* g_launch_record = nullptr;
int g_conv_row_mode = 1;

int cuda_fail(cudaError_t e) {
    g_last_cuda_error = static_cast<int>(e);
    cudaGetLastError();
    return DLF_E_CUDA;
}
int cuda_fail_drv(int e) {
    g_last_cuda_error = 100000 + e;
    return DLF_E_CUDA;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

int encode_tmap(void* out_map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                const uint32_t* box, const uint32_t* elem_strides) {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr);
        if (e != cudaSuccess) return cuda_fail(e);
        if (qr != cudaDriverEntryPointSuccess || !p) return cuda_fail_drv(999);
        fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    cuuint64_t gd[5], gs[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; i++) {
        gd[i] = dims[i];
        bx[i] = box[i];
        es[i] = elem_strides[i];
        if (i < rank - 1) gs[i] = strides_bytes[i];
    }
    CUresult r = fn(static_cast<CUtensorMap*>(out_map), CU_TENSOR_MAP_DATA_TYPE_FLOAT16, static_cast<cuuint32_t>(rank),
                    const_cast<void*>(base), gd, gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cuda_fail_drv(static_cast<int>(r));
    return DLF_OK;
}

enum Kind { K_CHAIN_TC, K_CONV_TC, K_CONV_DIRECT, K_DW, K_FC, K_MAXPOOL, K_GAVG, K_STEM_TC, K_MBCONV, K_CONV_SEQ, K_CONV_DUAL };
static const char* kKindName[] = {"chain_tc", "conv_tc", "conv_direct", "dw3x3", "fc", "maxpool", "gavgpool", "stem_tc", "mbconv_tc", "conv_seq", "conv_tc"};

struct Layer {
    dlf_layer_desc d;
    int64_t in[4], out[4];
    int ho_pre, wo_pre;  // before the fused pool
    int64_t ops_eq1, flops, w_elems;
    const void* w;
    const float* bias;
    size_t off, bytes;  // slot in the workspace
};

struct Group {
    int first, last, sms;
    Kind kind;
    ChainTiling tiling;
    MbconvTiling mb_tiling;
};

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// A captured plan: one kernel node per group, and the input and output the nodes' parameters hold at the moment.
constexpr int kHostParts = 4;

struct GraphCache {
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;
    std::vector<cudaGraphNode_t> nodes;
    const void* in = nullptr;
    void* out = nullptr;
    void drop() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
        nodes.clear();
    }
};

}  // namespace dlf

using namespace dlf;

struct dlf_net {
    int N, H, W, C;
    std::vector<Layer> layers;
    std::vector<Group> plan;
    uint8_t* ws = nullptr;
    size_t ws_bytes = 0, ws_need = 0, in_off = 0, in_bytes = 0, status_off = 0, splitk_off = 0;
    int dev_sms = 0;
    int opt_no_tc = 0, opt_single_chain = 0, opt_graph = 1, opt_group_kernel = 0;
    const void* last_out = nullptr;
    // One CUDA graph holds the whole plan and follows the caller's input and output pointers; a second, instrumented one
    // records an event after every group for per-group timing.
    dlf::GraphCache graph, graph_timed;
    // dlf_net_run_host on a large batch: the plan's first groups once per part of the batch, and the rest (see host_head)
    dlf::GraphCache host_part[dlf::kHostParts], host_rest;
    bool host_whole = false;   // the plan's groups could not be captured for parts of the batch
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t host_event[dlf::kHostParts + 1] = {};
    std::vector<cudaEvent_t> group_events;
    cudaStream_t capture_stream = nullptr;
    int* status_host = nullptr;   // page-locked copy of the status word
    ~dlf_net();
};

namespace dlf {

// Split-K scratch at the end of a net's workspace: 64 KB of counters and 16 MB of fp32 partial tiles.
constexpr size_t kSplitKCounterBytes = 65536;
constexpr size_t kSplitKBytes = kSplitKCounterBytes + (16u << 20);

static bool is_param(const Layer& l) { return l.d.op == DLF_CONV || l.d.op == DLF_DWCONV || l.d.op == DLF_FC; }

int query_sms(int* out) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e);
    *out = sms;
    return DLF_OK;
}

// ---- structure of fusable chains ----------------------------------------------------------------
// Layers first..last can be ONE fused kernel only if they form a chain of dense stride-1
// size-keeping convolutions (1x1 or 3x3), each reading its predecessor, with pooling / residual
// on the last layer only and no intermediate map used anywhere else.  Pure function of the list.
static bool chain_layer_ok(const Layer& l) {
    const dlf_layer_desc& d = l.d;
    return d.op == DLF_CONV && d.groups == 1 && d.stride == 1 && d.kh == d.kw && (d.kh == 1 || d.kh == 3) &&
           d.pad == d.kh / 2 && chain_tc_layer_supported(d.cin, d.cout, d.kh);
}

static bool span_is_chain(const dlf_net* net, int first, int last) {
    if (last - first + 1 > kMaxChain) return false;
    const int n = static_cast<int>(net->layers.size());
    for (int i = first; i <= last; i++) {
        const Layer& l = net->layers[i];
        if (!chain_layer_ok(l)) return false;
        if (i > first && l.d.src != i - 1) return false;
        if (i < last && (l.d.pool != 0 || l.d.res_src != -2)) return false;
        if (i == last && l.d.res_src >= first) return false;
    }
    // no outside use of an intermediate map
    for (int j = first + 1; j < n; j++) {
        const dlf_layer_desc& d = net->layers[j].d;
        const int refs[2] = {d.src, d.res_src};
        for (int r : refs) {
            if (r < first || r >= last) continue;        // not an intermediate of this span
            if (j <= last && r == j - 1 && r == d.src) {  // the chain edge itself
                if (d.res_src == r) return false;
                continue;
            }
            return false;
        }
    }
    return true;
}

// ---- inverted-residual pattern ------------------------------------------------------------------------
// [1x1 conv (expansion), depthwise 3x3, 1x1 conv (projection)] or, without expansion, [depthwise 3x3,
// 1x1 conv]: each layer reads its predecessor, no pooling, a residual only on the projection and
// from outside the span, the maps between the layers used nowhere else.  `prefix` accepts the
// pattern's first layers (a block that may still grow into the pattern).
static bool pointwise_ok(const dlf_layer_desc& d) {
    return d.op == DLF_CONV && d.groups == 1 && d.kh == 1 && d.kw == 1 && d.stride == 1 && d.pad == 0 && d.pool == 0;
}
static bool depthwise_ok(const dlf_layer_desc& d) {
    return d.op == DLF_DWCONV && d.kh == 3 && d.kw == 3 && d.pad == 1 && (d.stride == 1 || d.stride == 2) && d.pool == 0 &&
           d.res_src == -2;
}
static bool span_is_mbconv(const dlf_net* net, int first, int last, bool prefix) {
    const int len = last - first + 1;
    if (len < 2 || len > 3) return false;
    const dlf_layer_desc& d0 = net->layers[first].d;
    const bool has_expand = d0.op == DLF_CONV;
    const int n_full = has_expand ? 3 : 2;
    if (len > n_full || (!prefix && len != n_full)) return false;
    int idx = first;
    if (has_expand) {
        if (!pointwise_ok(d0) || d0.res_src != -2) return false;
        idx++;
    }
    const dlf_layer_desc& dd = net->layers[idx].d;
    if (!depthwise_ok(dd) || (idx > first && dd.src != idx - 1)) return false;
    int hid = dd.cin, cout = 8;  // no projection yet (a prefix): nothing to check on its width
    if (idx < last) {
        const dlf_layer_desc& dp = net->layers[idx + 1].d;
        if (!pointwise_ok(dp) || dp.src != idx || dp.res_src >= first) return false;
        cout = dp.cout;
    }
    MbconvArgs a;
    std::memset(&a, 0, sizeof(a));
    a.N = 1; a.H = 8; a.W = 8;
    a.Cin = has_expand ? d0.cin : hid; a.hid = hid; a.Cout = cout; a.stride = dd.stride; a.has_expand = has_expand ? 1 : 0;
    if (!mbconv_supported(a)) return false;
    // the maps between the layers are used nowhere else
    const int n = static_cast<int>(net->layers.size());
    for (int j = first + 1; j < n; j++) {
        const dlf_layer_desc& d = net->layers[j].d;
        const int refs[2] = {d.src, d.res_src};
        for (int k = 0; k < 2; k++) {
            const int r = refs[k];
            if (r < first || r >= last) continue;
            if (k == 0 && j <= last && r == j - 1) continue;
            return false;
        }
    }
    return true;
}

static inline const uint8_t* slot(const dlf_net* net, int idx) {
    return net->ws ? net->ws + net->layers[idx].off : nullptr;
}

static ChainArgs chain_args(const dlf_net* net, int first, int last, const void* in_dev, void* out_dev) {
    ChainArgs a;
    std::memset(&a, 0, sizeof(a));
    a.n_layers = last - first + 1;
    const Layer& f = net->layers[first];
    const Layer& z = net->layers[last];
    a.x = f.d.src < 0 ? in_dev : slot(net, f.d.src);
    for (int i = first; i <= last; i++) {
        const Layer& l = net->layers[i];
        a.w[i - first] = l.w;
        a.bias[i - first] = l.bias;
        a.cin[i - first] = l.d.cin;
        a.cout[i - first] = l.d.cout;
        a.k[i - first] = l.d.kh;
        a.act[i - first] = l.d.act;
    }
    a.res = z.d.res_src == -2 ? nullptr : (z.d.res_src < 0 ? in_dev : slot(net, z.d.res_src));
    a.y = out_dev;
    a.N = static_cast<int>(f.in[0]);
    a.H = static_cast<int>(f.in[1]);
    a.W = static_cast<int>(f.in[2]);
    a.pool = z.d.pool;
    return a;
}

static ConvArgs conv_args(const dlf_net* net, int i, const void* in_dev, void* out_dev) {
    const Layer& l = net->layers[i];
    ConvArgs a;
    std::memset(&a, 0, sizeof(a));
    a.x = l.d.src < 0 ? in_dev : slot(net, l.d.src);
    a.w = l.w;
    a.bias = l.bias;
    a.res = l.d.res_src == -2 ? nullptr : (l.d.res_src < 0 ? in_dev : slot(net, l.d.res_src));
    a.y = out_dev;
    a.N = static_cast<int>(l.in[0]); a.H = static_cast<int>(l.in[1]); a.W = static_cast<int>(l.in[2]);
    a.Cin = l.d.cin; a.Ho = l.ho_pre; a.Wo = l.wo_pre; a.Cout = l.d.cout;
    a.kh = l.d.kh; a.kw = l.d.kw; a.stride = l.d.stride; a.pad = l.d.pad; a.groups = l.d.groups;
    a.act = l.d.act; a.pool = l.d.pool;
    if (net->ws) {
        a.splitk_ws = net->ws + net->splitk_off;
        a.splitk_bytes = kSplitKBytes;
    }
    return a;
}

static MbconvArgs mbconv_args(const dlf_net* net, int first, int last, const void* in_dev, void* out_dev) {
    MbconvArgs a;
    std::memset(&a, 0, sizeof(a));
    const Layer& f = net->layers[first];
    const Layer& z = net->layers[last];
    const bool has_expand = f.d.op == DLF_CONV;
    const Layer& dwl = net->layers[has_expand ? first + 1 : first];
    a.x = f.d.src < 0 ? in_dev : slot(net, f.d.src);
    a.w1 = has_expand ? f.w : nullptr; a.b1 = has_expand ? f.bias : nullptr;
    a.wd = dwl.w; a.bd = dwl.bias;
    a.w2 = z.w; a.b2 = z.bias;
    a.res = z.d.res_src == -2 ? nullptr : (z.d.res_src < 0 ? in_dev : slot(net, z.d.res_src));
    a.y = out_dev;
    a.N = static_cast<int>(f.in[0]); a.H = static_cast<int>(f.in[1]); a.W = static_cast<int>(f.in[2]);
    a.Cin = f.d.cin; a.hid = dwl.d.cin; a.Cout = z.d.cout; a.stride = dwl.d.stride;
    a.has_expand = has_expand ? 1 : 0;
    a.act1 = has_expand ? f.d.act : 0; a.act2 = dwl.d.act; a.act3 = z.d.act;
    return a;
}

// A fully connected layer is a 1x1 convolution over a 1x1 image whose channels are the flattened
// input (NHWC order, which is how the map lies in memory): the tensor-core kernel then streams the
// weight matrix through its TMA ring, one slab of output features per CTA.
static ConvArgs fc_as_conv_args(const dlf_net* net, int i, const void* in_dev, void* out_dev) {
    const Layer& l = net->layers[i];
    ConvArgs a;
    std::memset(&a, 0, sizeof(a));
    a.x = l.d.src < 0 ? in_dev : slot(net, l.d.src);
    a.w = l.w;
    a.bias = l.bias;
    a.y = out_dev;
    a.N = static_cast<int>(l.in[0]); a.H = 1; a.W = 1;
    a.Cin = l.d.cin; a.Ho = 1; a.Wo = 1; a.Cout = l.d.cout;
    a.kh = 1; a.kw = 1; a.stride = 1; a.pad = 0; a.groups = 1;
    a.act = l.d.act; a.pool = 0;
    if (net->ws) {
        a.splitk_ws = net->ws + net->splitk_off;
        a.splitk_bytes = kSplitKBytes;
    }
    return a;
}

// ---- projection branch + expansion layer of a residual block as ONE product -----------------------------------------------
// [1x1 projection (stride 1 or 2, linear) of the block's input, 1x1 expansion of the block's 3x3 output + that projection as
// residual]: y = act(x_e * W_e + b_e + x_p * W_p + b_p) is one implicit GEMM whose K runs over both inputs' channels, so the
// projection's map is never written nor read back; it joins the fp32 accumulator without its own fp16 rounding (at most half
// an fp16 unit in the last place of the projection's value away from the layer-by-layer result).
static bool span_is_projadd(const dlf_net* net, int first, int last) {
    if (net->opt_no_tc || last != first + 1) return false;
    const int n = static_cast<int>(net->layers.size());
    const dlf_layer_desc& pj = net->layers[first].d;
    const dlf_layer_desc& ex = net->layers[last].d;
    if (pj.op != DLF_CONV || ex.op != DLF_CONV || pj.groups != 1 || ex.groups != 1) return false;
    if (pj.kh != 1 || pj.kw != 1 || pj.pad != 0 || pj.pool || pj.res_src != -2 || pj.act != DLF_ACT_NONE) return false;
    if (ex.kh != 1 || ex.kw != 1 || ex.pad != 0 || ex.stride != 1 || ex.pool) return false;
    if (ex.res_src != first || ex.src == first || ex.src >= first) return false;
    for (int j = first + 1; j < n; j++) {   // the projection's map is used by the expansion layer's sum alone
        const dlf_layer_desc& d = net->layers[j].d;
        if (d.src == first || (d.res_src == first && j != last)) return false;
    }
    ConvArgs a = conv_args(net, last, nullptr, nullptr);
    a.res = nullptr;
    const Layer& pl = net->layers[first];
    a.x2 = &a;   // only whether there is one matters here
    a.H2 = static_cast<int>(pl.in[1]); a.W2 = static_cast<int>(pl.in[2]); a.Cin2 = pj.cin; a.stride2 = pj.stride;
    return conv_tc_dual_supported(a);
}

static ConvArgs projadd_args(const dlf_net* net, int first, int last, const void* in_dev, void* out_dev) {
    ConvArgs a = conv_args(net, last, in_dev, out_dev);
    const Layer& pl = net->layers[first];
    a.res = nullptr;
    a.splitk_ws = nullptr;
    a.splitk_bytes = 0;
    a.x2 = pl.d.src < 0 ? in_dev : slot(net, pl.d.src);
    a.w2 = pl.w;
    a.bias2 = pl.bias;
    a.H2 = static_cast<int>(pl.in[1]); a.W2 = static_cast<int>(pl.in[2]); a.Cin2 = pl.d.cin; a.stride2 = pl.d.stride;
    return a;
}

// ---- groups handed over through L2 -------------------------------------------------------------------------------------
// Any run of dense convolutions the single-layer tensor-core kernel takes (any kernel size, stride 1 or 2, fused pool,
// residual from anywhere, a projection branch) can run as ONE persistent kernel whose CTAs walk the layers together with a
// device-wide barrier in between; every layer's map goes to its workspace slot.
static bool span_is_seq(const dlf_net* net, int first, int last) {
    if (net->opt_no_tc || last - first + 1 > conv_seq_max_layers()) return false;
    for (int i = first; i <= last; i++) {
        const Layer& l = net->layers[i];
        if (l.d.op != DLF_CONV || l.d.groups != 1) return false;
        ConvArgs a = conv_args(net, i, nullptr, nullptr);
        if (!conv_seq_layer_supported(a)) return false;
    }
    return true;
}

static bool single_kind(const dlf_net* net, int i, Kind* kind) {
    const Layer& l = net->layers[i];
    switch (l.d.op) {
        case DLF_CONV: {
            ConvArgs a = conv_args(net, i, nullptr, nullptr);
            if (l.d.res_src == -2) a.res = nullptr; else a.res = &a;  // only whether there is one matters here
            if (!net->opt_no_tc && conv_tc_supported(a)) { *kind = K_CONV_TC; return true; }
            if (!net->opt_no_tc && stem_tc_supported(a)) { *kind = K_STEM_TC; return true; }
            if (l.d.groups > 1 && (l.d.cout / l.d.groups) % 16 != 0) return false;
            *kind = K_CONV_DIRECT;
            return true;
        }
        case DLF_DWCONV:
            if (l.d.kh != 3 || l.d.kw != 3 || l.d.cin % 8 || l.d.pool) return false;
            *kind = K_DW;
            return true;
        case DLF_FC:
            if (l.d.cin % 8) return false;
            // the CUDA-core kernel re-reads the weights once per 8 images and keeps few bytes in flight: measured
            // faster only for small matrices at small batch
            if (!net->opt_no_tc && l.d.res_src == -2 && (l.in[0] > 8 || l.w_elems * 2 >= (16ll << 20)) &&
                conv_tc_supported(fc_as_conv_args(net, i, nullptr, nullptr))) { *kind = K_CONV_TC; return true; }
            *kind = K_FC;
            return true;
        case DLF_MAXPOOL:
            if (l.d.cin % 8) return false;
            *kind = K_MAXPOOL;
            return true;
        case DLF_GAVGPOOL:
            if (l.d.cin % 8) return false;
            *kind = K_GAVG;
            return true;
    }
    return false;
}

typedef std::map<std::pair<int, int>, double> SpanTimes;
static bool chain_pays(const dlf_net* net, int first, int last, int sms, ChainTiling* tiling, SpanTimes* memo = nullptr);

static bool make_group(const dlf_net* net, int first, int last, int sms, Group* g) {
    g->first = first; g->last = last; g->sms = sms;
    g->tiling = ChainTiling{};
    g->mb_tiling = MbconvTiling{};
    if (first == last) {
        // A single layer runs through the single-layer kernels unless the option asks for the fused-group kernel
        // (a narrow 3x3 layer: 20.5 us in the single-layer kernel's row mode against 26 us here at 56x56x64, batch 32).
        // ... or the layer is a narrow 3x3 layer on an image too wide for the single-layer kernel's row mode (more than 126
        // pixels) and without the whole 64-channel chunks of its column mode: that kernel then re-loads the input window for each
        // of the nine taps, the fused-group kernel loads the tile's frame once and shifts the operand window (64 -> 64 at 224x224
        // with a pool, batch 8: 74.5 us against 52.7; in the column mode 39.9).
        const Layer& l1 = net->layers[first];
        const bool wide_narrow = l1.d.op == DLF_CONV && l1.d.kh == 3 && l1.d.kw == 3 && l1.d.stride == 1 && l1.d.pad == 1 &&
                                 l1.d.cin < 64 && l1.d.cout <= 64 && l1.wo_pre + 2 > 128;
        const bool prefer_chain = net->opt_single_chain != 0 || wide_narrow;
        if (!(prefer_chain && !net->opt_no_tc && span_is_chain(net, first, last))) return single_kind(net, first, &g->kind);
    }
    if (net->opt_no_tc) return false;
    if (first < last && span_is_mbconv(net, first, last, false)) {
        g->mb_tiling = mbconv_tiling(mbconv_args(net, first, last, nullptr, nullptr), sms);
        g->kind = K_MBCONV;
        return g->mb_tiling.ok;
    }
    if (span_is_projadd(net, first, last)) {
        g->kind = K_CONV_DUAL;
        return true;
    }
    // Two ways to fuse dense convolutions: hand-over in shared memory (a chain of stride-1 1x1 / 3x3 layers, tile by tile) or
    // through L2 (any run of dense convolutions, layer by layer behind a device-wide barrier).  Unless an option says
    // otherwise the first is taken for narrow layers (at most 64 channels: there it was measured faster), the second elsewhere.
    const bool chain_ok = span_is_chain(net, first, last);
    const bool seq_ok = first < last && span_is_seq(net, first, last);
    bool narrow = true;
    for (int i = first; i <= last; i++) narrow = narrow && net->layers[i].d.cin <= 64 && net->layers[i].d.cout <= 64;
    bool want_chain = chain_ok && (first == last || net->opt_group_kernel == 1 || (net->opt_group_kernel == 0 && narrow) || !seq_ok);
    if (chain_ok && !want_chain && net->opt_group_kernel == 0) {   // wide layers: where the estimate says the kernel pays (few tiles per SM)
        want_chain = chain_pays(net, first, last, sms, &g->tiling);
        if (want_chain) {
            g->kind = K_CHAIN_TC;
            return true;
        }
        g->tiling = ChainTiling{};
    }
    if (want_chain) {
        ChainArgs a = chain_args(net, first, last, nullptr, nullptr);
        g->tiling = chain_tc_tiling(a, sms, net->dev_sms);
        g->kind = K_CHAIN_TC;
        if (g->tiling.ok) return true;
        if (first == last) return single_kind(net, first, &g->kind);
    }
    if (seq_ok) {
        g->kind = K_CONV_SEQ;
        return true;
    }
    return false;
}

// ---- what the tuner may propose as one group --------------------------------------------------------------------
// Algorithm 1 grows a block while the layers can run as one kernel AND that kernel is expected to pay (Sec. IV-B: fusing
// helps layers with few operations and hurts heavy ones).  For a dense chain the estimate is the fused kernel's own cost
// model (the tiler's SM clocks at 1.9 GHz: measured 0.85 to 1.3 times as long) against one kernel per layer: 2.4 us (3x3: 3.1)
// plus the slowest of the latency of its 64-channel chunks, its rounds of 128-pixel tiles (twice as long where a pixel's
// channels are no multiple of 32 bytes), its operations at 600 TFLOP/s and its bytes at 5.5 TB/s.  Fitted to 90 random chains
// of 2 to 8 layers timed both ways: 16 -> 16 3x3 at 5 images of 35x32 9.3 us fused against 12.3 for three layers, 24 -> 24 at
// 10 of 81x79 66 against 113 for four, 64 -> 64 1x1 at 5 of 41x38 7.3 against 6.4 for two.
// A chain may not swallow the expansion layer of an inverted-residual block (the layer a depthwise convolution reads):
// that block fuses better as a whole.  Inverted-residual blocks have an estimate of their own (mbconv_pays).  Groups
// handed over through L2 are proposed only when the option asks for them (measured: a device-wide barrier per layer is no
// cheaper than a kernel boundary).  `prefix`: the layers may also be the beginning of a pattern that can still grow.
// A layer of a dense chain as a kernel of its own inside a network (see above).
static double single_layer_us(const Layer& l, int sms) {
    const double chunks = static_cast<double>(l.d.kh * l.d.kw * ((l.d.cin + 63) / 64));
    const double rounds = static_cast<double>(l.in[0] * l.in[1] * l.in[2]) / (128.0 * sms) * ((l.d.cout + 255) / 256);
    const double bytes = static_cast<double>(l.in[0] * l.in[1] * l.in[2] * l.in[3] * 2) + static_cast<double>(l.bytes) + static_cast<double>(l.w_elems * 2) +
                         (l.d.res_src != -2 ? static_cast<double>(l.bytes) : 0.0);
    if (l.d.kh == 1 && l.d.cin <= 64 && l.d.cout <= 64) return 2.0 + bytes / 5e6;   // (streams its bytes: conv_narrow.cu)
    return 2.4 + (l.d.kh == 3 ? 0.7 : 0.0) +
           std::max({0.1 * chunks, rounds * (0.75 + 0.3 * chunks) * (l.d.cin % 16 ? 2.0 : 1.0), static_cast<double>(l.flops) / 600e6, bytes / 5.5e6});
}
static double tiling_us(const ChainTiling& t) { return 1.1 * t.cost / 1.9e3 + 0.3; }
// The chain first..last as one kernel; negative if it cannot run as one.
// (`memo`: the spans of one tuner pass, each asked for several times; tiling a span takes 0.1 ms)
static double chain_us(const dlf_net* net, int first, int last, int sms, ChainTiling* tiling, SpanTimes* memo = nullptr) {
    if (memo) {
        const auto it = memo->find({first, last});
        if (it != memo->end()) return it->second;
        return (*memo)[{first, last}] = chain_us(net, first, last, sms, tiling);
    }
    const ChainTiling t = chain_tc_tiling(chain_args(net, first, last, nullptr, nullptr), sms, net->dev_sms > 0 ? net->dev_sms : sms);
    if (tiling) *tiling = t;
    return t.ok ? tiling_us(t) : -1.0;
}
// True if the fused kernel is expected to beat one kernel per layer on `sms` SMs.  `tiling` receives the fused kernel's tiling.
static bool chain_pays(const dlf_net* net, int first, int last, int sms, ChainTiling* tiling, SpanTimes* memo) {
    const double fused = chain_us(net, first, last, sms, tiling, memo);
    double single = 0.0;
    for (int i = first; i <= last; i++) single += single_layer_us(net->layers[i], sms);
    return fused >= 0.0 && fused < 0.97 * single;
}
// True if a block that has reached layer last - 1 should go on: some longer chain from `first` beats the block so far and
// single layers behind it (two 1x1 layers may not pay where three do; the longest chain that pays is rarely the best one).
static bool chain_grows(const dlf_net* net, int first, int last, int sms, SpanTimes* memo) {
    double rest = last - 1 == first ? single_layer_us(net->layers[first], sms) : chain_us(net, first, last - 1, sms, nullptr, memo);
    if (rest < 0.0) return false;
    for (int e = last; e < static_cast<int>(net->layers.size()) && span_is_chain(net, first, e); e++) {
        rest += single_layer_us(net->layers[e], sms);
        const double fused = chain_us(net, first, e, sms, nullptr, memo);
        if (fused >= 0.0 && fused < 0.97 * rest) return true;
        if (fused < 0.0 || fused > 1.4 * rest) break;   // (longer ones only fall further behind)
    }
    return false;
}

// The estimate for an inverted-residual block: the fused kernel's own, launch included, against one kernel per layer.  Inside a network a
// layer's own kernel takes 3.3 us (a pointwise one of at most 64 channels on either side 2.8) plus its bytes at 3.6 TB/s (the depthwise
// one) or 3.2 TB/s (the pointwise ones): the best of the constants over 3400 random blocks, each timed both ways among nine others of
// its kind; what is proposed takes 2.4 % longer than the better of the two in the geometric mean, with 2.9 us a layer 3.1 %.
// On few images the clusters of mbconv_lat.cu win (14x14, 64 -> 384 -> 64 at one image 6.5 us against 10.4 by three kernels back to back),
// from a few images on maps of 14x14 and more the persistent kernel (24 -> 144 -> 24 at 56x56: 65 us against 96 at 64 images); wide blocks on
// small maps lose at many images (160 -> 960 -> 160 at 7x7: 23 us against 22 at 64), and so does a block without an expansion layer
// (32 -> 16 at 112x112, 64 images: 86 against 46).
// (`memo`: 1 or 0 for the blocks of one tuner pass, each asked for several times)
static bool mbconv_pays(const dlf_net* net, int first, int last, int sms, SpanTimes* memo = nullptr) {
    if (memo) {
        const auto it = memo->find({first, last});
        if (it != memo->end()) return it->second > 0.0;
        return ((*memo)[{first, last}] = mbconv_pays(net, first, last, sms) ? 1.0 : 0.0) > 0.0;
    }
    const MbconvTiling t = mbconv_tiling(mbconv_args(net, first, last, nullptr, nullptr), sms);
    if (!t.ok) return false;
    double single_us = 0.0;
    for (int i = first; i <= last; i++) {
        const Layer& l = net->layers[i];
        const double bytes = static_cast<double>(l.in[0] * l.in[1] * l.in[2] * l.in[3] * 2) + static_cast<double>(l.bytes) + static_cast<double>(l.w_elems * 2) +
                             (l.d.res_src != -2 ? static_cast<double>(l.bytes) : 0.0);
        const bool narrow = l.d.op == DLF_CONV && l.d.cin <= 64 && l.d.cout <= 64;
        single_us += std::max(static_cast<double>(l.flops) / 600e6, bytes / (l.d.op == DLF_DWCONV ? 3.6e6 : 3.2e6)) + (narrow ? 2.8 : 3.3);
    }
    return t.us < single_us;
}

static bool tuner_may_fuse(const dlf_net* net, int first, int last, bool prefix, int s_max, SpanTimes* memo = nullptr) {
    if (first == last) return true;
    if (net->opt_no_tc) return false;
    if (span_is_mbconv(net, first, last, prefix)) {
        // (the layers may be the beginning of the block: the estimate is made for the whole of it)
        const int full_last = first + (net->layers[first].d.op == DLF_CONV ? 2 : 1);
        return full_last < static_cast<int>(net->layers.size()) && span_is_mbconv(net, first, full_last, false) && mbconv_pays(net, first, full_last, s_max, memo);
    }
    // Not into a block that fuses better as a whole: with everything fused that can be, MobileNetV2 takes 0.56 ms in 25 groups at 64 images
    // and 0.12 in 22 at one; 1.04 and 0.41 in 37 where a projection and the next block's expansion are one of them.
    if (net->opt_group_kernel == 2 && span_is_seq(net, first, last)) {
        const int end = last + 2;
        return end >= static_cast<int>(net->layers.size()) || !span_is_mbconv(net, last, end, false) || !mbconv_pays(net, last, end, s_max, memo);
    }
    // a projection and the expansion layer it is added to are one product with a longer K: never slower than the two kernels
    if (span_is_projadd(net, first, last)) return true;
    if (!span_is_chain(net, first, last)) return false;
    if (net->opt_group_kernel == 1) return true;
    const int n = static_cast<int>(net->layers.size());
    for (int i = first; i <= last; i++)
        if (i + 1 < n && net->layers[i + 1].d.op == DLF_DWCONV && net->layers[i + 1].d.src == i) return false;
    return prefix ? chain_grows(net, first, last, s_max, memo) : chain_pays(net, first, last, s_max, nullptr, memo);
}

// Some of the batch's images: every map is one image after another, so a group's part of the batch is the same launch from
// another address with another N.
struct Part { int n0, n; };
static const void* part_ptr(const void* base, int64_t image_bytes, const Part* part) {
    return base ? static_cast<const uint8_t*>(base) + part->n0 * image_bytes : nullptr;
}
static void take_part(const Layer& first, const Layer& last, const void** x, const void** res, void** y, int* n, const Part* part) {
    *x = part_ptr(*x, first.in[1] * first.in[2] * first.in[3] * 2, part);
    *res = part_ptr(*res, static_cast<int64_t>(last.ho_pre) * last.wo_pre * last.d.cout * 2, part);   // (added before a pool)
    *y = const_cast<void*>(part_ptr(*y, static_cast<int64_t>(last.bytes) / first.in[0], part));
    *n = part->n;
}
// Launches a group for a part of the batch; the kinds that host_head() lets through.
static int launch_group_part(dlf_net* net, const Group& g, const void* in_dev, const Part& part, cudaStream_t s) {
    const Layer& f = net->layers[g.first];
    const Layer& z = net->layers[g.last];
    void* y = net->ws + z.off;
    int* status = reinterpret_cast<int*>(net->ws + net->status_off);
    switch (g.kind) {
        case K_CHAIN_TC: {
            ChainArgs a = chain_args(net, g.first, g.last, in_dev, y);
            take_part(f, z, &a.x, &a.res, &a.y, &a.N, &part);
            return launch_chain_tc(a, chain_tc_tiling(a, g.sms, net->dev_sms > 0 ? net->dev_sms : g.sms), g.sms, status, s);
        }
        case K_MBCONV: {
            MbconvArgs a = mbconv_args(net, g.first, g.last, in_dev, y);
            take_part(f, z, &a.x, &a.res, &a.y, &a.N, &part);
            return launch_mbconv_tc(a, mbconv_tiling(a, g.sms), g.sms, status, s);
        }
        case K_CONV_TC:
        case K_STEM_TC:
        case K_DW: {
            ConvArgs a = conv_args(net, g.first, in_dev, y);
            take_part(f, z, &a.x, &a.res, &a.y, &a.N, &part);
            return g.kind == K_CONV_TC ? launch_conv_tc(a, g.sms, status, s) : (g.kind == K_STEM_TC ? launch_stem_tc(a, g.sms, status, s) : launch_dw3x3(a, g.sms, s));
        }
        case K_CONV_DUAL: {
            ConvArgs a = projadd_args(net, g.first, g.last, in_dev, y);
            take_part(z, z, &a.x, &a.res, &a.y, &a.N, &part);   // (the expansion layer's input; the projection's beside it)
            a.x2 = part_ptr(a.x2, f.in[1] * f.in[2] * f.in[3] * 2, &part);
            return launch_conv_tc(a, g.sms, status, s);
        }
        case K_MAXPOOL: {
            const void* x = z.d.src < 0 ? in_dev : net->ws + net->layers[z.d.src].off;
            const void* none = nullptr;
            int n = 0;
            take_part(z, z, &x, &none, &y, &n, &part);
            return launch_maxpool(x, y, n, static_cast<int>(z.in[1]), static_cast<int>(z.in[2]), z.d.cin, z.d.kh, z.d.stride, z.d.pad,
                                  static_cast<int>(z.out[1]), static_cast<int>(z.out[2]), g.sms, s);
        }
        default: return DLF_E_UNSUPPORTED;
    }
}
// How many of the plan's first groups dlf_net_run_host works off part by part while the rest of the input is still on its way
// (0: the input is copied as a whole).  Only a batch whose copy takes long enough (8 MB are 150 us), and groups whose own time,
// about 0.64 of the copy's by the estimates, hides behind it: a part's launches are less efficient than the whole batch's, so a longer head
// costs more than it hides; and none whose part has neither 32 pixels nor two tiles of 32 pixels by 64 channels for each SM: its four
// launches then take almost four times the whole one's.  A layer by itself is taken to cost 3.3 us beside its bytes, as in mbconv_pays, and to
// reach 400 TFLOP/s.  From page-locked memory, some of 31 batches that were tried: MobileNetV2, 64 images 748 us (five groups; 800 with four,
// 740 with six), 48 images 616 (five; 653 with four); AlexNet, 28 images 302 (two convolutions; 348 with all five); ResNet-18, 28 images
// 399 (405 with one group more).  0.45 to 0.72, 0 to 128 pixels and 400 to 500 TFLOP/s were tried (at 0.72 ResNet-18 is 4 % slower).
static int host_head(const dlf_net* net) {
    if (!net->opt_graph || net->host_whole || net->N < 2 * kHostParts || net->in_bytes < (8u << 20)) return 0;
    const double copy_us = net->in_bytes / 50e3;
    double sum = 0.0;
    int count = 0;
    for (const Group& g : net->plan) {
        if (g.last == static_cast<int>(net->layers.size()) - 1) break;
        if (g.kind != K_CHAIN_TC && g.kind != K_MBCONV && g.kind != K_CONV_TC && g.kind != K_STEM_TC && g.kind != K_DW && g.kind != K_CONV_DUAL && g.kind != K_MAXPOOL) break;
        if (net->layers[g.last].d.op == DLF_FC) break;
        double bytes = static_cast<double>(net->layers[g.first].in[0] * net->layers[g.first].in[1] * net->layers[g.first].in[2] * net->layers[g.first].in[3] * 2), flops = 0.0;
        bytes += static_cast<double>(net->layers[g.last].bytes) * (net->layers[g.last].d.res_src != -2 ? 2 : 1);
        for (int i = g.first; i <= g.last; i++) flops += static_cast<double>(net->layers[i].flops);
        const double pixels = net->N / kHostParts * static_cast<double>(net->layers[g.last].ho_pre) * net->layers[g.last].wo_pre;
        if (pixels < 32.0 * net->dev_sms && pixels * net->layers[g.last].d.cout < 2.0 * 32 * 64 * net->dev_sms) break;
        sum += g.kind == K_MBCONV ? g.mb_tiling.us : (g.kind == K_CHAIN_TC ? tiling_us(g.tiling) : 3.3 + std::max(bytes / 3.5e6, flops / 400e6));
        if (sum > 0.64 * copy_us) break;
        count++;
    }
    return count;
}

static int launch_group(dlf_net* net, const Group& g, const void* in_dev, void* final_out, cudaStream_t s) {
    const int n = static_cast<int>(net->layers.size());
    const Layer& z = net->layers[g.last];
    void* y = (g.last == n - 1) ? final_out : static_cast<void*>(net->ws + z.off);
    int* status = reinterpret_cast<int*>(net->ws + net->status_off);
    switch (g.kind) {
        case K_CHAIN_TC: {
            ChainArgs a = chain_args(net, g.first, g.last, in_dev, y);
            return launch_chain_tc(a, g.tiling, g.sms, status, s);
        }
        case K_CONV_SEQ: {
            ConvArgs a[16];
            const int cnt = g.last - g.first + 1;
            if (cnt > 16) return DLF_E_PLAN;
            for (int i = g.first; i <= g.last; i++)
                a[i - g.first] = conv_args(net, i, in_dev, i == n - 1 ? final_out : static_cast<void*>(net->ws + net->layers[i].off));
            return launch_conv_seq(a, cnt, g.sms, status, reinterpret_cast<unsigned*>(status) + 2, s);
        }
        case K_MBCONV: return launch_mbconv_tc(mbconv_args(net, g.first, g.last, in_dev, y), g.mb_tiling, g.sms, status, s);
        case K_CONV_TC:
            if (z.d.op == DLF_FC) return launch_conv_tc(fc_as_conv_args(net, g.first, in_dev, y), g.sms, status, s);
            return launch_conv_tc(conv_args(net, g.first, in_dev, y), g.sms, status, s);
        case K_CONV_DUAL: return launch_conv_tc(projadd_args(net, g.first, g.last, in_dev, y), g.sms, status, s);
        case K_STEM_TC: return launch_stem_tc(conv_args(net, g.first, in_dev, y), g.sms, status, s);
        case K_CONV_DIRECT: return launch_conv_direct(conv_args(net, g.first, in_dev, y), g.sms, s);
        case K_DW: return launch_dw3x3(conv_args(net, g.first, in_dev, y), g.sms, s);
        case K_FC: {
            const void* x = z.d.src < 0 ? in_dev : net->ws + net->layers[z.d.src].off;
            return launch_fc(x, z.w, z.bias, y, static_cast<int>(z.in[0]), z.d.cin, z.d.cout, z.d.act, g.sms, s);
        }
        case K_MAXPOOL: {
            const void* x = z.d.src < 0 ? in_dev : net->ws + net->layers[z.d.src].off;
            return launch_maxpool(x, y, static_cast<int>(z.in[0]), static_cast<int>(z.in[1]), static_cast<int>(z.in[2]),
                                  z.d.cin, z.d.kh, z.d.stride, z.d.pad, static_cast<int>(z.out[1]),
                                  static_cast<int>(z.out[2]), g.sms, s);
        }
        case K_GAVG: {
            const void* x = z.d.src < 0 ? in_dev : net->ws + net->layers[z.d.src].off;
            return launch_gavgpool(x, y, static_cast<int>(z.in[0]), static_cast<int>(z.in[1]), static_cast<int>(z.in[2]),
                                   z.d.cin, g.sms, s);
        }
    }
    return DLF_E_UNSUPPORTED;
}

}  // namespace dlf
namespace dlf {
int kernels_init() {
    int rc = conv_tc_init();
    if (rc == DLF_OK) rc = chain_tc_init();
    if (rc == DLF_OK) rc = mbconv_tc_init();
    if (rc == DLF_OK) rc = mbconv_lat_init();
    return rc ? rc : stem_tc_init();
}

static void invalidate_graphs(dlf_net* net) {
    net->graph.drop();
    net->graph_timed.drop();
    for (GraphCache& gc : net->host_part) gc.drop();
    net->host_rest.drop();
    net->host_whole = false;
}

// Captures the launches of every group of the plan into one executable graph (thread-local
// capture on a stream the net owns, so that nothing else the caller's thread or other threads
// enqueue is swallowed).  With `timed`, an event is recorded before the first and after every group.  g_begin, g_end: these
// groups of the plan only (-1: to the end); `part`: for some of the images.
static int build_graph(dlf_net* net, GraphCache* gc, const void* in_dev, void* out_dev, bool timed, int g_begin = 0, int g_end = -1, const Part* part = nullptr) {
    gc->drop();
    cudaError_t e;
    if (!net->capture_stream) {
        e = cudaStreamCreateWithFlags(&net->capture_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    if (timed) {
        while (net->group_events.size() < net->plan.size() + 1) {
            cudaEvent_t ev;
            e = cudaEventCreate(&ev);
            if (e != cudaSuccess) return cuda_fail(e);
            net->group_events.push_back(ev);
        }
    }
    cudaStream_t cs = net->capture_stream;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(e);
    int rc = DLF_OK;
    if (timed) cudaEventRecordWithFlags(net->group_events[0], cs, cudaEventRecordExternal);
    const size_t end = g_end < 0 ? net->plan.size() : static_cast<size_t>(g_end);
    for (size_t g = g_begin; g < end && rc == DLF_OK; g++) {
        rc = part ? launch_group_part(net, net->plan[g], in_dev, *part, cs) : launch_group(net, net->plan[g], in_dev, out_dev, cs);
        if (rc == DLF_OK) {   // the group's kernel is what the capture would wait for next
            cudaStreamCaptureStatus cst;
            const cudaGraphNode_t* deps = nullptr;
            const cudaGraphEdgeData* edges = nullptr;
            size_t n_deps = 0;
            e = cudaStreamGetCaptureInfo_v3(cs, &cst, nullptr, nullptr, &deps, &edges, &n_deps);
            if (e != cudaSuccess) rc = cuda_fail(e);
            else gc->nodes.push_back(n_deps == 1 ? deps[0] : nullptr);
        }
        if (timed && rc == DLF_OK) cudaEventRecordWithFlags(net->group_events[g + 1], cs, cudaEventRecordExternal);
    }
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(cs, &graph);
    if (rc != DLF_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e);
    gc->graph = graph;
    e = cudaGraphInstantiate(&gc->exec, graph, 0);
    if (e != cudaSuccess) {
        gc->exec = nullptr;
        gc->drop();
        return cuda_fail(e);
    }
    gc->in = in_dev;
    gc->out = out_dev;
    return DLF_OK;
}

// True if the group's kernel is given the network's input or writes its output.
static bool group_touches_io(const dlf_net* net, const Group& g) {
    for (int i = g.first; i <= g.last; i++)
        if (net->layers[i].d.src == -1 || net->layers[i].d.res_src == -1) return true;
    return g.last == static_cast<int>(net->layers.size()) - 1;
}

// New input or output buffers: the few groups that see them get new kernel parameters (capturing and instantiating the
// whole plan again costs a caller with a buffer per batch more than the plan itself: 2.4 ms against 0.2 ms for ResNet-18 at
// batch 8).  Launches already enqueued keep the parameters they were enqueued with.
static int retarget_graph(dlf_net* net, GraphCache* gc, const void* in_dev, void* out_dev) {
    for (size_t g = 0; g < net->plan.size(); g++) {
        if (!group_touches_io(net, net->plan[g])) continue;
        if (!gc->nodes[g]) return DLF_E_CUDA;
        const GraphNodeUpdate update{gc->exec, gc->nodes[g]};
        g_node_update = &update;
        const int rc = launch_group(net, net->plan[g], in_dev, out_dev, net->capture_stream);
        g_node_update = nullptr;
        if (rc) return rc;
    }
    gc->in = in_dev;
    gc->out = out_dev;
    return DLF_OK;
}

static int run_graph(dlf_net* net, GraphCache* gc, const void* in_dev, void* out_dev, bool timed, cudaStream_t s) {
    if (gc->exec && (gc->in != in_dev || gc->out != out_dev) && retarget_graph(net, gc, in_dev, out_dev) != DLF_OK) gc->drop();
    if (!gc->exec) {
        int rc = build_graph(net, gc, in_dev, out_dev, timed);
        if (rc) return rc;
    }
    cudaError_t e = cudaGraphLaunch(gc->exec, s);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

// First image of every part, and one past the last part's.  A part starts on a multiple of four bytes, as the first-layer kernel
// reads its input in words (an odd number of 2-byte elements per image: the parts hold even numbers of images, but for the last).
static void host_part_bounds(const dlf_net* net, int (&n0)[kHostParts + 1]) {
    const int unit = net->in_bytes / net->N % 4 ? 2 : 1;
    for (int i = 0; i < kHostParts; i++) n0[i] = static_cast<int>(static_cast<int64_t>(net->N) * i / kHostParts) / unit * unit;
    n0[kHostParts] = net->N;
}

// What run_host_parts() launches; enqueues nothing.
static int build_host_parts(dlf_net* net, int head) {
    cudaError_t e = cudaSuccess;
    if (!net->copy_stream) e = cudaStreamCreateWithFlags(&net->copy_stream, cudaStreamNonBlocking);
    for (cudaEvent_t& ev : net->host_event)
        if (e == cudaSuccess && !ev) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(e);
    uint8_t* in_dev = net->ws + net->in_off;
    void* out_dev = net->ws + net->layers.back().off;
    int n0[kHostParts + 1];
    host_part_bounds(net, n0);
    for (int i = 0; i <= kHostParts; i++) {
        GraphCache* gc = i < kHostParts ? &net->host_part[i] : &net->host_rest;
        if (gc->exec) continue;
        const Part part{n0[i], i < kHostParts ? n0[i + 1] - n0[i] : 0};
        const int rc = i < kHostParts ? build_graph(net, gc, in_dev, out_dev, false, 0, head, &part) : build_graph(net, gc, in_dev, out_dev, false, head);
        if (rc) return rc;
    }
    return DLF_OK;
}

// The input in kHostParts copies on a stream of the net's own, the plan's first groups for a part as soon as it is there, then
// the other groups for the whole batch.  Leaves the output in its workspace slot.  Each part's groups are launched ahead of the
// next copy: one from pageable memory holds this thread until it is almost done.
static int run_host_parts(dlf_net* net, const void* in_host, cudaStream_t s) {
    uint8_t* in_dev = net->ws + net->in_off;
    const size_t image = net->in_bytes / net->N;
    int n0[kHostParts + 1];
    host_part_bounds(net, n0);
    cudaError_t e = cudaEventRecord(net->host_event[kHostParts], s);   // what the stream holds so far may still read the workspace or write the host buffer
    if (e == cudaSuccess) e = cudaStreamWaitEvent(net->copy_stream, net->host_event[kHostParts], 0);
    for (int i = 0; i < kHostParts && e == cudaSuccess; i++) {
        e = cudaMemcpyAsync(in_dev + n0[i] * image, static_cast<const uint8_t*>(in_host) + n0[i] * image, (n0[i + 1] - n0[i]) * image, cudaMemcpyHostToDevice, net->copy_stream);
        if (e == cudaSuccess) e = cudaEventRecord(net->host_event[i], net->copy_stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, net->host_event[i], 0);
        if (e == cudaSuccess) e = cudaGraphLaunch(net->host_part[i].exec, s);
    }
    if (e == cudaSuccess) e = cudaGraphLaunch(net->host_rest.exec, s);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(net->copy_stream);   // the caller's buffer is no longer read
        return cuda_fail(e);
    }
    net->last_out = net->ws + net->layers.back().off;
    return DLF_OK;
}

static int check_ready(const dlf_net* net) {
    if (!net->ws) return DLF_E_WORKSPACE;
    if (net->plan.empty()) return DLF_E_STATE;
    for (const Layer& l : net->layers)
        if (is_param(l) && (!l.w || !l.bias)) return DLF_E_STATE;
    return DLF_OK;
}

static int validate_plan(const dlf_net* net, int n_groups, const int32_t* ends, const int32_t* sms, std::vector<Group>* out) {
    const int n = static_cast<int>(net->layers.size());
    if (n_groups < 1 || n_groups > n) return DLF_E_PLAN;
    std::vector<char> is_end(n, 0);
    int prev = -1;
    for (int g = 0; g < n_groups; g++) {
        if (ends[g] <= prev || ends[g] >= n) return DLF_E_PLAN;
        if (sms[g] < 1 || sms[g] > net->dev_sms) return DLF_E_PLAN;
        prev = ends[g];
        is_end[prev] = 1;
    }
    if (prev != n - 1) return DLF_E_PLAN;
    int first = 0;
    out->clear();
    std::vector<char> stored(n, 0);   // the layer's map reaches its workspace slot: a group's last layer, any layer of an L2 group
    for (int g = 0; g < n_groups; g++) {
        Group grp;
        if (!make_group(net, first, ends[g], sms[g], &grp)) return DLF_E_PLAN;
        out->push_back(grp);
        for (int i = first; i <= ends[g]; i++) stored[i] = (i == ends[g] || grp.kind == K_CONV_SEQ) ? 1 : 0;
        first = ends[g] + 1;
    }
    // a tensor read across a group boundary must have been stored
    first = 0;
    for (int g = 0; g < n_groups; g++) {
        for (int i = first; i <= ends[g]; i++) {
            const int refs[2] = {net->layers[i].d.src, net->layers[i].d.res_src};
            for (int r : refs)
                if (r >= 0 && r < first && !stored[r]) return DLF_E_PLAN;
        }
        first = ends[g] + 1;
    }
    return DLF_OK;
}

// Eq. 5 mapped to an SM count.
static int layer_sms(const Layer& l, const dlf_tuner_params& p, int s_max) {
    const double score = p.alpha * std::log2(static_cast<double>(l.d.cout)) + p.beta * std::log2(static_cast<double>(l.flops));
    const double s = std::floor(p.kappa * score + p.kappa0 + 0.5);
    return static_cast<int>(std::min<double>(std::max<double>(s, 1.0), s_max));
}

}  // namespace dlf

namespace dlf {
// The search's second half: given the best time t[a][len-1] of every span a..a+len-1 (infinity: cannot run) and the SM
// count that reached it, the contiguous partition with the least total time (a plan's time is the sum of its groups').
static int solve_partition(int n, int max_len, const std::vector<std::vector<float>>& t, const std::vector<std::vector<int>>& ts, int* n_groups,
                           int32_t* group_end, int32_t* sm_count, float* best_ms) {
    const float inf = std::numeric_limits<float>::infinity();
    std::vector<float> best(n + 1, inf);
    std::vector<int> from(n + 1, -1);
    best[0] = 0.0f;
    for (int i = 1; i <= n; i++)
        for (int len = 1; len <= max_len && len <= i; len++) {
            const int a = i - len;
            if (best[a] == inf || t[a][len - 1] == inf) continue;
            if (best[a] + t[a][len - 1] < best[i]) { best[i] = best[a] + t[a][len - 1]; from[i] = a; }
        }
    if (best[n] == inf) return DLF_E_PLAN;
    std::vector<int> cuts;
    for (int i = n; i > 0; i = from[i]) cuts.push_back(i);
    std::reverse(cuts.begin(), cuts.end());
    int a = 0;
    for (size_t g = 0; g < cuts.size(); g++) {
        group_end[g] = cuts[g] - 1;
        sm_count[g] = ts[a][cuts[g] - a - 1];
        a = cuts[g];
    }
    *n_groups = static_cast<int>(cuts.size());
    if (best_ms) *best_ms = best[n];
    return DLF_OK;
}
}  // namespace dlf

dlf_net::~dlf_net() {
    graph.drop();
    graph_timed.drop();
    for (cudaEvent_t ev : group_events) cudaEventDestroy(ev);
    if (capture_stream) cudaStreamDestroy(capture_stream);
    for (dlf::GraphCache& gc : host_part) gc.drop();
    host_rest.drop();
    for (cudaEvent_t ev : host_event)
        if (ev) cudaEventDestroy(ev);
    if (copy_stream) cudaStreamDestroy(copy_stream);
    if (status_host) cudaFreeHost(status_host);
}

// ---- C ABI ------------------------------------------------------------------------------------------

extern "C" {

const char* dlf_strerror(int status) {
    switch (status) {
        case DLF_OK: return "ok";
        case DLF_E_INVALID_ARG: return "invalid argument";
        case DLF_E_SHAPE: return "layer list does not type-check";
        case DLF_E_PLAN: return "invalid fusion plan";
        case DLF_E_WORKSPACE: return "workspace missing, misaligned or too small";
        case DLF_E_UNSUPPORTED: return "unsupported layer";
        case DLF_E_CUDA: return "CUDA error";
        case DLF_E_TIMEOUT: return "device-side wait timed out";
        case DLF_E_STATE: return "call out of order (weights, plan or workspace missing)";
    }
    return "unknown status";
}

int dlf_last_cuda_error(void) { return g_last_cuda_error; }

int dlf_device_sm_count(void) {
    int sms = 0;
    int rc = query_sms(&sms);
    return rc ? rc : sms;
}

int dlf_net_create(const dlf_layer_desc* layers, int n_layers, int N, int H, int W, int C, dlf_net** out) {
    if (!layers || !out || n_layers <= 0 || N <= 0 || H <= 0 || W <= 0 || C <= 0) return DLF_E_INVALID_ARG;
    *out = nullptr;
    dlf_net* net = new (std::nothrow) dlf_net();
    if (!net) return DLF_E_INVALID_ARG;
    net->N = N; net->H = H; net->W = W; net->C = C;
    net->layers.resize(n_layers);
    int rc = DLF_OK;
    size_t off = 0;
    net->in_off = 0;
    net->in_bytes = static_cast<size_t>(N) * H * W * C * 2;
    off = align_up(net->in_bytes, 256);
    for (int i = 0; i < n_layers && rc == DLF_OK; i++) {
        Layer& l = net->layers[i];
        l.d = layers[i];
        l.w = nullptr; l.bias = nullptr;
        const dlf_layer_desc& d = l.d;
        if (d.op < DLF_CONV || d.op > DLF_GAVGPOOL || d.act < DLF_ACT_NONE || d.act > DLF_ACT_RELU6) { rc = DLF_E_INVALID_ARG; break; }
        if (d.src < -1 || d.src >= i || d.res_src < -2 || d.res_src >= i) { rc = DLF_E_SHAPE; break; }
        const int64_t* in = nullptr;
        int64_t net_in[4] = {N, H, W, C};
        in = d.src < 0 ? net_in : net->layers[d.src].out;
        std::memcpy(l.in, in, sizeof(l.in));
        l.ops_eq1 = l.flops = l.w_elems = 0;
        if (d.op == DLF_CONV || d.op == DLF_DWCONV || d.op == DLF_MAXPOOL) {
            if (d.kh <= 0 || d.kw <= 0 || d.stride <= 0 || d.pad < 0) { rc = DLF_E_INVALID_ARG; break; }
            if (d.cin != in[3]) { rc = DLF_E_SHAPE; break; }
            const int64_t ho = (in[1] + 2 * d.pad - d.kh) / d.stride + 1, wo = (in[2] + 2 * d.pad - d.kw) / d.stride + 1;
            if (in[1] + 2 * d.pad < d.kh || in[2] + 2 * d.pad < d.kw || ho <= 0 || wo <= 0) { rc = DLF_E_SHAPE; break; }
            l.ho_pre = static_cast<int>(ho); l.wo_pre = static_cast<int>(wo);
            if (d.op == DLF_MAXPOOL) {
                if (d.cout != d.cin || d.pad >= d.kh || d.pool != 0 || d.res_src != -2) { rc = DLF_E_SHAPE; break; }
                l.out[0] = in[0]; l.out[1] = ho; l.out[2] = wo; l.out[3] = d.cin;
            } else {
                if (d.groups <= 0 || d.cin % d.groups || d.cout % d.groups || d.cout <= 0) { rc = DLF_E_SHAPE; break; }
                if (d.op == DLF_DWCONV && !(d.groups == d.cin && d.cin == d.cout)) { rc = DLF_E_SHAPE; break; }
                if (d.pool != 0 && d.pool != 2) { rc = DLF_E_INVALID_ARG; break; }
                const int64_t hp = d.pool ? ho / 2 : ho, wp = d.pool ? wo / 2 : wo;
                if (hp <= 0 || wp <= 0) { rc = DLF_E_SHAPE; break; }
                l.out[0] = in[0]; l.out[1] = hp; l.out[2] = wp; l.out[3] = d.cout;
                l.ops_eq1 = 2 * ho * wo * d.kh * d.kw * static_cast<int64_t>(d.cin) * d.cout;
                l.flops = l.ops_eq1 * in[0] / d.groups;
                l.w_elems = static_cast<int64_t>(d.cout) * d.kh * d.kw * (d.cin / d.groups);
            }
        } else if (d.op == DLF_FC) {
            if (d.cin != in[1] * in[2] * in[3] || d.cout <= 0 || d.pool != 0) { rc = DLF_E_SHAPE; break; }
            l.out[0] = in[0]; l.out[1] = 1; l.out[2] = 1; l.out[3] = d.cout;
            l.ops_eq1 = 2 * static_cast<int64_t>(d.cin) * d.cout;
            l.flops = l.ops_eq1 * in[0];
            l.w_elems = static_cast<int64_t>(d.cin) * d.cout;
            l.ho_pre = l.wo_pre = 1;
        } else {  // global average pool
            if (d.cin != in[3] || d.cout != d.cin || d.pool != 0 || d.res_src != -2) { rc = DLF_E_SHAPE; break; }
            l.out[0] = in[0]; l.out[1] = 1; l.out[2] = 1; l.out[3] = d.cin;
            l.ho_pre = l.wo_pre = 1;
        }
        if (d.res_src != -2) {
            // the residual must have the shape of the pre-pool output
            int64_t rs[4];
            std::memcpy(rs, d.res_src < 0 ? net_in : net->layers[d.res_src].out, sizeof(rs));
            if (rs[0] != l.out[0] || rs[1] != l.ho_pre || rs[2] != l.wo_pre || rs[3] != l.out[3]) { rc = DLF_E_SHAPE; break; }
        }
        l.bytes = static_cast<size_t>(l.out[0] * l.out[1] * l.out[2] * l.out[3]) * 2;
        l.off = off;
        off = align_up(off + l.bytes, 256);
    }
    if (rc == DLF_OK) {
        // every layer must have a kernel
        for (int i = 0; i < n_layers; i++) {
            Kind k;
            if (!single_kind(net, i, &k)) { rc = DLF_E_UNSUPPORTED; break; }
        }
    }
    if (rc != DLF_OK) {
        delete net;
        return rc;
    }
    net->status_off = off;
    net->splitk_off = off + 256;
    net->ws_need = net->splitk_off + kSplitKBytes;
    *out = net;
    return DLF_OK;
}

void dlf_net_destroy(dlf_net* net) { delete net; }

int dlf_net_layer_info(const dlf_net* net, int layer, int64_t* ops_eq1, int64_t* flops, int64_t out_shape[4]) {
    if (!net || layer < 0 || layer >= static_cast<int>(net->layers.size())) return DLF_E_INVALID_ARG;
    const Layer& l = net->layers[layer];
    if (ops_eq1) *ops_eq1 = l.ops_eq1;
    if (flops) *flops = l.flops;
    if (out_shape) std::memcpy(out_shape, l.out, sizeof(l.out));
    return DLF_OK;
}

int dlf_net_set_weights(dlf_net* net, int layer, const void* w_f16_dev, const float* bias_dev) {
    if (!net || layer < 0 || layer >= static_cast<int>(net->layers.size()) || !w_f16_dev || !bias_dev) return DLF_E_INVALID_ARG;
    Layer& l = net->layers[layer];
    if (!is_param(l)) return DLF_E_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(w_f16_dev) & 15) || (reinterpret_cast<uintptr_t>(bias_dev) & 15)) return DLF_E_INVALID_ARG;
    l.w = w_f16_dev;
    invalidate_graphs(net);
    l.bias = bias_dev;
    return DLF_OK;
}

int dlf_net_workspace_bytes(const dlf_net* net, size_t* bytes) {
    if (!net || !bytes) return DLF_E_INVALID_ARG;
    *bytes = net->ws_need;
    return DLF_OK;
}

int dlf_net_bind_workspace(dlf_net* net, void* workspace_dev, size_t bytes) {
    if (!net) return DLF_E_INVALID_ARG;
    if (!workspace_dev || (reinterpret_cast<uintptr_t>(workspace_dev) & 255) || bytes < net->ws_need) return DLF_E_WORKSPACE;
    if (net->dev_sms == 0) {
        int rc = query_sms(&net->dev_sms);
        if (rc) return rc;
    }
    net->ws = static_cast<uint8_t*>(workspace_dev);
    invalidate_graphs(net);
    net->ws_bytes = bytes;
    if (!net->status_host && cudaHostAlloc(reinterpret_cast<void**>(&net->status_host), sizeof(int), cudaHostAllocDefault) != cudaSuccess) {
        net->status_host = nullptr;
        return cuda_fail(cudaErrorMemoryAllocation);
    }
    // the status block and, behind it, the split-K arrival counters (zero between launches)
    cudaError_t e = cudaMemset(net->ws + net->status_off, 0, 256 + kSplitKCounterBytes);
    if (e != cudaSuccess) return cuda_fail(e);
    return DLF_OK;
}

int dlf_net_set_plan(dlf_net* net, int n_groups, const int32_t* group_end, const int32_t* sm_count) {
    if (!net || !group_end || !sm_count) return DLF_E_INVALID_ARG;
    if (net->dev_sms == 0) {
        int rc = query_sms(&net->dev_sms);
        if (rc) return rc;
    }
    std::vector<Group> plan;
    int rc = validate_plan(net, n_groups, group_end, sm_count, &plan);
    if (rc) return rc;
    rc = kernels_init();
    if (rc) return rc;
    net->plan.swap(plan);
    invalidate_graphs(net);
    return DLF_OK;
}

int dlf_net_plan_unfused(dlf_net* net) {
    if (!net) return DLF_E_INVALID_ARG;
    if (net->dev_sms == 0) {
        int rc = query_sms(&net->dev_sms);
        if (rc) return rc;
    }
    const int n = static_cast<int>(net->layers.size());
    std::vector<int32_t> ends(n), sms(n, net->dev_sms);
    for (int i = 0; i < n; i++) ends[i] = i;
    return dlf_net_set_plan(net, n, ends.data(), sms.data());
}

int dlf_net_get_plan(const dlf_net* net, int* n_groups, int32_t* group_end, int32_t* sm_count) {
    if (!net || !n_groups || !group_end || !sm_count) return DLF_E_INVALID_ARG;
    *n_groups = static_cast<int>(net->plan.size());
    for (size_t g = 0; g < net->plan.size(); g++) {
        group_end[g] = net->plan[g].last;
        sm_count[g] = net->plan[g].sms;
    }
    return DLF_OK;
}

int dlf_net_group_is_legal(const dlf_net* net, int first, int last, int sm_count) {
    if (!net || first < 0 || last < first || last >= static_cast<int>(net->layers.size())) return DLF_E_INVALID_ARG;
    if (net->dev_sms == 0) {
        int rc = query_sms(&const_cast<dlf_net*>(net)->dev_sms);
        if (rc) return rc;
    }
    if (sm_count < 1 || sm_count > net->dev_sms) return 0;
    Group g;
    return make_group(net, first, last, sm_count, &g) ? 1 : 0;
}

int dlf_net_tuner_may_fuse(const dlf_net* net, int first, int last, int prefix, int s_max) {
    if (!net || first < 0 || last < first || last >= static_cast<int>(net->layers.size()) || s_max < 1) return DLF_E_INVALID_ARG;
    return tuner_may_fuse(net, first, last, prefix != 0, s_max) ? 1 : 0;
}

int dlf_net_autotune(const dlf_net* net, const dlf_tuner_params* params, int* n_groups, int32_t* group_end,
                     int32_t* sm_count) {
    if (!net || !params || !n_groups || !group_end || !sm_count) return DLF_E_INVALID_ARG;
    int s_max = params->s_max;
    if (s_max <= 0 || params->legalise) {
        int sms = net->dev_sms;
        if (sms == 0) {
            int rc = query_sms(&sms);
            if (rc) return rc;
            const_cast<dlf_net*>(net)->dev_sms = sms;
        }
        if (s_max <= 0 || s_max > sms) s_max = sms;
    }
    if (!(params->op_critical > 0.0)) return DLF_E_INVALID_ARG;
    const int n = static_cast<int>(net->layers.size());
    double sum_op = 0.0, sum_mp = 0.0;
    int block = 0, start = 0, ng = 0;
    SpanTimes memo;
    for (int i = 0; i < n; i++) {
        const Layer& l = net->layers[i];
        if (is_param(l)) {
            sum_op += static_cast<double>(l.flops);
            sum_mp += layer_sms(l, *params, s_max);
            block++;
        }
        // a block may grow while its layers are, or can still become, a group one kernel runs; it may
        // close only where they already are one (inside an inverted-residual block it keeps growing)
        bool forced = (i == n - 1) || !tuner_may_fuse(net, start, i + 1, true, s_max, &memo);
        const bool closable = (i == start) || tuner_may_fuse(net, start, i, false, s_max, &memo);
        if (!forced && params->legalise) {
            Group g;
            if (i + 1 > start && tuner_may_fuse(net, start, i + 1, false, s_max, &memo))
                forced = !make_group(net, start, i + 1, s_max, &g);
        }
        if (block > 0) {
            const double avg = sum_mp / block;
            if ((sum_op / avg >= params->op_critical && closable) || forced) {
                int mp = 1 << static_cast<int>(std::floor(std::log2(avg)));
                if (avg >= s_max) mp = s_max;  // the top step is the whole chip, as 32 of 32 cores in the paper
                mp = std::min(std::max(mp, 1), s_max);
                Group g;
                if (params->legalise && i > start && !make_group(net, start, i, mp, &g)) {
                    // the block cannot run as one kernel: one group per layer
                    for (int j = start; j <= i; j++) { group_end[ng] = j; sm_count[ng] = mp; ng++; }
                } else {
                    group_end[ng] = i;
                    sm_count[ng] = mp;
                    ng++;
                }
                sum_op = sum_mp = 0.0;
                block = 0;
                start = i + 1;
            }
        } else if (forced) {
            group_end[ng] = i;
            sm_count[ng] = s_max;
            ng++;
            start = i + 1;
        }
    }
    *n_groups = ng;
    return DLF_OK;
}

int dlf_net_run(dlf_net* net, const void* in_f16_dev, void* out_f16_dev, void* stream) {
    if (!net || !in_f16_dev || !out_f16_dev) return DLF_E_INVALID_ARG;
    int rc = check_ready(net);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (net->opt_graph) {
        rc = run_graph(net, &net->graph, in_f16_dev, out_f16_dev, false, s);
        if (rc) return rc;
    } else {
        for (const Group& g : net->plan) {
            g_stream_order = &g == &net->plan[0];
            rc = launch_group(net, g, in_f16_dev, out_f16_dev, s);
            g_stream_order = false;
            if (rc) return rc;
        }
    }
    net->last_out = out_f16_dev;
    return DLF_OK;
}

int dlf_net_sync(dlf_net* net, void* stream) {
    if (!net) return DLF_E_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    // the status word comes back behind the kernels, so that one wait is enough (a blocking copy after it costs 8 us)
    if (net->ws) e = cudaMemcpyAsync(net->status_host, net->ws + net->status_off, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return cuda_fail(e);
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e);
    if (net->ws) {
        const int st = *net->status_host;
        if (st != 0) {
            g_last_cuda_error = st;
            cudaMemset(net->ws + net->status_off, 0, 4 * sizeof(int));   // the status word and the multi-layer kernels' barrier counters
            // a launch that gave up may have left split-K arrival counters behind
            cudaMemset(net->ws + net->splitk_off, 0, kSplitKCounterBytes);
            return DLF_E_TIMEOUT;
        }
    }
    return DLF_OK;
}

int dlf_net_debug_stall(dlf_net* net, int limit_us, void* stream) {
    if (!net || limit_us < 1 || limit_us > 1000000) return DLF_E_INVALID_ARG;
    if (!net->ws) return DLF_E_WORKSPACE;
    return launch_stall(reinterpret_cast<int*>(net->ws + net->status_off), static_cast<unsigned long long>(limit_us) * 1000ull,
                        static_cast<cudaStream_t>(stream));
}

int dlf_net_run_host(dlf_net* net, const void* in_f16_host, void* out_f16_host, void* stream) {
    if (!net || !in_f16_host || !out_f16_host) return DLF_E_INVALID_ARG;
    int rc = check_ready(net);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const Layer& z = net->layers.back();
    cudaError_t e = cudaSuccess;
    int head = host_head(net);
    if (head > 0 && build_host_parts(net, head) != DLF_OK) {   // (a part is refused where the whole batch may not be)
        invalidate_graphs(net);
        net->host_whole = true;
        head = 0;
    }
    if (head > 0) {
        rc = run_host_parts(net, in_f16_host, s);
        if (rc) return rc;
    } else {
        e = cudaMemcpyAsync(net->ws + net->in_off, in_f16_host, net->in_bytes, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return cuda_fail(e);
        rc = dlf_net_run(net, net->ws + net->in_off, net->ws + z.off, s);
        if (rc) return rc;
    }
    e = cudaMemcpyAsync(out_f16_host, net->ws + z.off, z.bytes, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return cuda_fail(e);
    return dlf_net_sync(net, s);
}

static float median_of(std::vector<float> v) {
    std::sort(v.begin(), v.end());
    return v.empty() ? 0.0f : v[v.size() / 2];
}

int dlf_net_time(dlf_net* net, const void* in_dev, void* out_dev, void* stream, int warmup, int iters, void* flush_dev,
                 size_t flush_bytes, float* ms_median, float* ms_min, float* ms_per_group) {
    if (!net || !in_dev || !out_dev || warmup < 0 || iters < 1) return DLF_E_INVALID_ARG;
    int rc = check_ready(net);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t ng = net->plan.size();
    std::vector<cudaEvent_t> ev(2);
    for (auto& e : ev)
        if (cudaEventCreate(&e) != cudaSuccess) return cuda_fail(cudaGetLastError());
    auto cleanup = [&]() { for (auto& e : ev) cudaEventDestroy(e); };
    for (int i = 0; i < warmup; i++) {
        rc = dlf_net_run(net, in_dev, out_dev, s);
        if (rc) { cleanup(); return rc; }
    }
    std::vector<float> times;
    for (int i = 0; i < iters; i++) {
        if (flush_dev && flush_bytes) cudaMemsetAsync(flush_dev, i & 0xff, flush_bytes, s);
        cudaEventRecord(ev[0], s);
        rc = dlf_net_run(net, in_dev, out_dev, s);
        if (rc) { cleanup(); return rc; }
        cudaEventRecord(ev[1], s);
        cudaError_t e = cudaEventSynchronize(ev[1]);
        if (e != cudaSuccess) { cleanup(); return cuda_fail(e); }
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, ev[0], ev[1]);
        times.push_back(ms);
    }
    if (ms_median) *ms_median = median_of(times);
    if (ms_min) *ms_min = *std::min_element(times.begin(), times.end());
    if (ms_per_group) {
        std::vector<std::vector<float>> per(ng);
        const int reps = std::min(std::max(iters, 3), 20);
        for (int i = 0; i < reps; i++) {
            if (flush_dev && flush_bytes) cudaMemsetAsync(flush_dev, i & 0xff, flush_bytes, s);
            rc = run_graph(net, &net->graph_timed, in_dev, out_dev, true, s);
            if (rc) { cleanup(); return rc; }
            cudaError_t e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) { cleanup(); return cuda_fail(e); }
            for (size_t g = 0; g < ng; g++) {
                float ms = 0.0f;
                cudaEventElapsedTime(&ms, net->group_events[g], net->group_events[g + 1]);
                per[g].push_back(ms);
            }
        }
        for (size_t g = 0; g < ng; g++) ms_per_group[g] = median_of(per[g]);
    }
    cleanup();
    return dlf_net_sync(net, s);
}

// Median device time of ONE launch of group `g`: a graph of kReps back-to-back launches (which hides the
// host's launch cost) is timed `iters` times between two events after `warmup` untimed launches.
static int time_group(dlf_net* net, const Group& g, const void* in_dev, void* final_out, cudaStream_t s, cudaEvent_t e0,
                      cudaEvent_t e1, int warmup, int iters, float* ms_out) {
    const int kReps = 4;
    int rc = DLF_OK;
    cudaGraphExec_t exec = nullptr;
    if (!net->capture_stream && cudaStreamCreateWithFlags(&net->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
        return cuda_fail(cudaGetLastError());
    cudaGraph_t graph = nullptr;
    if (cudaStreamBeginCapture(net->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return cuda_fail(cudaGetLastError());
    for (int r = 0; r < kReps && rc == DLF_OK; r++) rc = launch_group(net, g, in_dev, final_out, net->capture_stream);
    cudaError_t e = cudaStreamEndCapture(net->capture_stream, &graph);
    if (rc == DLF_OK && e != cudaSuccess) rc = cuda_fail(e);
    if (rc == DLF_OK && cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
    if (graph) cudaGraphDestroy(graph);
    for (int i = 0; i < warmup && rc == DLF_OK; i++)
        if (cudaGraphLaunch(exec, s) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
    std::vector<float> v;
    for (int i = 0; i < iters && rc == DLF_OK; i++) {
        cudaEventRecord(e0, s);
        if (cudaGraphLaunch(exec, s) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
        cudaEventRecord(e1, s);
        if (rc == DLF_OK && cudaEventSynchronize(e1) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
        float ms = 0.0f;
        if (rc == DLF_OK) cudaEventElapsedTime(&ms, e0, e1);
        v.push_back(ms / kReps);
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (rc == DLF_OK) *ms_out = median_of(v);
    return rc;
}

int dlf_net_time_span(dlf_net* net, int first, int last, int sm_count, const void* in_dev, void* stream, int warmup,
                      int iters, int prepare, float* ms) {
    if (!net || !in_dev || !ms || first < 0 || last < first || last >= static_cast<int>(net->layers.size()) || warmup < 0 || iters < 1)
        return DLF_E_INVALID_ARG;
    if (!net->ws) return DLF_E_WORKSPACE;
    for (const Layer& l : net->layers)
        if (is_param(l) && (!l.w || !l.bias)) return DLF_E_STATE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void* final_out = net->ws + net->layers.back().off;
    int rc = DLF_OK;
    if (prepare) {   // every layer's slot filled once, so that the span finds its inputs in HBM
        std::vector<Group> saved = net->plan;
        rc = dlf_net_plan_unfused(net);
        if (rc == DLF_OK) rc = dlf_net_run(net, in_dev, final_out, s);
        if (rc == DLF_OK) rc = dlf_net_sync(net, s);
        net->plan = saved;
        invalidate_graphs(net);
        if (rc) return rc;
    }
    if (net->dev_sms == 0) {
        rc = query_sms(&net->dev_sms);
        if (rc) return rc;
    }
    if (sm_count < 1 || sm_count > net->dev_sms) return DLF_E_PLAN;
    Group g;
    if (!make_group(net, first, last, sm_count, &g)) return DLF_E_PLAN;
    rc = kernels_init();
    if (rc) return rc;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return cuda_fail(cudaGetLastError());
    rc = time_group(net, g, in_dev, final_out, s, e0, e1, warmup, iters, ms);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc ? rc : dlf_net_sync(net, s);
}

int dlf_net_bruteforce(dlf_net* net, const dlf_search_params* sp, const void* in_dev, void* stream, int* n_groups,
                       int32_t* group_end, int32_t* sm_count, float* best_ms) {
    if (!net || !sp || !in_dev || !n_groups || !group_end || !sm_count) return DLF_E_INVALID_ARG;
    if (sp->n_sm_choices < 1 || sp->n_sm_choices > 16 || sp->max_group_len < 1 || sp->iters < 1 || sp->warmup < 0) return DLF_E_INVALID_ARG;
    if (!net->ws) return DLF_E_WORKSPACE;
    for (const Layer& l : net->layers)
        if (is_param(l) && (!l.w || !l.bias)) return DLF_E_STATE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int n = static_cast<int>(net->layers.size());
    std::vector<Group> saved = net->plan;
    // fill every layer's slot once so that each candidate group finds its inputs in HBM
    int rc = dlf_net_plan_unfused(net);
    if (rc) { net->plan = saved; invalidate_graphs(net); return rc; }
    void* final_out = net->ws + net->layers.back().off;
    rc = dlf_net_run(net, in_dev, final_out, s);
    if (rc == DLF_OK) rc = dlf_net_sync(net, s);
    net->plan = saved;
    invalidate_graphs(net);   // the graph just built holds the no-fusion plan
    if (rc) return rc;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return cuda_fail(cudaGetLastError());
    const float inf = std::numeric_limits<float>::infinity();
    // t[a][len-1] = best time of span a..a+len-1 over the SM choices
    std::vector<std::vector<float>> t(n, std::vector<float>(sp->max_group_len, inf));
    std::vector<std::vector<int>> ts(n, std::vector<int>(sp->max_group_len, 0));
    for (int a = 0; a < n && rc == DLF_OK; a++)
        for (int len = 1; len <= sp->max_group_len && a + len <= n && rc == DLF_OK; len++)
            for (int c = 0; c < sp->n_sm_choices && rc == DLF_OK; c++) {
                const int S = sp->sm_choices[c];
                if (S < 1 || S > net->dev_sms) continue;
                Group g;
                if (!make_group(net, a, a + len - 1, S, &g)) continue;
                float m = 0.0f;
                rc = time_group(net, g, in_dev, final_out, s, e0, e1, sp->warmup, sp->iters, &m);
                if (rc == DLF_OK && m < t[a][len - 1]) { t[a][len - 1] = m; ts[a][len - 1] = S; }
            }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    rc = solve_partition(n, sp->max_group_len, t, ts, n_groups, group_end, sm_count, best_ms);
    if (rc) return rc;
    return dlf_net_sync(net, s);
}

int dlf_bruteforce_table(int n_layers, int max_group_len, int n_sm_choices, const int32_t* sm_choices, const float* ms, int* n_groups,
                         int32_t* group_end, int32_t* sm_count, float* best_ms) {
    if (n_layers < 1 || max_group_len < 1 || n_sm_choices < 1 || !sm_choices || !ms || !n_groups || !group_end || !sm_count) return DLF_E_INVALID_ARG;
    const float inf = std::numeric_limits<float>::infinity();
    std::vector<std::vector<float>> t(n_layers, std::vector<float>(max_group_len, inf));
    std::vector<std::vector<int>> ts(n_layers, std::vector<int>(max_group_len, 0));
    for (int a = 0; a < n_layers; a++)
        for (int len = 1; len <= max_group_len && a + len <= n_layers; len++)
            for (int c = 0; c < n_sm_choices; c++) {
                const float m = ms[(static_cast<size_t>(a) * max_group_len + (len - 1)) * n_sm_choices + c];
                if (m >= 0.0f && m < t[a][len - 1]) { t[a][len - 1] = m; ts[a][len - 1] = sm_choices[c]; }
            }
    return solve_partition(n_layers, max_group_len, t, ts, n_groups, group_end, sm_count, best_ms);

}

int dlf_net_boundary_tensor(const dlf_net* net, int layer, const void** dev_ptr, int64_t shape[4]) {
    if (!net || !dev_ptr || layer < 0 || layer >= static_cast<int>(net->layers.size())) return DLF_E_INVALID_ARG;
    if (!net->ws) return DLF_E_WORKSPACE;
    bool is_end = false;
    for (const Group& g : net->plan) is_end |= (g.last == layer);
    if (!is_end) return DLF_E_PLAN;
    const Layer& l = net->layers[layer];
    *dev_ptr = (layer == static_cast<int>(net->layers.size()) - 1) ? net->last_out : net->ws + l.off;
    if (shape) std::memcpy(shape, l.out, sizeof(l.out));
    return DLF_OK;
}

int dlf_net_group_model(const dlf_net* net, int group, int64_t* flops, int64_t* hbm_bytes, double* redundancy, int* launches) {
    if (!net || group < 0 || group >= static_cast<int>(net->plan.size())) return DLF_E_INVALID_ARG;
    const Group& g = net->plan[group];
    int64_t fl = 0, by = 0;
    const Layer& f = net->layers[g.first];
    const Layer& z = net->layers[g.last];
    by += f.in[0] * f.in[1] * f.in[2] * f.in[3] * 2;
    by += static_cast<int64_t>(z.bytes);
    for (int i = g.first; i <= g.last; i++) {
        const Layer& l = net->layers[i];
        fl += l.flops;
        by += l.w_elems * 2 + (is_param(l) ? l.d.cout * 4 : 0);
        if (l.d.res_src != -2 && l.d.res_src < g.first) by += l.out[0] * l.ho_pre * l.wo_pre * l.out[3] * 2;
        if (g.kind == K_CONV_DUAL && i > g.first) by += l.in[0] * l.in[1] * l.in[2] * l.in[3] * 2;   // the expansion layer's own input
        // a group handed over through L2 still writes every map to its slot and reads it back: counted like separate layers
        if (g.kind == K_CONV_SEQ) {
            if (i > g.first) by += l.in[0] * l.in[1] * l.in[2] * l.in[3] * 2;
            if (i < g.last) by += static_cast<int64_t>(l.bytes);
            if (l.d.res_src != -2 && l.d.res_src >= g.first) by += l.out[0] * l.ho_pre * l.wo_pre * l.out[3] * 2;
        }
    }
    if (flops) *flops = fl;
    if (hbm_bytes) *hbm_bytes = by;
    if (redundancy) *redundancy = g.kind == K_CHAIN_TC ? g.tiling.redundancy : (g.kind == K_MBCONV ? g.mb_tiling.redundancy : 1.0);
    if (launches) *launches = 1;
    return DLF_OK;
}

const char* dlf_net_group_kernel(const dlf_net* net, int group) {
    if (!net || group < 0 || group >= static_cast<int>(net->plan.size())) return "";
    return kKindName[net->plan[group].kind];
}

int dlf_net_group_launch(dlf_net* net, int group, char* name, size_t name_bytes, int* grid, int* block) {
    if (!net || group < 0 || group >= static_cast<int>(net->plan.size()) || (name && name_bytes == 0)) return DLF_E_INVALID_ARG;
    int rc = check_ready(net);
    if (rc) return rc;
    LaunchRecord rec{nullptr, 0, 0, ""};
    g_launch_record = &rec;
    rc = launch_group(net, net->plan[group], net->ws + net->in_off, net->ws + net->layers.back().off, nullptr);
    g_launch_record = nullptr;
    if (rc) return rc;
    if (grid) *grid = rec.grid;
    if (block) *block = rec.block;
    if (name) {
        const char* mangled = nullptr;
        cudaError_t e = cudaFuncGetName(&mangled, rec.func);
        if (e != cudaSuccess) return cuda_fail(e);
        // "void dlf::(anonymous namespace)::kernel<1, 2>(arguments)" -> "kernel<1, 2>"
        char* full = abi::__cxa_demangle(mangled, nullptr, nullptr, nullptr);
        std::string text = full ? full : mangled;
        std::free(full);
        const std::string anon = "(anonymous namespace)::";
        for (size_t at = text.find(anon); at != std::string::npos; at = text.find(anon)) text.erase(at, anon.size());
        text = text.substr(0, text.find('('));
        const size_t scope = text.substr(0, text.find('<')).rfind("::");
        if (scope != std::string::npos) text = text.substr(scope + 2);
        std::snprintf(name, name_bytes, "%s%s", text.c_str(), rec.note);
    }
    return DLF_OK;
}

int dlf_net_set_option(dlf_net* net, int option, int value) {
    if (!net) return DLF_E_INVALID_ARG;
    switch (option) {
        case DLF_OPT_NO_TENSOR_CORE: net->opt_no_tc = value != 0; break;
        case DLF_OPT_SINGLE_AS_CHAIN: net->opt_single_chain = value != 0; break;
        case DLF_OPT_GROUP_KERNEL:
            if (value < 0 || value > 2) return DLF_E_INVALID_ARG;
            net->opt_group_kernel = value;
            break;
        case DLF_OPT_CUDA_GRAPH: net->opt_graph = value != 0; return DLF_OK;
        case DLF_OPT_PDL: g_use_pdl = value != 0; invalidate_graphs(net); return DLF_OK;
        case DLF_OPT_CONV_ROW_MODE:
            if (value < 0 || value > 2) return DLF_E_INVALID_ARG;
            g_conv_row_mode = value;
            invalidate_graphs(net);
            return DLF_OK;
        default: return DLF_E_INVALID_ARG;
    }
    net->plan.clear();  // kernel choices depend on the options: the plan must be set again
    invalidate_graphs(net);
    return DLF_OK;
}

}  // extern "C"
