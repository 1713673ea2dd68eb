// Fused propagate (Sec. 3 "Message Passing": apply_edges + aggregate_neighbors combined into a
// generalised sparse x dense product) and its backward passes: host side of the segmented reduction
// (reduce_rows.cuh); the edge-wise dot products of the weight gradients are in edge_dots.cu.
#include <mutex>

#include "reduce_params.cuh"

namespace gnn {

bool pick_shape(int nvec, int* lpr, int* vpl) {
    if (nvec < 1 || nvec > 128) return false;
    if (nvec <= 4) { *lpr = 4; *vpl = 1; }
    else if (nvec <= 8) { *lpr = 8; *vpl = 1; }
    else if (nvec <= 16) { *lpr = 16; *vpl = 1; }
    else if (nvec <= 32) { *lpr = 32; *vpl = 1; }
    else if (nvec <= 64) { *lpr = 32; *vpl = 2; }
    else { *lpr = 32; *vpl = 4; }
    return true;
}

// one translation unit per element type and group of modes (reduce_*.cu)
template <typename T> void launch_reduce_sums(const PropParams& P, int mode, bool stream, cudaStream_t st);
template <typename T> void launch_reduce_others(const PropParams& P, int mode, bool stream, cudaStream_t st);
extern template void launch_reduce_sums<float>(const PropParams&, int, bool, cudaStream_t);
extern template void launch_reduce_sums<__nv_bfloat16>(const PropParams&, int, bool, cudaStream_t);
extern template void launch_reduce_others<float>(const PropParams&, int, bool, cudaStream_t);
extern template void launch_reduce_others<__nv_bfloat16>(const PropParams&, int, bool, cudaStream_t);

template <typename T>
static void launch_mode(const PropParams& P, int mode, bool stream, cudaStream_t st) {
    if (mode == MODE_SUM && (P.w || P.gscale_rowptr)) mode = MODE_WSUM;
    if (mode == MODE_HEADSUM && (P.gscale_rowptr || P.epi_l)) mode = P.epi_l ? MODE_HEADRANK : MODE_HEADSUM_W;
    if (mode == MODE_SUM || mode == MODE_WSUM || mode == MODE_HEADSUM || mode == MODE_HEADSUM_W || mode == MODE_HEADRANK) launch_reduce_sums<T>(P, mode, stream, st);
    else launch_reduce_others<T>(P, mode, stream, st);
}

struct ReduceWs {
    int32_t* tail_row;
    float* part_val;
    int32_t* part_arg;
    size_t bytes;
};
static ReduceWs carve(void* ws, int64_t pieces, int F, bool with_arg) {
    ReduceWs w;
    char* p = (char*)ws;
    size_t off = 0;
    w.tail_row = (int32_t*)(p + off); off += up256((size_t)pieces * 4);
    w.part_val = (float*)(p + off); off += up256((size_t)pieces * 2 * F * 4);
    w.part_arg = (int32_t*)(p + off); if (with_arg) off += up256((size_t)pieces * 2 * F * 4);
    w.bytes = off;
    return w;
}


// Positions per warp (see reduce_rows.cuh): a function of the shape alone, so that results are reproducible.
//  - From 2.5 M positions on 256, the most a warp stages.  Below that 256 leaves the machine with one wave of warps and a
//    nearly empty second: rows over 128 bytes then take 128 (1.36 M edges, 512-byte rows: 82 -> 75 us), narrower ones below
//    1 M (557k edges, 128-byte rows: 26 -> 18 us; above, the set-up of twice as many warps costs more than it gives).
//  - Where the mean row spans several pieces (pooling over a few large graphs), 256: every cut is one more partial row.
//  - Small graphs are bound by the longest chain of loads of a warp, so their shares shrink with them (80k edges with hubs,
//    512-byte rows: 15.8 us at 64, 11.8 us at 32; 64-byte rows have eight groups per warp and gain nothing below 64).
static int warp_positions(int32_t N, int64_t E, int row_bytes, bool stream) {
    if (E >= 512 * 1024) return E > 64 * (int64_t)N || E >= 2500 * 1000 || (row_bytes <= 128 && E >= 1000 * 1000) ? 256 : 128;
    if (!stream) return 64;
    // rows over 512 bytes run in slabs: the last one's eight lane groups, if it has 64 bytes or less, need 64 positions to pipeline
    const int narrowest = row_bytes > 512 && row_bytes % 512 != 0 ? row_bytes % 512 : row_bytes;
    return E >= 256 * 1024 ? 128 : E >= 128 * 1024 || narrowest <= 64 ? 64 : 32;
}

// Mean row length from which the reduction looks whether a batch of positions holds a row end at all before it tests each
// (lane groups side by side; a warp-wide row always does).  123 M edges, 51 per row, 128-byte rows: 1.96 -> 1.87 ms; 1.36 M edges, 8
// per row, 256-byte rows, where hardly a batch is without one: 2 % slower.
constexpr int VOTE_DEGREE = 24;

// Room for a partial row per 64, 128 or 1024 positions.  The streaming kernel, whose pieces are 256 to 2048 positions, needs a
// sixteenth to a quarter of that below 4 Mi edges and half above; the size is what callers have been told since the first
// version, and what decides which problems the built-in scratch takes.
size_t chunked_workspace(int64_t E, int F, bool with_arg) {
    if (E <= 0) return carve(nullptr, 1, F, with_arg).bytes;
    const int per = E >= (int64_t)4 * 1024 * 1024 ? 1024 : E >= 512 * 1024 ? 128 : 64;
    return carve(nullptr, ceil_div(E, (int64_t)per), F < 256 ? F : 256, with_arg).bytes;
}

int64_t gatv2_rows_pieces(int32_t N, int64_t E, int row_bytes) {
    return E > 0 ? ceil_div(E, (int64_t)warp_positions(N, E, row_bytes, true) * RR_WARPS) : 1;
}

size_t gatv2_rows_workspace(int32_t N, int64_t E, int F, int row_bytes) { return carve(nullptr, gatv2_rows_pieces(N, E, row_bytes), F, false).bytes; }

template <typename T> void launch_gatv2_rows(const PropParams& P, cudaStream_t st);  // reduce_gatv2.cu
extern template void launch_gatv2_rows<float>(const PropParams&, cudaStream_t);
extern template void launch_gatv2_rows<__nv_bfloat16>(const PropParams&, cudaStream_t);

gnn_status run_gatv2_rows(const char* who, int32_t N, int64_t E, const int64_t* rowptr, const int32_t* col, const int32_t* ds_index, const float* ds, int H,
                          const void* Xself, const void* Xother, const float* a, float slope, int F, gnn_dtype dtype, void* out, float* da_part, void* ws,
                          cudaStream_t st) {
    PropParams P = {};
    const int row_bytes = F * elem_size(dtype);
    P.rowptr = rowptr; P.col = col; P.X = Xother; P.out = out;
    P.N = N; P.E = E; P.nvec = row_bytes / 16; P.x_ld = P.out_ld = (uint32_t)row_bytes; P.F = P.arg_ld = F;
    P.sub = warp_positions(N, E, row_bytes, true);
    P.piece = P.sub * RR_WARPS;
    P.npieces = gatv2_rows_pieces(N, E, row_bytes);
    const ReduceWs w = carve(ws, P.npieces, F, false);
    P.tail_row = w.tail_row; P.part_val = w.part_val;
    P.wh = ds; P.wh_index = ds_index; P.H = H; P.fph = F / H; P.epi_a = a;
    P.vote = E > VOTE_DEGREE * (int64_t)N;
    P.v2_self = Xself; P.slope = slope; P.da_part = da_part;
    if (dtype == GNN_F32) launch_gatv2_rows<float>(P, st);
    else launch_gatv2_rows<__nv_bfloat16>(P, st);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

gnn_status run_chunked(const char* who, int mode, int32_t N, int64_t E, const int64_t* rowptr,
                       const int32_t* col, const float* w, const void* X, void* out,
                       int32_t* argmax, const int64_t* gscale_rowptr, const int32_t* route_arg,
                       const int32_t* route_pos, int mean, int F, gnn_dtype dtype, void* ws,
                       size_t ws_bytes, cudaStream_t st, const HeadExtra* hx, const RowExtra* rx) {
    const int s = elem_size(dtype), epc = 16 / s;
    GNN_REQUIRE(F > 0 && ((size_t)F * s) % 16 == 0, GNN_ERR_UNSUPPORTED,
                "%s: F*sizeof(element) = %d must be a multiple of 16 bytes", who, F * s);
    const int nvec = F * s / 16;
    GNN_REQUIRE(nvec <= 128, GNN_ERR_UNSUPPORTED, "%s: feature rows wider than 2048 bytes are not supported (F=%d)", who, F);
    GNN_REQUIRE(aligned16(X) && aligned16(out), GNN_ERR_INVALID_ARG, "%s: feature matrices must be 16-byte aligned", who);
    GNN_REQUIRE(E >= 0 && E < ((int64_t)1 << 31) - 1024, GNN_ERR_UNSUPPORTED, "%s: positions must fit 32 bits (E < 2^31)", who);
    const bool with_arg = (mode == MODE_MAX || mode == MODE_MIN);
    const size_t need = chunked_workspace(E, F, with_arg);
    GNN_REQUIRE(ws && ws_bytes >= need && aligned16(ws), GNN_ERR_WORKSPACE_TOO_SMALL,
                "%s: workspace of %zu bytes (16-byte aligned) needed, %zu given", who, need, ws_bytes);
    if (N == 0) return GNN_OK;
    PropParams P;
    P.rowptr = rowptr; P.col = col; P.w = w; P.argmax = argmax;
    P.gscale_rowptr = gscale_rowptr; P.route_arg = route_arg; P.route_pos = route_pos;
    P.N = N; P.E = E; P.mean = mean; P.arg_ld = F;
    P.vote = E > VOTE_DEGREE * (int64_t)N;
    P.v2_self = nullptr; P.slope = 0.f; P.da_part = nullptr;
    P.wh = nullptr; P.wh_index = nullptr; P.H = 1; P.fph = F; P.epi_l = P.epi_r = P.epi_a = P.epi_b = nullptr;
    if (hx) {
        GNN_REQUIRE(mode == MODE_HEADSUM && (hx->wh || E == 0) && hx->H >= 1 && F % hx->H == 0 && (F / hx->H) % epc == 0, GNN_ERR_UNSUPPORTED,
                    "%s: per-head weights need F divisible by H and F/H a multiple of %d elements", who, epc);
        P.wh = hx->wh; P.wh_index = hx->wh_index; P.H = hx->H; P.fph = F / hx->H;
        P.epi_l = hx->epi_l; P.epi_r = hx->epi_r; P.epi_a = hx->epi_a; P.epi_b = hx->epi_b;
    } else {
        GNN_REQUIRE(mode != MODE_HEADSUM, GNN_ERR_INVALID_ARG, "%s: per-head mode without weights", who);
    }
    P.x_ld = P.out_ld = P.self_ld = (uint32_t)nvec * 16;
    P.ef = nullptr; P.ef_ld = 0; P.has_epi = 0; P.agg_c = 1.0f; P.self_c = 0.f; P.self_mode = GNN_SELF_ALWAYS; P.relu = 0;
    P.self_X = nullptr; P.self_rowptr = rowptr; P.bias = nullptr; P.descending = 0;
    if (rx) {
        GNN_REQUIRE(mode == MODE_EFSUM ? (rx->ef != nullptr || E == 0) : rx->ef == nullptr, GNN_ERR_INVALID_ARG,
                    "%s: per-feature multipliers and mode disagree", who);
        GNN_REQUIRE(!rx->ef || (rx->ef_ld >= F && rx->ef_ld % 4 == 0 && aligned16(rx->ef)), GNN_ERR_INVALID_ARG,
                    "%s: per-feature multipliers must be 16-byte aligned rows of at least F floats", who);
        GNN_REQUIRE(!rx->self_X || aligned16(rx->self_X), GNN_ERR_INVALID_ARG, "%s: the self-term matrix must be 16-byte aligned", who);
        GNN_REQUIRE(rx->self_mode >= GNN_SELF_ALWAYS && rx->self_mode <= GNN_SELF_IF_NONEMPTY, GNN_ERR_INVALID_ARG, "%s: bad self mode", who);
        P.ef_ld = rx->ef_ld;
        P.agg_c = rx->agg_c; P.self_c = rx->self_c; P.self_mode = rx->self_mode;
        if (rx->self_rowptr) P.self_rowptr = rx->self_rowptr;
        P.relu = rx->relu;
        P.descending = rx->descending;
        P.has_epi = (rx->agg_c != 1.0f || rx->self_X || rx->bias || rx->relu) ? 1 : 0;
    } else {
        GNN_REQUIRE(mode != MODE_EFSUM, GNN_ERR_INVALID_ARG, "%s: per-feature mode without multipliers", who);
    }
    // Rows over 512 bytes run one 512-byte column slab at a time: every pass re-reads the index stream but gathers from a
    // narrower matrix, of which more rows stay in L2 (2048-byte fp32 rows on 123 M edges: 141 -> 77 GB of DRAM traffic).
    const int slab_vec = nvec < 32 ? nvec : 32, slab_f = slab_vec * epc;
    // Graphs of up to 128 Ki edges and a handful per row are bound by latency and take a row per lane group (13k nodes,
    // 69k edges, 512-byte rows: 8.7 us against 11.6 us positions first); higher mean degrees say that long rows carry the
    // edges (10k nodes, 80k edges with hubs: 13.4 against 11.8 us).
    // The routing mode fetches two rows per position and has fewer in flight per lane: always positions first (17 / 14 us).
    const bool stream = E >= 128 * 1024 || E > 6 * (int64_t)N || (mode == MODE_ROUTE && E > 0);
    P.sub = warp_positions(N, E, nvec * 16, stream);
    P.piece = stream ? P.sub * RR_WARPS : P.sub;
    P.npieces = E > 0 ? ceil_div(E, (int64_t)P.piece) : 1;
    const ReduceWs wsv = carve(ws, P.npieces, slab_f, with_arg);
    GNN_REQUIRE(wsv.bytes <= ws_bytes, GNN_ERR_WORKSPACE_TOO_SMALL, "%s: partial rows of %zu bytes exceed the workspace", who, wsv.bytes);
    P.tail_row = wsv.tail_row; P.part_val = wsv.part_val; P.part_arg = wsv.part_arg;
    for (int v0 = 0; v0 < nvec; v0 += 32) {
        P.vec0 = v0;
        P.nvec = nvec - v0 < 32 ? nvec - v0 : 32;
        P.F = P.nvec * epc;
        P.X = (const char*)X + (size_t)v0 * 16;
        P.out = (char*)out + (size_t)v0 * 16;
        P.argmax = argmax ? argmax + v0 * epc : nullptr;
        P.route_arg = route_arg ? route_arg + v0 * epc : nullptr;
        if (rx) {
            P.ef = rx->ef ? rx->ef + v0 * epc : nullptr;
            P.self_X = rx->self_X ? (const char*)rx->self_X + (size_t)v0 * 16 : nullptr;
            P.bias = rx->bias ? rx->bias + v0 * epc : nullptr;
        }
        if (dtype == GNN_F32) launch_mode<float>(P, mode, stream, st);
        else launch_mode<__nv_bfloat16>(P, mode, stream, st);
    }
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

// ------------------------------------------------------------------ built-in scratch
// Scratch for gnn_propagate_fused_static: lives in the library image, so every GPU that loads the
// library carries these bytes until the process exits.  Host code must not hand this name to a
// kernel: on the host it is only a handle for cudaGetSymbolAddress.
constexpr size_t STATIC_WS_BYTES = (size_t)8 << 20;  // 8 MiB
static __device__ __align__(256) unsigned char g_static_ws[STATIC_WS_BYTES];

constexpr int STATIC_MAX_DEVICES = 64;
static void* g_static_ws_addr[STATIC_MAX_DEVICES];  // device address of g_static_ws, per device ordinal
static std::mutex g_static_ws_mutex;

// device address of the built-in scratch on the current device (looked up once per device)
static gnn_status static_ws_address(const char* who, void** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: cudaGetDevice: %s", who, cudaGetErrorString(e));
    GNN_REQUIRE(dev >= 0 && dev < STATIC_MAX_DEVICES, GNN_ERR_UNSUPPORTED, "%s: device ordinal %d not supported", who, dev);
    std::lock_guard<std::mutex> lock(g_static_ws_mutex);
    if (!g_static_ws_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_ws);
        if (e != cudaSuccess || !p)
            GNN_FAIL(GNN_ERR_CUDA, "%s: cudaGetSymbolAddress failed: %s", who, cudaGetErrorString(e));
        g_static_ws_addr[dev] = p;
    }
    *out = g_static_ws_addr[dev];
    return GNN_OK;
}

}  // namespace gnn

using namespace gnn;

extern "C" {

size_t gnn_propagate_fused_workspace(int64_t E, int F, gnn_op op) {
    if (E < 0 || F <= 0) return 0;
    // MAX/MIN keep winner positions beside the partial values; their backward needs values
    // only, so the forward size always suffices for the backward call
    return chunked_workspace(E, F, op == GNN_MAX || op == GNN_MIN);
}

gnn_status gnn_propagate_fused(const gnn_csr* g, gnn_msg msg, gnn_op op, const void* X,
                               const float* w_csr, int F, gnn_dtype dtype, void* out,
                               int32_t* argmax, void* ws, size_t ws_bytes, gnn_stream stream) {
    GNN_REQUIRE(g && g->rowptr && X && out, GNN_ERR_INVALID_ARG, "gnn_propagate_fused: null argument");
    GNN_REQUIRE(g->E == 0 || g->col, GNN_ERR_INVALID_ARG, "gnn_propagate_fused: null col");
    GNN_REQUIRE(msg == GNN_MSG_COPY_XJ || msg == GNN_MSG_E_MUL_XJ, GNN_ERR_UNSUPPORTED,
                "gnn_propagate_fused: message must be COPY_XJ or E_MUL_XJ");
    GNN_REQUIRE(msg == GNN_MSG_COPY_XJ || w_csr, GNN_ERR_INVALID_ARG, "gnn_propagate_fused: E_MUL_XJ needs w_csr");
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "gnn_propagate_fused: bad dtype");
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "gnn_propagate_fused: bad op");
    GNN_REQUIRE(!argmax || aligned16(argmax), GNN_ERR_INVALID_ARG, "gnn_propagate_fused: argmax must be 16-byte aligned");
    const float* w = (msg == GNN_MSG_E_MUL_XJ) ? w_csr : nullptr;
    const int mode = op == GNN_MAX ? MODE_MAX : op == GNN_MIN ? MODE_MIN : MODE_SUM;
    return run_chunked("gnn_propagate_fused", mode, g->N, g->E, g->rowptr, g->col, w, X, out,
                       argmax, nullptr, nullptr, nullptr, op == GNN_MEAN, F, dtype, ws, ws_bytes,
                       as_stream(stream));
}

gnn_status gnn_propagate_fused_backward(const gnn_csr* g, gnn_msg msg, gnn_op op,
                                        const void* dOut, const void* X, const float* w_csrT,
                                        const int32_t* argmax, int F, gnn_dtype dtype, void* dX,
                                        float* dW, void* ws, size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_propagate_fused_backward";
    GNN_REQUIRE(g && g->rowptr && g->rowptrT && dOut, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(g->E == 0 || (g->col && g->colT), GNN_ERR_INVALID_ARG, "%s: null col", who);
    GNN_REQUIRE(msg == GNN_MSG_COPY_XJ || msg == GNN_MSG_E_MUL_XJ, GNN_ERR_UNSUPPORTED,
                "%s: message must be COPY_XJ or E_MUL_XJ", who);
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "%s: bad op", who);
    const bool mm = (op == GNN_MAX || op == GNN_MIN);
    cudaStream_t st = as_stream(stream);
    if (dX) {
        GNN_REQUIRE(msg == GNN_MSG_COPY_XJ || w_csrT, GNN_ERR_INVALID_ARG, "%s: E_MUL_XJ needs w_csrT for dX", who);
        const float* w = (msg == GNN_MSG_E_MUL_XJ) ? w_csrT : nullptr;
        gnn_status rc;
        if (mm) {
            GNN_REQUIRE(argmax && (g->E == 0 || g->t2f) && aligned16(argmax), GNN_ERR_INVALID_ARG,
                        "%s: MAX/MIN need the forward argmax (16-byte aligned) and t2f", who);
            rc = run_chunked(who, MODE_ROUTE, g->N, g->E, g->rowptrT, g->colT, w, dOut, dX, nullptr,
                             nullptr, argmax, g->t2f, 0, F, dtype, ws, ws_bytes, st);
        } else {
            rc = run_chunked(who, MODE_SUM, g->N, g->E, g->rowptrT, g->colT, w, dOut, dX, nullptr,
                             op == GNN_MEAN ? g->rowptr : nullptr, nullptr, nullptr, 0, F, dtype, ws,
                             ws_bytes, st);
        }
        if (rc != GNN_OK) return rc;
    }
    if (dW) {
        GNN_REQUIRE(!mm, GNN_ERR_UNSUPPORTED, "%s: dW is defined for SUM/MEAN only", who);
        GNN_REQUIRE(X, GNN_ERR_INVALID_ARG, "%s: dW needs X", who);
        gnn_status rc = run_sddmm(who, g, X, dOut, 1, F, op == GNN_MEAN, dtype, dW, st);
        if (rc != GNN_OK) return rc;
    }
    return GNN_OK;
}

static gnn_status copy_async(const char* who, void* dst, const void* src, size_t bytes,
                             cudaMemcpyKind kind, cudaStream_t st) {
    if (bytes == 0) return GNN_OK;
    cudaError_t e = cudaMemcpyAsync(dst, src, bytes, kind, st);
    if (e != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: copy failed: %s", who, cudaGetErrorString(e));
    return GNN_OK;
}

gnn_status gnn_propagate_fused_host(const gnn_csr* g, gnn_msg msg, gnn_op op, const void* h_X,
                                    const float* w_csr, int F, gnn_dtype dtype, void* h_out,
                                    int32_t* argmax, void* d_in, void* d_out, void* ws,
                                    size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_propagate_fused_host";
    GNN_REQUIRE(g && h_X && h_out && d_in && d_out, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(F > 0 && (dtype == GNN_F32 || dtype == GNN_BF16), GNN_ERR_INVALID_ARG, "%s: bad F or dtype", who);
    const size_t bytes = (size_t)g->N * F * elem_size(dtype);
    cudaStream_t st = as_stream(stream);
    gnn_status rc = copy_async(who, d_in, h_X, bytes, cudaMemcpyHostToDevice, st);
    if (rc != GNN_OK) return rc;
    rc = gnn_propagate_fused(g, msg, op, d_in, w_csr, F, dtype, d_out, argmax, ws, ws_bytes, stream);
    if (rc != GNN_OK) return rc;
    return copy_async(who, h_out, d_out, bytes, cudaMemcpyDeviceToHost, st);
}

gnn_status gnn_propagate_fused_backward_host(const gnn_csr* g, gnn_msg msg, gnn_op op,
                                             const void* h_dOut, const float* w_csrT,
                                             const int32_t* argmax, int F, gnn_dtype dtype,
                                             void* h_dX, void* d_in, void* d_out, void* ws,
                                             size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_propagate_fused_backward_host";
    GNN_REQUIRE(g && h_dOut && h_dX && d_in && d_out, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(F > 0 && (dtype == GNN_F32 || dtype == GNN_BF16), GNN_ERR_INVALID_ARG, "%s: bad F or dtype", who);
    const size_t bytes = (size_t)g->N * F * elem_size(dtype);
    cudaStream_t st = as_stream(stream);
    gnn_status rc = copy_async(who, d_in, h_dOut, bytes, cudaMemcpyHostToDevice, st);
    if (rc != GNN_OK) return rc;
    rc = gnn_propagate_fused_backward(g, msg, op, d_in, nullptr, w_csrT, argmax, F, dtype, d_out, nullptr, ws, ws_bytes, stream);
    if (rc != GNN_OK) return rc;
    return copy_async(who, h_dX, d_out, bytes, cudaMemcpyDeviceToHost, st);
}

size_t gnn_propagate_fused_static_max_bytes(void) { return STATIC_WS_BYTES; }

gnn_status gnn_propagate_fused_static(const gnn_csr* g, gnn_msg msg, gnn_op op, const void* X,
                                      const float* w_csr, int F, gnn_dtype dtype, void* out,
                                      int32_t* argmax, gnn_stream stream) {
    const char* who = "gnn_propagate_fused_static";
    GNN_REQUIRE(g && F > 0, GNN_ERR_INVALID_ARG, "%s: null graph or bad F", who);
    const size_t need = gnn_propagate_fused_workspace(g->E, F, op);
    GNN_REQUIRE(need <= STATIC_WS_BYTES, GNN_ERR_WORKSPACE_TOO_SMALL,
                "%s: E=%lld, F=%d needs %zu bytes of scratch; the built-in scratch holds %zu. "
                "Use gnn_propagate_fused with a caller-provided workspace", who, (long long)g->E, F, need, STATIC_WS_BYTES);
    void* ws = nullptr;
    gnn_status rc = static_ws_address(who, &ws);
    if (rc != GNN_OK) return rc;
    return gnn_propagate_fused(g, msg, op, X, w_csr, F, dtype, out, argmax, ws, STATIC_WS_BYTES, stream);
}

}  // extern "C"
