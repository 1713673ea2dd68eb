// Further fused (message, op) pairs of propagate (Sec. 3 "Message Passing": "specific message
// functions and aggregation operations"), the GIN aggregation and the row epilogue of the conv layers
// (Sec. 3 "Graph Convolutional Layers"), the XI_DOT_XJ message, and the set-up calls that turn a
// heterogeneous graph or a sequence of temporal snapshots (Sec. 3 "Graph Data Structures") into one
// sparse form.  Every reduction here runs through the chunked segmented reduction of propagate.cu:
// this file holds the host dispatch and the small element-wise kernels around it.
#include "propagate.cuh"

namespace gnn {


// ------------------------------------------------------------------ element-wise kernels
// out[i, chunk] = c(i) * D[i, chunk], c(i) = row length (times_degree) or [row length > 0]
template <typename T>
__global__ void row_scale_kernel(const int64_t* rowptr, int32_t N, int nvec, int times_degree,
                                 const uint4* D, uint4* __restrict__ out) {
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, total = (int64_t)N * nvec;
    for (; t < total; t += stride) {
        const int64_t i = t / nvec;
        const int64_t d = rowptr[i + 1] - rowptr[i];
        const float c = times_degree ? (float)d : (d > 0 ? 1.f : 0.f);
        float x[EPC];
        Chunk<T>::unpack(D[t], x);
#pragma unroll
        for (int j = 0; j < EPC; ++j) x[j] *= c;
        out[t] = Chunk<T>::pack(x);
    }
}

// de[p, f] = scale(i) * X[col[p], f] * D[i, f] for p in row i: the gradient of element-wise edge factors
template <typename T>
__global__ void edge_factor_grad_kernel(const int64_t* rowptr, const int32_t* col, int32_t N,
                                        int64_t E, int nvec, int mean, const uint4* X,
                                        const uint4* D, float* __restrict__ de) {
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, total = E * nvec;
    for (; t < total; t += stride) {
        const int64_t p = t / nvec;
        const int ci = (int)(t - p * nvec);
        const int i = lower_bound_i64(rowptr, N + 1, p + 1) - 1;
        const float sc = mean ? 1.0f / (float)(rowptr[i + 1] - rowptr[i]) : 1.0f;
        float x[EPC], d[EPC];
        Chunk<T>::unpack(X[(size_t)col[p] * nvec + ci], x);
        Chunk<T>::unpack(D[(size_t)i * nvec + ci], d);
        float4* o = reinterpret_cast<float4*>(de + (size_t)t * EPC);
#pragma unroll
        for (int j = 0; j < EPC; j += 4)
            o[j / 4] = make_float4(sc * (x[j] * d[j]), sc * (x[j + 1] * d[j + 1]), sc * (x[j + 2] * d[j + 2]), sc * (x[j + 3] * d[j + 3]));
    }
}

// <a, b> over n 16-byte chunks in a fixed order: every thread sums its grid-stride share, the block
// combines its threads by a shuffle / shared-memory tree, and a second launch adds the block results
constexpr int DOT_THREADS = 256, DOT_MAX_BLOCKS = 1184;
template <typename T>
__global__ void __launch_bounds__(DOT_THREADS) dot_partial_kernel(const uint4* a, const uint4* b,
                                                                  int64_t nvec, float* __restrict__ partial) {
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    __shared__ float s_w[DOT_THREADS / 32];
    float acc = 0.f;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nvec; t += stride) {
        float x[EPC], y[EPC];
        Chunk<T>::unpack(a[t], x);
        Chunk<T>::unpack(b[t], y);
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < EPC; ++j) s = fmaf(x[j], y[j], s);
        acc += s;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < DOT_THREADS / 32; ++w) s += s_w[w];
        partial[blockIdx.x] = s;
    }
}
// the partials' sum in a fixed order: a lane takes every 32nd, the lanes are added by an xor tree
__global__ void dot_final_kernel(const float* partial, int nb, float* __restrict__ out) {
    pdl_wait();
    float s = 0.f;
#pragma unroll 4
    for (int b = threadIdx.x; b < nb; b += 32) s += partial[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *out = s;
}

// dZ = dY where (!relu or Y > 0) else 0, and per-block column sums of dZ.  A block owns a contiguous
// range of rows; its threads form row groups of nvec threads (one 16-byte chunk each).
constexpr int EB_THREADS = 256, EB_MAX_BLOCKS = 592;
template <typename T>
__global__ void __launch_bounds__(EB_THREADS) epilogue_backward_kernel(const uint4* Y, const uint4* dY,
                                                                      int32_t N, int nvec, int relu, uint4* __restrict__ dZ,
                                                                      float* __restrict__ partial, int rows_per_block) {
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    extern __shared__ float s_acc[];  // [groups][nvec * EPC]
    const int groups = EB_THREADS / nvec;
    const int grp = threadIdx.x / nvec, ci = threadIdx.x % nvec;
    const bool active = grp < groups;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
    const int64_t r1 = r0 + rows_per_block < N ? r0 + rows_per_block : N;
    float acc[EPC];
#pragma unroll
    for (int j = 0; j < EPC; ++j) acc[j] = 0.f;
    if (active) {
        constexpr int U = 4;  // rows whose loads are in flight together
        for (int64_t r = r0 + grp; r < r1; r += U * groups) {
            uint4 dr[U], yr[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r + u * groups < r1) {
                    dr[u] = dY[(size_t)(r + u * groups) * nvec + ci];
                    if (relu) yr[u] = Y[(size_t)(r + u * groups) * nvec + ci];
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (r + u * groups >= r1) break;
                float d[EPC];
                Chunk<T>::unpack(dr[u], d);
                if (relu) {
                    float y[EPC];
                    Chunk<T>::unpack(yr[u], y);
#pragma unroll
                    for (int j = 0; j < EPC; ++j) d[j] = y[j] > 0.f ? d[j] : 0.f;
                }
                if (dZ) dZ[(size_t)(r + u * groups) * nvec + ci] = Chunk<T>::pack(d);
#pragma unroll
                for (int j = 0; j < EPC; ++j) acc[j] += d[j];
            }
        }
    }
    if (!partial) return;
    if (active) {
#pragma unroll
        for (int j = 0; j < EPC; ++j) s_acc[(size_t)grp * nvec * EPC + ci * EPC + j] = acc[j];
    }
    __syncthreads();
    if (grp == 0) {
#pragma unroll
        for (int j = 0; j < EPC; ++j) {
            float s = 0.f;
            for (int q = 0; q < groups; ++q) s += s_acc[(size_t)q * nvec * EPC + ci * EPC + j];
            partial[(size_t)blockIdx.x * nvec * EPC + ci * EPC + j] = s;
        }
    }
}
// out[f] = sum of the nb partials of column f: 8 walkers per column take every eighth partial, four loads in flight each, and
// are added in walker order (one thread per column walking them all took 14 us for 400 partials)
constexpr int CS_WALKERS = 8;
__global__ void __launch_bounds__(32 * CS_WALKERS) column_sum_final_kernel(const float* partial, int nb, int F, float* __restrict__ out) {
    pdl_wait();
    __shared__ float sums[CS_WALKERS][32];
    const int col = threadIdx.x & 31, w = threadIdx.x >> 5, f = blockIdx.x * 32 + col;
    float s = 0.f;
    if (f < F)
#pragma unroll 4
        for (int b = w; b < nb; b += CS_WALKERS) s += partial[(size_t)b * F + f];
    sums[w][col] = s;
    __syncthreads();
    if (w == 0 && f < F) {
#pragma unroll
        for (int k = 1; k < CS_WALKERS; ++k) s += sums[k][col];
        out[f] = s;
    }
}

// merged edge list of one segment: ids shifted by the segment's offsets
__global__ void merge_segment_kernel(const int32_t* src, const int32_t* dst, int64_t E,
                                     int32_t so, int32_t dof, int32_t seg, int32_t* __restrict__ src_out,
                                     int32_t* __restrict__ dst_out, int32_t* __restrict__ seg_out) {
    pdl_wait();
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; t < E; t += stride) {
        src_out[t] = src[t] + so;
        dst_out[t] = dst[t] + dof;
        if (seg_out) seg_out[t] = seg;
    }
}

// coef[p] = w[p] / max(1, number of positions of p's row in p's segment) for mean segments, else w[p].
// Inside a row the segments are contiguous and ascending, so the count comes from two binary searches.
__global__ void segment_coef_kernel(const int64_t* rowptr, int32_t N, int64_t E, const int32_t* seg,
                                    const float* w, const int32_t* seg_is_mean, int S,
                                    float* __restrict__ coef, int* __restrict__ flag) {
    pdl_wait();
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; p < E; p += stride) {
        const int sg = seg[p];
        float c = w ? w[p] : 1.0f;
        if (sg < 0 || sg >= S) {
            *flag = 1;
        } else if (seg_is_mean[sg]) {
            const int i = lower_bound_i64(rowptr, N + 1, p + 1) - 1;
            int64_t lo = rowptr[i], hi = p;  // first position of the row with segment >= sg
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (seg[mid] < sg) lo = mid + 1; else hi = mid;
            }
            const int64_t first = lo;
            lo = p + 1; hi = rowptr[i + 1];  // first position after p with a larger segment
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (seg[mid] <= sg) lo = mid + 1; else hi = mid;
            }
            c = c / (float)(lo - first);
        }
        coef[p] = c;
    }
}

static int mode_of(gnn_op op) { return op == GNN_MAX ? MODE_MAX : op == GNN_MIN ? MODE_MIN : MODE_SUM; }

static gnn_status check_msg_args(const char* who, const gnn_csr* g, gnn_msg msg, gnn_op op, int e_width, int F,
                                 gnn_dtype dtype) {
    GNN_REQUIRE(g && g->rowptr, GNN_ERR_INVALID_ARG, "%s: null graph", who);
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "%s: bad op", who);
    GNN_REQUIRE(msg == GNN_MSG_COPY_XJ || msg == GNN_MSG_E_MUL_XJ || msg == GNN_MSG_XI_SUB_XJ, GNN_ERR_UNSUPPORTED,
                "%s: message must be COPY_XJ, E_MUL_XJ or XI_SUB_XJ", who);
    GNN_REQUIRE(F > 0, GNN_ERR_INVALID_ARG, "%s: bad F", who);
    if (msg == GNN_MSG_E_MUL_XJ) {
        GNN_REQUIRE(e_width >= 1 && F % e_width == 0, GNN_ERR_INVALID_ARG, "%s: e_width must be 1, a divisor H of F, or F", who);
        GNN_REQUIRE(e_width == 1 || op == GNN_SUM || op == GNN_MEAN, GNN_ERR_UNSUPPORTED,
                    "%s: edge factors wider than 1 take SUM or MEAN only", who);
    }
    return GNN_OK;
}

}  // namespace gnn

using namespace gnn;

extern "C" {

gnn_status gnn_propagate_msg(const gnn_csr* g, gnn_msg msg, gnn_op op, const void* Xj, const void* Xi,
                             const float* e_csr, int e_width, int F, gnn_dtype dtype,
                             const gnn_row_epilogue* epi, void* out, int32_t* argmax, void* ws,
                             size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_propagate_msg";
    gnn_status rc = check_msg_args(who, g, msg, op, e_width, F, dtype);
    if (rc != GNN_OK) return rc;
    GNN_REQUIRE(Xj && out, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(g->E == 0 || g->col, GNN_ERR_INVALID_ARG, "%s: null col", who);
    GNN_REQUIRE(!argmax || aligned16(argmax), GNN_ERR_INVALID_ARG, "%s: argmax must be 16-byte aligned", who);
    RowExtra rx = {nullptr, 0, 1.0f, nullptr, 0.f, GNN_SELF_ALWAYS, g->rowptr, nullptr, 0};
    if (epi) {
        rx.self_X = epi->Xself; rx.self_c = epi->self_coef; rx.self_mode = epi->self_mode;
        rx.bias = epi->bias; rx.relu = epi->relu;
    }
    int mode = mode_of(op);
    const float* w = nullptr;
    HeadExtra hx = {nullptr, nullptr, 1, nullptr, nullptr, nullptr, nullptr};
    const HeadExtra* hxp = nullptr;
    if (msg == GNN_MSG_E_MUL_XJ) {
        GNN_REQUIRE(e_csr || g->E == 0, GNN_ERR_INVALID_ARG, "%s: E_MUL_XJ needs e_csr", who);
        if (e_width == 1) {
            w = e_csr;
        } else if (e_width == F) {
            mode = MODE_EFSUM; rx.ef = e_csr; rx.ef_ld = F;
        } else {
            mode = MODE_HEADSUM; hx.wh = e_csr; hx.H = e_width; hxp = &hx;
        }
    } else if (msg == GNN_MSG_XI_SUB_XJ) {
        GNN_REQUIRE(Xi, GNN_ERR_INVALID_ARG, "%s: XI_SUB_XJ needs Xi", who);
        GNN_REQUIRE(!rx.self_X, GNN_ERR_UNSUPPORTED, "%s: XI_SUB_XJ uses the self term itself; epi->Xself must be NULL", who);
        // sum_p (x_i - x_j) = deg * x_i - sum x_j; max_p (x_i - x_j) = x_i - min_j x_j (and the reverse)
        rx.agg_c = -1.0f; rx.self_X = Xi; rx.self_c = 1.0f;
        rx.self_mode = op == GNN_SUM ? GNN_SELF_TIMES_DEGREE : GNN_SELF_IF_NONEMPTY;
        if (op == GNN_MAX) mode = MODE_MIN;
        else if (op == GNN_MIN) mode = MODE_MAX;
    }
    return run_chunked(who, mode, g->N, g->E, g->rowptr, g->col, w, Xj, out, argmax, nullptr, nullptr, nullptr,
                       op == GNN_MEAN, F, dtype, ws, ws_bytes, as_stream(stream), hxp, &rx);
}

gnn_status gnn_propagate_msg_backward(const gnn_csr* g, gnn_msg msg, gnn_op op, const void* dOut,
                                      const void* Xj, const float* e_csrT, int e_width,
                                      const int32_t* argmax, int F, gnn_dtype dtype,
                                      const gnn_row_epilogue* self_grad, void* dXj, void* dXi,
                                      float* de_csr, void* ws, size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_propagate_msg_backward";
    gnn_status rc = check_msg_args(who, g, msg, op, e_width, F, dtype);
    if (rc != GNN_OK) return rc;
    GNN_REQUIRE(dOut && g->rowptrT, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(g->E == 0 || (g->col && g->colT), GNN_ERR_INVALID_ARG, "%s: null col", who);
    const bool mm = op == GNN_MAX || op == GNN_MIN;
    const int s = elem_size(dtype);
    GNN_REQUIRE(((size_t)F * s) % 16 == 0, GNN_ERR_UNSUPPORTED, "%s: F*sizeof(element) must be a multiple of 16 bytes", who);
    const int nvec = F * s / 16;
    cudaStream_t st = as_stream(stream);
    if (dXj) {
        RowExtra rx = {nullptr, 0, msg == GNN_MSG_XI_SUB_XJ ? -1.0f : 1.0f, nullptr, 0.f, GNN_SELF_ALWAYS, g->rowptr, nullptr, 0};
        if (self_grad) {
            GNN_REQUIRE(!self_grad->bias && !self_grad->relu, GNN_ERR_INVALID_ARG, "%s: self_grad takes a self term only", who);
            rx.self_X = self_grad->Xself; rx.self_c = self_grad->self_coef; rx.self_mode = self_grad->self_mode;
        }
        int mode = MODE_SUM;
        const float* w = nullptr;
        HeadExtra hx = {nullptr, nullptr, 1, nullptr, nullptr, nullptr, nullptr};
        const HeadExtra* hxp = nullptr;
        if (msg == GNN_MSG_E_MUL_XJ) {
            GNN_REQUIRE(e_csrT || g->E == 0, GNN_ERR_INVALID_ARG, "%s: E_MUL_XJ needs e_csrT for dXj", who);
            if (e_width == 1) w = e_csrT;
            else if (e_width == F) { mode = MODE_EFSUM; rx.ef = e_csrT; rx.ef_ld = F; }
            else { mode = MODE_HEADSUM; hx.wh = e_csrT; hx.H = e_width; hxp = &hx; }
        }
        if (mm) {
            GNN_REQUIRE(argmax && (g->E == 0 || g->t2f) && aligned16(argmax), GNN_ERR_INVALID_ARG,
                        "%s: MAX/MIN need the forward argmax (16-byte aligned) and t2f", who);
            rc = run_chunked(who, MODE_ROUTE, g->N, g->E, g->rowptrT, g->colT, w, dOut, dXj, nullptr, nullptr, argmax,
                             g->t2f, 0, F, dtype, ws, ws_bytes, st, nullptr, &rx);
        } else {
            rc = run_chunked(who, mode, g->N, g->E, g->rowptrT, g->colT, w, dOut, dXj, nullptr,
                             op == GNN_MEAN ? g->rowptr : nullptr, nullptr, nullptr, 0, F, dtype, ws, ws_bytes, st, hxp, &rx);
        }
        if (rc != GNN_OK) return rc;
    }
    if (dXi) {
        GNN_REQUIRE(msg == GNN_MSG_XI_SUB_XJ, GNN_ERR_INVALID_ARG, "%s: dXi exists for XI_SUB_XJ only", who);
        GNN_REQUIRE(aligned16(dOut) && aligned16(dXi), GNN_ERR_INVALID_ARG, "%s: misaligned matrix", who);
        if (g->N > 0) {
            const int grid = grid_for((int64_t)g->N * nvec, 256);
            if (dtype == GNN_F32) launch_overlapped(row_scale_kernel<float>, dim3((unsigned)(grid)), dim3(256), 0, st, g->rowptr, g->N, nvec, op == GNN_SUM, (const uint4*)dOut, (uint4*)dXi);
            else launch_overlapped(row_scale_kernel<__nv_bfloat16>, dim3((unsigned)(grid)), dim3(256), 0, st, g->rowptr, g->N, nvec, op == GNN_SUM, (const uint4*)dOut, (uint4*)dXi);
            GNN_CHECK_LAUNCH(who);
        }
    }
    if (de_csr) {
        GNN_REQUIRE(msg == GNN_MSG_E_MUL_XJ && !mm, GNN_ERR_UNSUPPORTED, "%s: de is defined for E_MUL_XJ with SUM/MEAN only", who);
        GNN_REQUIRE(Xj, GNN_ERR_INVALID_ARG, "%s: de needs Xj", who);
        if (e_width == F) {
            GNN_REQUIRE(aligned16(Xj) && aligned16(dOut) && aligned16(de_csr), GNN_ERR_INVALID_ARG, "%s: misaligned matrix", who);
            if (g->E > 0) {
                const int grid = grid_for(g->E * nvec, 256);
                if (dtype == GNN_F32)
                    launch_overlapped(edge_factor_grad_kernel<float>, dim3((unsigned)(grid)), dim3(256), 0, st, g->rowptr, g->col, g->N, g->E, nvec, op == GNN_MEAN, (const uint4*)Xj, (const uint4*)dOut, de_csr);
                else
                    launch_overlapped(edge_factor_grad_kernel<__nv_bfloat16>, dim3((unsigned)(grid)), dim3(256), 0, st, g->rowptr, g->col, g->N, g->E, nvec, op == GNN_MEAN, (const uint4*)Xj, (const uint4*)dOut, de_csr);
                GNN_CHECK_LAUNCH(who);
            }
        } else if (e_width == 1) {
            rc = run_sddmm(who, g, Xj, dOut, 1, F, op == GNN_MEAN, dtype, de_csr, st);
            if (rc != GNN_OK) return rc;
        } else {
            rc = run_sddmm(who, g, Xj, dOut, e_width, F / e_width, op == GNN_MEAN, dtype, de_csr, st);
            if (rc != GNN_OK) return rc;
        }
    }
    return GNN_OK;
}

size_t gnn_row_epilogue_backward_workspace(int32_t N, int F) {
    if (N < 0 || F <= 0) return 0;
    return up256((size_t)EB_MAX_BLOCKS * F * 4);
}

gnn_status gnn_row_epilogue_backward(const void* Y, const void* dY, int32_t N, int F, gnn_dtype dtype,
                                     int relu, void* dZ, float* dbias, void* ws, size_t ws_bytes,
                                     gnn_stream stream) {
    const char* who = "gnn_row_epilogue_backward";
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    const int s = elem_size(dtype);
    GNN_REQUIRE(N >= 0 && F > 0 && ((size_t)F * s) % 16 == 0 && F * s <= 2048, GNN_ERR_UNSUPPORTED,
                "%s: rows must be a multiple of 16 bytes and at most 2048 bytes", who);
    GNN_REQUIRE(dY && (!relu || Y) && (dZ || dbias), GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(aligned16(dY) && aligned16(Y) && aligned16(dZ), GNN_ERR_INVALID_ARG, "%s: misaligned matrix", who);
    const int nvec = F * s / 16;
    cudaStream_t st = as_stream(stream);
    // at least four rows per thread, so that a small graph does not leave hundreds of partials of one or two rows
    const int least = 4 * (EB_THREADS / nvec > 0 ? EB_THREADS / nvec : 1);
    const int spread = (int)ceil_div(N > 0 ? N : 1, EB_MAX_BLOCKS), rows_per_block = spread > least ? spread : least;
    const int nb = N > 0 ? (int)ceil_div(N, rows_per_block) : 0;
    float* partial = nullptr;
    if (dbias) {
        const size_t need = gnn_row_epilogue_backward_workspace(N, F);
        GNN_REQUIRE(ws && ws_bytes >= need && aligned16(ws), GNN_ERR_WORKSPACE_TOO_SMALL, "%s: workspace of %zu bytes needed, %zu given", who, need, ws_bytes);
        partial = (float*)ws;
    }
    if (nb > 0) {
        const size_t smem = (size_t)(EB_THREADS / nvec) * nvec * (16 / s) * 4;
        if (dtype == GNN_F32)
            launch_overlapped(epilogue_backward_kernel<float>, dim3((unsigned)(nb)), dim3(EB_THREADS), smem, st, (const uint4*)Y, (const uint4*)dY, N, nvec, relu, (uint4*)dZ, partial, rows_per_block);
        else
            launch_overlapped(epilogue_backward_kernel<__nv_bfloat16>, dim3((unsigned)(nb)), dim3(EB_THREADS), smem, st, (const uint4*)Y, (const uint4*)dY, N, nvec, relu, (uint4*)dZ, partial, rows_per_block);
        GNN_CHECK_LAUNCH(who);
    }
    if (dbias) {
        launch_overlapped(column_sum_final_kernel, dim3((unsigned)ceil_div(F, 32)), dim3(32 * CS_WALKERS), 0, st, partial, nb, F, dbias);
        GNN_CHECK_LAUNCH(who);
    }
    return GNN_OK;
}

size_t gnn_gin_workspace(int64_t E, int F) {
    if (E < 0 || F <= 0) return 0;
    return chunked_workspace(E, F, false) + up256((size_t)DOT_MAX_BLOCKS * 4);
}

gnn_status gnn_gin(const gnn_csr* g, const void* X, float eps, int F, gnn_dtype dtype, void* out,
                   void* ws, size_t ws_bytes, gnn_stream stream) {
    const gnn_row_epilogue epi = {X, 1.0f + eps, GNN_SELF_ALWAYS, nullptr, 0};
    return gnn_propagate_msg(g, GNN_MSG_COPY_XJ, GNN_SUM, X, nullptr, nullptr, 0, F, dtype, &epi, out, nullptr, ws,
                             ws_bytes, stream);
}

gnn_status gnn_gin_backward(const gnn_csr* g, const void* dOut, const void* X, float eps, int F,
                            gnn_dtype dtype, void* dX, float* deps, void* ws, size_t ws_bytes,
                            gnn_stream stream) {
    const char* who = "gnn_gin_backward";
    GNN_REQUIRE(g && dOut && F > 0, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    const size_t need = gnn_gin_workspace(g->E, F);
    GNN_REQUIRE(ws && ws_bytes >= need, GNN_ERR_WORKSPACE_TOO_SMALL, "%s: workspace of %zu bytes needed, %zu given", who, need, ws_bytes);
    if (dX) {
        const gnn_row_epilogue sg = {dOut, 1.0f + eps, GNN_SELF_ALWAYS, nullptr, 0};
        gnn_status rc = gnn_propagate_msg_backward(g, GNN_MSG_COPY_XJ, GNN_SUM, dOut, nullptr, nullptr, 0, nullptr, F, dtype,
                                                   &sg, dX, nullptr, nullptr, ws, ws_bytes, stream);
        if (rc != GNN_OK) return rc;
    }
    if (deps) {
        GNN_REQUIRE(X, GNN_ERR_INVALID_ARG, "%s: deps needs X", who);
        GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
        const int s = elem_size(dtype);
        GNN_REQUIRE(((size_t)F * s) % 16 == 0 && aligned16(X) && aligned16(dOut), GNN_ERR_UNSUPPORTED, "%s: rows must be 16-byte multiples, matrices aligned", who);
        const int64_t nvec = (int64_t)g->N * (F * s / 16);
        float* partial = (float*)((char*)ws + chunked_workspace(g->E, F, false));  // behind the reduction's scratch
        const int nb = (int)(nvec > 0 ? (ceil_div(nvec, DOT_THREADS) < DOT_MAX_BLOCKS ? ceil_div(nvec, DOT_THREADS) : DOT_MAX_BLOCKS) : 0);
        cudaStream_t st = as_stream(stream);
        if (nb > 0) {
            if (dtype == GNN_F32) launch_overlapped(dot_partial_kernel<float>, dim3((unsigned)(nb)), dim3(DOT_THREADS), 0, st, (const uint4*)dOut, (const uint4*)X, nvec, partial);
            else launch_overlapped(dot_partial_kernel<__nv_bfloat16>, dim3((unsigned)(nb)), dim3(DOT_THREADS), 0, st, (const uint4*)dOut, (const uint4*)X, nvec, partial);
        }
        launch_overlapped(dot_final_kernel, dim3((unsigned)(1)), dim3(32), 0, st, partial, nb, deps);
        GNN_CHECK_LAUNCH(who);
    }
    return GNN_OK;
}

gnn_status gnn_edge_dot(const gnn_csr* g, const void* Xj, const void* Xi, int H, int C,
                        gnn_dtype dtype, float* s_csr, gnn_stream stream) {
    const char* who = "gnn_edge_dot";
    GNN_REQUIRE(g && g->rowptr && Xj && Xi && (s_csr || g->E == 0), GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(g->E == 0 || g->col, GNN_ERR_INVALID_ARG, "%s: null col", who);
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    GNN_REQUIRE(H >= 1 && C >= 1, GNN_ERR_INVALID_ARG, "%s: bad H or C", who);
    if (H == 1) return run_sddmm(who, g, Xj, Xi, 1, C, 0, dtype, s_csr, as_stream(stream));
    return run_sddmm(who, g, Xj, Xi, H, C, 0, dtype, s_csr, as_stream(stream));
}

size_t gnn_edge_dot_backward_workspace(int64_t E, int H, int C) {
    if (E < 0 || H <= 0 || C <= 0) return 0;
    return chunked_workspace(E, H * C, false) + up256((size_t)(E > 0 ? E : 1) * H * 4);
}

gnn_status gnn_edge_dot_backward(const gnn_csr* g, const void* Xj, const void* Xi,
                                 const float* ds_csr, int H, int C, gnn_dtype dtype, void* dXj,
                                 void* dXi, void* ws, size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_edge_dot_backward";
    GNN_REQUIRE(g && g->rowptr && g->rowptrT && (ds_csr || g->E == 0), GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(g->E == 0 || (g->col && g->colT && g->t2f), GNN_ERR_INVALID_ARG, "%s: incomplete gnn_csr", who);
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    GNN_REQUIRE(H >= 1 && C >= 1, GNN_ERR_INVALID_ARG, "%s: bad H or C", who);
    const int F = H * C;
    const size_t red = chunked_workspace(g->E, F, false), need = gnn_edge_dot_backward_workspace(g->E, H, C);
    GNN_REQUIRE(ws && ws_bytes >= need && aligned16(ws), GNN_ERR_WORKSPACE_TOO_SMALL, "%s: workspace of %zu bytes needed, %zu given", who, need, ws_bytes);
    cudaStream_t st = as_stream(stream);
    gnn_status rc;
    if (dXi) {  // rows = targets, gathered rows = sources
        GNN_REQUIRE(Xj, GNN_ERR_INVALID_ARG, "%s: dXi needs Xj", who);
        if (H == 1) {
            rc = run_chunked(who, MODE_SUM, g->N, g->E, g->rowptr, g->col, ds_csr, Xj, dXi, nullptr, nullptr, nullptr, nullptr,
                             0, F, dtype, ws, red, st);
        } else {
            HeadExtra hx = {ds_csr, nullptr, H, nullptr, nullptr, nullptr, nullptr};
            rc = run_chunked(who, MODE_HEADSUM, g->N, g->E, g->rowptr, g->col, nullptr, Xj, dXi, nullptr, nullptr, nullptr,
                             nullptr, 0, F, dtype, ws, red, st, &hx);
        }
        if (rc != GNN_OK) return rc;
    }
    if (dXj) {  // rows = sources, gathered rows = targets; the factors in transposed order
        GNN_REQUIRE(Xi, GNN_ERR_INVALID_ARG, "%s: dXj needs Xi", who);
        float* dsT = (float*)((char*)ws + red);
        if (g->E > 0) {
            rc = gnn_permute_edge_data(g->t2f, g->E, H, 4, ds_csr, dsT, stream);
            if (rc != GNN_OK) return rc;
        }
        if (H == 1) {
            rc = run_chunked(who, MODE_SUM, g->N, g->E, g->rowptrT, g->colT, dsT, Xi, dXj, nullptr, nullptr, nullptr, nullptr,
                             0, F, dtype, ws, red, st);
        } else {
            HeadExtra hx = {dsT, nullptr, H, nullptr, nullptr, nullptr, nullptr};
            rc = run_chunked(who, MODE_HEADSUM, g->N, g->E, g->rowptrT, g->colT, nullptr, Xi, dXj, nullptr, nullptr, nullptr,
                             nullptr, 0, F, dtype, ws, red, st, &hx);
        }
        if (rc != GNN_OK) return rc;
    }
    return GNN_OK;
}

gnn_status gnn_merge_edge_lists(const gnn_edge_segment* segs, int S, int32_t* src_out,
                                int32_t* dst_out, int32_t* seg_out, gnn_stream stream) {
    const char* who = "gnn_merge_edge_lists";
    GNN_REQUIRE(segs && S >= 1, GNN_ERR_INVALID_ARG, "%s: no segments", who);
    int64_t total = 0;
    for (int k = 0; k < S; ++k) {
        GNN_REQUIRE(segs[k].E >= 0 && (segs[k].E == 0 || (segs[k].src && segs[k].dst)), GNN_ERR_INVALID_ARG, "%s: segment %d: bad edge list", who, k);
        GNN_REQUIRE(segs[k].src_offset >= 0 && segs[k].dst_offset >= 0, GNN_ERR_INVALID_ARG, "%s: segment %d: negative offset", who, k);
        total += segs[k].E;
    }
    GNN_REQUIRE(total < ((int64_t)1 << 31), GNN_ERR_UNSUPPORTED, "%s: the merged list must have fewer than 2^31 edges", who);
    GNN_REQUIRE(total == 0 || (src_out && dst_out), GNN_ERR_INVALID_ARG, "%s: null output", who);
    cudaStream_t st = as_stream(stream);
    int64_t base = 0;
    for (int k = 0; k < S; ++k) {
        if (segs[k].E == 0) continue;
        launch_overlapped(merge_segment_kernel, dim3((unsigned)(grid_for(segs[k].E, 256))), dim3(256), 0, st, segs[k].src, segs[k].dst, segs[k].E, segs[k].src_offset,
                                                                        segs[k].dst_offset, k, src_out + base, dst_out + base,
                                                                        seg_out ? seg_out + base : nullptr);
        base += segs[k].E;
    }
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

gnn_status gnn_segment_coef(const gnn_csr* g, const int32_t* seg_csr, const float* w_csr,
                            const int32_t* seg_is_mean, int S, float* coef_csr, float* coef_csrT,
                            gnn_stream stream) {
    const char* who = "gnn_segment_coef";
    GNN_REQUIRE(g && g->rowptr && S >= 1 && seg_is_mean, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(coef_csr, GNN_ERR_INVALID_ARG, "%s: coef_csr is needed (coef_csrT is derived from it)", who);
    if (g->E == 0) return GNN_OK;
    GNN_REQUIRE(seg_csr, GNN_ERR_INVALID_ARG, "%s: null seg_csr", who);
    cudaStream_t st = as_stream(stream);
    // an out-of-range segment id leaves its factor unscaled and is reported through the last word of coef_csrT's
    // pass below only if asked for; the ids come from gnn_merge_edge_lists, so this is a guard, not a path
    launch_overlapped(segment_coef_kernel, dim3((unsigned)(grid_for(g->E, 256))), dim3(256), 0, st, g->rowptr, g->N, g->E, seg_csr, w_csr, seg_is_mean, S, coef_csr, nullptr);
    GNN_CHECK_LAUNCH(who);
    if (coef_csrT) {
        GNN_REQUIRE(g->t2f, GNN_ERR_INVALID_ARG, "%s: coef_csrT needs t2f", who);
        return gnn_permute_edge_data(g->t2f, g->E, 1, 4, coef_csr, coef_csrT, stream);
    }
    return GNN_OK;
}

}  // extern "C"
