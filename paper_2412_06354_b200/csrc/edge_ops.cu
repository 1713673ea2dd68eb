// Unfused message-passing primitives (Sec. 3 "Message Passing"): gather, apply_edges,
// aggregate_neighbors and their backward passes, on explicit E x F message tensors.  These are
// the building blocks custom layers are written with; the fused propagate avoids their E x F
// traffic.  Edge tensors are in CSR order unless stated.
#include "reduce_params.cuh"

namespace gnn {

// row of the sparse form that contains position p: last r with rowptr[r] <= p
__device__ __forceinline__ int row_of_position(const int64_t* rowptr, int N, int64_t p) {
    return lower_bound_i64(rowptr, N + 1, p + 1) - 1;
}

// Row of position p for a thread whose positions only grow: a block owns a contiguous span of (position, chunk) pairs,
// so from one step to the next a thread's position moves on by blockDim / chunks-per-position and its row by a step or
// two.  A full search per 16-byte chunk made the calls below run at a sixth of the memory rate; now there is one full
// search per thread, and another only where more than eight rows (a run of empty ones) are skipped at once.
__device__ __forceinline__ int advance_row(const int64_t* rowptr, int N, int row, int64_t p) {
    if (row < 0) return row_of_position(rowptr, N, p);
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        if (rowptr[row + 1] > p) return row;  // rowptr[row] <= p holds throughout
        ++row;
    }
    return rowptr[row + 1] > p ? row : row_of_position(rowptr, N, p);
}
// first pair of this block's span and one past its last; spans are multiples of the block size
__device__ __forceinline__ void block_span(int64_t total, int64_t* t0, int64_t* t1) {
    const int64_t per = ((total + gridDim.x - 1) / gridDim.x + blockDim.x - 1) / blockDim.x * blockDim.x;
    *t0 = (int64_t)blockIdx.x * per;
    *t1 = *t0 + per < total ? *t0 + per : total;
}

// (position, 16-byte chunk) pairs t = p * nvec + ci, EO_U * 256 consecutive ones per block and EO_U per thread, so that a
// thread has as many dependent index -> row loads in flight.  One 64-bit division per thread for the block's first pair;
// the rest divide a number below nvec + EO_U * 256 by a multiplication (see over_nvec).  A thread that walked the grid's stride with one pair at a
// time took 86 us to gather 1.36 M rows of 256 bytes; floor for writing them 54 us.
constexpr int EO_U = 4;
// x / nvec; magic = 2^32 / nvec rounded up, which is exact while x * nvec < 2^32: the callers' x is below nvec + 1024, so
// rows of up to 4096 chunks have one and the others, and rows of one chunk, divide.
__device__ __forceinline__ uint32_t over_nvec(uint32_t x, uint32_t nvec, uint32_t magic) { return magic ? __umulhi(x, magic) : x / nvec; }
static uint32_t pair_magic(int nvec) { return nvec > 1 && nvec <= 4096 ? (uint32_t)((((uint64_t)1 << 32) + nvec - 1) / nvec) : 0; }
struct PairTile {
    int64_t p0, left;  // position of the block's first pair; pairs from it to the last of all
    uint32_t r0, nvec, magic;
    __device__ __forceinline__ PairTile(int64_t total, int nv, uint32_t mg) : nvec((uint32_t)nv), magic(mg) {
        const int64_t t0 = (int64_t)blockIdx.x * (EO_U * 256);
        p0 = t0 / nv;
        r0 = (uint32_t)(t0 - p0 * nv);
        left = total - t0;
    }
    __device__ __forceinline__ bool get(int u, int64_t* p, int* ci) const {  // this thread's u-th pair
        const uint32_t k = threadIdx.x + u * 256, x = r0 + k, q = over_nvec(x, nvec, magic);
        *p = p0 + q;
        *ci = (int)(x - q * nvec);
        return k < left;
    }
};
static dim3 pair_grid(int64_t total) { return dim3((unsigned)ceil_div(total, (int64_t)EO_U * 256)); }

// out[k, chunk] = X[idx[k], chunk]
__global__ void __launch_bounds__(256) gather_rows_kernel(const int32_t* idx, int64_t E, const uint4* X,
                                                          int nvec, uint32_t magic, uint4* __restrict__ out) {
    pdl_wait();
    const PairTile tile(E * nvec, nvec, magic);
    const uint64_t pol_keep = policy_evict_last();
    uint4* const o = out + (int64_t)blockIdx.x * (EO_U * 256) + threadIdx.x;
    size_t at[EO_U];
    bool ok[EO_U];
#pragma unroll
    for (int u = 0; u < EO_U; ++u) {
        int64_t p;
        int ci;
        ok[u] = tile.get(u, &p, &ci);
        at[u] = (size_t)(ok[u] ? idx[p] : 0) * nvec + ci;
    }
    uint4 v[EO_U];
#pragma unroll
    for (int u = 0; u < EO_U; ++u)
        if (ok[u]) v[u] = ld_hint16(reinterpret_cast<const char*>(X + at[u]), pol_keep);
#pragma unroll
    for (int u = 0; u < EO_U; ++u)
        if (ok[u]) o[u * 256] = v[u];
}

// m[p, f] = e[p, g(f)] * X[col[p], f]   (e == nullptr: plain copy of the source row)
template <typename T>
__global__ void __launch_bounds__(256) apply_edges_mul_kernel(const int32_t* col, int64_t E, const uint4* X,
                                                              int nvec, uint32_t magic, const float* e, int ew, int feats_per_e,
                                                              uint4* __restrict__ m) {
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    const PairTile tile(E * nvec, nvec, magic);
    const uint64_t pol_keep = policy_evict_last();
    uint4* const o = m + (int64_t)blockIdx.x * (EO_U * 256) + threadIdx.x;
    const bool chunk_in_one = feats_per_e % EPC == 0;  // every 16-byte chunk lies under one multiplier
    int64_t p[EO_U];
    int ci[EO_U], from[EO_U];
    bool ok[EO_U];
#pragma unroll
    for (int u = 0; u < EO_U; ++u) {
        ok[u] = tile.get(u, &p[u], &ci[u]);
        from[u] = ok[u] ? col[p[u]] : 0;
    }
    uint4 v[EO_U];
    float f[EO_U];
#pragma unroll
    for (int u = 0; u < EO_U; ++u) {
        f[u] = 1.0f;
        if (!ok[u]) continue;
        v[u] = ld_hint16(reinterpret_cast<const char*>(X + (size_t)from[u] * nvec + ci[u]), pol_keep);
        if (e && chunk_in_one) f[u] = e[p[u] * ew + (ew == 1 ? 0 : (ci[u] * EPC) / feats_per_e)];
    }
#pragma unroll
    for (int u = 0; u < EO_U; ++u) {
        if (!ok[u]) continue;
        if (e) {
            float x[EPC];
            Chunk<T>::unpack(v[u], x);
#pragma unroll
            for (int j = 0; j < EPC; ++j) x[j] *= chunk_in_one ? f[u] : e[p[u] * ew + (ci[u] * EPC + j) / feats_per_e];
            v[u] = Chunk<T>::pack(x);
        }
        o[u * 256] = v[u];
    }
}

// s[p, h] = LeakyReLU_slope(al[col[p], h] + ar[row(p), h]), fp32
__global__ void gat_logit_kernel(const int64_t* rowptr, const int32_t* col, int N,
                                 int64_t E, int H, const float* al, const float* ar,
                                 float slope, float* __restrict__ s) {
    pdl_wait();
    int64_t t0, t1;
    block_span(E * H, &t0, &t1);
    int i = -1;
    for (int64_t t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
        const int64_t p = t / H;
        const int h = (int)(t - p * H);
        i = advance_row(rowptr, N, i, p);
        const float z = al[(size_t)col[p] * H + h] + ar[(size_t)i * H + h];
        s[t] = z > 0.f ? z : slope * z;
    }
}

// backward of aggregate w.r.t. the messages: dm[p, :] from dOut[row(p), :].  A warp looks up the rows of its share of
// positions once; lpr lanes cover a row (of more than 32 chunks: 32 of them at a time) and its lane groups take equal runs
// of the share, each row's dOut and winners held in registers while its positions are written, the next row's on their way.
// Bound by the writes.  1.36 M rows of 256 bytes, max: 160 us with a search per chunk, 119 us with a load of dOut and
// winners per position and chunk (the L1 path was busy 77 % of the time), 86 us now; writing them takes 54 us.
constexpr int AB_SUB = 128;  // most positions per warp
template <typename T>
__global__ void __launch_bounds__(256) aggregate_backward_kernel(const int64_t* rowptr, int N, int64_t E, int op, int sub, int lpr, bool wide,
                                                                 const uint4* dOut, const int32_t* argmax,
                                                                 int nvec, uint4* __restrict__ dm) {
    constexpr int EPC = Chunk<T>::N;
    __shared__ int s_rows[8][AB_SUB + 1];
    __shared__ uint16_t s_start[8][AB_SUB + 2];
    pdl_wait();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, g = lane / lpr;
    const int64_t c = (int64_t)blockIdx.x * 8 + wib;
    if (c * sub >= E) return;
    const int cs = (int)(c * sub), n = (int)min((int64_t)sub, E - cs);
    const int* const row = s_rows[wib];
    const uint16_t* const start = s_start[wib];
    bool began_before;
    const int m = stage_rows(rowptr, N, E, cs, n, lane, s_rows[wib], s_start[wib], began_before);
    __syncwarp();
    const int L = sub * lpr / 32, a = g * L, b = min(a + L, n);
    if (a >= b) return;
    int q0 = 0, hi = m;  // start[q0] <= a < start[hi]
    while (hi - q0 > 1) {
        const int mid = (q0 + hi) >> 1;
        if (start[mid] <= a) q0 = mid; else hi = mid;
    }
    const bool route = op == GNN_MAX || op == GNN_MIN;
    struct Row { uint4 v, win[EPC / 4]; float deg; };
    for (int ci = lane % lpr; ci < nvec; ci += lpr) {
        auto load = [&](int q, Row& R) {
            const int r = max(row[q], 0);
            const size_t from = (size_t)r * nvec + ci;
            R.v = ld_16(dOut + from);
            if (op == GNN_MEAN) R.deg = (float)(rowptr[r + 1] - rowptr[r]);
            if (route) {
#pragma unroll
                for (int j = 0; j < EPC / 4; ++j) {
                    const int32_t* w = argmax + from * EPC + 4 * j;  // wide: 16-byte aligned
                    if (wide) R.win[j] = ld_16(w);
                    else R.win[j] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        };
        Row R, next;
        load(q0, R);
        uint4* const o = dm + (size_t)cs * nvec + ci;
        for (int q = q0, p = a;; ++q) {
            const int e = min((int)start[q + 1], b);
            if (e < b) load(q + 1, next);
            if (op == GNN_MEAN) {
                float x[EPC];
                Chunk<T>::unpack(R.v, x);
#pragma unroll
                for (int j = 0; j < EPC; ++j) x[j] = x[j] / R.deg;
                R.v = Chunk<T>::pack(x);
            }
            if (row[q] < 0) R.v = make_uint4(0u, 0u, 0u, 0u);  // positions of no row (not where they are loaded: it would wait)
            for (; p < e; ++p) {
                uint4 v = R.v;
                if (route) {  // zero where another position won
                    const uint32_t at = (uint32_t)(cs + p);
                    if (EPC == 4) {
                        v.x = R.win[0].x == at ? v.x : 0u; v.y = R.win[0].y == at ? v.y : 0u; v.z = R.win[0].z == at ? v.z : 0u; v.w = R.win[0].w == at ? v.w : 0u;
                    } else {
                        const uint4 &lo = R.win[0], &up = R.win[EPC / 4 - 1];
                        v.x &= (lo.x == at ? 0xffffu : 0u) | (lo.y == at ? 0xffff0000u : 0u); v.y &= (lo.z == at ? 0xffffu : 0u) | (lo.w == at ? 0xffff0000u : 0u);
                        v.z &= (up.x == at ? 0xffffu : 0u) | (up.y == at ? 0xffff0000u : 0u); v.w &= (up.z == at ? 0xffffu : 0u) | (up.w == at ? 0xffff0000u : 0u);
                    }
                }
                o[(size_t)p * nvec] = v;
            }
            if (e >= b) break;
            R = next;
        }
    }
}
// Share of positions: 128 once they fill the machine, fewer below so that every SM has warps (13k positions, 512-byte rows:
// 12.5 us at 32, 5.3 us at 8).
static gnn_status launch_aggregate_backward(const char* who, const int64_t* rowptr, int32_t N, int64_t E, gnn_op op, const void* dOut,
                                            const int32_t* argmax, int nvec, gnn_dtype dtype, void* dm, cudaStream_t st) {
    const int sub = E >= 512 * 1024 ? AB_SUB : E >= 128 * 1024 ? 64 : E >= 64 * 1024 ? 32 : 8;
    const int lpr = nvec <= 4 ? 4 : nvec <= 8 ? 8 : nvec <= 16 ? 16 : 32;
    const dim3 grid((unsigned)ceil_div(E, (int64_t)sub * 8));
    auto launch = [&](auto kernel) {
        launch_overlapped(kernel, grid, dim3(256), 0, st, rowptr, N, E, (int)op, sub, lpr, aligned16(argmax), (const uint4*)dOut, argmax, nvec, (uint4*)dm);
    };
    if (dtype == GNN_F32) launch(aggregate_backward_kernel<float>);
    else launch(aggregate_backward_kernel<__nv_bfloat16>);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

static gnn_status check_rows(const char* who, int F, gnn_dtype dtype, int* nvec) {
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    const int s = elem_size(dtype);
    GNN_REQUIRE(F > 0 && ((size_t)F * s) % 16 == 0, GNN_ERR_UNSUPPORTED,
                "%s: F*sizeof(element) = %d must be a multiple of 16 bytes", who, F * s);
    *nvec = F * s / 16;
    return GNN_OK;
}

// graph_ptr[g] = first node whose graph id is >= g; flag set if ids are unsorted or out of range
__global__ void graph_ptr_kernel(const int32_t* gid, int32_t N, int32_t G,
                                 int64_t* __restrict__ gptr, int* __restrict__ flag) {
    pdl_wait();
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t n = t; n < N; n += stride) {
        const int a = gid[n];
        if (a < 0 || a >= G || (n + 1 < N && gid[n + 1] < a)) *flag = 1;
    }
    for (int64_t g = t; g <= G; g += stride) {
        int lo = 0, hi = N;
        while (lo < hi) {
            int mid = (lo + hi) >> 1;
            if (gid[mid] < (int32_t)g) lo = mid + 1; else hi = mid;
        }
        gptr[g] = lo;
    }
}

// out = alpha*a + beta*b, element-wise in fp32 (self terms of layers: W1*x_i + W2*agg, (1+eps)*x_i + sum).  From the end: a and b
// were usually written just before, in ascending order, and L2 holds their ends; what reads `out` next begins with the part written last.  A GraphConv step of
// 512 graphs 110.5 -> 108.8 us; of 13 other layers one 1.7 % slower, the rest level.
template <typename T>
__global__ void axpby_kernel(float alpha, const uint4* a, float beta, const uint4* b,
                             int64_t nvec, uint4* __restrict__ out) {
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (t = nvec - 1 - t; t >= 0; t -= stride) {
        float x[EPC], y[EPC];
        Chunk<T>::unpack(a[t], x);
        Chunk<T>::unpack(b[t], y);
#pragma unroll
        for (int j = 0; j < EPC; ++j) x[j] = fmaf(alpha, x[j], beta * y[j]);
        out[t] = Chunk<T>::pack(x);
    }
}

// out[k, :] = X[idx[k], :], rows of nvec 16-byte chunks
void launch_gather_rows(const int32_t* idx, int64_t E, const void* X, int nvec, void* out, cudaStream_t st) {
    launch_overlapped(gather_rows_kernel, pair_grid(E * nvec), dim3(256), 0, st, idx, E, (const uint4*)X, nvec, pair_magic(nvec), (uint4*)out);
}

}  // namespace gnn

using namespace gnn;

extern "C" {

gnn_status gnn_gather(const int32_t* idx, int64_t E, const void* X, int32_t N, int F,
                      gnn_dtype dtype, void* out, gnn_stream stream) {
    const char* who = "gnn_gather";
    int nvec;
    gnn_status rc = check_rows(who, F, dtype, &nvec);
    if (rc != GNN_OK) return rc;
    GNN_REQUIRE(E >= 0 && N >= 0, GNN_ERR_INVALID_ARG, "%s: negative size", who);
    if (E == 0) return GNN_OK;
    GNN_REQUIRE(idx && X && out && aligned16(X) && aligned16(out), GNN_ERR_INVALID_ARG,
                "%s: null or misaligned argument", who);
    launch_gather_rows(idx, E, X, nvec, out, as_stream(stream));
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

gnn_status gnn_gather_backward(const gnn_csr* g, int by_src, const void* dOut_EF, int F,
                               gnn_dtype dtype, void* dX, void* ws, size_t ws_bytes,
                               gnn_stream stream) {
    const char* who = "gnn_gather_backward";
    GNN_REQUIRE(g && dOut_EF && dX, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    const int64_t* rp = by_src ? g->rowptrT : g->rowptr;
    const int32_t* rows = by_src ? g->eidT : g->eid;  // COO row of dOut for each position
    GNN_REQUIRE(rp && (g->E == 0 || rows), GNN_ERR_INVALID_ARG, "%s: incomplete gnn_csr", who);
    // The edge tensor is usually larger than L2 and has just been written in ascending order: its end is what L2 still holds (message passes by separate
    // calls 673 -> 668 us at 1.36 M edges, 0.9 to 1.5 % on four of ten others, none slower).
    RowExtra rx = {};
    rx.agg_c = 1.0f;
    rx.descending = 1;
    return run_chunked(who, MODE_SUM, g->N, g->E, rp, rows, nullptr, dOut_EF, dX, nullptr, nullptr,
                       nullptr, nullptr, 0, F, dtype, ws, ws_bytes, as_stream(stream), nullptr, &rx);
}

gnn_status gnn_apply_edges(const gnn_csr* g, gnn_msg msg, const void* X_or_al, const void* ar,
                           const float* e, int e_width, int F, gnn_dtype dtype, float slope,
                           void* m_out, gnn_stream stream) {
    const char* who = "gnn_apply_edges";
    GNN_REQUIRE(g && g->rowptr && X_or_al && m_out, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    if (g->E == 0) return GNN_OK;
    GNN_REQUIRE(g->col, GNN_ERR_INVALID_ARG, "%s: null col", who);
    cudaStream_t st = as_stream(stream);
    if (msg == GNN_MSG_GAT_LOGIT) {
        GNN_REQUIRE(dtype == GNN_F32, GNN_ERR_UNSUPPORTED, "%s: GAT_LOGIT works on fp32 scores", who);
        GNN_REQUIRE(ar && F > 0, GNN_ERR_INVALID_ARG, "%s: GAT_LOGIT needs ar and F = heads", who);
        launch_overlapped(gat_logit_kernel, dim3((unsigned)(grid_for(g->E * F, 256))), dim3(256), 0, st, g->rowptr, g->col, g->N, g->E, F, (const float*)X_or_al,
                                                                  (const float*)ar, slope, (float*)m_out);
        GNN_CHECK_LAUNCH(who);
        return GNN_OK;
    }
    GNN_REQUIRE(msg == GNN_MSG_COPY_XJ || msg == GNN_MSG_E_MUL_XJ, GNN_ERR_INVALID_ARG, "%s: bad message", who);
    int nvec;
    gnn_status rc = check_rows(who, F, dtype, &nvec);
    if (rc != GNN_OK) return rc;
    GNN_REQUIRE(aligned16(X_or_al) && aligned16(m_out), GNN_ERR_INVALID_ARG, "%s: misaligned matrix", who);
    int feats_per_e = 1;
    if (msg == GNN_MSG_E_MUL_XJ) {
        GNN_REQUIRE(e && e_width >= 1 && F % e_width == 0, GNN_ERR_INVALID_ARG,
                    "%s: E_MUL_XJ needs e of width 1, H (dividing F) or F", who);
        feats_per_e = F / e_width;
    } else {
        e = nullptr;
        e_width = 1;
    }
    auto launch = [&](auto kernel) {
        launch_overlapped(kernel, pair_grid(g->E * nvec), dim3(256), 0, st, g->col, g->E, (const uint4*)X_or_al, nvec, pair_magic(nvec), e, e_width, feats_per_e, (uint4*)m_out);
    };
    if (dtype == GNN_F32) launch(apply_edges_mul_kernel<float>);
    else launch(apply_edges_mul_kernel<__nv_bfloat16>);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

gnn_status gnn_aggregate(const gnn_csr* g, gnn_op op, const void* m_EF, int F, gnn_dtype dtype,
                         void* out, int32_t* argmax, void* ws, size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_aggregate";
    GNN_REQUIRE(g && g->rowptr && m_EF && out, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "%s: bad op", who);
    GNN_REQUIRE(!argmax || aligned16(argmax), GNN_ERR_INVALID_ARG, "%s: argmax must be 16-byte aligned", who);
    const int mode = op == GNN_MAX ? MODE_MAX : op == GNN_MIN ? MODE_MIN : MODE_SUM;
    // position p reads row p of the message tensor: the segmented reduction without a gather
    return run_chunked(who, mode, g->N, g->E, g->rowptr, nullptr, nullptr, m_EF, out, argmax, nullptr,
                       nullptr, nullptr, op == GNN_MEAN, F, dtype, ws, ws_bytes, as_stream(stream));
}

gnn_status gnn_aggregate_backward(const gnn_csr* g, gnn_op op, const void* dOut_NF,
                                  const int32_t* argmax, int F, gnn_dtype dtype, void* dm_EF,
                                  gnn_stream stream) {
    const char* who = "gnn_aggregate_backward";
    GNN_REQUIRE(g && g->rowptr && dOut_NF && dm_EF, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "%s: bad op", who);
    GNN_REQUIRE((op != GNN_MAX && op != GNN_MIN) || argmax, GNN_ERR_INVALID_ARG, "%s: MAX/MIN need the forward argmax", who);
    int nvec;
    gnn_status rc = check_rows(who, F, dtype, &nvec);
    if (rc != GNN_OK) return rc;
    if (g->E == 0) return GNN_OK;
    GNN_REQUIRE(aligned16(dOut_NF) && aligned16(dm_EF), GNN_ERR_INVALID_ARG, "%s: misaligned matrix", who);
    return launch_aggregate_backward(who, g->rowptr, g->N, g->E, op, dOut_NF, argmax, nvec, dtype, dm_EF, as_stream(stream));
}

gnn_status gnn_graph_ptr_from_ids(const int32_t* graph_id, int32_t N, int32_t G, int64_t* graph_ptr,
                                  void* ws, size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_graph_ptr_from_ids";
    GNN_REQUIRE(N >= 0 && G >= 0 && graph_ptr && (N == 0 || graph_id), GNN_ERR_INVALID_ARG, "%s: bad argument", who);
    GNN_REQUIRE(ws && ws_bytes >= 4, GNN_ERR_WORKSPACE_TOO_SMALL, "%s: 4 bytes of workspace needed", who);
    cudaStream_t st = as_stream(stream);
    int* flag = (int*)ws;
    if (cudaMemsetAsync(flag, 0, 4, st) != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: memset failed", who);
    launch_overlapped(graph_ptr_kernel, dim3((unsigned)(grid_for((N > G ? N : G) + 1, 256))), dim3(256), 0, st, graph_id, N, G, graph_ptr, flag);
    GNN_CHECK_LAUNCH(who);
    int h = 0;
    if (cudaMemcpyAsync(&h, flag, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        GNN_FAIL(GNN_ERR_CUDA, "%s: reading the validation flag failed", who);
    GNN_REQUIRE(h == 0, GNN_ERR_NOT_SORTED, "%s: graph ids must be sorted and inside [0, %d)", who, G);
    return GNN_OK;
}

gnn_status gnn_reduce_nodes(const int64_t* graph_ptr, int32_t G, int32_t N, gnn_op op, const void* X,
                            int F, gnn_dtype dtype, void* out_GF, int32_t* argmax, void* ws,
                            size_t ws_bytes, gnn_stream stream) {
    const char* who = "gnn_reduce_nodes";
    GNN_REQUIRE(graph_ptr && X && out_GF && G >= 0 && N >= 0, GNN_ERR_INVALID_ARG, "%s: bad argument", who);
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "%s: bad op", who);
    GNN_REQUIRE(!argmax || aligned16(argmax), GNN_ERR_INVALID_ARG, "%s: argmax must be 16-byte aligned", who);
    const int mode = op == GNN_MAX ? MODE_MAX : op == GNN_MIN ? MODE_MIN : MODE_SUM;
    // graphs are the rows, nodes the positions: the same segmented reduction as aggregate
    return run_chunked(who, mode, G, N, graph_ptr, nullptr, nullptr, X, out_GF, argmax, nullptr, nullptr,
                       nullptr, op == GNN_MEAN, F, dtype, ws, ws_bytes, as_stream(stream));
}

gnn_status gnn_reduce_nodes_backward(const int64_t* graph_ptr, int32_t G, int32_t N, gnn_op op,
                                     const void* dOut_GF, const int32_t* argmax, int F,
                                     gnn_dtype dtype, void* dX_NF, gnn_stream stream) {
    const char* who = "gnn_reduce_nodes_backward";
    GNN_REQUIRE(graph_ptr && dOut_GF && dX_NF && G >= 0 && N >= 0, GNN_ERR_INVALID_ARG, "%s: bad argument", who);
    GNN_REQUIRE(op >= GNN_SUM && op <= GNN_MIN, GNN_ERR_INVALID_ARG, "%s: bad op", who);
    GNN_REQUIRE((op != GNN_MAX && op != GNN_MIN) || argmax, GNN_ERR_INVALID_ARG, "%s: MAX/MIN need the forward argmax", who);
    int nvec;
    gnn_status rc = check_rows(who, F, dtype, &nvec);
    if (rc != GNN_OK) return rc;
    if (N == 0) return GNN_OK;
    GNN_REQUIRE(aligned16(dOut_GF) && aligned16(dX_NF), GNN_ERR_INVALID_ARG, "%s: misaligned matrix", who);
    if (G == 0) {
        if (cudaMemsetAsync(dX_NF, 0, (size_t)N * F * elem_size(dtype), as_stream(stream)) != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: memset failed", who);
        return GNN_OK;
    }
    return launch_aggregate_backward(who, graph_ptr, G, N, op, dOut_GF, argmax, nvec, dtype, dX_NF, as_stream(stream));
}

gnn_status gnn_axpby(float alpha, const void* a, float beta, const void* b, int64_t n, gnn_dtype dtype,
                     void* out, gnn_stream stream) {
    const char* who = "gnn_axpby";
    GNN_REQUIRE(n >= 0 && (dtype == GNN_F32 || dtype == GNN_BF16), GNN_ERR_INVALID_ARG, "%s: bad argument", who);
    if (n == 0) return GNN_OK;
    const int epc = 16 / elem_size(dtype);
    GNN_REQUIRE(n % epc == 0, GNN_ERR_UNSUPPORTED, "%s: the element count must be a multiple of %d", who, epc);
    GNN_REQUIRE(a && b && out && aligned16(a) && aligned16(b) && aligned16(out), GNN_ERR_INVALID_ARG, "%s: null or misaligned argument", who);
    const int64_t nvec = n / epc;
    cudaStream_t st = as_stream(stream);
    if (dtype == GNN_F32) launch_overlapped(axpby_kernel<float>, dim3((unsigned)(grid_for(nvec, 256))), dim3(256), 0, st, alpha, (const uint4*)a, beta, (const uint4*)b, nvec, (uint4*)out);
    else launch_overlapped(axpby_kernel<__nv_bfloat16>, dim3((unsigned)(grid_for(nvec, 256))), dim3(256), 0, st, alpha, (const uint4*)a, beta, (const uint4*)b, nvec, (uint4*)out);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

}  // extern "C"
