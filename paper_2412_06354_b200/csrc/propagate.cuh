// Declarations shared by the calls that reduce gathered rows.
#pragma once
#include "common.cuh"

namespace gnn {

enum { MODE_SUM = 0, MODE_MAX = 1, MODE_MIN = 2, MODE_ROUTE = 3, MODE_HEADSUM = 4, MODE_EFSUM = 5, MODE_WSUM = 6, MODE_V2 = 7, MODE_HEADSUM_W = 8, MODE_HEADRANK = 9 };

// MODE_HEADSUM extras: multipliers per (position, head) and an optional rank-1 row epilogue
//   out[r,f] += epi_l[r,h(f)] * epi_a[f] + epi_r[r,h(f)] * epi_b[f]
struct HeadExtra {
    const float* wh;  // [E,H]
    const int32_t* wh_index;  // nullptr: position p uses row p of wh; else row wh_index[p]
    int H;
    const float *epi_l, *epi_r;  // [rows,H] or nullptr
    const float *epi_a, *epi_b;  // [F]
};

// per-feature multipliers (MODE_EFSUM) and the optional row epilogue of run_chunked:
//   v = agg_c * v + self_c * c(r) * self_X[r,f] + bias[f], then max(v, 0) if relu
// c(r) = 1, the length of row r in self_rowptr, or [that length > 0] (gnn_self_mode)
struct RowExtra {
    const float* ef;  // MODE_EFSUM: [E, ef_ld] fp32, or nullptr
    int ef_ld;
    float agg_c;      // multiplier of the reduced value: 1 or -1
    const void* self_X;  // [rows, F] of the call's dtype, or nullptr
    float self_c;
    int self_mode;
    const int64_t* self_rowptr;
    const float* bias;  // [F] or nullptr
    int relu;
    int descending = 0;  // positions from the last to the first: the gathered matrix was just written in ascending order
};

// lanes per row (4..32) and 16-byte vectors per lane (1, 2, 4) for rows of nvec 16-byte chunks
bool pick_shape(int nvec, int* lpr, int* vpl);

size_t chunked_workspace(int64_t E, int F, bool with_arg);

// out[r,:] = reduce over positions p of row r of  w[p] * X[col[p],:]   (see reduce_rows.cuh)
gnn_status run_chunked(const char* who, int mode, int32_t N, int64_t E, const int64_t* rowptr,
                       const int32_t* col, const float* w, const void* X, void* out,
                       int32_t* argmax, const int64_t* gscale_rowptr, const int32_t* route_arg,
                       const int32_t* route_pos, int mean, int F, gnn_dtype dtype, void* ws,
                       size_t ws_bytes, cudaStream_t st, const HeadExtra* hx = nullptr, const RowExtra* rx = nullptr);

// Gradient of the GATv2 logits with respect to the rows of one sparse form (see PropParams): out [N,F], and with da_part one
// partial of da per piece.  gatv2_rows_pieces: how many pieces; ws: gatv2_rows_workspace bytes.
int64_t gatv2_rows_pieces(int32_t N, int64_t E, int row_bytes);
size_t gatv2_rows_workspace(int32_t N, int64_t E, int F, int row_bytes);
gnn_status run_gatv2_rows(const char* who, int32_t N, int64_t E, const int64_t* rowptr, const int32_t* col, const int32_t* ds_index, const float* ds, int H,
                          const void* Xself, const void* Xother, const float* a, float slope, int F, gnn_dtype dtype, void* out, float* da_part, void* ws,
                          cudaStream_t st);

// s[p,h] = sum over the features f of head h of a[f] * LeakyReLU(X[col[p],f] + D[i,f]) for p in row i
gnn_status run_gatv2_logits(const char* who, const gnn_csr* g, const void* X, const void* D, const float* a, int H, int C, float slope, gnn_dtype dtype,
                            float* s, cudaStream_t st);

// dW[p,h] = <X[col[p],h,:], D[i,h,:]> for p in row i (H = 1, lph = 0: one dot product per edge, times 1/row length if mean)
gnn_status run_sddmm(const char* who, const gnn_csr* g, const void* X, const void* D, int H, int C, int mean,
                     gnn_dtype dtype, float* dW, cudaStream_t st);

}  // namespace gnn
