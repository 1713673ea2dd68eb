// Arguments of the segmented reduction (reduce_rows.cuh) and what its launch rules share.
#pragma once
#include "propagate.cuh"

namespace gnn {

constexpr int RR_WARPS = 8;    // warps per block
constexpr int RR_SHORT = 32;   // longest row that one lane group reduces alone (row-per-group kernel)

struct PropParams {
    const int64_t* rowptr;  // rows of the output
    const int32_t* col;     // gathered row of X per position (nullptr: position p gathers row p)
    const float* w;         // per-position multiplier or nullptr
    const void* X;          // gathered matrix [N,F]
    void* out;              // [N,F]
    int32_t* argmax;        // MODE_MAX/MIN: winner positions [N,F] or nullptr
    const int64_t* gscale_rowptr;  // if set: each gathered row c is divided by max(1, length of
                                   // row c in this other sparse form) -- backward of MEAN
    const int32_t* route_arg;  // MODE_ROUTE: forward argmax [N,F]
    const int32_t* route_pos;  // MODE_ROUTE: forward position of each transposed position
    int32_t N;
    int64_t E;
    int nvec;  // 16-byte chunks per feature row (of the column slab this launch covers)
    int vec0;  // first 16-byte chunk of the slab within the full row
    uint32_t x_ld, out_ld;  // bytes between consecutive rows of X and of out (>= nvec*16)
    int F;                  // features of the slab
    int arg_ld;             // features between rows of argmax / route_arg
    int mean;               // divide the finished row by max(1, row length)
    int sub, piece;         // positions per warp, and per piece (the unit of partial rows): sub, or RR_WARPS * sub
    int64_t npieces;
    int32_t* tail_row;  // [npieces] row whose partial lives in slot 1, or -1
    float* part_val;    // [npieces][2][F]
    int32_t* part_arg;  // [npieces][2][F] (MODE_MAX/MIN)
    // MODE_HEADSUM: multiplier per (position, head), features of head h = [h*fph, (h+1)*fph)
    const float* wh;  // [E,H]
    const int32_t* wh_index;  // row of wh per position, or nullptr (= the position)
    int H, fph;
    // optional rank-1 epilogue: out[r,f] += epi_l[r,h(f)]*epi_a[f] + epi_r[r,h(f)]*epi_b[f]
    const float *epi_l, *epi_r, *epi_a, *epi_b;
    // MODE_EFSUM: multiplier per (position, feature), fp32 [E, ef_ld]
    const float* ef;
    int ef_ld;
    // optional row epilogue (has_epi), applied in fp32 to a finished row before its single rounding:
    //   v = agg_c * v + self_c * c(r) * self_X[r,f] + bias[f], then max(v, 0) if relu
    // c(r) = 1 (GNN_SELF_ALWAYS), the length of row r in self_rowptr (GNN_SELF_TIMES_DEGREE), or 1 if that
    // length is positive else 0 (GNN_SELF_IF_NONEMPTY)
    int has_epi;
    float agg_c, self_c;
    int self_mode, relu;
    const void* self_X;
    uint32_t self_ld;  // bytes between rows of self_X
    const int64_t* self_rowptr;
    const float* bias;  // [F] or nullptr
};

// Smallest row r in [lo, N) with rowptr[r + 1] > v, or N: the first row at or after lo that has a
// position beyond v.  Warp-cooperative (every lane must call it with the same arguments): a look at the
// next 32 rows, then a 32-way search.
__device__ __forceinline__ int first_row_ending_after(const int64_t* __restrict__ rowptr, int lo, int N, int64_t v, int lane) {
    {  // the common case, one coalesced load: the row is among the next 32
        const int r = lo + lane;
        const unsigned m = __ballot_sync(0xffffffffu, r >= N || rowptr[r + 1] > v);
        if (m) return min(lo + __ffs(m) - 1, N);
        lo += 32;
    }
    int hi = N;
    while (hi > lo) {
        const int step = (hi - lo + 31) / 32;
        const int idx = lo + lane * step;
        const bool le = idx < hi && rowptr[idx + 1] <= v;  // true for a prefix of the lanes
        const int k = __popc(__ballot_sync(0xffffffffu, le));
        if (k == 0) { hi = lo; break; }
        const int nlo = lo + (k - 1) * step + 1;
        hi = min(lo + k * step, hi);
        lo = nlo;
    }
    return lo;
}

}  // namespace gnn
