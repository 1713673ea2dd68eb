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
    int descending;  // pieces from the last to the first
    int vote;  // rows are long enough on average that whole batches without a row end are common
    int has_epi;
    float agg_c, self_c;
    int self_mode, relu;
    const void* self_X;
    uint32_t self_ld;  // bytes between rows of self_X
    const int64_t* self_rowptr;
    const float* bias;  // [F] or nullptr
    // MODE_V2 (gradient of GATv2 logits): out[r,f] = epi_a[f] * sum over p of wh[p,h(f)] * LeakyReLU'(X[col[p],f] + v2_self[r,f])
    const void* v2_self;
    float slope;
    float* da_part;  // [npieces][F]: per piece, sum over p of wh[p,h(f)] * LeakyReLU(X[col[p],f] + v2_self[r,f]); or nullptr
};

// d.xy += w.xy * x.xy as one packed fp32x2 FMA (each half is an IEEE fused multiply-add)
__device__ __forceinline__ void fma2(float& a0, float& a1, float x0, float x1, float w0, float w1) {
    asm("{\n\t.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mov.b64 rc, {%0, %1};\n\tfma.rn.f32x2 rc, ra, rb, rc;\n\tmov.b64 {%0, %1}, rc;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "f"(x0), "f"(x1), "f"(w0), "f"(w1));
}

// d.xy *= w.xy
__device__ __forceinline__ void mul2(float& a0, float& a1, float w0, float w1) {
    asm("{\n\t.reg .b64 ra, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rc, {%0, %1};\n\tmul.rn.f32x2 rc, ra, rc;\n\tmov.b64 {%0, %1}, rc;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "f"(w0), "f"(w1));
}

// d.xy += x.xy
__device__ __forceinline__ void add2(float& a0, float& a1, float x0, float x1) {
    asm("{\n\t.reg .b64 ra, rc;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rc, {%0, %1};\n\tadd.rn.f32x2 rc, ra, rc;\n\tmov.b64 {%0, %1}, rc;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "f"(x0), "f"(x1));
}

// t0 += x.lo * d.lo, t1 += x.hi * d.hi for pairs of bf16: the fused multiply-adds of the unpacked values, without unpacking
__device__ __forceinline__ void fma_bf16(float& t0, float& t1, uint32_t x, uint32_t d) {
    asm("{\n\t.reg .b16 xl, xh, dl, dh;\n\tmov.b32 {xl, xh}, %2;\n\tmov.b32 {dl, dh}, %3;\n\t"
        "fma.rn.f32.bf16 %0, xl, dl, %0;\n\tfma.rn.f32.bf16 %1, xh, dh, %1;\n\t}"
        : "+f"(t0), "+f"(t1)
        : "r"(x), "r"(d));
}
// t0 += x.lo, t1 += x.hi
__device__ __forceinline__ void add_bf16(float& t0, float& t1, uint32_t x) {
    asm("{\n\t.reg .b16 xl, xh;\n\tmov.b32 {xl, xh}, %2;\n\tadd.rn.f32.bf16 %0, xl, %0;\n\tadd.rn.f32.bf16 %1, xh, %1;\n\t}" : "+f"(t0), "+f"(t1) : "r"(x));
}

// Smallest row r in [lo, N) with rowptr[r + 1] > v, or N: the first row at or after lo that has a
// position beyond v.  Warp-cooperative (every lane must call it with the same arguments): a look at the
// next 32 rows, then a 32-way search.
__device__ __forceinline__ int first_row_ending_after(const int64_t* rowptr, int lo, int N, int64_t v, int lane) {
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

// Position holding `pos`: the last row r with rowptr[r] <= pos (0 <= pos < E), or row 0 if there is none.  Warp-cooperative.  The
// first look is at 32 rows spaced 64 apart around the row that even degrees would give, then 32-way steps, then 64 rows at once.
__device__ __forceinline__ int row_of_position(const int64_t* rowptr, int N, int64_t E, int64_t pos, int lane) {
    int lo = 0, hi = N;  // rowptr[lo] <= pos < rowptr[hi]
    if (N > 1024) {
        const int guess = (int)((double)pos * ((double)N / (double)E));
        const int idx = guess + (lane - 16) * 64;
        const bool le = idx <= 0 || (idx < N && rowptr[idx] <= pos);
        const int c = __popc(__ballot_sync(0xffffffffu, le));
        if (c > 0) lo = max(lo, guess + (c - 1 - 16) * 64);
        if (c < 32) hi = min(hi, guess + (c - 16) * 64);
    }
    while (hi - lo > 64) {
        const int step = (hi - lo + 31) / 32;
        const int idx = lo + lane * step;
        const bool le = idx < hi && rowptr[idx] <= pos;  // true for a prefix of the lanes; for none if pos lies before the first row
        const int c = __popc(__ballot_sync(0xffffffffu, le));
        lo = lo + max(c - 1, 0) * step;
        hi = min(lo + step, hi);
    }
    const int a = lo + 1 + lane, b = a + 32;
    const bool la = a < hi && rowptr[a] <= pos, lb = b < hi && rowptr[b] <= pos;
    return lo + __popc(__ballot_sync(0xffffffffu, la)) + __popc(__ballot_sync(0xffffffffu, lb));
}

// The rows with positions in [cs, cs + n), n > 0: their ids to row[], their first positions relative to cs to start[] (0 for a
// row that began before), start[count] = the last one's end, or n + 1 if it goes on.  Positions before the first row or after the
// last (row pointers of a caller that leave some uncovered, as nodes outside graph_ptr) are staged as a row of id -1 that counts
// as begun before, if it is the first, and never ends, if it is the last: no caller finishes it, and none needs to look (a look
// at every row end cost 1 to 3 % of the segmented reduction).  Returns the count, at most n.  Warp-cooperative.
__device__ __forceinline__ int stage_rows(const int64_t* rowptr, int N, int64_t E, int cs, int n, int lane, int* row, uint16_t* start,
                                          bool& began_before) {
    const int r0 = row_of_position(rowptr, N, E, cs, lane);
    int m = 1;
    const int64_t s0 = rowptr[r0], e0 = rowptr[r0 + 1];
    const bool none = s0 > cs || e0 <= cs;  // the first position is in no row
    int64_t last_end = none ? (int64_t)cs + n + 1 : e0;
    began_before = none || s0 < cs;
    if (lane == 0) { row[0] = none ? -1 : r0; start[0] = 0; }
    for (int rb = s0 > cs ? r0 : r0 + 1; rb < N;) {
        const int r = rb + lane;
        int64_t s = 0, e = 0;
        bool in = false;
        if (r < N) {
            s = rowptr[r];
            in = s < cs + n;
            if (in) e = rowptr[r + 1];
        }
        const bool live = in && e > s;
        const unsigned lm = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int q = m + __popc(lm & ((1u << lane) - 1u));
            row[q] = r;
            start[q] = (uint16_t)(s - cs);
        }
        m += __popc(lm);
        if (lm) last_end = __shfl_sync(0xffffffffu, e, 31 - __clz(lm));
        if (!__all_sync(0xffffffffu, in)) break;
        if (lm == 0) rb = first_row_ending_after(rowptr, rb + 32, N, __shfl_sync(0xffffffffu, s, 0), lane);  // over a run of empty rows
        else rb += 32;
    }
    if (last_end < (int64_t)cs + n) {  // no row holds the rest
        if (lane == 0) { row[m] = -1; start[m] = (uint16_t)(last_end - cs); }
        ++m;
        last_end = (int64_t)cs + n + 1;
    }
    if (lane == 0) start[m] = (uint16_t)min(last_end - cs, (int64_t)n + 1);
    return m;
}

}  // namespace gnn
