// The segmented reduction behind propagate, aggregate, gather_backward, pooling and the attention sums:
//   out[r,:] = op over positions p of row r of  m(p) * X[col[p],:]
//
// Two kernels.  stream_rows_kernel (all but small graphs) splits the positions, a warp per piece, and lets the gathers run
// ahead of the rows.  reduce_rows_kernel (graphs of up to 128 Ki edges with short rows, which latency bounds) gives every
// row a lane group: three dependent loads and a store in all.  Both leave rows that are cut by a piece as fp32 partials
// (slot 0: the row began in an earlier piece, slot 1: it begins here), which fixup_rows_kernel adds in ascending order.
//
// Inside a warp a feature row of up to 512 bytes is covered by LPR lanes x 16 bytes, so NG = 32/LPR groups work side by
// side; wider rows are reduced in column slabs of 512 bytes.
//
// What bounds it: instruction issue (about 20 per position and lane group, the unpacking of bf16 and the store of a row
// among them) and the loads in flight on narrow rows, the L2 -> SM return path (64 B/clk/SM) on rows of 512 bytes.
// Every order of additions is a fixed function of the graph and (F, dtype): results are bit-reproducible, no atomics.
#pragma once
#include "reduce_params.cuh"

namespace gnn {

// does candidate (cv, ca) beat the incumbent (v, a)?  ties go to the smaller position
template <int MODE>
__device__ __forceinline__ bool beats(float cv, int32_t ca, float v, int32_t a) {
    if (ca < 0) return false;
    if (a < 0) return true;
    bool better = (MODE == MODE_MAX) ? (cv > v) : (cv < v);
    return better || (cv == v && ca < a);
}

// Everything between the reduced values of a row and its stored 16-byte column ci (of the slab): division of the mean,
// rank-1 epilogue of the per-head mode and row epilogue (only with EPI), rounding, winners.
// r1 (READY): the rank-1 epilogue's factors, which the caller has at hand; loaded here, where the row ends, they are waited for
// once per row.
struct RankOne {
    float l, r;          // this row's and head's
    const float *a, *b;  // this column's, in shared memory
};
template <typename T, int MODE, bool EPI, bool READY = false>
__device__ __forceinline__ void finish_row(const PropParams& P, int row, int64_t len, int ci, float* v, const int32_t* a, const RankOne& r1 = RankOne()) {
    constexpr int EPC = Chunk<T>::N;
    constexpr bool ARG = MODE == MODE_MAX || MODE == MODE_MIN;
    if (P.mean) {
        const float f = 1.0f / (float)(len > 1 ? len : 1);
#pragma unroll
        for (int j = 0; j < EPC; ++j) v[j] *= f;
    }
    if (MODE == MODE_V2 && len > 0) {  // (a row without positions stays zero, whatever a holds)
#pragma unroll
        for (int j = 0; j < EPC; ++j) v[j] *= P.epi_a[ci * EPC + j];
    }
    if (READY) {
#pragma unroll
        for (int j = 0; j < EPC; j += 4) {
            const float4 x = *reinterpret_cast<const float4*>(r1.a + j), y = *reinterpret_cast<const float4*>(r1.b + j);
            v[j] += r1.l * x.x + r1.r * y.x;
            v[j + 1] += r1.l * x.y + r1.r * y.y;
            v[j + 2] += r1.l * x.z + r1.r * y.z;
            v[j + 3] += r1.l * x.w + r1.r * y.w;
        }
    } else if (MODE == MODE_HEADRANK) {
        const int f0 = (P.vec0 + ci) * EPC, h = f0 / P.fph;  // a 16-byte chunk lies inside one head
        const float el = P.epi_l[(size_t)row * P.H + h], er = P.epi_r[(size_t)row * P.H + h];
#pragma unroll
        for (int j = 0; j < EPC; ++j) v[j] += el * P.epi_a[f0 + j] + er * P.epi_b[f0 + j];
    }
    if (EPI && P.has_epi) {
        if (P.agg_c != 1.0f) {
#pragma unroll
            for (int j = 0; j < EPC; ++j) v[j] *= P.agg_c;
        }
        if (P.self_X) {
            float c = P.self_c;
            if (P.self_mode != GNN_SELF_ALWAYS) {
                const int64_t d = P.self_rowptr[row + 1] - P.self_rowptr[row];
                c = (P.self_mode == GNN_SELF_TIMES_DEGREE) ? c * (float)d : (d > 0 ? c : 0.f);
            }
            float x[EPC];
            Chunk<T>::unpack(*reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(P.self_X) + (size_t)row * P.self_ld + (size_t)ci * 16), x);
#pragma unroll
            for (int j = 0; j < EPC; ++j) v[j] = fmaf(c, x[j], v[j]);
        }
        if (P.bias) {
#pragma unroll
            for (int j = 0; j < EPC; ++j) v[j] += P.bias[ci * EPC + j];
        }
        if (P.relu) {
#pragma unroll
            for (int j = 0; j < EPC; ++j) v[j] = fmaxf(v[j], 0.f);
        }
    }
    st_stream16(reinterpret_cast<char*>(P.out) + (size_t)row * P.out_ld + (size_t)ci * 16, Chunk<T>::pack(v));
    if (ARG && P.argmax) {
        int32_t* ap = P.argmax + (size_t)row * P.arg_ld + (size_t)ci * EPC;
#pragma unroll
        for (int j = 0; j < EPC; j += 4) *reinterpret_cast<int4*>(ap + j) = make_int4(a[j], a[j + 1], a[j + 2], a[j + 3]);
    }
}


template <typename T, int LPR, int MODE>
struct RowReducer {
    static constexpr int EPC = Chunk<T>::N, NG = 32 / LPR;
    static constexpr bool ARG = MODE == MODE_MAX || MODE == MODE_MIN, EF = MODE == MODE_EFSUM, ROUTE = MODE == MODE_ROUTE;
    static constexpr bool HEAD = MODE == MODE_HEADSUM || MODE == MODE_HEADSUM_W || MODE == MODE_HEADRANK;
    static constexpr bool PLAIN = MODE == MODE_SUM || MODE == MODE_HEADSUM || MODE == MODE_HEADRANK;  // no multiplier per position (MODE_WSUM, MODE_HEADSUM_W: one)
    static constexpr int U = 4;  // gathers in flight per lane
    static constexpr int MW = EF ? EPC : 1;

    const PropParams& P;
    const int lane, g, li, ci;
    const bool col_lane;
    const uint64_t pol_keep;
    const char* const Xl;
    const float* const wh_l;  // HEAD: this lane's head column of the multiplier matrix
    float acc[EPC];
    int32_t arg[ARG ? EPC : 1];

    __device__ __forceinline__ RowReducer(const PropParams& p)
        : P(p), lane(threadIdx.x & 31), g((threadIdx.x & 31) / LPR), li((threadIdx.x & 31) % LPR), ci(li < p.nvec ? li : 0), col_lane(li < p.nvec),
          pol_keep(policy_evict_last()), Xl(reinterpret_cast<const char*>(p.X) + (size_t)(li < p.nvec ? li : 0) * 16),
          wh_l(HEAD ? p.wh + ((p.vec0 + (li < p.nvec ? li : 0)) * EPC) / p.fph : nullptr) {}

    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < EPC; ++j) {
            acc[j] = 0.f;
            if (ARG) arg[ARG ? j : 0] = -1;
        }
    }

    // one position per lane: gathered row, multiplier, and the forward position (ROUTE) or row of the multiplier matrix (HEAD)
    struct Entry { int c; float w; int t; };
    __device__ __forceinline__ Entry entry(int p, bool ok) const {
        Entry e = {0, 1.0f, 0};
        if (ok) {
            e.c = P.col ? ld_stream_i32(P.col + p) : p;
            if (!PLAIN && P.w) e.w = ld_stream_f32(P.w + p);
            if (ROUTE) e.t = ld_stream_i32(P.route_pos + p);
            if (HEAD) e.t = P.wh_index ? ld_stream_i32(P.wh_index + p) : p;
            if (!PLAIN && P.gscale_rowptr) {
                const int64_t d = P.gscale_rowptr[e.c + 1] - P.gscale_rowptr[e.c];
                e.w = e.w / (float)(d > 1 ? d : 1);
            }
        }
        return e;
    }

    // gather and add the entries j .. j + n - 1 (at most U) that the group's lanes hold; the first is at position pos
    __device__ __forceinline__ void batch(const Entry& e, int j, int n, int pos) {
        uint4 buf[U];
        float hw[(HEAD || EF) ? U : 1][MW];
        int4 win[ROUTE ? U : 1][ROUTE ? EPC / 4 : 1];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = __shfl_sync(0xffffffffu, e.c, j + u, LPR);
            const int t = HEAD ? __shfl_sync(0xffffffffu, e.t, j + u, LPR) : 0;
            if (u < n) {
                buf[u] = ld_hint16(Xl + (size_t)(uint32_t)c * P.x_ld, pol_keep);
                if (HEAD) hw[HEAD ? u : 0][0] = ld_f32(wh_l + (size_t)(uint32_t)t * P.H);
                if (EF) {
                    const float4* q = reinterpret_cast<const float4*>(P.ef + (size_t)(pos + u) * P.ef_ld + (size_t)ci * EPC);
#pragma unroll
                    for (int k = 0; k < MW / 4; ++k) {
                        const float4 a4 = __ldcs(q + k);
                        float* d = hw[EF ? u : 0] + 4 * k;
                        d[0] = a4.x; d[EF ? 1 : 0] = a4.y; d[EF ? 2 : 0] = a4.z; d[EF ? 3 : 0] = a4.w;
                    }
                }
                if (ROUTE) {
                    const int4* q = reinterpret_cast<const int4*>(P.route_arg + (size_t)(uint32_t)c * P.arg_ld + (size_t)ci * EPC);
#pragma unroll
                    for (int k = 0; k < EPC / 4; ++k) win[ROUTE ? u : 0][ROUTE ? k : 0] = ld_int4(q + k);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float w = PLAIN ? 1.0f : __shfl_sync(0xffffffffu, e.w, j + u, LPR);
            const int t = ROUTE ? __shfl_sync(0xffffffffu, e.t, j + u, LPR) : 0;
            if (u < n) {
                float x[EPC];
                Chunk<T>::unpack(buf[u], x);
                if (ARG) {
#pragma unroll
                    for (int k = 0; k < EPC; ++k) {
                        const float m = w * x[k];  // w = 1 where there are no multipliers: exact
                        // positions ascend within a group: a strict comparison keeps the first of equal values
                        const bool take = arg[ARG ? k : 0] < 0 || (MODE == MODE_MAX ? m > acc[k] : m < acc[k]);
                        if (take) { acc[k] = m; arg[ARG ? k : 0] = pos + u; }
                    }
                } else if (ROUTE) {  // keep dOut only where this edge was the winner
#pragma unroll
                    for (int k = 0; k < EPC / 4; ++k) {
                        const int4 a = win[ROUTE ? u : 0][ROUTE ? k : 0];
                        if (a.x == t) acc[4 * k] = fmaf(w, x[4 * k], acc[4 * k]);
                        if (a.y == t) acc[4 * k + 1] = fmaf(w, x[4 * k + 1], acc[4 * k + 1]);
                        if (a.z == t) acc[4 * k + 2] = fmaf(w, x[4 * k + 2], acc[4 * k + 2]);
                        if (a.w == t) acc[4 * k + 3] = fmaf(w, x[4 * k + 3], acc[4 * k + 3]);
                    }
                } else if (EF) {
#pragma unroll
                    for (int k = 0; k < EPC; k += 2)
                        fma2(acc[k], acc[k + 1], x[k], x[k + 1], hw[EF ? u : 0][EF ? k : 0] * w, hw[EF ? u : 0][EF ? k + 1 : 0] * w);
                } else if (PLAIN && !HEAD) {
#pragma unroll
                    for (int k = 0; k < EPC; k += 2) add2(acc[k], acc[k + 1], x[k], x[k + 1]);
                } else {
                    const float h = hw[HEAD ? u : 0][0], m = !HEAD ? w : PLAIN ? h : h * w;
#pragma unroll
                    for (int k = 0; k < EPC; k += 2) fma2(acc[k], acc[k + 1], x[k], x[k + 1], m, m);
                }
            }
        }
    }

    // positions [a, b) of one row, all groups together: of every 32 positions, whose entries the lanes load together,
    // group g adds LPR; afterwards every lane holds the result of its chunk
    __device__ __forceinline__ void whole_warp(int a, int b) {
        clear();
        Entry cur = entry(a + lane, a + lane < b);
        for (int q = a; q < b; q += 32) {
            const Entry nxt = entry(q + 32 + lane, q + 32 + lane < b);
            const int n = b - q - g * LPR;
#pragma unroll 1
            for (int j = 0; j < LPR && j < b - q; j += U) batch(cur, j, n - j, q + g * LPR + j);
            cur = nxt;
        }
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            const bool low = (lane & o) == 0;
#pragma unroll
            for (int j = 0; j < EPC; ++j) {
                const float mine = acc[j], ov = __shfl_xor_sync(0xffffffffu, mine, o);
                if (ARG) {
                    const int32_t ma = arg[ARG ? j : 0], oa = __shfl_xor_sync(0xffffffffu, ma, o);
                    if (beats<MODE>(ov, oa, mine, ma)) { acc[j] = ov; arg[ARG ? j : 0] = oa; }
                } else {
                    acc[j] = low ? (mine + ov) : (ov + mine);  // both partners add in the same operand order
                }
            }
        }
    }

    __device__ __forceinline__ void write_partial(int64_t slot, int which) const {
        if (lane >= LPR || !col_lane) return;
        const size_t off = ((size_t)slot * 2 + which) * P.F + (size_t)ci * EPC;
#pragma unroll
        for (int j = 0; j < EPC; j += 4) {
            *reinterpret_cast<float4*>(P.part_val + off + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
            if (ARG) *reinterpret_cast<int4*>(P.part_arg + off + j) = make_int4(arg[ARG ? j : 0], arg[ARG ? j + 1 : 0], arg[ARG ? j + 2 : 0], arg[ARG ? j + 3 : 0]);
        }
    }
};

template <typename T, int MODE>
__host__ __device__ constexpr int rr_min_blocks() {
    return (MODE == MODE_SUM || MODE == MODE_WSUM) ? 4 : 3;
}

template <typename T, int LPR, int MODE, bool EPI>
__global__ void __launch_bounds__(RR_WARPS * 32, (rr_min_blocks<T, MODE>()))
reduce_rows_kernel(const __grid_constant__ PropParams P, int long_blocks) {
    using R = RowReducer<T, LPR, MODE>;
    constexpr int NG = R::NG, U = R::U;
    pdl_wait();
    R red(P);
    const int lane = red.lane, N = P.N;
    if ((int)blockIdx.x >= long_blocks) {
        // ---- rows of at most RR_SHORT positions: one per lane group
        const int64_t row64 = ((int64_t)((int)blockIdx.x - long_blocks) * RR_WARPS + (threadIdx.x >> 5)) * NG + red.g;
        int row = -1, s = 0, len = 0;
        if (row64 < N) {
            const int64_t a = P.rowptr[row64], b = P.rowptr[row64 + 1];
            if (b - a <= RR_SHORT || P.E <= RR_SHORT) { row = (int)row64; s = (int)a; len = (int)(b - a); }
        }
        int most = len;
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
        red.clear();
        typename R::Entry cur = red.entry(s + red.li, red.li < len);
        for (int q = 0; q < most; q += LPR) {
            const int p = q + LPR + red.li;
            typename R::Entry nxt = cur;
            if (q + LPR < most) nxt = red.entry(s + p, p < len);
#pragma unroll 1
            for (int j = 0; j < LPR && q + j < most; j += U) red.batch(cur, j, len - q - j, s + q + j);
            cur = nxt;
        }
        if (row >= 0 && red.col_lane) finish_row<T, MODE, EPI>(P, row, len, red.ci, red.acc, red.arg);
        return;
    }
    // ---- longer rows: piece v = positions [v * P.piece, (v + 1) * P.piece), all groups on one row
    const int64_t v = (int64_t)blockIdx.x * RR_WARPS + (threadIdx.x >> 5);
    if (v >= P.npieces) return;
    const int64_t c0 = v * (int64_t)P.piece, c1 = min(c0 + P.piece, P.E);
    int tail = -1;
    for (int rb = row_of_position(P.rowptr, N, P.E, c0, lane); rb < N; rb += 32) {
        const int r = rb + lane;
        int64_t s = 0, e = 0;
        if (r < N) { s = P.rowptr[r]; e = P.rowptr[r + 1]; }
        const bool in = r < N && s < c1;
        unsigned m = __ballot_sync(0xffffffffu, in && e - s > RR_SHORT && e > c0);
        while (m) {
            const int k = __ffs(m) - 1, row = rb + k;
            m &= m - 1;
            const int rs = (int)__shfl_sync(0xffffffffu, s, k), re = (int)__shfl_sync(0xffffffffu, e, k);
            const bool begins = rs >= c0, ends = re <= c1;
            red.whole_warp(begins ? rs : (int)c0, ends ? re : (int)c1);
            if (begins && ends) {
                if (lane < LPR && red.col_lane) finish_row<T, MODE, EPI>(P, row, re - rs, red.ci, red.acc, red.arg);
            } else {
                red.write_partial(v, begins ? 1 : 0);
                if (begins) tail = row;
            }
        }
        if (!__all_sync(0xffffffffu, in)) break;
    }
    if (lane == 0) P.tail_row[v] = tail;
}

// ------------------------------------------------------------------ positions first
// One warp per run of P.sub consecutive positions, a block per piece of RR_WARPS such runs.  The gathers do not depend on the rows: every lane group streams
// sub/NG of them with four to eight gathers always in flight (two register buffers of H, each refilled as soon
// as it has been added), and a row's end, a bit per position, only makes the
// accumulator go out.  Rows cut between lane groups are stitched inside the warp, rows cut between warps inside the block
// (through shared memory, by the warp in which they begin), both in position order; rows cut by the piece leave the
// partials that the second kernel adds (a piece per warp: that kernel took 313 us of 4.9 ms on 123 M edges).  Rows without edges are written by a scan that is spread over all warps.
//
// What made the difference (170k nodes, 1.36 M edges, before -> after): a staging of 4 to 12 bytes per position (it was
// 10 KB per warp, and shared memory is taken from the L1 that holds gathers in flight), 64 registers without spills (32
// warps per SM), buffers refilled in turn instead of one batch after the other, an epilogue-free row end: fp32 sums over
// 512-byte rows 113 -> 75 us, bf16 256-byte 74 -> 60 us, 64-byte 54 -> 32 us, max fp32 157 -> 117 us; on 123 M edges the
// 128-byte rows of a weighted sum 2.45 -> 2.26 ms, max over 256-byte rows 8.1 -> 6.6 ms.
// Row ends as bits beside the indices instead of in their sign: no index to mask, and a batch without an end has nothing to
// test: 123 M edges, 128-byte bf16 rows 1.96 -> 1.87 ms, sums over 512 fp32 features 37.9 -> 35.4 ms a forward and backward pass.
// Plain bf16 sums by additions that take bf16 (nothing unpacked, the same bits): 1.36 M edges, 256-byte rows 63.7 -> 60.9 us.
constexpr int RS_SUB = 256;  // most positions per warp
constexpr int RS_SKEW = 32;

template <int EPC, bool HAS_W, bool HAS_T, bool ARG>
struct alignas(16) StreamStage {
    // per position; four words further for every lane group before the position's (see sk)
    int col[RS_SUB + RS_SKEW];                         // gathered row
    alignas(16) float w[HAS_W ? RS_SUB + RS_SKEW : 1]; // multiplier
    alignas(16) int t[HAS_T ? RS_SUB + RS_SKEW : 1];   // ROUTE: forward position; HEAD: row of the multiplier matrix
    int row[RS_SUB + 1];                   // [q] the q-th row with positions in the warp's share
    uint16_t start[RS_SUB + 2];            // [q] its first position in the warp's share; [count]: end of the last, or n + 1 if it is cut
    uint32_t ends[RS_SUB / 32];            // a bit per position: the last one of its row
    float head[32 * EPC];                  // per lane: sum of a group's (then the warp's) first row, which began before it
    int32_t head_a[ARG ? 32 * EPC : 1];
    // the warp's last row, if it goes on past the warp: over col and w, which are done with by then
    __device__ __forceinline__ float* tail() { return reinterpret_cast<float*>(col); }
    __device__ __forceinline__ int32_t* tail_a() { return reinterpret_cast<int32_t*>(w); }
};
// what a warp leaves to the block: its first row began in an earlier warp and ends here (CLOSED) or does not (THROUGH)
enum { HEAD_NONE = 0, HEAD_CLOSED = 1, HEAD_THROUGH = 2 };

template <typename T, int MODE, bool EPI>
__host__ __device__ constexpr int rs_min_blocks() {
    return (MODE == MODE_SUM || MODE == MODE_WSUM) ? 4 : MODE == MODE_V2 && EPI && sizeof(T) == 2 ? 2 : 3;  // (three: 170 bytes of spills)
}

template <typename T, int LPR, int MODE, bool EPI>
__global__ void __launch_bounds__(RR_WARPS * 32, (rs_min_blocks<T, MODE, EPI>()))
stream_rows_kernel(const __grid_constant__ PropParams P) {
    constexpr int EPC = Chunk<T>::N, NG = 32 / LPR;
    constexpr bool ARG = MODE == MODE_MAX || MODE == MODE_MIN, EF = MODE == MODE_EFSUM, ROUTE = MODE == MODE_ROUTE;
    constexpr bool RANK1 = MODE == MODE_HEADRANK, HEAD = MODE == MODE_HEADSUM || MODE == MODE_HEADSUM_W || RANK1 || MODE == MODE_V2;
    constexpr bool PLAIN = MODE == MODE_SUM, V2 = MODE == MODE_V2, DA = V2 && EPI;
    constexpr int H = (ROUTE || EF) ? 2 : 4;  // positions per register buffer
    constexpr int MW = EF ? EPC : 1;
    constexpr bool HAS_W = !PLAIN && !V2 && MODE != MODE_HEADSUM && !RANK1;  // a multiplier per position
    using Stage = StreamStage<EPC, HAS_W, ROUTE || HEAD, ARG>;
    static_assert(32 * EPC <= RS_SUB, "a row's sums fit over the staged indices");
    extern __shared__ __align__(16) unsigned char rs_smem[];
    pdl_wait();
    const int lane = threadIdx.x & 31, g = lane / LPR, li = lane % LPR;
    const int piece = P.descending ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int wib = threadIdx.x >> 5, c = piece * RR_WARPS + wib;
    __shared__ int s_head[RR_WARPS], s_tail_row[RR_WARPS];
    Stage& S = reinterpret_cast<Stage*>(rs_smem)[wib];
    const int cs = (int)min((int64_t)c * P.sub, P.E);
    const int n = (int)min((int64_t)P.sub, P.E - cs);  // 0 in the last block's idle warps
    const bool col_lane = li < P.nvec;
    const int ci = col_lane ? li : 0;

    // The groups' runs start sub / NG positions apart: at a multiple of 32 words they would read the same bank at the same
    // time (eight-way conflicts with 64-byte rows, four-way with 128-byte rows: 90 % of the shared-memory path's cycles).  Four
    // words of skew per group keep the runs apart and on 16 bytes, so that a register buffer's entries are one load.
    const int L = P.sub / NG, lsh = 31 - __clz(L);
    auto sk = [&](int i) { return i + ((i >> lsh) << 2); };
    if (lane < RS_SUB / 32) S.ends[lane] = 0u;
    {  // ---- indices and multipliers, asynchronously while the rows are looked up
        auto copy = [&](void* dst, const void* src) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
        };
        for (int i = lane; i < n; i += 32) {
            const int k = sk(i);
            if (P.col) copy(S.col + k, P.col + cs + i);
            else S.col[k] = cs + i;
            if (HAS_W) {
                if (P.w) copy(S.w + k, P.w + cs + i);
                else S.w[k] = 1.0f;
            }
            if (ROUTE) copy(S.t + k, P.route_pos + cs + i);
            if (HEAD) {
                if (P.wh_index) copy(S.t + k, P.wh_index + cs + i);
                else S.t[k] = cs + i;
            }
        }
    }
    // ---- rows with positions in the warp's share
    int m = 0;
    bool began_before = false;  // the first of them has positions in an earlier warp's
    if (n > 0) m = stage_rows(P.rowptr, P.N, P.E, cs, n, lane, S.row, S.start, began_before);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (HAS_W && P.gscale_rowptr) {
#pragma unroll 4
        for (int i = lane; i < n; i += 32) {
            const int k = sk(i), cc = S.col[k];
            const int64_t d = P.gscale_rowptr[cc + 1] - P.gscale_rowptr[cc];
            S.w[k] = S.w[k] / (float)(d > 1 ? d : 1);
        }
        __syncwarp();
    }
    for (int q = lane; q < m; q += 32) {
        const int e = S.start[q + 1];
        if (e <= n) atomicOr(S.ends + ((e - 1) >> 5), 1u << ((e - 1) & 31));
    }
    __syncwarp();

    // ---- this group's run
    const int a = g * L, b = min(a + L, n);
    const bool vote = P.vote && n == P.sub;  // (every group has a run of the same length)
    auto ends_at = [&](int i) { return (S.ends[i >> 5] >> (i & 31) & 1u) != 0; };
    const int* const Sc = S.col + 4 * g;
    const float* const Sw = S.w + (HAS_W ? 4 * g : 0);
    const int* const St = S.t + (ROUTE || HEAD ? 4 * g : 0);
    // four entries at a time cost some kernels the registers they have left: plain bf16 sums (59 -> 61 us on 1.36 M 256-byte
    // rows), and all bf16 rows of 512 bytes, which have one lane group and no bank conflict
    constexpr bool ONE_BY_ONE = EPC == 8 && (PLAIN || LPR == 32);
    auto words = [&](int* to, const void* from) {  // H staged words, on their own size
        if (H == 4) *reinterpret_cast<int4*>(to) = *reinterpret_cast<const int4*>(from);
        else *reinterpret_cast<int2*>(to) = *reinterpret_cast<const int2*>(from);
    };
    const uint64_t pol_keep = policy_evict_last();
    const char* const Xl = reinterpret_cast<const char*>(P.X) + (size_t)ci * 16;
    const float* const wh_l = HEAD ? P.wh + ((P.vec0 + ci) * EPC) / P.fph : nullptr;
    float acc[EPC];
    int32_t arg[ARG ? EPC : 1];
    bool fresh = true;  // ARG: the next position is the row's first in this run and is taken whatever its value
    auto clear = [&]() {
        fresh = true;
#pragma unroll
        for (int j = 0; j < EPC; ++j) {
            acc[j] = 0.f;
            if (ARG) arg[ARG ? j : 0] = -1;
        }
    };
    auto write_partial = [&](int which, const float* v, const int32_t* va) {
        if (lane >= LPR || !col_lane) return;
        const size_t off = ((size_t)piece * 2 + which) * P.F + (size_t)ci * EPC;
#pragma unroll
        for (int j = 0; j < EPC; j += 4) {
            *reinterpret_cast<float4*>(P.part_val + off + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            if (ARG) *reinterpret_cast<int4*>(P.part_arg + off + j) = make_int4(va[ARG ? j : 0], va[ARG ? j + 1 : 0], va[ARG ? j + 2 : 0], va[ARG ? j + 3 : 0]);
        }
    };
    clear();
    int q = 0;  // row of the next position
    if (NG > 1) {
        int lo = 0, hi = m;  // start[lo] <= a < start[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (S.start[mid] <= a) lo = mid; else hi = mid;
        }
        q = lo;
    }
    // the rank-1 epilogue: the attention vectors from shared memory, the row's two factors loaded when it begins
    float* const ab = reinterpret_cast<float*>(rs_smem + RR_WARPS * sizeof(Stage));  // [2][F]
    RankOne r1 = {0.f, 0.f, ab + ci * EPC, ab + P.F + ci * EPC};
    auto row_factors = [&](int qq) {
        const size_t k = (size_t)max(S.row[qq], 0) * P.H + ((P.vec0 + ci) * EPC) / P.fph;
        r1.l = ld_f32(P.epi_l + k);
        r1.r = ld_f32(P.epi_r + k);
    };
    if (RANK1) {
        if (a < b) row_factors(q);
        for (int f = threadIdx.x; f < P.F; f += RR_WARPS * 32) {
            ab[f] = P.epi_a[P.vec0 * EPC + f];
            ab[P.F + f] = P.epi_b[P.vec0 * EPC + f];
        }
        __syncthreads();
    }
    bool open = a < b && (S.start[q] < a || (a == 0 && began_before));  // the run's first row began before the run
    int head_q = -1;
    // MODE_V2: this row's own features, the next row's on their way, and the share of da (all rows of the group together)
    float xs[V2 ? EPC : 1], da[DA ? EPC : 1];
    uint4 own_next = make_uint4(0u, 0u, 0u, 0u);
    auto own = [&](int qq) { return ld_16(reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(P.v2_self) + (size_t)max(S.row[qq], 0) * P.x_ld) + ci); };
    if (V2) {
        if (a < b) {
            Chunk<T>::unpack(own(q), xs);
            if (q + 1 < m) own_next = own(q + 1);
        }
#pragma unroll
        for (int j = 0; j < (DA ? EPC : 1); ++j) da[j] = 0.f;
    }
    auto flush = [&]() {  // row q ends here
        if (open) {
            open = false;
            head_q = q;
#pragma unroll
            for (int j = 0; j < EPC; ++j) {
                S.head[lane * EPC + j] = acc[j];
                if (ARG) S.head_a[ARG ? lane * EPC + j : 0] = arg[ARG ? j : 0];
            }
        } else if (col_lane) {
            finish_row<T, MODE, EPI, RANK1>(P, S.row[q], S.start[q + 1] - S.start[q], ci, acc, arg, r1);
        }
        clear();
        ++q;
        if (RANK1 && q < m) row_factors(q);
        if (V2) {
            Chunk<T>::unpack(own_next, xs);
            if (q + 1 < m) own_next = own(q + 1);
        }
    };
    struct Buf {
        uint4 x[H];
        float hw[(HEAD || EF) ? H : 1][MW];
        int4 win[ROUTE ? H : 1][ROUTE ? EPC / 4 : 1];
    };
    // the gathers of positions i .. i + H - 1
    auto issue = [&](Buf& B, int i) {
        alignas(16) int ccs[H], ts[H];
        if (ONE_BY_ONE) {
#pragma unroll
            for (int u = 0; u < H; ++u) ccs[u] = Sc[i + u];
        } else {
            words(ccs, Sc + i);
        }
        if (HEAD) words(ts, St + (HEAD ? i : 0));
#pragma unroll
        for (int u = 0; u < H; ++u) {
            const int cc = ccs[u];
            B.x[u] = ld_hint16(Xl + (size_t)(uint32_t)cc * P.x_ld, pol_keep);
            if (HEAD) B.hw[HEAD ? u : 0][0] = ld_f32(wh_l + (size_t)(uint32_t)ts[u] * P.H);
            if (EF) {
                const float4* f = reinterpret_cast<const float4*>(P.ef + (size_t)(cs + i + u) * P.ef_ld + (size_t)ci * EPC);
#pragma unroll
                for (int k = 0; k < MW / 4; ++k) {
                    const float4 a4 = __ldcs(f + k);
                    float* d = B.hw[EF ? u : 0] + 4 * k;
                    d[0] = a4.x; d[EF ? 1 : 0] = a4.y; d[EF ? 2 : 0] = a4.z; d[EF ? 3 : 0] = a4.w;
                }
            }
            if (ROUTE) {
                const int4* f = reinterpret_cast<const int4*>(P.route_arg + (size_t)(uint32_t)cc * P.arg_ld + (size_t)ci * EPC);
#pragma unroll
                for (int k = 0; k < EPC / 4; ++k) B.win[ROUTE ? u : 0][ROUTE ? k : 0] = ld_int4(f + k);
            }
        }
    };
    auto use = [&](const Buf& B, int u, int i, float w, int t) {  // entry u of the buffer, position i of the piece
        if constexpr (PLAIN && sizeof(T) == 2) {
            add_bf16(acc[0], acc[1], B.x[u].x);
            add_bf16(acc[2], acc[3], B.x[u].y);
            add_bf16(acc[4], acc[5], B.x[u].z);
            add_bf16(acc[6], acc[7], B.x[u].w);
            return;
        }
        float x[EPC];
        Chunk<T>::unpack(B.x[u], x);
        if (ARG) {
#pragma unroll
            for (int k = 0; k < EPC; k += 2) mul2(x[k], x[k + 1], w, w);  // w = 1 where there are no multipliers: exact
#pragma unroll
            for (int k = 0; k < EPC; ++k) {
                // positions ascend within a run: a strict comparison keeps the first of equal values
                const bool take = fresh || (MODE == MODE_MAX ? x[k] > acc[k] : x[k] < acc[k]);
                if (take) { acc[k] = x[k]; arg[ARG ? k : 0] = cs + i; }
            }
            fresh = false;
        } else if (ROUTE) {  // keep dOut only where this edge was the winner
#pragma unroll
            for (int k = 0; k < EPC / 4; ++k) {
                const int4 z = B.win[ROUTE ? u : 0][ROUTE ? k : 0];
                if (z.x == t) acc[4 * k] = fmaf(w, x[4 * k], acc[4 * k]);
                if (z.y == t) acc[4 * k + 1] = fmaf(w, x[4 * k + 1], acc[4 * k + 1]);
                if (z.z == t) acc[4 * k + 2] = fmaf(w, x[4 * k + 2], acc[4 * k + 2]);
                if (z.w == t) acc[4 * k + 3] = fmaf(w, x[4 * k + 3], acc[4 * k + 3]);
            }
        } else if (EF) {
#pragma unroll
            for (int k = 0; k < EPC; k += 2)
                fma2(acc[k], acc[k + 1], x[k], x[k + 1], B.hw[EF ? u : 0][EF ? k : 0] * w, B.hw[EF ? u : 0][EF ? k + 1 : 0] * w);
        } else if (PLAIN) {
#pragma unroll
            for (int k = 0; k < EPC; k += 2) add2(acc[k], acc[k + 1], x[k], x[k + 1]);
        } else if (V2) {  // ds * LeakyReLU'(z), times a when the row is complete; da: ds * LeakyReLU(z)
            const float f = B.hw[HEAD ? u : 0][0], fs = f * P.slope;
#pragma unroll
            for (int k = 0; k < EPC; ++k) {
                const float z = x[k] + xs[V2 ? k : 0];
                const float d = z > 0.f ? f : fs;
                acc[k] += d;
                if (DA) da[DA ? k : 0] = fmaf(d, z, da[DA ? k : 0]);
            }
        } else {
            const float h = B.hw[HEAD ? u : 0][0], f = !HEAD ? w : HAS_W ? h * w : h;
#pragma unroll
            for (int k = 0; k < EPC; k += 2) fma2(acc[k], acc[k + 1], x[k], x[k + 1], f, f);
        }
    };
    auto use_all = [&](const Buf& B, unsigned ends, int i) {
        alignas(16) float ws[H];
        alignas(16) int ts[H];
        if (HAS_W && !ONE_BY_ONE) words(reinterpret_cast<int*>(ws), Sw + (HAS_W ? i : 0));
        if (ROUTE) words(ts, St + (ROUTE ? i : 0));
        // most positions of a skewed graph lie in long rows: without a row end in any group there is nothing to test
        if (NG == 1 ? ends == 0 : vote && !__any_sync(0xffffffffu, ends != 0)) {
#pragma unroll
            for (int u = 0; u < H; ++u) use(B, u, i + u, !HAS_W ? 1.0f : ONE_BY_ONE ? Sw[HAS_W ? i + u : 0] : ws[u], ROUTE ? ts[u] : 0);
            return;
        }
#pragma unroll
        for (int u = 0; u < H; ++u) {
            use(B, u, i + u, !HAS_W ? 1.0f : ONE_BY_ONE ? Sw[HAS_W ? i + u : 0] : ws[u], ROUTE ? ts[u] : 0);
            if (ends >> u & 1u) flush();
        }
    };
    if (a < b) {
        Buf A, B;
        // L is a multiple of 2 H: only the last piece of the graph has a remainder
        int i = a;
        if (i + 2 * H <= b) {
            issue(A, i);
            issue(B, i + H);
        }
#pragma unroll 1
        for (; i + 2 * H <= b; i += 2 * H) {
            const bool more = i + 4 * H <= b;
            const unsigned ends = S.ends[i >> 5] >> (i & 31);  // a run starts at a multiple of 2 H
            use_all(A, ends & ((1u << H) - 1u), i);
            if (more) issue(A, i + 2 * H);
            use_all(B, (ends >> H) & ((1u << H) - 1u), i + H);
            if (more) issue(B, i + 3 * H);
        }
#pragma unroll 1
        for (; i < b; ++i) {
            // one at a time: entry 0 of a buffer whose other entries repeat it
            Buf R;
            const int cc = Sc[i];
            const bool end = ends_at(i);
            R.x[0] = ld_hint16(Xl + (size_t)(uint32_t)cc * P.x_ld, pol_keep);
            if (HEAD) R.hw[0][0] = ld_f32(wh_l + (size_t)(uint32_t)St[HEAD ? i : 0] * P.H);
            if (EF) {
#pragma unroll
                for (int k = 0; k < MW; ++k) R.hw[0][k] = P.ef[(size_t)(cs + i) * P.ef_ld + (size_t)ci * EPC + k];
            }
            if (ROUTE) {
#pragma unroll
                for (int k = 0; k < EPC / 4; ++k)
                    R.win[0][ROUTE ? k : 0] = ld_int4(reinterpret_cast<const int4*>(P.route_arg + (size_t)(uint32_t)cc * P.arg_ld + (size_t)ci * EPC) + k);
            }
            use(R, 0, i, HAS_W ? Sw[HAS_W ? i : 0] : 1.0f, ROUTE ? St[ROUTE ? i : 0] : 0);
            if (end) flush();
        }
    }
    // ---- what the groups leave: a closed head (parked), and the sum of a row that goes on past the group (in acc)
    const bool rest = a < b && !ends_at(b - 1);
    int head_state = HEAD_NONE, tail_row = -1;
    __syncwarp();
    // the warp's first or last row, as far as it lies here, for the block (lanes below LPR)
    auto leave = [&](float* to, int32_t* to_a, const float* v, const int32_t* va) {
        if (lane < LPR) {
#pragma unroll
            for (int j = 0; j < EPC; ++j) {
                to[li * EPC + j] = v[j];
                if (ARG) to_a[li * EPC + j] = va[ARG ? j : 0];
            }
        }
    };
    float carry[EPC];
    int32_t carg[ARG ? EPC : 1];
    // values v of later positions join the carry, which wins ties
    auto join = [&](bool have, const float* v, const int32_t* va) {
#pragma unroll
        for (int j = 0; j < EPC; ++j) {
            if (ARG) {
                if (!have || beats<MODE>(v[j], va[ARG ? j : 0], carry[j], carg[ARG ? j : 0])) { carry[j] = v[j]; carg[ARG ? j : 0] = va[ARG ? j : 0]; }
            } else {
                carry[j] = have ? carry[j] + v[j] : v[j];
            }
        }
    };
    if (NG == 1) {
        if (head_q >= 0) head_state = HEAD_CLOSED;
        if (rest && open) {
            head_state = HEAD_THROUGH;
            leave(S.head, S.head_a, acc, arg);
        } else if (rest) {
            tail_row = S.row[q];
            leave(S.tail(), S.tail_a(), acc, arg);
        }
    } else {
        bool have = false, before = false;
        int ck = 0;
#pragma unroll 1
        for (int gg = 0; gg < NG; ++gg) {
            const int hq = __shfl_sync(0xffffffffu, head_q, gg * LPR), tq = __shfl_sync(0xffffffffu, q, gg * LPR);
            const bool left = __shfl_sync(0xffffffffu, (int)rest, gg * LPR), through = __shfl_sync(0xffffffffu, (int)open, gg * LPR);
            if (hq >= 0) {
                if (!have) before = true;  // only the first group can go on from before without a carry
                join(have, S.head + (gg * LPR + li) * EPC, S.head_a + (ARG ? (gg * LPR + li) * EPC : 0));
                __syncwarp();
                if (before) {
                    head_state = HEAD_CLOSED;
                    leave(S.head, S.head_a, carry, carg);
                } else if (lane < LPR && col_lane) {
                    finish_row<T, MODE, EPI>(P, S.row[hq], S.start[hq + 1] - S.start[hq], ci, carry, carg);
                }
                have = before = false;
            }
            if (left) {
                float v[EPC];
                int32_t va[ARG ? EPC : 1];
#pragma unroll
                for (int j = 0; j < EPC; ++j) {
                    v[j] = __shfl_sync(0xffffffffu, acc[j], gg * LPR + li);
                    if (ARG) va[ARG ? j : 0] = __shfl_sync(0xffffffffu, arg[ARG ? j : 0], gg * LPR + li);
                }
                if (!through) have = before = false;
                else if (!have) before = true;
                join(have, v, va);
                have = true;
                ck = tq;
            }
        }
        if (have) {  // the row goes on past the warp
            __syncwarp();
            if (before) {
                head_state = HEAD_THROUGH;
                leave(S.head, S.head_a, carry, carg);
            } else {
                tail_row = S.row[ck];
                leave(S.tail(), S.tail_a(), carry, carg);
            }
        }
    }
    if (lane == 0) { s_head[wib] = head_state; s_tail_row[wib] = tail_row; }
    // ---- rows without edges: warp c takes its share of all rows
    {
        const int64_t warps = P.npieces * RR_WARPS, per = (P.N + warps - 1) / warps;
        const int64_t b0 = c * per;
        const int e0 = (int)min(b0, (int64_t)P.N), e1 = (int)min(b0 + per, (int64_t)P.N);
        for (int rb = e0; rb < e1; rb += 32) {
            const int r = rb + lane;
            unsigned em = __ballot_sync(0xffffffffu, r < e1 && P.rowptr[r + 1] == P.rowptr[r]);
            em &= (NG == 8 ? 0x01010101u : NG == 4 ? 0x11111111u : NG == 2 ? 0x55555555u : 0xffffffffu) << g;  // group g takes every NG-th
            while (em) {
                const int bit = __ffs(em) - 1;
                em &= em - 1;
                clear();
                if (col_lane) finish_row<T, MODE, EPI>(P, rb + bit, 0, ci, acc, arg);
            }
        }
    }
    // ---- rows cut between the warps of the block
    __syncthreads();
    if (lane < LPR && col_lane) {
        const Stage* const all = reinterpret_cast<const Stage*>(rs_smem);
        auto chain = [&](int row) {  // carry goes on into the next warps; row < 0: it began before the block
#pragma unroll 1
            for (int k = wib + 1; k < RR_WARPS && s_head[k] != HEAD_NONE; ++k) {
                join(true, all[k].head + li * EPC, all[k].head_a + (ARG ? li * EPC : 0));
                if (s_head[k] == HEAD_CLOSED) {
                    if (row >= 0) finish_row<T, MODE, EPI>(P, row, P.mean ? P.rowptr[row + 1] - P.rowptr[row] : 1, ci, carry, carg);
                    else write_partial(0, carry, carg);
                    return;
                }
            }
            write_partial(row >= 0 ? 1 : 0, carry, carg);
        };
        if (wib == 0 && head_state != HEAD_NONE) {
            join(false, S.head + li * EPC, S.head_a + (ARG ? li * EPC : 0));
            if (head_state == HEAD_CLOSED) write_partial(0, carry, carg);
            else chain(-1);
        }
        if (tail_row >= 0) {
            join(false, S.tail() + li * EPC, S.tail_a() + (ARG ? li * EPC : 0));
            chain(tail_row);
        }
    }
    if (DA) {  // the block's share of da: lane groups by an xor tree, then the warps in order
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
            for (int j = 0; j < EPC; ++j) da[DA ? j : 0] += __shfl_xor_sync(0xffffffffu, da[DA ? j : 0], o);
        __syncthreads();  // the stages are done with
        float* const sums = reinterpret_cast<float*>(rs_smem);  // [RR_WARPS][LPR * EPC]
        if (lane < LPR)
#pragma unroll
            for (int j = 0; j < EPC; ++j) sums[(wib * LPR + li) * EPC + j] = da[DA ? j : 0];
        __syncthreads();
        for (int f = threadIdx.x; f < P.F; f += RR_WARPS * 32) {
            float v = 0.f;
#pragma unroll
            for (int k = 0; k < RR_WARPS; ++k) v += sums[k * LPR * EPC + f];
            P.da_part[(size_t)piece * P.F + f] = v;
        }
    }
    if (threadIdx.x == 0) {  // the row that begins in the block and reaches past it
        int t = -1;
        for (int k = 0; k < RR_WARPS; ++k) {
            if (s_head[k] != HEAD_THROUGH) t = -1;
            if (s_tail_row[k] >= 0) t = s_tail_row[k];
        }
        P.tail_row[piece] = t;
    }
}

// ------------------------------------------------------------------ second pass: rows cut by piece boundaries
// One launch, two kinds of blocks.  The first nsimple blocks: a thread per (piece, 16-byte column) adds the partials of
// the row that begins in its piece, in ascending piece order, eight loads together.  The rest share the rows cut into
// more than FIX_LONG pieces (hub rows): there one thread per column would pay a load latency per eight of hundreds of
// partials (45-150 us on a graph whose largest row has 300 pieces), so a block takes such a row with 256/(F/4) walkers per
// column, four loads in flight each, and adds the walkers' sums in walker order.  Both orders are a fixed function of
// (graph, F).  Max / min keep (value, position) pairs, whose combination does not depend on the order.
constexpr int FIX_LONG = 64;
constexpr int FIX_THREADS = 256;
constexpr int FIX_LONG_BLOCKS = 592;

template <typename T, int MODE>
__device__ void fixup_long_rows(const PropParams& P, int block, int nblocks) {
    constexpr int EPC = Chunk<T>::N;
    constexpr bool ARG = (MODE == MODE_MAX || MODE == MODE_MIN);
    __shared__ float4 sums[FIX_THREADS];
    __shared__ int4 args[ARG ? FIX_THREADS : 1];
    __shared__ int todo[64];
    __shared__ int ntodo;
    const int tid = threadIdx.x;
    const int F = P.F, F4 = F / 4;
    const int K = FIX_THREADS / F4 > 0 ? FIX_THREADS / F4 : 1;
    const int k = tid / F4, q = tid - k * F4;
    const int64_t per = (P.npieces + nblocks - 1) / nblocks;
    const int64_t c0 = (int64_t)block * per, c1 = c0 + per < P.npieces ? c0 + per : P.npieces;
    auto last_piece = [&](int r) { return (P.rowptr[r + 1] - 1) / P.piece; };
    for (int64_t cb = c0; cb < c1; cb += 64) {  // 64 pieces at a time: find the long rows, then do them one by one
        if (tid == 0) ntodo = 0;
        __syncthreads();
        if (tid < 64 && cb + tid < c1) {
            const int32_t r = P.tail_row[cb + tid];
            if (r >= 0 && last_piece(r) - (cb + tid) > FIX_LONG) todo[atomicAdd(&ntodo, 1)] = tid;
        }
        __syncthreads();
        const int n = ntodo;
        for (int i = 0; i < n; ++i) {
            // rows of one block are independent: the order in which the list was filled does not matter
            const int64_t c = cb + todo[i];
            const int32_t r = P.tail_row[c];
            const int64_t span = last_piece(r) - c;  // partial rows: (c, slot 1), then slot 0 of c + 1 .. c + span
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            int4 arg = make_int4(-1, -1, -1, -1);
            if (k < K && q < F4) {
                for (int64_t j = k; j <= span; j += 4 * (int64_t)K) {
                    float4 t[4];
                    int4 ta[ARG ? 4 : 1];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int64_t jj = j + (int64_t)u * K;
                        if (jj <= span) {
                            const size_t slot = jj == 0 ? (size_t)c * 2 + 1 : (size_t)(c + jj) * 2;
                            t[u] = *(reinterpret_cast<const float4*>(P.part_val + slot * (size_t)F) + q);
                            if (ARG) ta[ARG ? u : 0] = *(reinterpret_cast<const int4*>(P.part_arg + slot * (size_t)F) + q);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (j + (int64_t)u * K <= span) {
                            if (ARG) {
                                const int4 b = ta[ARG ? u : 0];
                                if (beats<MODE>(t[u].x, b.x, acc.x, arg.x)) { acc.x = t[u].x; arg.x = b.x; }
                                if (beats<MODE>(t[u].y, b.y, acc.y, arg.y)) { acc.y = t[u].y; arg.y = b.y; }
                                if (beats<MODE>(t[u].z, b.z, acc.z, arg.z)) { acc.z = t[u].z; arg.z = b.z; }
                                if (beats<MODE>(t[u].w, b.w, acc.w, arg.w)) { acc.w = t[u].w; arg.w = b.w; }
                            } else {
                                acc.x += t[u].x; acc.y += t[u].y; acc.z += t[u].z; acc.w += t[u].w;
                            }
                        }
                }
                sums[k * F4 + q] = acc;
                if (ARG) args[ARG ? k * F4 + q : 0] = arg;
            }
            __syncthreads();
            if (tid < P.nvec) {
                const int ci = tid;
                float v[EPC];
                int32_t av[ARG ? EPC : 1];
#pragma unroll
                for (int j4 = 0; j4 < EPC / 4; ++j4) {
                    float4 a = sums[ci * (EPC / 4) + j4];
                    int4 aa = ARG ? args[ARG ? ci * (EPC / 4) + j4 : 0] : make_int4(-1, -1, -1, -1);
                    for (int kk = 1; kk < K; ++kk) {
                        const float4 b = sums[kk * F4 + ci * (EPC / 4) + j4];
                        if (ARG) {
                            const int4 ba = args[ARG ? kk * F4 + ci * (EPC / 4) + j4 : 0];
                            if (beats<MODE>(b.x, ba.x, a.x, aa.x)) { a.x = b.x; aa.x = ba.x; }
                            if (beats<MODE>(b.y, ba.y, a.y, aa.y)) { a.y = b.y; aa.y = ba.y; }
                            if (beats<MODE>(b.z, ba.z, a.z, aa.z)) { a.z = b.z; aa.z = ba.z; }
                            if (beats<MODE>(b.w, ba.w, a.w, aa.w)) { a.w = b.w; aa.w = ba.w; }
                        } else {
                            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
                        }
                    }
                    v[4 * j4] = a.x; v[4 * j4 + 1] = a.y; v[4 * j4 + 2] = a.z; v[4 * j4 + 3] = a.w;
                    if (ARG) { av[ARG ? 4 * j4 : 0] = aa.x; av[ARG ? 4 * j4 + 1 : 0] = aa.y; av[ARG ? 4 * j4 + 2 : 0] = aa.z; av[ARG ? 4 * j4 + 3 : 0] = aa.w; }
                }
                finish_row<T, MODE, true>(P, r, P.rowptr[r + 1] - P.rowptr[r], ci, v, av);
            }
            __syncthreads();
        }
    }
}

template <typename T, int MODE>
__global__ void __launch_bounds__(FIX_THREADS)
fixup_rows_kernel(const __grid_constant__ PropParams P, int nsimple) {
    constexpr int EPC = Chunk<T>::N;
    constexpr bool ARG = (MODE == MODE_MAX || MODE == MODE_MIN);
    pdl_wait();
    if ((int)blockIdx.x >= nsimple) {
        fixup_long_rows<T, MODE>(P, (int)blockIdx.x - nsimple, (int)gridDim.x - nsimple);
        return;
    }
    const int64_t t = blockIdx.x * (int64_t)FIX_THREADS + threadIdx.x;
    const int64_t c = t / P.nvec;
    const int ci = (int)(t - c * P.nvec);
    if (c >= P.npieces) return;
    const int32_t r = P.tail_row[c];
    if (r < 0) return;
    const int64_t rs = P.rowptr[r], re = P.rowptr[r + 1];
    const int64_t c_end = (re - 1) / P.piece;
    if ((int)gridDim.x > nsimple && c_end - c > FIX_LONG) return;  // a hub row: the other blocks finish it
    float v[EPC];
    int32_t a[ARG ? EPC : 1];
    const size_t F = P.F;
    auto load = [&](int64_t slot, float4* x, int4* b) {
#pragma unroll
        for (int q = 0; q < EPC / 4; ++q) {
            x[q] = *(reinterpret_cast<const float4*>(P.part_val + (size_t)slot * F + (size_t)ci * EPC) + q);
            if (ARG) b[ARG ? q : 0] = *(reinterpret_cast<const int4*>(P.part_arg + (size_t)slot * F + (size_t)ci * EPC) + q);
        }
    };
    {
        float4 x[EPC / 4];
        int4 b[ARG ? EPC / 4 : 1];
        load(c * 2 + 1, x, b);
#pragma unroll
        for (int q = 0; q < EPC / 4; ++q) {
            v[4 * q] = x[q].x; v[4 * q + 1] = x[q].y; v[4 * q + 2] = x[q].z; v[4 * q + 3] = x[q].w;
            if (ARG) { a[ARG ? 4 * q : 0] = b[ARG ? q : 0].x; a[ARG ? 4 * q + 1 : 0] = b[ARG ? q : 0].y; a[ARG ? 4 * q + 2 : 0] = b[ARG ? q : 0].z; a[ARG ? 4 * q + 3 : 0] = b[ARG ? q : 0].w; }
        }
    }
    constexpr int UF = ARG ? 4 : 8;  // partial rows whose loads are in flight together
    for (int64_t cc = c + 1; cc <= c_end; cc += UF) {
        float4 x[UF][EPC / 4];
        int4 b[ARG ? UF : 1][ARG ? EPC / 4 : 1];
#pragma unroll
        for (int u = 0; u < UF; ++u)
            if (cc + u <= c_end) load((cc + u) * 2, x[u], b[ARG ? u : 0]);
#pragma unroll
        for (int u = 0; u < UF; ++u) {
            if (cc + u > c_end) break;
#pragma unroll
            for (int q = 0; q < EPC / 4; ++q) {
                const float y[4] = {x[u][q].x, x[u][q].y, x[u][q].z, x[u][q].w};
                if (ARG) {
                    const int4 w = b[ARG ? u : 0][ARG ? q : 0];
                    const int32_t z[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (beats<MODE>(y[j], z[j], v[4 * q + j], a[ARG ? 4 * q + j : 0])) { v[4 * q + j] = y[j]; a[ARG ? 4 * q + j : 0] = z[j]; }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[4 * q + j] += y[j];
                }
            }
        }
    }
    finish_row<T, MODE, true>(P, r, re - rs, ci, v, a);
}

// ------------------------------------------------------------------ launches
template <typename T, int MODE, bool EPI, int L>
static void launch_width(const PropParams& P, bool stream, cudaStream_t st) {
    if (stream) {
        constexpr bool rank1 = MODE == MODE_HEADRANK, head = MODE == MODE_HEADSUM || MODE == MODE_HEADSUM_W || MODE == MODE_V2 || rank1;
        constexpr size_t stages = RR_WARPS * sizeof(StreamStage<Chunk<T>::N, MODE != MODE_SUM && MODE != MODE_V2 && MODE != MODE_HEADSUM && !rank1,
                                                               MODE == MODE_ROUTE || head, MODE == MODE_MAX || MODE == MODE_MIN>);
        static_assert(stages + (rank1 ? 2 * 256 * sizeof(float) : 0) <= 48 * 1024, "staging fits the default shared memory");
        const size_t smem = stages + (rank1 ? 2 * P.F * sizeof(float) : 0);
        launch_overlapped(stream_rows_kernel<T, L, MODE, EPI>, dim3((unsigned)P.npieces), dim3(RR_WARPS * 32), smem, st, P);
    } else if constexpr (MODE != MODE_V2) {
        const int long_blocks = P.E > RR_SHORT ? (int)ceil_div(P.npieces, RR_WARPS) : 0;
        launch_overlapped(reduce_rows_kernel<T, L, MODE, EPI>, dim3((unsigned)(long_blocks + ceil_div(P.N, RR_WARPS * (32 / L)))), dim3(RR_WARPS * 32), 0, st, P,
                          long_blocks);
    }
}

template <typename T, int MODE>
static void launch_reduce(const PropParams& P, bool stream, cudaStream_t st) {
    constexpr bool EPI = MODE != MODE_HEADRANK;  // (the rank-1 epilogue comes alone)
    const bool epi = MODE == MODE_V2 ? P.da_part != nullptr : P.has_epi;
#define GNN_WIDTH(L) epi && EPI ? launch_width<T, MODE, EPI, L>(P, stream, st) : launch_width<T, MODE, false, L>(P, stream, st)
    if (P.nvec <= 4) GNN_WIDTH(4);
    else if (P.nvec <= 8) GNN_WIDTH(8);
    else if (P.nvec <= 16) GNN_WIDTH(16);
    else GNN_WIDTH(32);
#undef GNN_WIDTH
    if (P.E <= RR_SHORT && !stream) return;  // no row can have been cut
    // a row of more than FIX_LONG pieces exists only where a row can be that long
    const int nsimple = (int)ceil_div(P.npieces * P.nvec, FIX_THREADS);
    const bool hubs = P.E > (int64_t)FIX_LONG * P.piece;
    const int64_t nlong = hubs ? (P.npieces < 64 * (int64_t)FIX_LONG_BLOCKS ? ceil_div(P.npieces, 64) : FIX_LONG_BLOCKS) : 0;
    launch_overlapped(fixup_rows_kernel<T, MODE>, dim3((unsigned)(nsimple + nlong)), dim3(FIX_THREADS), 0, st, P, nsimple);
}

template <typename T>
void launch_reduce_sums(const PropParams& P, int mode, bool stream, cudaStream_t st) {
    if (mode == MODE_SUM) launch_reduce<T, MODE_SUM>(P, stream, st);
    else if (mode == MODE_WSUM) launch_reduce<T, MODE_WSUM>(P, stream, st);
    else if (mode == MODE_HEADSUM) launch_reduce<T, MODE_HEADSUM>(P, stream, st);
    else if (mode == MODE_HEADRANK) launch_reduce<T, MODE_HEADRANK>(P, stream, st);
    else launch_reduce<T, MODE_HEADSUM_W>(P, stream, st);
}

template <typename T>
void launch_reduce_others(const PropParams& P, int mode, bool stream, cudaStream_t st) {
    if (mode == MODE_MAX) launch_reduce<T, MODE_MAX>(P, stream, st);
    else if (mode == MODE_MIN) launch_reduce<T, MODE_MIN>(P, stream, st);
    else if (mode == MODE_EFSUM) launch_reduce<T, MODE_EFSUM>(P, stream, st);
    else launch_reduce<T, MODE_ROUTE>(P, stream, st);
}

}  // namespace gnn
