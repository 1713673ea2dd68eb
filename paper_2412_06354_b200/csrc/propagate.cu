// Fused propagate (Sec. 3 "Message Passing": apply_edges + aggregate_neighbors combined into a
// generalised sparse x dense product) and its backward passes: host side of the segmented reduction
// (reduce_rows.cuh) and the edge-wise dot products of the weight gradients.
#include <mutex>

#include "reduce_params.cuh"

namespace gnn {

// ------------------------------------------------------------------ edge-weight gradient (SDDMM)
// dW[p] = scale(i) * <X[col[p],:], dOut[i,:]> for p in row i.  Same chunking; every edge is
// independent, so no partials.  The dOut row stays in registers along the row.
struct SddmmParams {
    const int64_t* rowptr;
    const int32_t* col;
    const void* X;
    const void* dOut;
    float* dW;
    int32_t N;
    int64_t E;
    int nvec;
    int mean;
    int64_t nchunks;
    int H, lph;  // lph > 0: one result per (edge, head), a head = lph adjacent 16-byte chunks
};

template <typename T, int LPR, int VPL>
__global__ void __launch_bounds__(PF_WARPS * 32)
sddmm_chunk_kernel(const SddmmParams P) {
    constexpr int EPC = Chunk<T>::N;
    constexpr int NG = 32 / LPR;
    constexpr int U = (LPR >= 16) ? (8 / VPL) : 4;
    const int lane = threadIdx.x & 31, g = lane / LPR, li = lane % LPR;
    const int64_t c = (int64_t)blockIdx.x * PF_WARPS + (threadIdx.x >> 5);
    if (c >= P.nchunks) return;
    const int64_t cs = c * PF_SLAB;
    const int64_t ce = (cs + PF_SLAB < P.E) ? cs + PF_SLAB : P.E;
    if (cs >= ce) return;
    const uint64_t pol_keep = policy_evict_last(), pol_stream = policy_evict_first();
    const size_t row_bytes = (size_t)P.nvec * 16;
    const char* Xb = reinterpret_cast<const char*>(P.X);
    const char* Db = reinterpret_cast<const char*>(P.dOut);
    // row containing position cs: last row with rowptr[r] <= cs
    int r = lower_bound_i64(P.rowptr, P.N + 1, cs + 1) - 1;
    int64_t pos = cs;
    while (pos < ce) {
        r = first_row_ending_after(P.rowptr, r, P.N, pos, lane);  // skip rows that end at or before pos
        const int64_t rs = P.rowptr[r], re = P.rowptr[r + 1];
        const int64_t b = re < ce ? re : ce;
        float d[VPL][EPC];
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int ci = v * LPR + li;
            if (ci < P.nvec) {
                Chunk<T>::unpack(ld_hint16(Db + (size_t)r * row_bytes + (size_t)ci * 16, pol_stream), d[v]);
            } else {
#pragma unroll
                for (int j = 0; j < EPC; ++j) d[v][j] = 0.f;
            }
        }
        const float scale = P.mean ? 1.0f / (float)(re - rs) : 1.0f;
        for (int64_t base = pos; base < b; base += 32) {
            const int n = (int)((b - base) < 32 ? (b - base) : 32);
            int myc = lane < n ? ld_hint_i32(P.col + base + lane, pol_stream) : 0;
            const int rounds = (n + NG - 1) / NG;
            for (int r0 = 0; r0 < rounds; r0 += U) {
                uint4 buf[U][VPL];
                bool ok[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int e = (r0 + u) * NG + g;
                    ok[u] = e < n;
                    int cv = __shfl_sync(0xffffffffu, myc, e & 31);
                    if (ok[u]) {
#pragma unroll
                        for (int v = 0; v < VPL; ++v) {
                            const int ci = v * LPR + li;
                            if (ci < P.nvec) buf[u][v] = ld_hint16(Xb + (size_t)cv * row_bytes + (size_t)ci * 16, pol_keep);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float dotv[VPL];
#pragma unroll
                    for (int v = 0; v < VPL; ++v) {
                        dotv[v] = 0.f;
                        const int ci = v * LPR + li;
                        if (ok[u] && ci < P.nvec) {
                            float x[EPC];
                            Chunk<T>::unpack(buf[u][v], x);
#pragma unroll
                            for (int j = 0; j < EPC; ++j) dotv[v] = fmaf(x[j], d[v][j], dotv[v]);
                        }
                    }
                    const int64_t p = base + (r0 + u) * NG + g;
                    if (P.lph == 0) {  // one dot product per edge over the whole row
                        float dot = dotv[0];
#pragma unroll
                        for (int v = 1; v < VPL; ++v) dot += dotv[v];
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                        if (ok[u] && li == 0) P.dW[p] = scale * dot;
                    } else {  // one per (edge, head): a head covers lph adjacent lanes
#pragma unroll
                        for (int v = 0; v < VPL; ++v) {
                            float dot = dotv[v];
                            for (int o = P.lph >> 1; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                            const int ci = v * LPR + li;
                            if (ok[u] && ci < P.nvec && (li % P.lph) == 0) P.dW[p * P.H + ci / P.lph] = scale * dot;
                        }
                    }
                }
            }
        }
        pos = b;
    }
}

// ------------------------------------------------------------------ flat SDDMM for short rows
// Same idea as propagate_flat_kernel: positions first, rows second.  The warp stages the gathered
// rows of its 256 positions and finds, by marking row starts and a prefix maximum, the row of every
// position; each lane group then takes a contiguous run and issues, per batch of 4 positions, the
// independent loads of X[col[p]] and, where the row changes, dOut[row(p)].  Every position is independent, so there are no partials and no second pass.
constexpr int SF_U = 4;
constexpr int FL_WARPS = 4;

struct SddmmFlatSmem {
    int2 e[PF_SLAB];        // x: gathered row of X, y: start entry of the position's row
    int32_t srow[PF_SLAB];  // [k] row starting at position k of the chunk ([0]: the row holding position 0)
    float sinv[PF_SLAB];    // [k] 1, or 1 / row length for the mean
};

template <typename T, int LPR>
__global__ void __launch_bounds__(FL_WARPS * 32, 8)
sddmm_flat_kernel(const SddmmParams P) {
    constexpr int EPC = Chunk<T>::N, NG = 32 / LPR, U = SF_U, L = PF_SLAB / NG;
    __shared__ SddmmFlatSmem s_all[FL_WARPS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.x * FL_WARPS + wib;
    if (c >= P.nchunks) return;
    SddmmFlatSmem& S = s_all[wib];
    const uint64_t pol_keep = policy_evict_last(), pol_stream = policy_evict_first();
    const int64_t cs = c * PF_SLAB;
    const int n = (int)((cs + PF_SLAB < P.E ? cs + PF_SLAB : P.E) - cs);
    const int g = lane / LPR, li = lane % LPR;
    const bool col_lane = li < P.nvec;

    // the row holding position cs: largest r with rowptr[r] <= cs (32-way search)
    int lo = 0, hi = P.N;
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32;
        const int idx = min(lo + (lane + 1) * step, hi);
        const bool le = idx < hi && P.rowptr[idx] <= cs;
        const int k = __popc(__ballot_sync(0xffffffffu, le));
        const int nlo = lo + k * step;
        hi = min(nlo + step, hi);
        lo = nlo;
    }
    const int cur0 = lo;
    auto row_factor = [&](int64_t len) { return P.mean ? 1.0f / (float)(len > 1 ? len : 1) : 1.0f; };
    for (int i = lane; i < n; i += 32) S.e[i] = make_int2(ld_hint_i32(P.col + cs + i, pol_stream), 0);
    if (lane == 0) { S.srow[0] = cur0; S.sinv[0] = row_factor(P.rowptr[cur0 + 1] - P.rowptr[cur0]); }
    __syncwarp();
    for (int rb = cur0 + 1; rb < P.N;) {  // non-empty rows starting inside the chunk
        const int r = rb + lane;
        int64_t rs = 0, re = 0;
        bool live = false;
        if (r < P.N) {
            rs = P.rowptr[r];
            live = rs < cs + n;
            if (live) re = P.rowptr[r + 1];
        }
        if (live && re > rs) {
            const int k = (int)(rs - cs);
            S.srow[k] = r;
            S.sinv[k] = row_factor(re - rs);
            S.e[k].y = k;
        }
        if (!__all_sync(0xffffffffu, live)) break;
        // 32 rows without edges: jump over the rest of the run
        if (__all_sync(0xffffffffu, re == rs)) rb = first_row_ending_after(P.rowptr, rb + 32, P.N, __shfl_sync(0xffffffffu, rs, 0), lane);
        else rb += 32;
    }
    __syncwarp();
    {  // prefix maximum of the start marks: lane owns positions 8*lane .. 8*lane+7
        int m[8];
        int run = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = lane * 8 + q;
            run = max(run, i < n ? S.e[i].y : 0);
            m[q] = run;
        }
        int incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl = max(incl, t);
        }
        int before = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) before = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = lane * 8 + q;
            if (i < n) S.e[i].y = max(before, m[q]);
        }
    }
    __syncwarp();

    const int a = g * L, b = min(a + L, n);
    const size_t row_bytes = (size_t)P.nvec * 16;
    const char* Xl = reinterpret_cast<const char*>(P.X) + (size_t)(col_lane ? li : 0) * 16;
    const char* Dl = reinterpret_cast<const char*>(P.dOut) + (size_t)(col_lane ? li : 0) * 16;
    const int span = P.lph == 0 ? LPR : P.lph;  // lanes per result: the whole row, or one head
    const bool writer = col_lane && (li % span) == 0;
    const int head = P.lph == 0 ? 0 : li / P.lph, wstride = P.lph == 0 ? 1 : P.H;
    const uint32_t row_bytes32 = (uint32_t)row_bytes;
    int kprev = -1;   // start entry of the position before this batch
    uint4 dcur = make_uint4(0, 0, 0, 0);  // this lane's chunk of the current row of dOut: reloaded only when the row changes
    for (int i = a; i < a + L; i += U) {  // same trip count in every lane: the shuffles below are warp-wide
        uint4 xb[U], db[U];
        int k[U];
        bool fresh[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = i + u < b;
            const int2 e = S.e[ok ? i + u : 0];
            k[u] = ok ? e.y : -1;
            fresh[u] = ok && k[u] != (u == 0 ? kprev : k[u - 1]);
            if (ok) xb[u] = ld_hint16(Xl + (size_t)((uint32_t)e.x) * row_bytes32, pol_keep);
            if (fresh[u]) db[u] = __ldg(reinterpret_cast<const uint4*>(Dl + (size_t)((uint32_t)S.srow[e.y]) * row_bytes32));
        }
        kprev = k[U - 1];
        static_assert(SF_U == 4, "the reductions below fold four positions at a time");
        float dot[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (fresh[u]) dcur = db[u];
            dot[u] = 0.f;
            if (k[u] >= 0 && col_lane) {
                float x[EPC], d[EPC];
                Chunk<T>::unpack(xb[u], x);
                Chunk<T>::unpack(dcur, d);
#pragma unroll
                for (int j = 0; j < EPC; ++j) dot[u] = fmaf(x[j], d[j], dot[u]);
            }
        }
        if (span >= 4) {
            // fold the four positions while reducing over the span lanes: the first two levels halve the values
            // a lane carries (2 + 1 shuffles), the rest reduce the one left; the quarter of the span a lane
            // sits in decides which position it ends up with: 6 shuffles for 32 lanes instead of 20
            const int h1 = span >> 1, h2 = span >> 2;
            const bool up1 = (li & h1) != 0, up2 = (li & h2) != 0;
            const float s0 = up1 ? dot[0] : dot[2], s1 = up1 ? dot[1] : dot[3];
            const float r0 = (up1 ? dot[2] : dot[0]) + __shfl_xor_sync(0xffffffffu, s0, h1);
            const float r1 = (up1 ? dot[3] : dot[1]) + __shfl_xor_sync(0xffffffffu, s1, h1);
            float v = (up2 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, up2 ? r0 : r1, h2);
            for (int o = span >> 3; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            const int mine = (up1 ? 2 : 0) + (up2 ? 1 : 0);  // the position of the batch this lane holds
            const int km = mine == 0 ? k[0] : mine == 1 ? k[1] : mine == 2 ? k[2] : k[3];
            // any lane of the span may end up holding a result (with whole-row results also a lane past a narrow row)
            if ((P.lph == 0 || col_lane) && (li & (h2 - 1)) == 0 && km >= 0) P.dW[(cs + i + mine) * wstride + head] = S.sinv[km] * v;
        } else {  // heads of one or two 16-byte chunks
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float v = dot[u];
                for (int o = span >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (k[u] >= 0 && writer) P.dW[(cs + i + u) * wstride + head] = S.sinv[k[u]] * v;
            }
        }
    }
}

// ------------------------------------------------------------------ host dispatch
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
    if (mode == MODE_SUM || mode == MODE_WSUM || mode == MODE_HEADSUM) launch_reduce_sums<T>(P, mode, stream, st);
    else launch_reduce_others<T>(P, mode, stream, st);
}

template <typename T>
static void launch_sddmm(const SddmmParams& P, int lpr, int vpl, cudaStream_t st) {
    if (vpl == 1) {  // positions first
        const int grid = (int)ceil_div(P.nchunks, FL_WARPS);
        switch (lpr) {
            case 4: sddmm_flat_kernel<T, 4><<<grid, FL_WARPS * 32, 0, st>>>(P); break;
            case 8: sddmm_flat_kernel<T, 8><<<grid, FL_WARPS * 32, 0, st>>>(P); break;
            case 16: sddmm_flat_kernel<T, 16><<<grid, FL_WARPS * 32, 0, st>>>(P); break;
            default: sddmm_flat_kernel<T, 32><<<grid, FL_WARPS * 32, 0, st>>>(P); break;
        }
        return;
    }
    const int grid = (int)ceil_div(P.nchunks, PF_WARPS);
    const int thr = PF_WARPS * 32;
#define GNN_SD_CASE(L, V) \
    if (lpr == L && vpl == V) { sddmm_chunk_kernel<T, L, V><<<grid, thr, 0, st>>>(P); }
    GNN_SD_CASE(4, 1) GNN_SD_CASE(8, 1) GNN_SD_CASE(16, 1) GNN_SD_CASE(32, 1) GNN_SD_CASE(32, 2) GNN_SD_CASE(32, 4)
#undef GNN_SD_CASE
}

static int64_t num_slabs(int64_t E) { return E > 0 ? ceil_div(E, PF_SLAB) : 1; }

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
    if (E >= (int64_t)4 * 1024 * 1024) return 256;
    if (E >= 512 * 1024) return E > 64 * (int64_t)N || E >= 2500 * 1000 || (row_bytes <= 128 && E >= 1000 * 1000) ? 256 : 128;
    if (!stream) return 64;
    return E >= 256 * 1024 ? 128 : E >= 128 * 1024 || row_bytes <= 64 ? 64 : 32;
}

// Room for a partial row per 64 to 256 positions.  The streaming kernel needs an eighth of that; the size is what callers
// have been told since the first version, and what decides which problems the built-in scratch takes.
size_t chunked_workspace(int64_t E, int F, bool with_arg) {
    if (E <= 0) return carve(nullptr, 1, F, with_arg).bytes;
    const int per = E >= (int64_t)4 * 1024 * 1024 ? 1024 : E >= 512 * 1024 ? 128 : 64;
    return carve(nullptr, ceil_div(E, (int64_t)per), F < 256 ? F : 256, with_arg).bytes;
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
    GNN_REQUIRE(E >= 0 && E < ((int64_t)1 << 31) - 4 * PF_SLAB, GNN_ERR_UNSUPPORTED, "%s: positions must fit 32 bits (E < 2^31)", who);
    const bool with_arg = (mode == MODE_MAX || mode == MODE_MIN);
    const size_t need = chunked_workspace(E, F, with_arg);
    GNN_REQUIRE(ws && ws_bytes >= need && aligned16(ws), GNN_ERR_WORKSPACE_TOO_SMALL,
                "%s: workspace of %zu bytes (16-byte aligned) needed, %zu given", who, need, ws_bytes);
    if (N == 0) return GNN_OK;
    PropParams P;
    P.rowptr = rowptr; P.col = col; P.w = w; P.argmax = argmax;
    P.gscale_rowptr = gscale_rowptr; P.route_arg = route_arg; P.route_pos = route_pos;
    P.N = N; P.E = E; P.mean = mean; P.arg_ld = F;
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
    P.self_X = nullptr; P.self_rowptr = rowptr; P.bias = nullptr;
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

// dW[p,h] = <X[col[p],h,:], dOut[i,h,:]> for p in row i: the per-head edge dot products of the
// attention backward pass
gnn_status sddmm_heads(const char* who, const gnn_csr* g, const void* X, const void* dOut, int H, int C,
                       gnn_dtype dtype, float* dW_EH, cudaStream_t st, int mean) {
    const int s = elem_size(dtype), F = H * C;
    GNN_REQUIRE(((size_t)C * s) % 16 == 0, GNN_ERR_UNSUPPORTED, "%s: a head must be a multiple of 16 bytes wide", who);
    const int lph = C * s / 16;
    GNN_REQUIRE(lph <= 32 && (lph & (lph - 1)) == 0, GNN_ERR_UNSUPPORTED,
                "%s: a head must span a power-of-two number (<= 32) of 16-byte chunks (C=%d)", who, C);
    int lpr, vpl;
    GNN_REQUIRE(pick_shape(F * s / 16, &lpr, &vpl), GNN_ERR_UNSUPPORTED, "%s: feature rows wider than 2048 bytes", who);
    GNN_REQUIRE(lph <= lpr, GNN_ERR_UNSUPPORTED, "%s: head wider than the row layout", who);
    GNN_REQUIRE(aligned16(X) && aligned16(dOut), GNN_ERR_INVALID_ARG, "%s: feature matrices must be 16-byte aligned", who);
    if (g->E == 0) return GNN_OK;
    SddmmParams S;
    S.rowptr = g->rowptr; S.col = g->col; S.X = X; S.dOut = dOut; S.dW = dW_EH;
    S.N = g->N; S.E = g->E; S.nvec = F * s / 16; S.mean = mean; S.nchunks = num_slabs(g->E); S.H = H; S.lph = lph;
    if (dtype == GNN_F32) launch_sddmm<float>(S, lpr, vpl, st);
    else launch_sddmm<__nv_bfloat16>(S, lpr, vpl, st);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

// one dot product per edge (H == 1; scaled by 1 / row length if mean) or per edge and head
gnn_status run_sddmm(const char* who, const gnn_csr* g, const void* X, const void* D, int H, int C, int mean,
                     gnn_dtype dtype, float* dW, cudaStream_t st) {
    if (H > 1) {
        return sddmm_heads(who, g, X, D, H, C, dtype, dW, st, mean);
    }
    const int s = elem_size(dtype), F = C;
    GNN_REQUIRE(F > 0 && ((size_t)F * s) % 16 == 0, GNN_ERR_UNSUPPORTED, "%s: F*sizeof(element) must be a multiple of 16 bytes", who);
    int lpr, vpl;
    GNN_REQUIRE(pick_shape(F * s / 16, &lpr, &vpl), GNN_ERR_UNSUPPORTED, "%s: feature rows wider than 2048 bytes", who);
    GNN_REQUIRE(aligned16(X) && aligned16(D), GNN_ERR_INVALID_ARG, "%s: feature matrices must be 16-byte aligned", who);
    if (g->E == 0) return GNN_OK;
    SddmmParams S;
    S.rowptr = g->rowptr; S.col = g->col; S.X = X; S.dOut = D; S.dW = dW;
    S.N = g->N; S.E = g->E; S.nvec = F * s / 16; S.mean = mean; S.nchunks = num_slabs(g->E); S.H = 1; S.lph = 0;
    if (dtype == GNN_F32) launch_sddmm<float>(S, lpr, vpl, st);
    else launch_sddmm<__nv_bfloat16>(S, lpr, vpl, st);
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
