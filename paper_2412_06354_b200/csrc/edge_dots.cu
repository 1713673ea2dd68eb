// One value per edge (and head) from the two rows that meet there:
//   dot      dW[p,h] = scale(i) * <X[col[p],h,:], D[i,h,:]>                      (edge-weight gradients, XI_DOT_XJ, attention)
//   GATv2    s[p,h]  = sum_c a[h,c] * LeakyReLU(X[col[p],h,c] + D[i,h,c])         for p in row i
// Every edge is independent, so there are no partials and no second pass.
#include "reduce_params.cuh"

namespace gnn {

struct EdgeParams {
    const int64_t* rowptr;
    const int32_t* col;
    const void* X;  // gathered rows
    const void* D;  // rows of the sparse form
    const float* a;  // GATv2: [F]
    float* out;
    int32_t N;
    int64_t E;
    int nvec, sub;  // 16-byte chunks per row; positions per warp
    int H, lph;     // lph > 0: one result per (edge, head), a head = lph adjacent 16-byte chunks
    float slope;
};

enum { EDGE_DOT = 0, EDGE_DOT_MEAN = 1, EDGE_GATV2 = 2 };

// ------------------------------------------------------------------ rows of up to 512 bytes
// Positions first, as in the segmented reduction: a warp stages the gathered rows' indices of its share of positions and
// the rows they lie in; each of its lane groups streams a run of them with four to eight gathers in flight (two register
// buffers, each refilled as soon as it is used).  The row's own chunk stays in registers while the row lasts (row ends
// are bits; a batch of positions without one has nothing to test), the next row's is fetched meanwhile.  The lanes' shares of four positions
// are folded together: two levels halve the values a lane carries, the rest reduce the one left (32 lanes: 6 shuffles per
// four positions instead of 20).
// Bound by instruction issue for narrow rows and by the gathers (L2 -> SM) for rows of 512 bytes.  Before (4 positions per
// batch, one batch after the other, 8-byte entries, the row's chunk loaded when it changes) -> now:
//   100k nodes / 1.6 M edges, 512-byte rows, 8 heads bf16 150 -> 105 us; 123 M edges, 128-byte bf16 rows 2.86 -> 2.4 ms;
//   bf16 dots by multiply-adds that take bf16 (nothing unpacked, the same bits): 105 -> 96 us and 2.33 -> 2.10 ms there, and with
//   the registers that frees four blocks per SM for rows up to 256 bytes, 1.96 ms with 12 bytes of spills (512 bytes: 96 -> 98 us, three it stays); bf16 logits 81 -> 77 us;
//   GATv2 logits of 100k nodes / 1.6 M edges, 512-byte fp32 rows (a gather per index load, four at a time) 358 -> 113 us.
constexpr int ED_SUB = 256;  // most positions per warp
constexpr int ED_H = 4;      // positions per register buffer

template <bool MEAN>
struct EdgeStage {
    alignas(16) int col[ED_SUB + 32];  // gathered row; four words further for every lane group before it
    uint32_t ends[ED_SUB / 32];        // a bit per position: the last one of its row
    int row[ED_SUB + 1];       // [q] the q-th row with positions in the warp's share
    uint16_t start[ED_SUB + 2];
    float inv[MEAN ? ED_SUB + 1 : 1];  // [q] 1 / length of that row
};

// VB: 16-byte chunks per lane.  With two, half as many lanes cover a row, and what is done per position and lane (index, address,
// load, fold, row end) is done half as often.
template <typename T, int LPR, int KIND, int VB>
__global__ void __launch_bounds__(RR_WARPS * 32, VB == 2 ? 2 : sizeof(T) == 4 || (KIND == EDGE_DOT && LPR <= 16) ? 4 : 3)
edge_rows_kernel(const __grid_constant__ EdgeParams P) {
    constexpr int EPL = Chunk<T>::N, EPC = VB * EPL, NG = 32 / LPR, H = ED_H;
    using Raw = Vec16<VB>;
    auto unpack = [](const Raw& r, float* f) {
#pragma unroll
        for (int k = 0; k < VB; ++k) Chunk<T>::unpack(r.v[k], f + k * EPL);
    };
    constexpr bool MEAN = KIND == EDGE_DOT_MEAN, V2 = KIND == EDGE_GATV2;
    __shared__ EdgeStage<MEAN> s_all[RR_WARPS];
    pdl_wait();
    const int lane = threadIdx.x & 31, g = lane / LPR, li = lane % LPR;
    const int c = (int)blockIdx.x * RR_WARPS + (threadIdx.x >> 5);
    EdgeStage<MEAN>& S = s_all[threadIdx.x >> 5];
    if ((int64_t)c * P.sub >= P.E) return;
    const int cs = c * P.sub, n = (int)min((int64_t)P.sub, P.E - cs);
    const bool col_lane = li * VB < P.nvec;
    const int ci = col_lane ? li : 0;
    // skewed as in the segmented reduction: the groups' runs are in different banks, and four entries are one load
    const int L = P.sub / NG, lsh = 31 - __clz(L);
    auto sk = [&](int i) { return i + ((i >> lsh) << 2); };
    if (lane < ED_SUB / 32) S.ends[lane] = 0u;
    for (int i = lane; i < n; i += 32)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(S.col + sk(i))), "l"(P.col + cs + i) : "memory");
    bool began_before;
    const int m = stage_rows(P.rowptr, P.N, P.E, cs, n, lane, S.row, S.start, began_before);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    for (int q = lane; q < m; q += 32) {
        const int e = S.start[q + 1];
        if (e <= n) atomicOr(S.ends + ((e - 1) >> 5), 1u << ((e - 1) & 31));
        if (MEAN) {
            const int r = max(S.row[q], 0);
            S.inv[MEAN ? q : 0] = 1.0f / (float)(P.rowptr[r + 1] - P.rowptr[r]);
        }
    }
    __syncwarp();

    const int a = g * L, b = min(a + L, n);
    const int* const Sc = S.col + 4 * g;
    const uint64_t pol_keep = policy_evict_last();
    const uint32_t row_bytes = (uint32_t)P.nvec * 16;
    const char* const Xl = reinterpret_cast<const char*>(P.X) + (size_t)ci * (16 * VB);
    const char* const Dl = reinterpret_cast<const char*>(P.D) + (size_t)ci * (16 * VB);
    const int span = P.lph == 0 ? LPR : P.lph / VB;  // lanes per result: the whole row, or one head
    const int head = P.lph == 0 ? 0 : li / span, wstride = P.lph == 0 ? 1 : P.H;
    float av[V2 ? EPC : 1];
#pragma unroll
    for (int j = 0; j < (V2 ? EPC : 1); ++j) av[j] = V2 ? P.a[ci * EPC + j] : 0.f;
    int q = 0;  // row of the next position
    if (NG > 1 && a < b) {
        int lo = 0, hi = m;  // start[lo] <= a < start[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (S.start[mid] <= a) lo = mid; else hi = mid;
        }
        q = lo;
    }
    auto own = [&](int qq) {
        Raw r;
        const char* const p = Dl + (size_t)(uint32_t)max(S.row[qq], 0) * row_bytes;
#pragma unroll
        for (int k = 0; k < VB; ++k) r.v[k] = ld_16(p + 16 * k);
        return r;
    };
    constexpr bool MIXED = sizeof(T) == 2 && !V2;  // dots of bf16 need no unpacked values
    float d[MIXED ? 1 : EPC], sc = 1.0f;
    Raw dr = {}, own_next = {};
    auto take = [&](const Raw& r) {
        if constexpr (MIXED) dr = r;
        else unpack(r, d);
    };
    if (a < b) {
        take(own(q));
        if (MEAN) sc = S.inv[MEAN ? q : 0];
        if (q + 1 < m) own_next = own(q + 1);
    }
    auto next_row = [&]() {
        ++q;
        take(own_next);
        if (MEAN && q < m) sc = S.inv[MEAN ? q : 0];
        if (q + 1 < m) own_next = own(q + 1);
    };
    for (int i = n + lane; i < P.sub; i += 32) S.col[sk(i)] = 0;  // the last warp: positions past the end gather row 0
    __syncwarp();
    auto issue = [&](Raw* x, int i) {
        const int4 c4 = V2 ? make_int4(Sc[i], Sc[i + 1], Sc[i + 2], Sc[i + 3]) : *reinterpret_cast<const int4*>(Sc + i);
        const int ccs[H] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
        for (int u = 0; u < H; ++u) ld_hint(x[u], Xl + (size_t)(uint32_t)ccs[u] * row_bytes, pol_keep);
    };
    auto use = [&](const Raw* xr, unsigned ends, int i) {
        float dot[H], scale[MEAN ? H : 1];
        auto one = [&](int u) {
            float x[EPC], t = 0.f, t1 = 0.f;
            if constexpr (MIXED) {
#pragma unroll
                for (int k = 0; k < VB; ++k) {
                    fma_bf16(t, t1, xr[u].v[k].x, dr.v[k].x);
                    fma_bf16(t, t1, xr[u].v[k].y, dr.v[k].y);
                    fma_bf16(t, t1, xr[u].v[k].z, dr.v[k].z);
                    fma_bf16(t, t1, xr[u].v[k].w, dr.v[k].w);
                }
            } else if constexpr (V2 && sizeof(T) == 2) {  // x + d, of which only the sum is used
#pragma unroll
                for (int j = 0; j < EPC; ++j) x[j] = d[j];
#pragma unroll
                for (int k = 0; k < VB; ++k) {
                    add_bf16(x[8 * k], x[8 * k + 1], xr[u].v[k].x);
                    add_bf16(x[8 * k + 2], x[8 * k + 3], xr[u].v[k].y);
                    add_bf16(x[8 * k + 4], x[8 * k + 5], xr[u].v[k].z);
                    add_bf16(x[8 * k + 6], x[8 * k + 7], xr[u].v[k].w);
                }
            } else {
                unpack(xr[u], x);
            }
#pragma unroll
            for (int j = 0; j < (MIXED ? 0 : EPC); j += 2) {
                if (V2) {  // single FMAs: packed ones measured 126 us instead of 119 (register pairs)
                    const float z = sizeof(T) == 2 ? x[j] : x[j] + d[j], z1 = sizeof(T) == 2 ? x[j + 1] : x[j + 1] + d[j + 1];
                    t = fmaf(av[V2 ? j : 0], z > 0.f ? z : P.slope * z, t);
                    t = fmaf(av[V2 ? j + 1 : 0], z1 > 0.f ? z1 : P.slope * z1, t);
                } else {
                    fma2(t, t1, x[j], x[j + 1], d[j], d[j + 1]);
                }
            }
            dot[u] = col_lane ? t + t1 : 0.f;
            if (MEAN) scale[MEAN ? u : 0] = sc;
        };
        if (V2 || __any_sync(0xffffffffu, ends != 0)) {  // (GATv2: two copies of the loop spill)
#pragma unroll
            for (int u = 0; u < H; ++u) {
                one(u);
                if (ends >> u & 1u) next_row();
            }
            __syncwarp();
        } else {  // most positions of a skewed graph lie in long rows: nothing to test
#pragma unroll
            for (int u = 0; u < H; ++u) one(u);
        }
        if (span >= 4) {
            const int h1 = span >> 1, h2 = span >> 2;
            const bool up1 = (li & h1) != 0, up2 = (li & h2) != 0;
            const float s0 = up1 ? dot[0] : dot[2], s1 = up1 ? dot[1] : dot[3];
            const float r0 = (up1 ? dot[2] : dot[0]) + __shfl_xor_sync(0xffffffffu, s0, h1);
            const float r1 = (up1 ? dot[3] : dot[1]) + __shfl_xor_sync(0xffffffffu, s1, h1);
            float v = (up2 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, up2 ? r0 : r1, h2);
            for (int o = span >> 3; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            const int mine = (up1 ? 2 : 0) + (up2 ? 1 : 0);  // the position of the batch this lane holds
            if (MEAN) v *= up1 ? (up2 ? scale[MEAN ? 3 : 0] : scale[MEAN ? 2 : 0]) : (up2 ? scale[MEAN ? 1 : 0] : scale[0]);
            // any lane of the span may end up holding a result (with whole-row results also a lane past a narrow row)
            if ((P.lph == 0 || col_lane) && (li & (h2 - 1)) == 0 && i + mine < b) P.out[(int64_t)(cs + i + mine) * wstride + head] = v;
        } else {  // heads of one or two 16-byte chunks
#pragma unroll
            for (int u = 0; u < H; ++u) {
                float v = dot[u];
                for (int o = span >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (MEAN) v *= scale[MEAN ? u : 0];
                if (col_lane && (li % span) == 0 && i + u < b) P.out[(int64_t)(cs + i + u) * wstride + head] = v;
            }
        }
    };
    // same trip count in every group (the shuffles are warp-wide); L is a multiple of 2 H
    Raw A[H], B[H];
    issue(A, a);
    issue(B, a + H);
#pragma unroll 1
    for (int i = a; i < a + L; i += 2 * H) {
        const bool more = i + 2 * H < a + L;
        const unsigned ends = S.ends[i >> 5] >> (i & 31);
        use(A, ends & ((1u << H) - 1u), i);
        if (more) issue(A, i + 2 * H);
        use(B, (ends >> H) & ((1u << H) - 1u), i + H);
        if (more) issue(B, i + 3 * H);
    }
}

// ------------------------------------------------------------------ rows of up to 2048 bytes
// A warp per 256 positions walks the rows, the own row's chunks held in registers along the row.
constexpr int EC_POSITIONS = 256;

template <typename T, int VPL, bool MEAN>
__global__ void __launch_bounds__(RR_WARPS * 32)
edge_wide_rows_kernel(const __grid_constant__ EdgeParams P) {
    constexpr int LPR = 32;
    pdl_wait();
    constexpr int EPC = Chunk<T>::N;
    constexpr int NG = 32 / LPR;
    constexpr int U = (LPR >= 16) ? (8 / VPL) : 4;
    const int lane = threadIdx.x & 31, g = lane / LPR, li = lane % LPR;
    const int64_t c = (int64_t)blockIdx.x * RR_WARPS + (threadIdx.x >> 5);
        const int64_t cs = c * EC_POSITIONS;
    const int64_t ce = (cs + EC_POSITIONS < P.E) ? cs + EC_POSITIONS : P.E;
    if (cs >= ce) return;
    const uint64_t pol_keep = policy_evict_last(), pol_stream = policy_evict_first();
    const size_t row_bytes = (size_t)P.nvec * 16;
    const char* Xb = reinterpret_cast<const char*>(P.X);
    const char* Db = reinterpret_cast<const char*>(P.D);
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
        const float scale = MEAN ? 1.0f / (float)(re - rs) : 1.0f;
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
                        if (ok[u] && li == 0) P.out[p] = scale * dot;
                    } else {  // one per (edge, head): a head covers lph adjacent lanes
#pragma unroll
                        for (int v = 0; v < VPL; ++v) {
                            float dot = dotv[v];
                            for (int o = P.lph >> 1; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                            const int ci = v * LPR + li;
                            if (ok[u] && ci < P.nvec && (li % P.lph) == 0) P.out[p * P.H + ci / P.lph] = scale * dot;
                        }
                    }
                }
            }
        }
        pos = b;
    }
}

template <typename T>
static void launch_edge_rows(EdgeParams& P, int kind, cudaStream_t st) {
    if (P.nvec > 32) {
        const dim3 grid((unsigned)ceil_div(P.E, (int64_t)EC_POSITIONS * RR_WARPS)), block(RR_WARPS * 32);
#define GNN_WIDE(V) \
    kind == EDGE_DOT_MEAN ? launch_overlapped(edge_wide_rows_kernel<T, V, true>, grid, block, 0, st, P) : launch_overlapped(edge_wide_rows_kernel<T, V, false>, grid, block, 0, st, P)
        if (P.nvec <= 64) GNN_WIDE(2);
        else GNN_WIDE(4);
#undef GNN_WIDE
        return;
    }
    // positions per warp: fewer on small graphs, so that all SMs have warps
    P.sub = P.E >= 2500 * 1000 ? 256 : P.E >= 512 * 1024 ? 128 : 64;
    const dim3 grid((unsigned)ceil_div(P.E, (int64_t)P.sub * RR_WARPS)), block(RR_WARPS * 32);
#define GNN_EDGE(L, VB)                                                                                             \
    kind == EDGE_DOT ? launch_overlapped(edge_rows_kernel<T, L, EDGE_DOT, VB>, grid, block, 0, st, P)               \
    : kind == EDGE_DOT_MEAN ? launch_overlapped(edge_rows_kernel<T, L, EDGE_DOT_MEAN, VB>, grid, block, 0, st, P)   \
                            : launch_overlapped(edge_rows_kernel<T, L, EDGE_GATV2, VB>, grid, block, 0, st, P)
    // GATv2 logits of fp32 rows over 256 bytes: 32 bytes to a lane, where rows, heads and matrices are whole multiples of that (1.6 M edges
    // of 512 bytes: 113 -> 100 us).  Not the plain dots, which have less to do per value (600 k edges: 53 -> 57 us), nor bf16, whose
    // sixteen values a lane leave no room for a second buffer's worth of loads (512 bytes, eight heads: 105 -> 154 us), nor heads of fewer
    // than four such lanes, whose sums cannot be folded together (3 M edges, eight heads of 64 bytes: 188 -> 247 us).
    if constexpr (sizeof(T) == 4)
        if (kind == EDGE_GATV2 && P.nvec > 16 && P.nvec % 2 == 0 && (P.lph == 0 || P.lph >= 8) && ((reinterpret_cast<uintptr_t>(P.X) | reinterpret_cast<uintptr_t>(P.D)) & 31) == 0) {
            launch_overlapped(edge_rows_kernel<T, 16, EDGE_GATV2, 2>, grid, block, 0, st, P);
            return;
        }
    if (P.nvec <= 4) GNN_EDGE(4, 1);
    else if (P.nvec <= 8) GNN_EDGE(8, 1);
    else if (P.nvec <= 16) GNN_EDGE(16, 1);
    else GNN_EDGE(32, 1);
#undef GNN_EDGE
}

static gnn_status run_edges(const char* who, const gnn_csr* g, const void* X, const void* D, const float* a, int H, int C, int kind, float slope,
                            gnn_dtype dtype, float* out, cudaStream_t st) {
    const int s = elem_size(dtype), F = H * C;
    GNN_REQUIRE(C > 0 && ((size_t)C * s) % 16 == 0, GNN_ERR_UNSUPPORTED, "%s: a head must be a multiple of 16 bytes wide", who);
    const int nvec = F * s / 16, lph = C * s / 16;
    GNN_REQUIRE(nvec <= 128, GNN_ERR_UNSUPPORTED, "%s: feature rows wider than 2048 bytes", who);
    GNN_REQUIRE(H == 1 || (lph <= 32 && (lph & (lph - 1)) == 0), GNN_ERR_UNSUPPORTED,
                "%s: a head must span a power-of-two number (<= 32) of 16-byte chunks (C=%d)", who, C);
    GNN_REQUIRE(aligned16(X) && aligned16(D), GNN_ERR_INVALID_ARG, "%s: feature matrices must be 16-byte aligned", who);
    GNN_REQUIRE(g->E < ((int64_t)1 << 31), GNN_ERR_UNSUPPORTED, "%s: positions must fit 32 bits (E < 2^31)", who);
    if (g->E == 0) return GNN_OK;
    EdgeParams P = {};
    P.rowptr = g->rowptr; P.col = g->col; P.X = X; P.D = D; P.a = a; P.out = out;
    P.N = g->N; P.E = g->E; P.nvec = nvec; P.H = H; P.lph = H > 1 ? lph : 0; P.slope = slope;
    if (dtype == GNN_F32) launch_edge_rows<float>(P, kind, st);
    else launch_edge_rows<__nv_bfloat16>(P, kind, st);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

// one dot product per edge (H == 1) or per edge and head, scaled by 1 / row length if mean
gnn_status run_sddmm(const char* who, const gnn_csr* g, const void* X, const void* D, int H, int C, int mean,
                     gnn_dtype dtype, float* dW, cudaStream_t st) {
    return run_edges(who, g, X, D, nullptr, H, C, mean ? EDGE_DOT_MEAN : EDGE_DOT, 0.f, dtype, dW, st);
}

gnn_status run_gatv2_logits(const char* who, const gnn_csr* g, const void* X, const void* D, const float* a, int H, int C, float slope, gnn_dtype dtype,
                            float* s, cudaStream_t st) {
    return run_edges(who, g, X, D, a, H, C, EDGE_GATV2, slope, dtype, s, st);
}

}  // namespace gnn
