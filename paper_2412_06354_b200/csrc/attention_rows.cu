// Row-wise parts of attention with 4 and 8 heads, positions first: the edge softmax and the softmax of GAT logits over a row's
// positions, and their gradients.  A block takes NT / HV * 8 consecutive positions whatever rows they lie in (HV = heads / 4): a
// thread has eight consecutive positions of four heads, the rows' ends are bits, and a row's maximum or sum is a segmented
// scan: inside the thread, over the threads of a warp by shuffles, over the warps through shared memory.  Rows that lie inside the
// block are finished there.  GAT: a row that is cut leaves its maximum and sum per block, and a second kernel, again a block per
// chunk, combines a row's shares in ascending order and finishes the chunk's positions of it.  Edge softmax, which has no
// workspace: the blocks that a row is cut into read all of it, out of L2.
// Rows of more than AR_SPAN chunks are left to clusters (softmax.cu), which read them once per pass: the blocks together would read a row of k chunks
// k times (8 heads fp32, a row of 330 k positions among 1.9 M edges 632 -> 200 us, of 2.4 M among 7.2 M 20 -> 1.8 ms).
// What bounds it: the latency of a chunk (search, gathers, four to six barriers) at two or three blocks per SM, and instruction issue (an exponential and
// a division per value).
// Before: a row per 8 threads, per warp or per block, three kernels side by side on streams of their own, as long as their
// longest row and mostly idle warps.  100k nodes, 1.6 M edges, R-MAT: softmax of GAT logits of 8 heads 97 -> 43 us (tiers of rows side
// by side -> both kernels), its gradient 104 -> 100 us; edge softmax 80 -> 41 us and 55 -> 27 us (4 heads fp32), 113 -> 72 us and 83 -> 50 us (8).
// Distance to 64 bits as before (alpha 4.1e-8, 4.0e-8 by tiers; da_src 2.3e-7, 2.1e-7).
#include <atomic>
#include <cfloat>

#include "reduce_params.cuh"
#include "tc_common.cuh"

namespace gnn {

constexpr int AR_RUN = 8;  // positions per thread
template <int NT> __host__ __device__ constexpr int ar_blocks() { return 768 / NT; }  // per SM: 80 registers

template <int NT, int HV>
struct RowsTile {
    static constexpr int W = NT / 32, RPW = 32 / HV, WP = RPW * AR_RUN, RUNS = W * RPW, CHUNK = W * WP;
    struct Rows {
        int row[WP + 1];
        uint16_t start[WP + 2];
        uint32_t ends[WP / 32];  // a bit per position: the last one of its row
    };
    // a run's float4s begin HV further than the run before them ends: eight lanes read eight different 16-byte banks
    static __device__ __forceinline__ int at(int p, int v) { return (p / AR_RUN) * ((AR_RUN + 1) * HV) + (p % AR_RUN) * HV + v; }
    static constexpr int TILE = RUNS * (AR_RUN + 1) * HV;  // float4s of the block
    Rows rows[W];
    float4 total[RUNS * HV];     // [run][quad] total of the row that ends first in the run
    float4 open_total[HV];       // of the row that goes on past the chunk
    float4 warp_open[W * HV];    // what a warp's open tail comes to
    uint8_t warp_closed[W];      // whether a row ends in the warp
    uint32_t has_end[(RUNS + 31) / 32];  // a bit per run: a row ends in it
    uint8_t whole[RUNS];         // gradients: the run's positions whose rows lie inside the chunk
    int head_row, tail_row;      // row that began before the chunk / that begins here and goes on, or -1
    int began, open;             // the first position's row began before the chunk; the last one's goes on
};

template <bool MAX> __device__ __forceinline__ float comb(float x, float y) { return MAX ? fmaxf(x, y) : x + y; }
template <bool MAX> __device__ __forceinline__ float4 comb4(float4 x, float4 y) {
    if (!MAX) {  // two packed additions
        add2(x.x, x.y, y.x, y.y);
        add2(x.z, x.w, y.z, y.w);
        return x;
    }
    return make_float4(comb<MAX>(x.x, y.x), comb<MAX>(x.y, y.y), comb<MAX>(x.z, y.z), comb<MAX>(x.w, y.w));
}
__device__ __forceinline__ float4 shfl4(float4 v, int from) {
    return make_float4(__shfl_sync(0xffffffffu, v.x, from), __shfl_sync(0xffffffffu, v.y, from), __shfl_sync(0xffffffffu, v.z, from), __shfl_sync(0xffffffffu, v.w, from));
}
__device__ __forceinline__ float4 shfl_xor4(float4 v, int o) {
    return make_float4(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o), __shfl_xor_sync(0xffffffffu, v.z, o), __shfl_xor_sync(0xffffffffu, v.w, o));
}
__device__ __forceinline__ float4 mul4(float4 x, float4 y) { return make_float4(x.x * y.x, x.y * y.y, x.z * y.z, x.w * y.w); }
__device__ __forceinline__ float4 exp_of(float4 x, float4 m) { return make_float4(expf(x.x - m.x), expf(x.y - m.y), expf(x.z - m.z), expf(x.w - m.w)); }
__device__ __forceinline__ float4 over(float4 x, float4 s) { return make_float4(x.x / s.x, x.y / s.y, x.z / s.z, x.w / s.w); }
__device__ __forceinline__ float4 ld_float4(const float* p) {
    const uint4 u = ld_16(p);
    return make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z), __uint_as_float(u.w));
}

// stage_rows for these kernels, which latency bounds: the 64 row pointers of the search's last step serve the scan behind it, so that a
// warp whose rows lie among them waits for two loads, one after the other, instead of six.  (In the reductions, which issue bounds,
// its instructions cost more than the waits: 123 M edges of 128-byte rows 6.13 -> 6.22 ms, 170k bf16 sums over 256-byte rows 271 -> 290 us.)
__device__ __forceinline__ int stage_rows_early(const int64_t* rowptr, int N, int64_t E, int cs, int n, int lane, int* row, uint16_t* start,
                                                bool& began_before) {
    int lo = 0, hi = N;  // the row that holds cs is one of [lo, hi): row_of_position up to its last step
    if (N > 1024) {
        const int guess = (int)((double)cs * ((double)N / (double)E));
        const int idx = guess + (lane - 16) * 64;
        const bool le = idx <= 0 || (idx < N && rowptr[idx] <= cs);
        const int c = __popc(__ballot_sync(0xffffffffu, le));
        if (c > 0) lo = max(lo, guess + (c - 1 - 16) * 64);
        if (c < 32) hi = min(hi, guess + (c - 16) * 64);
    }
    while (hi - lo > 64) {
        const int step = (hi - lo + 31) / 32;
        const int idx = lo + lane * step;
        const bool le = idx < hi && rowptr[idx] <= cs;
        const int c = __popc(__ballot_sync(0xffffffffu, le));
        lo = lo + max(c - 1, 0) * step;
        hi = min(lo + step, hi);
    }
    constexpr int64_t NONE = (int64_t)1 << 62;
    const int ra = lo + 1 + lane, rb32 = ra + 32;
    const int64_t v0 = rowptr[lo], va = ra <= N ? rowptr[ra] : NONE, vb = rb32 <= N ? rowptr[rb32] : NONE;
    const int before = __popc(__ballot_sync(0xffffffffu, ra < hi && va <= cs)) + __popc(__ballot_sync(0xffffffffu, rb32 < hi && vb <= cs));  // < 64
    const int r0 = lo + before;
    auto pointer = [&](int k) {  // rowptr[lo + 1 + k]
        const int64_t x = __shfl_sync(0xffffffffu, va, k & 31), y = __shfl_sync(0xffffffffu, vb, k & 31);
        return k < 32 ? x : y;
    };
    const int64_t sk = pointer(before > 0 ? before - 1 : 0), s0 = before > 0 ? sk : v0, e0 = pointer(before);
    int m = 1;
    const bool none = s0 > cs || e0 <= cs;  // the first position is in no row
    int64_t last_end = none ? (int64_t)cs + n + 1 : e0;
    began_before = none || s0 < cs;
    if (lane == 0) { row[0] = none ? -1 : r0; start[0] = 0; }
    // rows [s, e) that begin in [cs, cs + n), ascending over the lanes; false when one of them does not: the scan is over
    auto take = [&](int r, int64_t s, int64_t e, bool skip) {
        const bool in = !skip && r < N && s < (int64_t)cs + n, live = in && e > s;
        const unsigned lm = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int q = m + __popc(lm & ((1u << lane) - 1u));
            row[q] = r;
            start[q] = (uint16_t)(s - cs);
        }
        m += __popc(lm);
        if (lm) last_end = __shfl_sync(0xffffffffu, e, 31 - __clz(lm));
        return __all_sync(0xffffffffu, skip || in) != 0;
    };
    int rb = s0 > cs ? r0 : N;
    if (s0 <= cs) {
        const int64_t na = __shfl_down_sync(0xffffffffu, va, 1), first_b = __shfl_sync(0xffffffffu, vb, 0), nb = __shfl_down_sync(0xffffffffu, vb, 1);
        if (take(ra, va, lane == 31 ? first_b : na, ra <= r0) && take(rb32, vb, nb, rb32 <= r0 || lane == 31)) rb = lo + 64;  // r0 < lo + 64
    }
    while (rb < N) {
        const int r = rb + lane;
        const int64_t s = r < N ? rowptr[r] : NONE, e = r < N ? rowptr[r + 1] : NONE;
        const int had = m;
        if (!take(r, s, e, false)) break;
        if (m == had) rb = first_row_ending_after(rowptr, rb + 32, N, __shfl_sync(0xffffffffu, s, 0), lane);  // over a run of empty rows
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

// The rows of the warp's share [cs, cs + n) of the chunk, their ends as bits, and what the chunk's ends are; a block barrier
// has to follow before head_row, tail_row, began and open are read.
template <int NT, int HV>
__device__ __forceinline__ void chunk_rows(RowsTile<NT, HV>& S, const int64_t* rowptr, int N, int64_t E, int64_t cs, int n, int n_chunk) {
    using Tile = RowsTile<NT, HV>;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    typename Tile::Rows& R = S.rows[w];
    if (lane < Tile::WP / 32) R.ends[lane] = 0u;
    if (n_chunk <= 0 && threadIdx.x == 0) { S.head_row = S.tail_row = -1; S.began = S.open = 0; }
    if (n <= 0) { __syncwarp(); return; }
    bool began = false;
    const int m = stage_rows_early(rowptr, N, E, (int)cs, n, lane, R.row, R.start, began);
    __syncwarp();
    for (int q = lane; q < m; q += 32) {
        const int e = R.start[q + 1];
        if (e <= n) atomicOr(R.ends + ((e - 1) >> 5), 1u << ((e - 1) & 31));
    }
    if (lane == 0 && w == 0) { S.began = began; S.head_row = began ? R.row[0] : -1; }
    if (lane == 0 && w * Tile::WP + n == n_chunk) {  // the chunk's last warp
        const int last = R.row[m - 1];
        const bool open = R.start[m] > n;
        S.open = open;
        S.tail_row = open && last >= 0 && rowptr[last] >= cs - (int64_t)w * Tile::WP ? last : -1;
    }
    __syncwarp();
}

// this thread's eight end bits
template <int NT, int HV>
__device__ __forceinline__ unsigned run_ends(const RowsTile<NT, HV>& S) {
    const int p = ((threadIdx.x & 31) / HV) * AR_RUN;
    return S.rows[threadIdx.x >> 5].ends[p >> 5] >> (p & 31) & 0xffu;
}

// p[i], i < 8: values of the thread's positions -> totals of their rows inside the chunk.  ends: the run's eight bits.
// The order of a row's additions is fixed: inside the runs, then over the runs of a warp (a scan tree), then over the warps.
// head_part, open_part: where the shares of the chunk's head row (cut_head) and of the row that goes on are written; `one`: their
// positions get 1 (a row that is cut is not divided yet).  Two block barriers.
template <int NT, int HV, bool MAX>
__device__ __forceinline__ void row_totals(RowsTile<NT, HV>& S, float4 (&p)[AR_RUN], unsigned ends, bool cut_head, float* head_part, float* open_part, bool one) {
    using Tile = RowsTile<NT, HV>;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, v = lane % HV, rw = lane / HV, run = w * Tile::RPW + rw;
    const float id = MAX ? -INFINITY : 0.f;
    const float4 none = make_float4(id, id, id, id);
#pragma unroll
    for (int i = 1; i < AR_RUN; ++i)
        if (!(ends >> (i - 1) & 1u)) p[i] = comb4<MAX>(p[i - 1], p[i]);
    // open tails: inclusive segmented scan over the runs
    bool f = ends != 0;
    float4 x = ends >> (AR_RUN - 1) & 1u ? none : p[AR_RUN - 1];
#pragma unroll
    for (int d = HV; d < 32; d <<= 1) {
        const int from = lane >= d ? lane - d : lane;
        const bool g = __shfl_sync(0xffffffffu, (int)f, from) != 0;
        const float4 y = shfl4(x, from);
        if (lane >= d) {
            if (!f) x = comb4<MAX>(y, x);
            f = f || g;
        }
    }
    const unsigned any = __ballot_sync(0xffffffffu, ends != 0);
    if (lane >= 32 - HV) S.warp_open[w * HV + v] = x;
    if (lane == 31) S.warp_closed[w] = f;
    if (lane == 0) {
        unsigned bits = any;
        static_assert(HV <= 2, "one or two lanes per run");
        if (HV == 2) {  // one bit per run: the even bits, together
            bits &= 0x55555555u;
            bits = (bits | bits >> 1) & 0x33333333u;
            bits = (bits | bits >> 2) & 0x0f0f0f0fu;
            bits = (bits | bits >> 4) & 0x00ff00ffu;
            bits = (bits | bits >> 8) & 0x0000ffffu;
        }
        if (Tile::RPW == 32) S.has_end[w] = bits;
        else reinterpret_cast<uint16_t*>(S.has_end)[w] = (uint16_t)bits;
    }
    __syncthreads();
    // what the warps before leave open, then the runs before in this warp
    float4 before = none;
    for (int k = w - 1; k >= 0; --k) {
        before = comb4<MAX>(S.warp_open[k * HV + v], before);
        if (S.warp_closed[k]) break;
    }
    const int left = lane >= HV ? lane - HV : lane;
    const float4 y = shfl4(x, left);
    const bool gl = __shfl_sync(0xffffffffu, (int)f, left) != 0;
    const float4 cin = lane < HV ? before : gl ? y : comb4<MAX>(before, y);
    const int fe = __ffs(ends) - 1;
    float4 first = p[AR_RUN - 1];
#pragma unroll
    for (int i = AR_RUN - 2; i >= 0; --i)
        if (ends >> i & 1u) first = p[i];
    first = comb4<MAX>(cin, first);
    const float4 ones = make_float4(1.f, 1.f, 1.f, 1.f);
    if (ends != 0) {
        bool earlier = false;  // a row ends in the chunk before this run
        for (int k = 0; k <= run / 32; ++k) earlier |= (S.has_end[k] & (k < run / 32 ? 0xffffffffu : (1u << (run & 31)) - 1u)) != 0;
        if (cut_head && !earlier) {
            *reinterpret_cast<float4*>(head_part + 4 * v) = first;
            if (one) first = ones;
        }
        S.total[run * HV + v] = first;
    }
    if (run == Tile::RUNS - 1) {  // the row that goes on past the chunk, if one does
        float4 t = f ? x : comb4<MAX>(before, x);
        if (S.open) {
            *reinterpret_cast<float4*>(open_part + 4 * v) = t;
            if (one) t = ones;
        }
        S.open_total[v] = t;
    }
    __syncthreads();
    float4 cur = none;
    if (!(ends >> (AR_RUN - 1) & 1u)) {  // the row of the last position ends in a later run, or past the chunk
        int e = -1;
        for (int k = (run + 1) / 32; k < (Tile::RUNS + 31) / 32; ++k) {
            const uint32_t bits = S.has_end[k] & (k == (run + 1) / 32 ? 0xffffffffu << ((run + 1) & 31) : 0xffffffffu);
            if (bits) { e = k * 32 + __ffs(bits) - 1; break; }
        }
        cur = e >= 0 ? S.total[e * HV + v] : S.open_total[v];
    }
#pragma unroll
    for (int i = AR_RUN - 1; i >= 0; --i) {
        if (ends >> i & 1u) cur = i == fe ? first : p[i];
        p[i] = cur;
    }
}

// The positions of the thread's run (`here` of them) that lie in rows wholly inside the chunk: not before the chunk's first row end, if
// its first row began before it, and not after the last, if its last row goes on.  (After row_totals.)
template <int NT, int HV>
__device__ __forceinline__ unsigned whole_rows(const RowsTile<NT, HV>& S, int run, unsigned ends, int here) {
    bool earlier = false, later = false;  // a row ends in a run before / after this one
    for (int k = 0; k < (RowsTile<NT, HV>::RUNS + 31) / 32; ++k) {
        const uint32_t bits = S.has_end[k], below = k < run / 32 ? 0xffffffffu : k == run / 32 ? (1u << (run & 31)) - 1u : 0u;
        const uint32_t self = k == run / 32 ? 1u << (run & 31) : 0u;
        earlier |= (bits & below) != 0;
        later |= (bits & ~below & ~self) != 0;
    }
    unsigned mine = (1u << here) - 1u;
    if (S.began && !earlier) mine &= ends ? ~((2u << (__ffs(ends) - 1)) - 1u) : 0u;
    if (S.open && !later) mine &= ends ? (2u << (31 - __clz(ends))) - 1u : 0u;
    return mine;
}
// rows of the warp's share that end before the thread's run
template <int NT, int HV>
__device__ __forceinline__ int rows_before_run(const RowsTile<NT, HV>& S) {
    using Tile = RowsTile<NT, HV>;
    const typename Tile::Rows& R = S.rows[threadIdx.x >> 5];
    const int p0 = ((threadIdx.x & 31) / HV) * AR_RUN;
    int q = 0;
    for (int k = 0; k < Tile::WP / 32; ++k) q += __popc(R.ends[k] & (k < p0 >> 5 ? 0xffffffffu : k == p0 >> 5 ? (1u << (p0 & 31)) - 1u : 0u));
    return q;
}

// ------------------------------------------------------------------ GAT
struct AttnParts {
    int32_t *head_row, *tail_row;  // [chunks]
    float *a, *b;                  // [chunks][2][H]: forward maximum and sum; gradient sum of alpha * dalpha and of dz
};

struct AttnArgs {
    const int64_t* rowptr;
    const int32_t* col;
    const float *al, *ar;
    float slope;
    int32_t N;
    int64_t E;
    float* alpha;   // forward: the result; gradient: read
    float* dz;      // gradient: dalpha, replaced by dz
    float* dar;     // gradient
    AttnParts parts;
};

__device__ __forceinline__ float lrelu(float z, float slope) { return z > 0.f ? z : slope * z; }

// al[col[p]] of the warp's share, lanes over (position, quad): issued before the rows are looked up, all in flight together
template <int HV>
__device__ __forceinline__ void gather_sources(const AttnArgs& A, int64_t cs, int n, float4 (&x)[AR_RUN]) {
    const int lane = threadIdx.x & 31;
    int c[AR_RUN];
#pragma unroll
    for (int k = 0; k < AR_RUN; ++k) {
        const int p = (lane + 32 * k) / HV;
        c[k] = p < n ? ld_stream_i32(A.col + cs + p) : 0;
    }
#pragma unroll
    for (int k = 0; k < AR_RUN; ++k) x[k] = ld_float4(A.al + (size_t)(uint32_t)c[k] * (4 * HV) + 4 * (lane % HV));
}
// body(item, position, z = al[col[p]] + ar[row of p]) for the lane's items (lane + 32 k)
template <int NT, int HV, class Body>
__device__ __forceinline__ void chunk_logits(const AttnArgs& A, const RowsTile<NT, HV>& S, int n, const float4 (&x)[AR_RUN], Body body) {
    const int lane = threadIdx.x & 31;
    const typename RowsTile<NT, HV>::Rows& R = S.rows[threadIdx.x >> 5];
    float4 y[AR_RUN];
    int q = 0;  // rows that end before the word
#pragma unroll
    for (int k = 0; k < AR_RUN; ++k) {
        const int p = (lane + 32 * k) / HV;
        const uint32_t word = R.ends[k / HV];
        const int r = p < n ? max(R.row[q + __popc(word & ((1u << (p & 31)) - 1u))], 0) : 0;
        y[k] = ld_float4(A.ar + (size_t)(uint32_t)r * (4 * HV) + 4 * (lane % HV));
        if (k % HV == HV - 1) q += __popc(word);
    }
#pragma unroll
    for (int k = 0; k < AR_RUN; ++k)
        if ((lane + 32 * k) / HV < n) body(k, (lane + 32 * k) / HV, make_float4(x[k].x + y[k].x, x[k].y + y[k].y, x[k].z + y[k].z, x[k].w + y[k].w));
}

template <int NT, int HV>
__global__ void __launch_bounds__(NT, ar_blocks<NT>())
attention_softmax_kernel(const __grid_constant__ AttnArgs A) {
    using Tile = RowsTile<NT, HV>;
    constexpr int H = 4 * HV;
    extern __shared__ __align__(16) unsigned char ar_smem[];
    Tile& S = *reinterpret_cast<Tile*>(ar_smem);
    float4* const tile = reinterpret_cast<float4*>(ar_smem + sizeof(Tile));
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, v = lane % HV, run = w * Tile::RPW + lane / HV;
    const int64_t c0 = (int64_t)blockIdx.x * Tile::CHUNK;
    const int n_chunk = (int)min((int64_t)Tile::CHUNK, A.E - c0), n = min(max(n_chunk - w * Tile::WP, 0), Tile::WP);
    const int64_t cs = c0 + w * Tile::WP;
    {
        float4 x[AR_RUN];
        gather_sources<HV>(A, cs, n, x);
        chunk_rows<NT, HV>(S, A.rowptr, A.N, A.E, cs, n, n_chunk);
        chunk_logits<NT, HV>(A, S, n, x, [&](int, int p, float4 z) {
            tile[Tile::at(w * Tile::WP + p, v)] = make_float4(lrelu(z.x, A.slope), lrelu(z.y, A.slope), lrelu(z.z, A.slope), lrelu(z.w, A.slope));
        });
    }
    const unsigned ends = run_ends<NT, HV>(S);
    __syncthreads();
    const int here = min(max(n_chunk - run * AR_RUN, 0), AR_RUN);  // positions of this run
    float4 t[AR_RUN];  // (the values stay in the tile: with them in registers too an SM holds two blocks)
    float4* const own = tile + Tile::at(run * AR_RUN, v);  // positions HV apart
    // The maximum of nothing but -inf counts as the lowest finite value: the exponentials are 0 then, not NaN, and so is the share that a
    // row has in a chunk where all its logits are -inf.  A row of nothing else comes to 0 / 0.
    const float4 lowest = make_float4(-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX);
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i) t[i] = i < here ? comb4<true>(lowest, own[i * HV]) : lowest;
    const bool cut_head = S.head_row >= 0;
    // the open row's share is the chunk's tail where the row begins here, else its head
    float* const head = A.parts.a + (size_t)blockIdx.x * 2 * H;
    float* const open = A.parts.a + ((size_t)blockIdx.x * 2 + (S.tail_row >= 0 ? 1 : 0)) * H;
    const size_t to_sums = A.parts.b - A.parts.a;
    row_totals<NT, HV, true>(S, t, ends, cut_head, head, open, false);
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i) {
        t[i] = i < here ? exp_of(own[i * HV], t[i]) : make_float4(0.f, 0.f, 0.f, 0.f);
        own[i * HV] = t[i];
    }
    __syncthreads();  // the totals of the maxima have been read
    row_totals<NT, HV, false>(S, t, ends, cut_head, head + to_sums, open + to_sums, true);
    float* const out = A.alpha + (size_t)(c0 + run * AR_RUN) * H + 4 * v;
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i)
        if (i < here) *reinterpret_cast<float4*>(out + (size_t)i * H) = over(own[i * HV], t[i]);
    if (threadIdx.x == 0) {
        A.parts.head_row[blockIdx.x] = S.head_row;
        A.parts.tail_row[blockIdx.x] = S.tail_row;
    }
}

// the shares that a row has in the chunks c0 .. c1 (slot 1 in c0, where it begins, else 0), lane / HV-th of the warp's (lane % HV: the quad)
template <int HV, class Body>
__device__ __forceinline__ void for_shares(const AttnParts& P, int c0, int c1, Body body) {
    constexpr int H = 4 * HV;
    const int lane = threadIdx.x & 31, v = lane % HV;
    for (int k = c0 + lane / HV; k <= c1; k += 32 / HV) {
        const size_t o = ((size_t)k * 2 + (k == c0 ? 1 : 0)) * H + 4 * v;
        body(P.a + o, P.b + o);
    }
}

// A row in more than AR_MANY chunks has its shares combined once, before the kernels that finish its positions, which else do it in every block
// (a row of k chunks: k * k shares of 64 bytes and more).  The result lies where the shares of the second chunk's other end would: the row
// goes through all of that chunk.  A block per 32 chunks, for the rows that begin in them.  8 heads fp32, one row of 20 M positions: GAT 19.6 -> 2.6 ms, its
// gradient 13.2 -> 8.3 ms, of 2.4 M 1160 -> 890 us and 2325 -> 2260 us; 3 us of 222 on 3 M edges without such a row.
constexpr int AR_MANY = 2048;
__device__ __forceinline__ size_t combined_at(int c0, int H) { return ((size_t)(c0 + 1) * 2 + 1) * H; }

template <int CHUNK, int HV, bool GRADIENT>
__global__ void __launch_bounds__(256)
attention_combine_kernel(const __grid_constant__ AttnArgs A, int chunks) {
    constexpr int H = 4 * HV, W = 8;
    __shared__ float4 part[W][HV];
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, v = lane % HV;
    auto over_block = [&](float4 x, auto op) {
#pragma unroll
        for (int o = 16; o >= HV; o >>= 1) x = op(x, shfl_xor4(x, o));
        __syncthreads();
        if (lane < HV) part[w][lane] = x;
        __syncthreads();
        x = part[0][v];
#pragma unroll
        for (int k = 1; k < W; ++k) x = op(x, part[k][v]);
        return x;
    };
    const auto most = [](float4 x, float4 y) { return comb4<true>(x, y); };
    const auto sum = [](float4 x, float4 y) { return comb4<false>(x, y); };
    int last = 0;  // lane k < 32: the last chunk of the row that begins in the block's k-th chunk, if it reaches far enough
    {
        const int c = (int)blockIdx.x * 32 + lane, r = c < chunks ? A.parts.tail_row[c] : -1;
        if (r >= 0) {
            const int c1 = (int)((A.rowptr[r + 1] - 1) / CHUNK);
            last = c1 - c >= AR_MANY ? c1 : 0;
        }
    }
    for (unsigned mask = __ballot_sync(0xffffffffu, last > 0); mask; mask &= mask - 1) {  // the same in every warp
        const int k0 = __ffs(mask) - 1, c0 = (int)blockIdx.x * 32 + k0, c1 = __shfl_sync(0xffffffffu, last, k0);
        auto share = [&](const float* p, int k) { return ld_float4(p + ((size_t)k * 2 + (k == c0 ? 1 : 0)) * H + 4 * v); };
        const int first = c0 + (int)threadIdx.x / HV, step = 256 / HV;
        float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (GRADIENT) {
#pragma unroll 8
            for (int k = first; k <= c1; k += step) s = sum(s, share(A.parts.a, k));
            s = over_block(s, sum);
            if (threadIdx.x < HV) *reinterpret_cast<float4*>(A.parts.a + combined_at(c0, H) + 4 * v) = s;
        } else {
#pragma unroll 8
            for (int k = first; k <= c1; k += step) m = most(m, share(A.parts.a, k));
            m = over_block(m, most);
#pragma unroll 4
            for (int k = first; k <= c1; k += step) s = sum(s, mul4(share(A.parts.b, k), exp_of(share(A.parts.a, k), m)));
            s = over_block(s, sum);
            if (threadIdx.x < HV) {
                *reinterpret_cast<float4*>(A.parts.a + combined_at(c0, H) + 4 * v) = m;
                *reinterpret_cast<float4*>(A.parts.b + combined_at(c0, H) + 4 * v) = s;
            }
        }
    }
}

// Second kernel of the softmax: a block per (chunk, end of it), for the row that it cuts.
template <int NT, int HV>
__global__ void __launch_bounds__(NT)
attention_softmax_cut_kernel(const __grid_constant__ AttnArgs A) {
    constexpr int H = 4 * HV, CHUNK = RowsTile<NT, HV>::CHUNK;
    pdl_wait();
    const int v = threadIdx.x % HV, c = (int)blockIdx.x, slot = (int)blockIdx.y;
    const int r = slot ? A.parts.tail_row[c] : A.parts.head_row[c];
    if (r < 0) return;
    const int64_t rs = A.rowptr[r], re = A.rowptr[r + 1];
    const int c0 = (int)(rs / CHUNK), c1 = (int)((re - 1) / CHUNK);
    float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c1 - c0 >= AR_MANY) {
        m = ld_float4(A.parts.a + combined_at(c0, H) + 4 * v);
        s = ld_float4(A.parts.b + combined_at(c0, H) + 4 * v);
    } else {
        for_shares<HV>(A.parts, c0, c1, [&](const float* a, const float*) { m = comb4<true>(m, ld_float4(a)); });
#pragma unroll
        for (int o = 16; o >= HV; o >>= 1) m = comb4<true>(m, shfl_xor4(m, o));
        for_shares<HV>(A.parts, c0, c1, [&](const float* a, const float* b) { s = comb4<false>(s, mul4(ld_float4(b), exp_of(ld_float4(a), m))); });
#pragma unroll
        for (int o = 16; o >= HV; o >>= 1) s = comb4<false>(s, shfl_xor4(s, o));
    }
    const float4 f = over(exp_of(ld_float4(A.parts.a + ((size_t)c * 2 + slot) * H + 4 * v), m), s);
    const int64_t p0 = max(rs, (int64_t)c * CHUNK), p1 = min(re, (int64_t)(c + 1) * CHUNK);
    float4* const al = reinterpret_cast<float4*>(A.alpha);
#pragma unroll 4
    for (int64_t t = p0 * HV + threadIdx.x; t < p1 * HV; t += NT) al[t] = mul4(al[t], f);  // NT and p0 * HV are multiples of HV: the quad stays
}

// dz = alpha * (dalpha - d) * LeakyReLU'(z), d = sum over the row of alpha * dalpha; pos: bits of z > 0
__device__ __forceinline__ float4 attn_dz(float4 a, float4 b, float4 d, unsigned pos, float slope) {
    return make_float4(a.x * (b.x - d.x) * (pos & 1u ? 1.f : slope), a.y * (b.y - d.y) * (pos & 2u ? 1.f : slope),
                       a.z * (b.z - d.z) * (pos & 4u ? 1.f : slope), a.w * (b.w - d.w) * (pos & 8u ? 1.f : slope));
}
__device__ __forceinline__ unsigned sign_bits(float4 z) { return (z.x > 0.f ? 1u : 0u) | (z.y > 0.f ? 2u : 0u) | (z.z > 0.f ? 4u : 0u) | (z.w > 0.f ? 8u : 0u); }

template <int NT, int HV>
__global__ void __launch_bounds__(NT, 512 / NT)
attention_gradient_kernel(const __grid_constant__ AttnArgs A) {
    using Tile = RowsTile<NT, HV>;
    constexpr int H = 4 * HV;
    extern __shared__ __align__(16) unsigned char ar_smem[];
    Tile& S = *reinterpret_cast<Tile*>(ar_smem);
    float4* const tile = reinterpret_cast<float4*>(ar_smem + sizeof(Tile));
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, v = lane % HV, run = w * Tile::RPW + lane / HV;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t c0 = (int64_t)blockIdx.x * Tile::CHUNK;
    const int n_chunk = (int)min((int64_t)Tile::CHUNK, A.E - c0), n = min(max(n_chunk - w * Tile::WP, 0), Tile::WP);
    const int64_t cs = c0 + w * Tile::WP;
    // the lane's items: (position, quad) lane + 32 k of the warp's share; all loads of the chunk are on their way before its rows are
    // looked up, and alpha and dalpha stay in registers but for 52 to 60 bytes (read again for dz, at three blocks per SM: 1.05 times as long)
    const float* const alpha = A.alpha + (size_t)cs * H;
    float* const dz = A.dz + (size_t)cs * H;
    unsigned pos = 0;  // four bits per item: z > 0
    float4 a[AR_RUN], b[AR_RUN];
    {
        float4 x[AR_RUN];
        gather_sources<HV>(A, cs, n, x);
#pragma unroll
        for (int k = 0; k < AR_RUN; ++k)
            if ((lane + 32 * k) / HV < n) {
                a[k] = ld_float4(alpha + 4 * (lane + 32 * k));
                b[k] = ld_float4(dz + 4 * (lane + 32 * k));
            }
        chunk_rows<NT, HV>(S, A.rowptr, A.N, A.E, cs, n, n_chunk);
        chunk_logits<NT, HV>(A, S, n, x, [&](int k, int, float4 z) { pos |= sign_bits(z) << (4 * k); });
    }
#pragma unroll
    for (int k = 0; k < AR_RUN; ++k)
        if ((lane + 32 * k) / HV < n) tile[Tile::at(w * Tile::WP + (lane + 32 * k) / HV, v)] = mul4(a[k], b[k]);
    const unsigned ends = run_ends<NT, HV>(S);
    __syncthreads();
    const int here = min(max(n_chunk - run * AR_RUN, 0), AR_RUN);
    float4 t[AR_RUN];
    float4* const own = tile + Tile::at(run * AR_RUN, v);  // positions HV apart
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i) t[i] = i < here ? own[i * HV] : zero;
    const bool cut_head = S.head_row >= 0;
    float* const head_part = A.parts.a + (size_t)blockIdx.x * 2 * H;
    float* const open_part = A.parts.a + ((size_t)blockIdx.x * 2 + (S.tail_row >= 0 ? 1 : 0)) * H;
    row_totals<NT, HV, false>(S, t, ends, cut_head, head_part, open_part, false);
    const unsigned mine = whole_rows<NT, HV>(S, run, ends, here);  // the others are left to the second kernel
    if (v == 0) S.whole[run] = (uint8_t)mine;
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i) own[i * HV] = t[i];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < AR_RUN; ++k) {
        const int p = w * Tile::WP + (lane + 32 * k) / HV;
        if (p - w * Tile::WP < n) {
            float4& d = tile[Tile::at(p, v)];
            float4 o = zero;
            if (S.whole[p / AR_RUN] >> (p % AR_RUN) & 1u) {
                o = attn_dz(a[k], b[k], d, pos >> (4 * k) & 15u, A.slope);
                *reinterpret_cast<float4*>(dz + 4 * (lane + 32 * k)) = o;
            }
            d = o;
        }
    }
    __syncthreads();  // also: the totals have been read
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i) t[i] = i < here ? own[i * HV] : zero;
    // (the shares of the cut rows are zero here; the second kernel writes them, into b)
    row_totals<NT, HV, false>(S, t, ends, false, nullptr, A.parts.b + ((size_t)blockIdx.x * 2) * H, false);
    const typename Tile::Rows& R = S.rows[w];
    int q = rows_before_run<NT, HV>(S);
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i)
        if (ends >> i & 1u) {
            const int r = R.row[q++];
            if (r >= 0 && (mine >> i & 1u)) *reinterpret_cast<float4*>(A.dar + (size_t)r * H + 4 * v) = t[i];
        }
    if (threadIdx.x == 0 && n_chunk > 0) {
        A.parts.head_row[blockIdx.x] = S.head_row;
        A.parts.tail_row[blockIdx.x] = S.tail_row;
    }
    {  // rows without edges: the blocks share them
        const int64_t per = ((int64_t)A.N + gridDim.x - 1) / gridDim.x, r0 = per * blockIdx.x, r1 = min(r0 + per, (int64_t)A.N);
        for (int64_t r = r0 + threadIdx.x; r < r1; r += NT)
            if (A.rowptr[r + 1] == A.rowptr[r])
#pragma unroll
                for (int q = 0; q < HV; ++q) *reinterpret_cast<float4*>(A.dar + (size_t)r * H + 4 * q) = zero;
    }
}

// Second kernel of the gradient: dz of the chunk's positions of the rows that its ends cut, and its share of their dar.
template <int NT, int HV>
__global__ void __launch_bounds__(NT)
attention_gradient_cut_kernel(const __grid_constant__ AttnArgs A) {
    constexpr int H = 4 * HV, CHUNK = RowsTile<NT, HV>::CHUNK;
    __shared__ float4 sums[NT / 32][HV];
    pdl_wait();
    const int v = threadIdx.x % HV, c = (int)blockIdx.x, slot = (int)blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int r = slot ? A.parts.tail_row[c] : A.parts.head_row[c];
    if (r < 0) return;
    const int64_t rs = A.rowptr[r], re = A.rowptr[r + 1];
    const int c0 = (int)(rs / CHUNK), c1 = (int)((re - 1) / CHUNK);
    float4 d = make_float4(0.f, 0.f, 0.f, 0.f), s = d;
    if (c1 - c0 >= AR_MANY) {
        d = ld_float4(A.parts.a + combined_at(c0, H) + 4 * v);
    } else {
        for_shares<HV>(A.parts, c0, c1, [&](const float* a, const float*) { d = comb4<false>(d, ld_float4(a)); });
#pragma unroll
        for (int o = 16; o >= HV; o >>= 1) d = comb4<false>(d, shfl_xor4(d, o));
    }
    const float4 arv = ld_float4(A.ar + (size_t)r * H + 4 * v);
    const int64_t p0 = max(rs, (int64_t)c * CHUNK), p1 = min(re, (int64_t)(c + 1) * CHUNK);
#pragma unroll 4
    for (int64_t t = p0 * HV + threadIdx.x; t < p1 * HV; t += NT) {
        const float4 x = ld_float4(A.al + (size_t)(uint32_t)A.col[t / HV] * H + 4 * v);
        const float4 a = ld_float4(A.alpha + 4 * t), b = ld_float4(A.dz + 4 * t);
        const float4 o = attn_dz(a, b, d, sign_bits(make_float4(x.x + arv.x, x.y + arv.y, x.z + arv.z, x.w + arv.w)), A.slope);
        *reinterpret_cast<float4*>(A.dz + 4 * t) = o;
        s = comb4<false>(s, o);
    }
#pragma unroll
    for (int o = 16; o >= HV; o >>= 1) s = comb4<false>(s, shfl_xor4(s, o));
    if (lane < HV) sums[w][lane] = s;
    __syncthreads();
    if (threadIdx.x < HV) {
        float4 t = sums[0][threadIdx.x];
#pragma unroll
        for (int k = 1; k < NT / 32; ++k) t = comb4<false>(t, sums[k][threadIdx.x]);
        *reinterpret_cast<float4*>(A.parts.b + ((size_t)c * 2 + slot) * H + 4 * threadIdx.x) = t;
    }
}

// third: dar of the rows that are cut, a warp per chunk in which one begins
template <int NT, int HV>
__global__ void __launch_bounds__(256)
attention_gradient_sums_kernel(const __grid_constant__ AttnArgs A, int chunks) {
    constexpr int H = 4 * HV, CHUNK = RowsTile<NT, HV>::CHUNK;
    pdl_wait();
    const int c = (int)blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= chunks) return;
    const int r = A.parts.tail_row[c];
    if (r < 0) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for_shares<HV>(A.parts, c, (int)((A.rowptr[r + 1] - 1) / CHUNK), [&](const float*, const float* b) { s = comb4<false>(s, ld_float4(b)); });
#pragma unroll
    for (int o = 16; o >= HV; o >>= 1) s = comb4<false>(s, shfl_xor4(s, o));
    if (lane < HV) *reinterpret_cast<float4*>(A.dar + (size_t)r * H + 4 * lane) = s;
}

// ------------------------------------------------------------------ edge softmax: values given, no workspace
template <typename T> __device__ __forceinline__ float4 ld_quad(const T* p);
template <> __device__ __forceinline__ float4 ld_quad<float>(const float* p) { return ld_float4(p); }
template <> __device__ __forceinline__ float4 ld_quad<__nv_bfloat16>(const __nv_bfloat16* p) {
    uint2 u;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(u.x), "=r"(u.y) : "l"(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
}
template <typename T> __device__ __forceinline__ void st_quad(T* p, float4 v);
template <> __device__ __forceinline__ void st_quad<float>(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
template <> __device__ __forceinline__ void st_quad<__nv_bfloat16>(__nv_bfloat16* p, float4 v) {
    *reinterpret_cast<uint2*>(p) = make_uint2(Chunk<__nv_bfloat16>::pack2(v.x, v.y), Chunk<__nv_bfloat16>::pack2(v.z, v.w));
}

struct SoftmaxArgs {
    const int64_t* rowptr;
    const void *x, *y;  // forward: logits; backward: alpha, dalpha
    void* out;          // alpha; dlogits
    float *rowmax, *rowsum;  // [N,H] or nullptr
    int32_t N;
    int64_t E;
    int64_t over;  // rows of more positions are left to others
};

// v over the threads of a quad: lanes, then warps in order
template <int NT, int HV, bool MAX>
__device__ __forceinline__ float4 block_quads(RowsTile<NT, HV>& S, float4 v) {
#pragma unroll
    for (int o = 16; o >= HV; o >>= 1) v = comb4<MAX>(v, shfl_xor4(v, o));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane < HV) S.warp_open[w * HV + lane] = v;
    __syncthreads();
    v = S.warp_open[lane % HV];
#pragma unroll
    for (int k = 1; k < NT / 32; ++k) v = comb4<MAX>(v, S.warp_open[k * HV + lane % HV]);
    return v;
}
__device__ __forceinline__ void put_stats(float* to, size_t at, float4 v) {  // (any alignment)
    if (!to) return;
    if ((reinterpret_cast<uintptr_t>(to) & 15) == 0) *reinterpret_cast<float4*>(to + at) = v;
    else { to[at] = v.x; to[at + 1] = v.y; to[at + 2] = v.z; to[at + 3] = v.w; }
}
__device__ __forceinline__ float4 softmax_grad(float4 a, float4 b, float4 d) {
    return make_float4(a.x * (b.x - d.x), a.y * (b.y - d.y), a.z * (b.z - d.z), a.w * (b.w - d.w));
}

template <typename T, int NT, int HV, bool BACKWARD>
__global__ void __launch_bounds__(NT, ar_blocks<NT>())
edge_softmax_chunk_kernel(const __grid_constant__ SoftmaxArgs A) {
    using Tile = RowsTile<NT, HV>;
    constexpr int H = 4 * HV, HALF = AR_RUN / 2;
    extern __shared__ __align__(16) unsigned char ar_smem[];
    __shared__ __align__(16) float unused[H];  // shares of cut rows
    Tile& S = *reinterpret_cast<Tile*>(ar_smem);
    float4* const tile = reinterpret_cast<float4*>(ar_smem + sizeof(Tile));
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, v = lane % HV, run = w * Tile::RPW + lane / HV;
    const T* const X = reinterpret_cast<const T*>(A.x);
    const T* const Y = reinterpret_cast<const T*>(A.y);
    T* const O = reinterpret_cast<T*>(A.out);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f), least = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (!BACKWARD && (A.rowmax || A.rowsum)) {  // rows without edges: the blocks share them
        const int64_t per = ((int64_t)A.N + gridDim.x - 1) / gridDim.x, r0 = per * blockIdx.x, r1 = min(r0 + per, (int64_t)A.N);
        for (int64_t r = r0 + threadIdx.x; r < r1; r += NT)
            if (A.rowptr[r + 1] == A.rowptr[r])
                for (int q = 0; q < HV; ++q) { put_stats(A.rowmax, (size_t)r * H + 4 * q, zero); put_stats(A.rowsum, (size_t)r * H + 4 * q, zero); }
    }
    const int64_t c0 = (int64_t)blockIdx.x * Tile::CHUNK;
    const int n_chunk = (int)min((int64_t)Tile::CHUNK, A.E - c0), n = min(max(n_chunk - w * Tile::WP, 0), Tile::WP);
    const int64_t cs = c0 + w * Tile::WP;
    const T* const x = X + (size_t)cs * H;
    const T* const y = BACKWARD ? Y + (size_t)cs * H : nullptr;
    // the lane's items, (position, quad) lane + 32 k of the warp's share, half of them at a time
    auto pairs = [&](int k0, float4 (&a)[HALF], float4 (&b)[HALF]) {
#pragma unroll
        for (int k = 0; k < HALF; ++k)
            if ((lane + 32 * (k0 + k)) / HV < n) {
                a[k] = ld_quad(x + 4 * (lane + 32 * (k0 + k)));
                if (BACKWARD) b[k] = ld_quad(y + 4 * (lane + 32 * (k0 + k)));
            }
    };
    {
        float4 a0[HALF], b0[HALF], a1[HALF], b1[HALF];
        pairs(0, a0, b0);
        if (!BACKWARD) pairs(HALF, a1, b1);
        chunk_rows<NT, HV>(S, A.rowptr, A.N, A.E, cs, n, n_chunk);
#pragma unroll
        for (int k = 0; k < HALF; ++k)
            if ((lane + 32 * k) / HV < n) tile[Tile::at(w * Tile::WP + (lane + 32 * k) / HV, v)] = BACKWARD ? mul4(a0[k], b0[k]) : a0[k];
        if (BACKWARD) pairs(HALF, a1, b1);
#pragma unroll
        for (int k = 0; k < HALF; ++k)
            if ((lane + 32 * (HALF + k)) / HV < n) tile[Tile::at(w * Tile::WP + (lane + 32 * (HALF + k)) / HV, v)] = BACKWARD ? mul4(a1[k], b1[k]) : a1[k];
    }
    const unsigned ends = run_ends<NT, HV>(S);
    __syncthreads();
    const int here = min(max(n_chunk - run * AR_RUN, 0), AR_RUN);
    float4* const own = tile + Tile::at(run * AR_RUN, v);  // positions HV apart
    float4 t[AR_RUN];
#pragma unroll
    for (int i = 0; i < AR_RUN; ++i) t[i] = i < here ? own[i * HV] : BACKWARD ? zero : least;
    row_totals<NT, HV, !BACKWARD>(S, t, ends, false, unused, unused, false);
    const unsigned mine = whole_rows<NT, HV>(S, run, ends, here);
    if (BACKWARD) {
        if (v == 0) S.whole[run] = (uint8_t)mine;
#pragma unroll
        for (int i = 0; i < AR_RUN; ++i) own[i * HV] = t[i];
        __syncwarp();
#pragma unroll
        for (int k0 = 0; k0 < AR_RUN; k0 += HALF) {
            float4 a[HALF], b[HALF];
            pairs(k0, a, b);
#pragma unroll
            for (int k = 0; k < HALF; ++k) {
                const int p = w * Tile::WP + (lane + 32 * (k0 + k)) / HV;
                if (p - w * Tile::WP < n && (S.whole[p / AR_RUN] >> (p % AR_RUN) & 1u))
                    st_quad(O + (size_t)cs * H + 4 * (lane + 32 * (k0 + k)), softmax_grad(a[k], b[k], tile[Tile::at(p, v)]));
            }
        }
    } else {
        const int q0 = rows_before_run<NT, HV>(S);
        const typename Tile::Rows& R = S.rows[w];
        auto stats = [&](float* to) {  // at the ends of whole rows
            if (!to) return;
            int q = q0;
#pragma unroll
            for (int i = 0; i < AR_RUN; ++i)
                if (ends >> i & 1u) {
                    const int r = R.row[q++];
                    if (r >= 0 && (mine >> i & 1u)) put_stats(to, (size_t)r * H + 4 * v, t[i]);
                }
        };
        stats(A.rowmax);
#pragma unroll
        for (int i = 0; i < AR_RUN; ++i) {
            t[i] = i < here ? exp_of(own[i * HV], t[i]) : zero;
            if (mine >> i & 1u) own[i * HV] = t[i];
        }
        __syncthreads();  // the totals of the maxima have been read
        row_totals<NT, HV, false>(S, t, ends, false, unused, unused, false);
        stats(A.rowsum);
        T* const out = O + (size_t)(c0 + run * AR_RUN) * H + 4 * v;
#pragma unroll
        for (int i = 0; i < AR_RUN; ++i)
            if (mine >> i & 1u) st_quad(out + (size_t)i * H, over(own[i * HV], t[i]));
    }
    // ---- the rows that the chunk's ends cut: all of the row is read, this chunk's positions of it are written
    const int head_row = S.head_row, tail_row = S.tail_row;
#pragma unroll 1
    for (int slot = 0; slot < 2; ++slot) {
        const int r = slot ? tail_row : head_row;  // the same in every thread
        if (r < 0) continue;
        const int64_t rs = A.rowptr[r], re = A.rowptr[r + 1], t0 = rs * HV + threadIdx.x, t1 = re * HV;  // NT, rs * HV: multiples of HV
        if (re - rs > A.over) continue;
        float4 m = least, s = zero;
        if (BACKWARD) {
#pragma unroll 4
            for (int64_t k = t0; k < t1; k += NT) {
                const float4 a = ld_quad(X + 4 * k), b = ld_quad(Y + 4 * k);
                s = make_float4(fmaf(a.x, b.x, s.x), fmaf(a.y, b.y, s.y), fmaf(a.z, b.z, s.z), fmaf(a.w, b.w, s.w));
            }
        } else {
#pragma unroll 8
            for (int64_t k = t0; k < t1; k += NT) m = comb4<true>(m, ld_quad(X + 4 * k));
            m = block_quads<NT, HV, true>(S, m);
#pragma unroll 8
            for (int64_t k = t0; k < t1; k += NT) s = comb4<false>(s, exp_of(ld_quad(X + 4 * k), m));
        }
        s = block_quads<NT, HV, false>(S, s);
        const int64_t p0 = max(rs, c0), p1 = min(re, c0 + n_chunk);
#pragma unroll 4
        for (int64_t k = p0 * HV + threadIdx.x; k < p1 * HV; k += NT) {
            const float4 a = ld_quad(X + 4 * k);
            if (BACKWARD) st_quad(O + 4 * k, softmax_grad(a, ld_quad(Y + 4 * k), s));
            else st_quad(O + 4 * k, over(exp_of(a, m), s));
        }
        if (!BACKWARD && slot && threadIdx.x < HV) {
            put_stats(A.rowmax, (size_t)r * H + 4 * threadIdx.x, m);
            put_stats(A.rowsum, (size_t)r * H + 4 * threadIdx.x, s);
        }
    }
}

// ------------------------------------------------------------------ launches
constexpr int AR_SLOT = 20;  // of allow_big_smem: 24 of them
// Chunks of 256 threads are 1024 (8 heads) or 2048 (4 heads) positions; small graphs take a quarter, so that all SMs have work.  A quarter / whole, us, R-MAT
// of mean length 12, graphs replayed, edges * heads / 8 of 100, 200, 300, 400 and 600 Ki: edge softmax of 8 heads 14.5 / 15.8, 19.6 / 20.2, 21.6 / 21.8,
// 26.9 / 22.9, 37.9 / 34.0, of 4 heads 17.3 / 13.8, 20.9 / 19.5, 22.1 / 22.1, 27.5 / 22.4, 39.6 / 32.4; GAT of 8 heads 28.0 / 29.0, 35.8 / 35.9, 42.4 / 41.4,
// 42.3 / 41.8, 60.2 / 61.6, its gradient within 2 % throughout.
constexpr int64_t AR_SMALL = 400 * 1024;  // edges * heads / 8
// Edge softmax: rows of up to so many chunks' positions are read by every block that they reach, longer ones by a cluster (1.6 M edges, R-MAT, 8
// heads fp32, of 2, 4, 8 and 16 chunks: 80, 78, 75 and 74 us; 300 k edges: 46, 31, 25 and 24 us; 160 k: 24, 24, 20 and 27 us).
constexpr int AR_SPAN = 8;

template <int NT, int HV>
static gnn_status softmax_launch(const char* who, const AttnArgs& A, int chunks, cudaStream_t st) {
    using Tile = RowsTile<NT, HV>;
    constexpr size_t smem = sizeof(Tile) + Tile::TILE * 16;
    const gnn_status rc = allow_big_smem(who, (const void*)attention_softmax_kernel<NT, HV>, AR_SLOT + (NT == 256) * 2 + HV - 1, smem);
    if (rc != GNN_OK) return rc;
    launch_overlapped(attention_softmax_kernel<NT, HV>, dim3(chunks), dim3(NT), smem, st, A);
    if constexpr (NT == 256)  // (small graphs have at most 1600 chunks)
        if (chunks > AR_MANY) launch_overlapped(attention_combine_kernel<Tile::CHUNK, HV, false>, dim3((unsigned)ceil_div(chunks, 32)), dim3(256), 0, st, A, chunks);
    launch_overlapped(attention_softmax_cut_kernel<NT, HV>, dim3(chunks, 2), dim3(NT), 0, st, A);
    return GNN_OK;
}

template <int NT, int HV>
static gnn_status gradient_launch(const char* who, const AttnArgs& A, int chunks, cudaStream_t st) {
    using Tile = RowsTile<NT, HV>;
    constexpr size_t smem = sizeof(Tile) + Tile::TILE * 16;
    const gnn_status rc = allow_big_smem(who, (const void*)attention_gradient_kernel<NT, HV>, AR_SLOT + 4 + (NT == 256) * 2 + HV - 1, smem);
    if (rc != GNN_OK) return rc;
    launch_overlapped(attention_gradient_kernel<NT, HV>, dim3(chunks > 0 ? chunks : 1), dim3(NT), smem, st, A);
    if (chunks == 0) return GNN_OK;
    if constexpr (NT == 256)  // (small graphs have at most 1600 chunks)
        if (chunks > AR_MANY) launch_overlapped(attention_combine_kernel<Tile::CHUNK, HV, true>, dim3((unsigned)ceil_div(chunks, 32)), dim3(256), 0, st, A, chunks);
    launch_overlapped(attention_gradient_cut_kernel<NT, HV>, dim3(chunks, 2), dim3(NT), 0, st, A);
    launch_overlapped(attention_gradient_sums_kernel<NT, HV>, dim3((unsigned)ceil_div(chunks, 8)), dim3(256), 0, st, A, chunks);
    return GNN_OK;
}

static int ar_chunk(int64_t E, int H) { return (E * H / 8 < AR_SMALL ? 64 : 256) / (H / 4) * AR_RUN; }

// The shares of the cut rows fit the workspace of the chunked reduction, which the attention calls are given and whose smallest room is a partial row per 1024
// positions: a head has four features or more, so 4 heads need 72 bytes per 512 or 2048 positions of at least 132 per 1024, 8 heads 136 per 256 or 1024 of at
// least 260 per 1024.
// dz and dar null: alpha = softmax over each row of LeakyReLU(al[col] + ar[row]).  Else dz (dalpha on entry) and dar from alpha.
gnn_status attention_rows(const char* who, const gnn_csr* g, const float* al, const float* ar, float slope, int H, float* alpha, float* dz, float* dar,
                          void* ws, size_t ws_bytes, cudaStream_t st) {
    const int chunk = ar_chunk(g->E, H);
    const int64_t chunks = ceil_div(g->E, (int64_t)chunk);
    const bool small = chunk == 64 / (H / 4) * AR_RUN;
    const size_t rows = ((size_t)chunks * 8 + 15) & ~(size_t)15, part = (size_t)chunks * 2 * H * 4;
    GNN_REQUIRE(ws && aligned16(ws) && ws_bytes >= rows + 2 * part, GNN_ERR_WORKSPACE_TOO_SMALL, "%s: %zu bytes needed for the rows that chunks cut", who, rows + 2 * part);
    GNN_REQUIRE(g->E < ((int64_t)1 << 31) - 1024, GNN_ERR_UNSUPPORTED, "%s: positions must fit 32 bits (E < 2^31)", who);
    AttnArgs A = {};
    A.rowptr = g->rowptr; A.col = g->col; A.al = al; A.ar = ar; A.slope = slope; A.N = g->N; A.E = g->E;
    A.alpha = alpha; A.dz = dz; A.dar = dar;
    char* p = (char*)ws;
    A.parts.head_row = (int32_t*)p; A.parts.tail_row = A.parts.head_row + chunks;
    A.parts.a = (float*)(p + rows); A.parts.b = (float*)(p + rows + part);
    gnn_status rc;
#define GNN_AR(NT, HV) rc = dz ? gradient_launch<NT, HV>(who, A, (int)chunks, st) : softmax_launch<NT, HV>(who, A, (int)chunks, st)
    if (H == 4) { if (small) GNN_AR(64, 1); else GNN_AR(256, 1); }
    else { if (small) GNN_AR(64, 2); else GNN_AR(256, 2); }
#undef GNN_AR
    if (rc != GNN_OK) return rc;
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

template <typename T, int NT, int HV, bool BACKWARD>
static gnn_status edge_softmax_launch(const char* who, const SoftmaxArgs& A, cudaStream_t st) {
    using Tile = RowsTile<NT, HV>;
    constexpr size_t smem = sizeof(Tile) + Tile::TILE * 16;
    const gnn_status rc = allow_big_smem(who, (const void*)edge_softmax_chunk_kernel<T, NT, HV, BACKWARD>,
                                         AR_SLOT + 8 + (sizeof(T) == 2) * 8 + (NT == 256) * 4 + (HV - 1) * 2 + BACKWARD, smem);
    if (rc != GNN_OK) return rc;
    launch_overlapped(edge_softmax_chunk_kernel<T, NT, HV, BACKWARD>, dim3((unsigned)ceil_div(A.E, (int64_t)Tile::CHUNK)), dim3(NT), smem, st, A);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

template <typename T, bool BACKWARD>
static gnn_status edge_softmax_dispatch(const char* who, const SoftmaxArgs& A, int H, cudaStream_t st) {
    const bool small = A.E * H / 8 < AR_SMALL;
    if (H == 4) return small ? edge_softmax_launch<T, 64, 1, BACKWARD>(who, A, st) : edge_softmax_launch<T, 256, 1, BACKWARD>(who, A, st);
    return small ? edge_softmax_launch<T, 64, 2, BACKWARD>(who, A, st) : edge_softmax_launch<T, 256, 2, BACKWARD>(who, A, st);
}

// Few edges on many nodes: a warp here walks the runs of empty rows between its positions, where the kernels that take every row on its own spread
// them over the machine.  Rows / chunks, us, graphs replayed: 8 Ki edges on 128 Ki nodes, 4 heads, edge softmax 29 / 54, GAT 44 / 86, its gradient
// 92 / 146; 100 Ki edges on 1.6 M nodes 203 / 61, 395 / 316, 648 / 550; 1000 edges on 2 M nodes, statistics of the softmax 0.23 / 6.7 ms.
static bool mostly_empty(int32_t N, int64_t E, int H) { return N > E && E * H < 150 * 1000; }
bool attention_by_chunks(int32_t N, int64_t E, int H) { return (H == 4 || H == 8) && E > 0 && !mostly_empty(N, E, H); }

// The GAT gradient by chunks is a chain of three kernels; on small graphs the three that take rows by length, side by side, are done sooner, and where
// rows are long and many they read faster.  The call by rows / by chunks, us.  R-MAT, graphs replayed, 4 heads: 8 k edges 36 / 45, 40 k 40 / 52 (calls in
// a row 53 / 56), 160 k 52 / 60 with rows up to 4820, 53 / 63, 320 k 74 / 76; 8 heads: 8 k 44 / 54, 160 k 67 / 69.  The line lies as low as it does for graphs
// with one row of all edges: 4 heads, 32 k 62 / 54, 64 k 103 / 64; 8 heads, 16 k 74 / 58, 32 k 118 / 65.  Long rows, 8 heads: 24 M edges of mean
// length 64 3290 / 3690, 48 M, 32 7440 / 8110, 24 M of even length 64 3300 / 3780.
bool attention_gradient_by_chunks(int32_t N, int64_t E, int H) {
    const double mean = (double)E / (N > 0 ? N : 1);
    return attention_by_chunks(N, E, H) && E * H / 8 >= 24 * 1024 && E * mean * mean < (H == 8 ? 1.5e10 : 9e10);
}

// Long rows on average: the edge softmax by chunks keeps 32 to 47 us per million edges of 8 heads whatever the rows' lengths, a warp or block
// per row falls to 18 there.  Rows by length / by chunks, us, R-MAT if not said otherwise.  8 heads, forward: 12 M edges of mean length 16 548 / 533,
// 32 488 / 546; 24 M, 8 1282 / 1040, 16 1017 / 1070; 3 M of even length 32 75 / 102; gradient: 12 M, 32 382 / 356, 24 M, 16 769 / 701, 32 635 / 703.
// 4 heads, forward: 24 M, 32 673 / 553, 64 527 / 564; gradient: 48 M, 32 808 / 713, 64 656 / 715.
static bool long_on_average(int32_t N, int64_t E, int H, bool backward) {
    const double mean = (double)E / N;
    return E >= 2000 * 1000 && mean >= 12 && E * mean * mean >= (H == 8 ? (backward ? 2e10 : 3e9) : (backward ? 1e11 : 4e10));
}

// 4 and 8 heads, four values to an access, results that do not lie over what other blocks still read, and rows that chunks suit
bool edge_softmax_chunks_fit(int32_t N, int64_t E, int H, gnn_dtype dtype, const void* x, const void* y, const void* out) {
    if (!attention_by_chunks(N, E, H) || E >= ((int64_t)1 << 31) - 1024 || long_on_average(N, E, H, y != nullptr)) return false;
    const size_t bytes = (size_t)E * H * elem_size(dtype), quad = 4 * elem_size(dtype);
    auto apart = [&](const void* p) { return (const char*)p + bytes <= (const char*)out || (const char*)out + bytes <= (const char*)p; };
    return ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(out)) & (quad - 1)) == 0 && apart(x) && (!y || apart(y));
}

// Up to 8 Ki edges without the clusters, whose launch beside this one is 2 us of 9 there; a single row of 8000 positions of 8 heads takes 29 us (one block
// for all of it: 37 us).
int64_t edge_softmax_chunk_rows(int64_t E, int H) { return E <= 8192 ? E : (int64_t)AR_SPAN * ar_chunk(E, H); }

// y null: out = softmax of x over each row; else out = x * (y - sum over the row of x * y)
gnn_status edge_softmax_chunks(const char* who, const gnn_csr* g, const void* x, const void* y, int H, gnn_dtype dtype, void* out, float* rowmax, float* rowsum,
                               cudaStream_t st) {
    const SoftmaxArgs A = {g->rowptr, x, y, out, rowmax, rowsum, g->N, g->E, edge_softmax_chunk_rows(g->E, H)};
    if (dtype == GNN_F32) return y ? edge_softmax_dispatch<float, true>(who, A, H, st) : edge_softmax_dispatch<float, false>(who, A, H, st);
    return y ? edge_softmax_dispatch<__nv_bfloat16, true>(who, A, H, st) : edge_softmax_dispatch<__nv_bfloat16, false>(who, A, H, st);
}

}  // namespace gnn
