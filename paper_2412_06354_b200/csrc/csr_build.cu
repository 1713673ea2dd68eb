// Graph set-up: COO -> sparse forms (stable LSD radix sort), degrees, GCN normalisation,
// self-loops, edge-data permutation.  Integer results are unique and bit-exact.
#include <stdarg.h>

#include "flag_slots.h"
#include "reduce_params.cuh"

namespace gnn {

static thread_local char g_err[512] = "";
void set_error(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

// ------------------------------------------------------------------ validation of a caller-built sparse form
// Bits of the result word; every read stays in bounds whatever the arrays hold (an index is used only after its
// range check, row look-ups search rowptr[0..N] by position).
enum : int {
    CSR_BAD_ROWPTR = 1,     // rowptr / rowptrT: first entry 0, last entry E, non-decreasing
    CSR_BAD_NODE = 2,       // col / colT outside [0, N)
    CSR_BAD_EDGE = 4,       // eid / eidT / t2f outside [0, E)
    CSR_BAD_PERM = 8,       // eid, eidT or t2f holds a value twice
    CSR_BAD_ORDER = 16,     // edge ids not ascending inside a row (the order that makes the forms unique)
    CSR_BAD_CROSS = 32,     // the two forms disagree: position t2f[q] is not the same edge as transposed position q
};

__device__ __forceinline__ int csr_row_of(const int64_t* __restrict__ rowptr, int32_t N, int64_t p) {
    int lo = 0, hi = N;  // largest i in [0, N) with rowptr[i] <= p (rowptr[0] = 0 <= p when the pointers are sound)
    while (hi - lo > 1) {
        const int mid = lo + (hi - lo) / 2;
        if (rowptr[mid] <= p) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void csr_validate_pointers_kernel(int32_t N, int64_t E, const int64_t* __restrict__ rowptr,
                                             const int64_t* __restrict__ rowptrT, int* __restrict__ flag) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i > N) return;
    bool bad = false;
    const int64_t a = rowptr[i], b = rowptrT[i];
    bad |= a < 0 || a > E || b < 0 || b > E;
    if (i == 0) bad |= a != 0 || b != 0;
    if (i == N) bad |= a != E || b != E;
    if (i < N) bad |= rowptr[i + 1] < a || rowptrT[i + 1] < b;
    if (bad) atomicOr(flag, CSR_BAD_ROWPTR);
}

// runs only when the pointers passed: one thread per position of either form
__global__ void csr_validate_positions_kernel(int32_t N, int64_t E, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                              const int32_t* __restrict__ eid, const int64_t* __restrict__ rowptrT,
                                              const int32_t* __restrict__ colT, const int32_t* __restrict__ eidT,
                                              const int32_t* __restrict__ t2f, unsigned* __restrict__ seen, int64_t words,
                                              int* __restrict__ flag) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= E) return;
    int bad = 0;
    const int32_t c = col[p], cT = colT[p], e = eid[p], eT = eidT[p], f = t2f[p];
    if (c < 0 || c >= N || cT < 0 || cT >= N) bad |= CSR_BAD_NODE;
    const bool e_ok = e >= 0 && e < E, eT_ok = eT >= 0 && eT < E, f_ok = f >= 0 && f < E;
    if (!e_ok || !eT_ok || !f_ok) bad |= CSR_BAD_EDGE;
    // each of the three arrays must hold every value once: a bit per value and array
    if (e_ok && (atomicOr(seen + (e >> 5), 1u << (e & 31)) >> (e & 31)) & 1u) bad |= CSR_BAD_PERM;
    if (eT_ok && (atomicOr(seen + words + (eT >> 5), 1u << (eT & 31)) >> (eT & 31)) & 1u) bad |= CSR_BAD_PERM;
    if (f_ok && (atomicOr(seen + 2 * words + (f >> 5), 1u << (f & 31)) >> (f & 31)) & 1u) bad |= CSR_BAD_PERM;
    // ascending edge ids inside a row, in both forms
    const int i = csr_row_of(rowptr, N, p), j = csr_row_of(rowptrT, N, p);
    if (p + 1 < rowptr[i + 1] && e_ok && eid[p + 1] <= e) bad |= CSR_BAD_ORDER;
    if (p + 1 < rowptrT[j + 1] && eT_ok && eidT[p + 1] <= eT) bad |= CSR_BAD_ORDER;
    // transposed position p (row j = the edge's source, colT = its target) and position t2f[p] are one edge
    if (f_ok && eT_ok) {
        if (eid[f] != eT || col[f] != j || csr_row_of(rowptr, N, f) != cT) bad |= CSR_BAD_CROSS;
    }
    if (bad) atomicOr(flag, bad);
}

constexpr int SCAN_THREADS = 256;

// exclusive scan of one value per thread over a 256-thread block; *total = block sum
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
    __shared__ uint32_t warp_sums[SCAN_THREADS / 32];
    __shared__ uint32_t block_total;
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_sums[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = lane < SCAN_THREADS / 32 ? warp_sums[lane] : 0;
        uint32_t si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += t;
        }
        if (lane < SCAN_THREADS / 32) warp_sums[lane] = si - s;
        if (lane == 31) block_total = si;
    }
    __syncthreads();
    uint32_t r = warp_sums[wid] + inc - v;
    *total = block_total;
    __syncthreads();
    return r;
}

// ------------------------------------------------------------------ stable LSD radix sort of (endpoint, edge index)
// Three launches per digit: a histogram per tile, an exclusive scan of every digit's row of tile counts, and a scatter that
// ranks a tile's keys (warp match, one pass: the rank is kept in a register) and writes (key, index) pairs of 8 bytes.
// Below SORT_BOTH edges the two sorts (by target, by source) share their launches, and digits are as wide as divides the key
// evenly in few passes (up to 10 bits: 2 passes for up to 1 M nodes); above, they run one after the other in one pair of
// buffers with 8-bit digits, whose runs per tile are longer.  The last pass writes the sparse form itself (edge index, other
// endpoint, and for the form by target each edge's position); row pointers come from the sorted keys' steps.
// 1.53 M edges, 170k nodes: 6 sorts' passes of 5 launches each and the forms 340 us -> 165 us.
constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_MAX_BINS = 1024;
constexpr int64_t SORT_BOTH = (int64_t)8 << 20;

struct SortJob {
    const int32_t* keys;   // first pass: the endpoints
    const int32_t* other;  // the other endpoint of each edge
    const uint2* in;       // later passes: (key, edge index)
    uint2* out;
    int32_t* ksorted;      // last pass: keys in order
    int32_t *col, *eid, *pos;  // last pass: the sparse form; pos[edge] = its position (or nullptr)
    uint32_t *table, *totals;  // [bins][ntiles] counts, then their exclusive scans per digit; [bins] totals
    int64_t* rowptr;
};
struct SortArgs {
    SortJob j[2];
    int64_t E;
    int32_t N;
    int shift, bits;
    uint32_t ntiles;
    int both;        // the first histogram of this launch sees the keys of both forms; otherwise it also checks the other endpoints
    int* flag;       // set if an endpoint is out of range
    int* host_flag;  // the same word for the waiting host
    const int32_t* pos;  // finalize: position of each edge in the form by target
    int32_t* t2f;
};

// element order inside a tile: warp-major, then round, then lane
template <int ROUNDS>
__device__ __forceinline__ int64_t rs_index(int64_t tile0, int warp, int round, int lane) {
    return tile0 + (int64_t)warp * (32 * ROUNDS) + round * 32 + lane;
}

template <int ROUNDS, bool FIRST>
__global__ void __launch_bounds__(RS_THREADS) radix_hist_kernel(const __grid_constant__ SortArgs A) {
    __shared__ uint32_t cnt[RS_MAX_BINS];
    pdl_wait();
    const SortJob& J = A.j[blockIdx.y];
    const int bins = 1 << A.bits;
    for (int d = threadIdx.x; d < bins; d += RS_THREADS) cnt[d] = 0;
    __syncthreads();
    const int64_t tile0 = (int64_t)blockIdx.x * (RS_THREADS * ROUNDS);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t key[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t i = rs_index<ROUNDS>(tile0, warp, r, lane);
        key[r] = i < A.E ? (FIRST ? J.keys[i] : (int32_t)J.in[i].x) : 0;
    }
    bool bad = false;
    if (FIRST && !A.both) {
        int32_t oth[ROUNDS];
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) {
            const int64_t i = rs_index<ROUNDS>(tile0, warp, r, lane);
            oth[r] = i < A.E ? J.other[i] : 0;
        }
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) bad |= oth[r] < 0 || oth[r] >= A.N;
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        if (FIRST) bad |= key[r] < 0 || key[r] >= A.N;
        if (rs_index<ROUNDS>(tile0, warp, r, lane) < A.E) atomicAdd(&cnt[((uint32_t)key[r] >> A.shift) & (bins - 1)], 1u);
    }
    if (FIRST && bad) {  // benign race: every writer stores the same value
        *A.flag = 1;
        *(volatile int*)A.host_flag = 1;
    }
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += RS_THREADS) J.table[(size_t)d * A.ntiles + blockIdx.x] = cnt[d];
}

// block (d, job): exclusive scan of digit d's row of tile counts, in place; its sum to totals[d]
__global__ void __launch_bounds__(RS_THREADS) radix_scan_kernel(const __grid_constant__ SortArgs A) {
    pdl_wait();
    const SortJob& J = A.j[blockIdx.y];
    uint32_t* const row = J.table + (size_t)blockIdx.x * A.ntiles;
    uint32_t carry = 0;
    for (uint32_t b0 = 0; b0 < A.ntiles; b0 += 4 * RS_THREADS) {
        const uint32_t i0 = b0 + threadIdx.x * 4;
        uint32_t v[4], s = 0, total;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = i0 + u < A.ntiles ? row[i0 + u] : 0;
            s += v[u];
        }
        uint32_t run = carry + block_exclusive_scan(s, &total);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i0 + u < A.ntiles) row[i0 + u] = run;
            run += v[u];
        }
        carry += total;
    }
    if (threadIdx.x == 0) J.totals[blockIdx.x] = carry;
}

template <int ROUNDS, bool FIRST, bool LAST>
__global__ void __launch_bounds__(RS_THREADS) radix_scatter_kernel(const __grid_constant__ SortArgs A) {
    __shared__ uint16_t wcnt[RS_WARPS][RS_MAX_BINS];  // counts, then prefixes, of a warp's keys per digit: at most 4096
    __shared__ uint32_t gbase[RS_MAX_BINS];
    pdl_wait();
    const SortJob& J = A.j[blockIdx.y];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, bins = 1 << A.bits;
    const int64_t tile0 = (int64_t)blockIdx.x * (RS_THREADS * ROUNDS);
    const int refused = LAST ? *(const volatile int*)A.flag : 0;  // an endpoint out of range: the outputs stay as they are
    uint2 kv[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t i = rs_index<ROUNDS>(tile0, warp, r, lane);
        kv[r] = make_uint2(0u, 0u);
        if (i < A.E) kv[r] = FIRST ? make_uint2((uint32_t)J.keys[i], (uint32_t)i) : J.in[i];
    }
    if (refused) return;
    for (int d = threadIdx.x; d < RS_WARPS * RS_MAX_BINS / 2; d += RS_THREADS) reinterpret_cast<uint32_t*>(wcnt)[d] = 0;
    {  // where each digit's keys of this tile begin: digits before, then tiles before
        const int per = RS_MAX_BINS / RS_THREADS;
        uint32_t v[per], s = 0, total;
#pragma unroll
        for (int u = 0; u < per; ++u) {
            const int d = threadIdx.x * per + u;
            v[u] = d < bins ? J.totals[d] : 0;
            s += v[u];
        }
        uint32_t run = block_exclusive_scan(s, &total);  // its barriers also close the zeroing above
#pragma unroll
        for (int u = 0; u < per; ++u) {
            const int d = threadIdx.x * per + u;
            if (d < bins) gbase[d] = run + J.table[(size_t)d * A.ntiles + blockIdx.x];
            run += v[u];
        }
    }
    const uint32_t lt = (1u << lane) - 1u;
    uint16_t rank[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {  // stable rank among the warp's keys of the same digit
        const bool ok = rs_index<ROUNDS>(tile0, warp, r, lane) < A.E;
        const int d = ok ? (int)((kv[r].x >> A.shift) & (uint32_t)(bins - 1)) : bins;  // lanes past the end form their own group
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = ok ? wcnt[warp][d] : 0;
        rank[r] = (uint16_t)(before + __popc(peers & lt));
        __syncwarp();
        if (ok && (peers & lt) == 0) wcnt[warp][d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += RS_THREADS) {  // prefix over the warps of the block
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            const uint32_t t = wcnt[w][d];
            wcnt[w][d] = (uint16_t)run;
            run += t;
        }
    }
    __syncthreads();
    uint32_t where[ROUNDS];
    int32_t oth[LAST ? ROUNDS : 1];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int d = (int)((kv[r].x >> A.shift) & (uint32_t)(bins - 1));
        where[r] = gbase[d] + wcnt[warp][d] + rank[r];
        if (LAST && rs_index<ROUNDS>(tile0, warp, r, lane) < A.E) oth[LAST ? r : 0] = J.other[kv[r].y];
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        if (rs_index<ROUNDS>(tile0, warp, r, lane) >= A.E) continue;
        const uint32_t p = where[r];
        if (LAST) {
            J.ksorted[p] = (int32_t)kv[r].x;
            J.eid[p] = (int32_t)kv[r].y;
            J.col[p] = oth[LAST ? r : 0];
            if (J.pos) J.pos[kv[r].y] = (int32_t)p;
        } else {
            J.out[p] = kv[r];
        }
    }
}

// row pointers from the sorted keys (rowptr[i] = first position whose key is >= i) and, with the form by source, t2f.  A
// thread fills the rows between its key and the one before; gaps of more than 32 rows (isolated nodes) by the whole block.
__global__ void __launch_bounds__(256) csr_finalize_kernel(const __grid_constant__ SortArgs A) {
    __shared__ int64_t gap_p[256];
    __shared__ int gap_a[256], gap_b[256], gaps;
    pdl_wait();
    if (*A.flag) return;  // endpoints out of range: the keys are not in order
    const SortJob& J = A.j[blockIdx.y];
    if (threadIdx.x == 0) gaps = 0;
    __syncthreads();
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;  // p == E: the rows after the last key
    if (p <= A.E) {
        const int a = p > 0 ? J.ksorted[p - 1] + 1 : 0, b = p < A.E ? J.ksorted[p] + 1 : A.N + 1;  // rows [a, b) begin at p
        if (b - a > 32) {
            const int k = atomicAdd(&gaps, 1);
            gap_a[k] = a; gap_b[k] = b; gap_p[k] = p;
        } else {
            for (int i = a; i < b; ++i) J.rowptr[i] = p;
        }
        if (J.pos == nullptr && p < A.E) A.t2f[p] = A.pos[J.eid[p]];
    }
    __syncthreads();
    for (int k = 0; k < gaps; ++k)
        for (int i = gap_a[k] + (int)threadIdx.x; i < gap_b[k]; i += 256) J.rowptr[i] = gap_p[k];
}

struct SortPlan {
    bool both;
    int rounds, bits, passes;
    uint32_t ntiles;
    uint2 *a[2], *b[2];
    uint32_t *table[2], *totals[2];
    int32_t* pos;
    int* flag;
    size_t bytes;
};

// Both sorts at once need twice the buffers.  A workspace that was sized for a graph of more edges, whose sorts run one after
// the other, may lack them: then a smaller graph's do so too (`both` is a wish).  So a size that serves E serves fewer edges.
static SortPlan sort_plan(void* ws, int32_t N, int64_t E, bool both = true) {
    SortPlan s;
    s.both = both && E < SORT_BOTH;
    s.rounds = s.both ? 8 : 16;
    int bits = 1;
    while (bits < 31 && ((int64_t)1 << bits) < (int64_t)N) ++bits;
    const int most = s.both ? 10 : 8;
    s.passes = (bits + most - 1) / most;
    s.bits = (bits + s.passes - 1) / s.passes;
    s.ntiles = (uint32_t)ceil_div(E > 0 ? E : 1, RS_THREADS * s.rounds);
    char* p = (char*)ws;
    // the flag, then everything else: pairs are read and written as 8 bytes, also in a workspace that begins between two of them
    s.flag = (int*)p;
    size_t off = 256 - reinterpret_cast<uintptr_t>(ws) % 8;
    const size_t pairs = up256((size_t)(E > 0 ? E : 1) * 8), bins = (size_t)1 << most;
    for (int k = 0; k < 2; ++k) {
        if (k == 1 && !s.both) { s.a[1] = s.a[0]; s.b[1] = s.b[0]; s.table[1] = s.table[0]; s.totals[1] = s.totals[0]; continue; }
        s.a[k] = (uint2*)(p + off); off += pairs;
        s.b[k] = (uint2*)(p + off); off += pairs;
        s.table[k] = (uint32_t*)(p + off); off += up256(bins * s.ntiles * 4);
        s.totals[k] = (uint32_t*)(p + off); off += up256(bins * 4);
    }
    s.pos = (int32_t*)(p + off); off += up256((size_t)(E > 0 ? E : 1) * 4);
    s.bytes = off;
    return s;
}

template <int ROUNDS>
static cudaError_t launch_sort(SortArgs A, const SortPlan& s, int first, int jobs, cudaEvent_t validated, cudaStream_t st) {
    if (first) A.j[0] = A.j[1];
    A.both = jobs == 2 || first;  // (the sort by target has checked all endpoints by then)
    for (int p = 0; p < s.passes; ++p) {
        A.shift = s.bits * p;
        A.bits = s.bits;
        const bool f = p == 0, l = p == s.passes - 1;
        for (int k = 0; k < jobs; ++k) {
            A.j[k].in = p % 2 ? s.a[k + first] : s.b[k + first];
            A.j[k].out = p % 2 ? s.b[k + first] : s.a[k + first];
            A.j[k].ksorted = (int32_t*)A.j[k].out;  // the last pass writes no pairs
        }
        const dim3 tiles(s.ntiles, jobs), block(RS_THREADS);
        if (f) launch_overlapped(radix_hist_kernel<ROUNDS, true>, tiles, block, 0, st, A);
        else launch_overlapped(radix_hist_kernel<ROUNDS, false>, tiles, block, 0, st, A);
        if (f && !first) {
            const cudaError_t e = cudaEventRecord(validated, st);
            if (e != cudaSuccess) return e;
        }
        launch_overlapped(radix_scan_kernel, dim3(1u << s.bits, jobs), block, 0, st, A);
        if (f && l) launch_overlapped(radix_scatter_kernel<ROUNDS, true, true>, tiles, block, 0, st, A);
        else if (f) launch_overlapped(radix_scatter_kernel<ROUNDS, true, false>, tiles, block, 0, st, A);
        else if (l) launch_overlapped(radix_scatter_kernel<ROUNDS, false, true>, tiles, block, 0, st, A);
        else launch_overlapped(radix_scatter_kernel<ROUNDS, false, false>, tiles, block, 0, st, A);
    }
    launch_overlapped(csr_finalize_kernel, dim3((unsigned)ceil_div(A.E + 1, 256), jobs), dim3(256), 0, st, A);
    return cudaGetLastError();
}

// The host waits for the validation of the endpoints, which is done long before the sorts that are queued behind it.
struct CudaSlots {
    using Event = cudaEvent_t;
    static bool make_word(int** w) { return cudaHostAlloc((void**)w, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess; }
    static void free_word(int* w) { cudaFreeHost(w); }
    static bool make_event(Event* e) { return cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess; }
    static void free_event(Event e) { cudaEventDestroy(e); }
};
static FlagSlots<CudaSlots> g_slots;

// ------------------------------------------------------------------ degrees / GCN coefficients
__global__ void degree_count_kernel(int32_t N, const int64_t* rowptr,
                                    int32_t* __restrict__ deg) {
    pdl_wait();
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < N) deg[i] = (int32_t)(rowptr[i + 1] - rowptr[i]);
}

// Sum of w over each row: eight lanes per row (four rows per warp), rows over DEG_LONG positions by the whole block (a hub
// of 10^5 positions walked by a warp alone takes milliseconds).  Fixed orders.  170k rows of nine positions on average:
// 31 us with a warp per row, 14 us.
constexpr int DEG_LONG = 512;
__global__ void __launch_bounds__(256) degree_weighted_kernel(int32_t N, const int64_t* rowptr,
                                                             const float* w, float* __restrict__ deg) {
    __shared__ int todo[32], ntodo;
    __shared__ float sums[8];
    pdl_wait();
    if (threadIdx.x == 0) ntodo = 0;
    __syncthreads();
    const int64_t row = blockIdx.x * (int64_t)32 + (threadIdx.x >> 3);
    const int li = threadIdx.x & 7;
    float s = 0.f;
    bool lng = false;
    if (row < N) {
        const int64_t a = rowptr[row], b = rowptr[row + 1];
        lng = b - a > DEG_LONG;
        if (!lng) {
#pragma unroll 4
            for (int64_t p = a + li; p < b; p += 8) s += w[p];
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (row < N && li == 0) {
        if (lng) todo[atomicAdd(&ntodo, 1)] = (int)row;  // rows are independent: their order does not matter
        else deg[row] = s;
    }
    __syncthreads();
    for (int k = 0; k < ntodo; ++k) {
        const int r = todo[k];
        const int64_t a = rowptr[r], b = rowptr[r + 1];
        s = 0.f;
#pragma unroll 4
        for (int64_t p = a + threadIdx.x; p < b; p += 256) s += w[p];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < 8; ++q) s += sums[q];
            deg[r] = s;
        }
        __syncthreads();
    }
}

__global__ void degree_unit_kernel(int32_t N, const int64_t* rowptr,
                                   float* __restrict__ deg) {
    pdl_wait();
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < N) deg[i] = (float)(rowptr[i + 1] - rowptr[i]);
}

// coef[p] = w[p] / sqrt(deg[row(p)] * deg[col[p]]), for the form by target (blockIdx.y = 0) and, with w through t2f, for the
// transposed one: the degrees of an edge's two ends meet in a product, so both forms give the same bits.  Positions first: a
// warp stages the rows of its 256 positions and every lane finds the row of its first of eight there and steps on, whatever
// the rows' lengths (a warp per row and a second pass for hubs: 58 + 35 + 9 us on 170k rows / 1.53 M positions).
struct CoefForm {
    const int64_t* rowptr;
    const int32_t *col, *w_index;
    float* out;
    int vec;  // all three on 16 bytes
};
struct CoefArgs {
    CoefForm f[2];
    const float *w, *deg;
    int32_t N;
    int64_t E;
};
__device__ __forceinline__ float gcn_coef(float wp, float di, float dj) {
    // IEEE sqrt and division (no approximate rsqrt): ~1e-7 relative
    return (di > 0.f && dj > 0.f) ? __fdiv_rn(wp, __fsqrt_rn(di * dj)) : 0.f;
}
__global__ void __launch_bounds__(256) gcn_coef_kernel(const __grid_constant__ CoefArgs A) {
    constexpr int SUB = 256, PER = SUB / 32;  // a lane takes eight consecutive positions
    __shared__ int s_row[8][SUB + 1];
    __shared__ uint16_t s_start[8][SUB + 2];
    pdl_wait();
    const CoefForm& F = A.f[blockIdx.y];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t cs64 = ((int64_t)blockIdx.x * 8 + warp) * SUB;
    if (cs64 >= A.E) return;
    const int cs = (int)cs64, n = (int)min((int64_t)SUB, A.E - cs64), i0 = lane * PER;
    const bool vec = F.vec && n == SUB;  // whole, aligned vectors
    __align__(16) int c[PER], wi[PER];
    float wp[PER], dj[PER], r[PER];
    if (vec) {
        *reinterpret_cast<int4*>(c) = __ldcs(reinterpret_cast<const int4*>(F.col + cs + i0));
        *reinterpret_cast<int4*>(c + 4) = __ldcs(reinterpret_cast<const int4*>(F.col + cs + i0) + 1);
        if (A.w && F.w_index) {
            *reinterpret_cast<int4*>(wi) = __ldcs(reinterpret_cast<const int4*>(F.w_index + cs + i0));
            *reinterpret_cast<int4*>(wi + 4) = __ldcs(reinterpret_cast<const int4*>(F.w_index + cs + i0) + 1);
        }
    } else {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            c[u] = i0 + u < n ? F.col[cs + i0 + u] : 0;
            wi[u] = A.w && F.w_index && i0 + u < n ? F.w_index[cs + i0 + u] : 0;
        }
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        wp[u] = 1.0f;
        if (A.w && i0 + u < n) wp[u] = A.w[F.w_index ? wi[u] : cs + i0 + u];
        dj[u] = i0 + u < n ? A.deg[c[u]] : 0.f;
        r[u] = 0.f;
    }
    bool began_before;
    const int m = stage_rows(F.rowptr, A.N, A.E, cs, n, lane, s_row[warp], s_start[warp], began_before);
    __syncwarp();
    if (i0 >= n) return;
    int q = 0, hi = m;  // start[q] <= i0 < start[hi]
    while (hi - q > 1) {
        const int mid = (q + hi) >> 1;
        if (s_start[warp][mid] <= i0) q = mid; else hi = mid;
    }
    float di = A.deg[max(s_row[warp][q], 0)];
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (i0 + u < n) {
            if (i0 + u >= s_start[warp][q + 1]) di = A.deg[max(s_row[warp][++q], 0)];  // staged rows have positions: one step is enough
            r[u] = gcn_coef(wp[u], di, dj[u]);
        }
    if (vec) {
        *reinterpret_cast<float4*>(F.out + cs + i0) = make_float4(r[0], r[1], r[2], r[3]);
        *reinterpret_cast<float4*>(F.out + cs + i0 + 4) = make_float4(r[4], r[5], r[6], r[7]);
    } else {
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (i0 + u < n) F.out[cs + i0 + u] = r[u];
    }
}

// rows of one element: four index -> element chains in flight per thread
template <typename T>
__global__ void __launch_bounds__(256) permute_elements_kernel(int64_t E, const int32_t* perm, const T* in, T* __restrict__ out) {
    pdl_wait();
    const int64_t t0 = blockIdx.x * (int64_t)1024 + threadIdx.x;
    int32_t p[4];
    T v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) p[u] = t0 + u * 256 < E ? perm[t0 + u * 256] : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = in[p[u]];
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (t0 + u * 256 < E) out[t0 + u * 256] = v[u];
}

template <typename T>
__global__ void permute_rows_kernel(int64_t E, int width, const int32_t* perm,
                                    const T* in, T* __restrict__ out) {
    pdl_wait();
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t total = E * width;
    for (; t < total; t += stride) {
        int64_t p = t / width;
        int c = (int)(t - p * width);
        out[t] = in[(int64_t)perm[p] * width + c];
    }
}

__global__ void add_self_loops_kernel(int32_t N, int64_t E, const int32_t* src,
                                      const int32_t* dst, int32_t* __restrict__ so,
                                      int32_t* __restrict__ dout) {
    pdl_wait();
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; k < E + N; k += stride) {
        if (k < E) {
            const int32_t s = src[k], d = dst[k];
            so[k] = s; dout[k] = d;
        }
        else { so[k] = (int32_t)(k - E); dout[k] = (int32_t)(k - E); }
    }
}

void launch_gather_rows(const int32_t* idx, int64_t E, const void* X, int nvec, void* out, cudaStream_t st);  // edge_ops.cu

template <typename T>
static void launch_permute(int64_t E, int width, const int32_t* perm, const void* in, void* out, cudaStream_t st) {
    if (width == 1) launch_overlapped(permute_elements_kernel<T>, dim3((unsigned)ceil_div(E, 1024)), dim3(256), 0, st, E, perm, (const T*)in, (T*)out);
    else launch_overlapped(permute_rows_kernel<T>, dim3((unsigned)grid_for(E * width, 256)), dim3(256), 0, st, E, width, perm, (const T*)in, (T*)out);
}

}  // namespace gnn

using namespace gnn;

extern "C" {

const char* gnn_status_string(gnn_status s) {
    switch (s) {
        case GNN_OK: return "ok";
        case GNN_ERR_INVALID_ARG: return "invalid argument";
        case GNN_ERR_INDEX_OUT_OF_RANGE: return "index out of range";
        case GNN_ERR_NOT_SORTED: return "not sorted";
        case GNN_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case GNN_ERR_UNSUPPORTED: return "unsupported";
        case GNN_ERR_CUDA: return "CUDA error";
        case GNN_ERR_TIMEOUT: return "timeout";
    }
    return "unknown status";
}
const char* gnn_last_error_string(void) { return g_err; }
int gnn_version(void) { return 100; }

size_t gnn_coo_to_csr_workspace(int32_t N, int64_t E) {
    if (E < 0) return 0;
    return sort_plan(nullptr, N, E).bytes;
}

gnn_status gnn_coo_to_csr(int32_t N, int64_t E, const int32_t* src, const int32_t* dst,
                          gnn_csr* out, void* ws, size_t ws_bytes, gnn_stream stream) {
    GNN_REQUIRE(N >= 0 && E >= 0, GNN_ERR_INVALID_ARG, "gnn_coo_to_csr: negative size");
    GNN_REQUIRE(E <= 0x7FFFFFFFLL - 1, GNN_ERR_UNSUPPORTED, "gnn_coo_to_csr: E must be < 2^31");
    GNN_REQUIRE(out && out->rowptr && out->rowptrT, GNN_ERR_INVALID_ARG, "gnn_coo_to_csr: null output");
    GNN_REQUIRE(E == 0 || (src && dst && out->col && out->eid && out->colT && out->eidT && out->t2f),
                GNN_ERR_INVALID_ARG, "gnn_coo_to_csr: null edge array");
    const bool both = ws_bytes >= gnn_coo_to_csr_workspace(N, E);
    GNN_REQUIRE(ws && ws_bytes >= sort_plan(nullptr, N, E, both).bytes, GNN_ERR_WORKSPACE_TOO_SMALL,
                "gnn_coo_to_csr: workspace of %zu bytes needed", gnn_coo_to_csr_workspace(N, E));
    cudaStream_t st = as_stream(stream);
    out->N = N;
    out->E = E;
    if (E == 0) {
        if (cudaMemsetAsync(out->rowptr, 0, ((size_t)N + 1) * 8, st) != cudaSuccess || cudaMemsetAsync(out->rowptrT, 0, ((size_t)N + 1) * 8, st) != cudaSuccess)
            GNN_FAIL(GNN_ERR_CUDA, "gnn_coo_to_csr: memset failed (are the outputs device pointers?)");
        return GNN_OK;
    }
    GNN_REQUIRE(N > 0, GNN_ERR_INDEX_OUT_OF_RANGE, "gnn_coo_to_csr: an edge endpoint is outside [0, %d)", N);
    const SortPlan s = sort_plan(ws, N, E, both);
    FlagSlots<CudaSlots>::Slot slot;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || !g_slots.take(dev, &slot)) GNN_FAIL(GNN_ERR_CUDA, "gnn_coo_to_csr: no pinned memory for the validation word: %s", cudaGetErrorString(cudaGetLastError()));
    *(volatile int*)slot.word = 0;
    SortArgs A = {};
    A.E = E; A.N = N; A.ntiles = s.ntiles; A.flag = s.flag; A.host_flag = slot.word; A.pos = s.pos; A.t2f = out->t2f;
    A.j[0].keys = dst; A.j[0].other = src; A.j[0].col = out->col; A.j[0].eid = out->eid; A.j[0].pos = s.pos; A.j[0].rowptr = out->rowptr;
    A.j[1].keys = src; A.j[1].other = dst; A.j[1].col = out->colT; A.j[1].eid = out->eidT; A.j[1].pos = nullptr; A.j[1].rowptr = out->rowptrT;
    for (int k = 0; k < 2; ++k) { A.j[k].table = s.table[k]; A.j[k].totals = s.totals[k]; }
    cudaError_t e = cudaMemsetAsync(s.flag, 0, sizeof(int), st);
    if (e == cudaSuccess) {
        if (s.both) {
            e = launch_sort<8>(A, s, 0, 2, slot.event, st);
        } else {
            e = launch_sort<16>(A, s, 0, 1, slot.event, st);
            if (e == cudaSuccess) e = launch_sort<16>(A, s, 1, 1, slot.event, st);
        }
    }
    if (e == cudaSuccess) e = cudaEventSynchronize(slot.event);
    const int bad = *(volatile int*)slot.word;
    // on any error nothing of the call is left running on the caller's buffers, or on the slot, when it returns
    cudaError_t quiet = cudaSuccess;
    if (e != cudaSuccess || bad) quiet = cudaStreamSynchronize(st);
    g_slots.give(slot, quiet == cudaSuccess);
    if (e == cudaSuccess) e = quiet;
    if (e != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "gnn_coo_to_csr: %s", cudaGetErrorString(e));
    GNN_REQUIRE(bad == 0, GNN_ERR_INDEX_OUT_OF_RANGE,
                "gnn_coo_to_csr: an edge endpoint is outside [0, %d)", N);
    return GNN_OK;
}

size_t gnn_csr_validate_workspace(int64_t E) {
    if (E < 0) return 0;
    return 256 + up256((size_t)3 * (size_t)((E + 31) / 32) * 4);
}

gnn_status gnn_csr_validate(const gnn_csr* g, void* ws, size_t ws_bytes, gnn_stream stream) {
    GNN_REQUIRE(g, GNN_ERR_INVALID_ARG, "gnn_csr_validate: null graph");
    GNN_REQUIRE(g->N >= 0 && g->E >= 0 && g->E <= 0x7FFFFFFFLL - 1, GNN_ERR_INVALID_ARG, "gnn_csr_validate: bad sizes (N=%d, E=%lld)", g->N, (long long)g->E);
    GNN_REQUIRE(g->rowptr && g->rowptrT, GNN_ERR_INVALID_ARG, "gnn_csr_validate: null row pointers");
    GNN_REQUIRE(g->E == 0 || (g->col && g->eid && g->colT && g->eidT && g->t2f), GNN_ERR_INVALID_ARG, "gnn_csr_validate: null edge array");
    const size_t need = gnn_csr_validate_workspace(g->E);
    GNN_REQUIRE(ws && ws_bytes >= need, GNN_ERR_WORKSPACE_TOO_SMALL, "gnn_csr_validate: workspace of %zu bytes needed", need);
    cudaStream_t st = as_stream(stream);
    int* flag = (int*)ws;
    unsigned* seen = (unsigned*)((char*)ws + 256);
    const int64_t words = (g->E + 31) / 32;
    if (cudaMemsetAsync(ws, 0, need, st) != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "gnn_csr_validate: memset failed (is ws a device pointer?)");
    auto read_flag = [&](int* h) {
        return cudaMemcpyAsync(h, flag, sizeof(int), cudaMemcpyDeviceToHost, st) == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess;
    };
    csr_validate_pointers_kernel<<<(int)ceil_div((int64_t)g->N + 1, 256), 256, 0, st>>>(g->N, g->E, g->rowptr, g->rowptrT, flag);
    GNN_CHECK_LAUNCH("csr_validate_pointers");
    int h = 0;
    if (!read_flag(&h)) GNN_FAIL(GNN_ERR_CUDA, "gnn_csr_validate: reading the result failed: %s", cudaGetErrorString(cudaGetLastError()));
    if (h == 0 && g->E > 0 && g->N > 0) {  // the position checks look rows up through the pointers: only once those are sound
        csr_validate_positions_kernel<<<(int)ceil_div(g->E, 256), 256, 0, st>>>(g->N, g->E, g->rowptr, g->col, g->eid, g->rowptrT, g->colT,
                                                                           g->eidT, g->t2f, seen, words, flag);
        GNN_CHECK_LAUNCH("csr_validate_positions");
        if (!read_flag(&h)) GNN_FAIL(GNN_ERR_CUDA, "gnn_csr_validate: reading the result failed: %s", cudaGetErrorString(cudaGetLastError()));
    }
    GNN_REQUIRE(h == 0, GNN_ERR_INVALID_ARG, "gnn_csr_validate: not a sparse form of one edge list:%s%s%s%s%s%s",
                (h & CSR_BAD_ROWPTR) ? " row pointers (0 .. E, non-decreasing);" : "", (h & CSR_BAD_NODE) ? " node index outside [0, N);" : "",
                (h & CSR_BAD_EDGE) ? " edge index outside [0, E);" : "", (h & CSR_BAD_PERM) ? " eid / eidT / t2f not a permutation;" : "",
                (h & CSR_BAD_ORDER) ? " edge ids not ascending inside a row;" : "", (h & CSR_BAD_CROSS) ? " the two forms describe different edges;" : "");
    return GNN_OK;
}

gnn_status gnn_degree(const gnn_csr* g, int transposed, const float* w, void* deg_out,
                      gnn_stream stream) {
    GNN_REQUIRE(g && deg_out, GNN_ERR_INVALID_ARG, "gnn_degree: null argument");
    const int64_t* rp = transposed ? g->rowptrT : g->rowptr;
    GNN_REQUIRE(rp, GNN_ERR_INVALID_ARG, "gnn_degree: null rowptr");
    if (g->N == 0) return GNN_OK;
    cudaStream_t st = as_stream(stream);
    if (!w)
        launch_overlapped(degree_count_kernel, dim3((unsigned)ceil_div(g->N, 256)), dim3(256), 0, st, g->N, rp, (int32_t*)deg_out);
    else
        launch_overlapped(degree_weighted_kernel, dim3((unsigned)ceil_div(g->N, 32)), dim3(256), 0, st, g->N, rp, w, (float*)deg_out);
    GNN_CHECK_LAUNCH("gnn_degree");
    return GNN_OK;
}

gnn_status gnn_add_self_loops(int32_t N, int64_t E, const int32_t* src, const int32_t* dst,
                              int32_t* src_out, int32_t* dst_out, gnn_stream stream) {
    GNN_REQUIRE(N >= 0 && E >= 0, GNN_ERR_INVALID_ARG, "gnn_add_self_loops: negative size");
    GNN_REQUIRE(E + N <= 0x7FFFFFFFLL - 1, GNN_ERR_UNSUPPORTED, "gnn_add_self_loops: E+N must be < 2^31");
    if (E + N == 0) return GNN_OK;
    GNN_REQUIRE(src_out && dst_out && (E == 0 || (src && dst)), GNN_ERR_INVALID_ARG,
                "gnn_add_self_loops: null argument");
    launch_overlapped(add_self_loops_kernel, dim3((unsigned)(grid_for(E + N, 256))), dim3(256), 0, as_stream(stream), N, E, src, dst, src_out, dst_out);
    GNN_CHECK_LAUNCH("gnn_add_self_loops");
    return GNN_OK;
}

gnn_status gnn_gcn_norm(const gnn_csr* g, const float* w_csr, float* deg_out, float* coef_csr,
                        float* coef_csrT, gnn_stream stream) {
    GNN_REQUIRE(g && g->rowptr && deg_out, GNN_ERR_INVALID_ARG, "gnn_gcn_norm: null argument");
    GNN_REQUIRE(!coef_csrT || coef_csr, GNN_ERR_INVALID_ARG,
                "gnn_gcn_norm: coef_csrT is derived from coef_csr, which is NULL");
    if (g->N == 0) return GNN_OK;
    cudaStream_t st = as_stream(stream);
    if (w_csr)
        launch_overlapped(degree_weighted_kernel, dim3((unsigned)ceil_div(g->N, 32)), dim3(256), 0, st, g->N, g->rowptr, w_csr, deg_out);
    else
        launch_overlapped(degree_unit_kernel, dim3((unsigned)ceil_div(g->N, 256)), dim3(256), 0, st, g->N, g->rowptr, deg_out);
    if (coef_csr && g->E > 0) {
        GNN_REQUIRE(g->col, GNN_ERR_INVALID_ARG, "gnn_gcn_norm: null col");
        GNN_REQUIRE(!coef_csrT || g->t2f, GNN_ERR_INVALID_ARG, "gnn_gcn_norm: null t2f");
        // both forms in one launch need the transposed form's rows, and weights that neither output overwrites; else the
        // second is the first, reordered
        auto apart = [&](const float* out) { return !w_csr || w_csr + g->E <= out || out + g->E <= w_csr; };
        const bool both = coef_csrT && g->rowptrT && g->colT && apart(coef_csr) && apart(coef_csrT);
        CoefArgs A = {};
        A.f[0] = {g->rowptr, g->col, nullptr, coef_csr, aligned16(g->col) && aligned16(coef_csr)};
        A.f[1] = {g->rowptrT, g->colT, g->t2f, coef_csrT, aligned16(g->colT) && aligned16(g->t2f) && aligned16(coef_csrT)};
        A.w = w_csr; A.deg = deg_out; A.N = g->N; A.E = g->E;
        launch_overlapped(gcn_coef_kernel, dim3((unsigned)ceil_div(g->E, 256 * 8), both ? 2 : 1), dim3(256), 0, st, A);
        if (coef_csrT && !both)
            launch_permute<uint32_t>(g->E, 1, g->t2f, coef_csr, coef_csrT, st);
    }
    GNN_CHECK_LAUNCH("gnn_gcn_norm");
    return GNN_OK;
}

gnn_status gnn_permute_edge_data(const int32_t* perm, int64_t E, int width, int elem_bytes,
                                 const void* in, void* out, gnn_stream stream) {
    GNN_REQUIRE(E >= 0 && width >= 1, GNN_ERR_INVALID_ARG, "gnn_permute_edge_data: bad size");
    if (E == 0) return GNN_OK;
    GNN_REQUIRE(perm && in && out && in != out, GNN_ERR_INVALID_ARG, "gnn_permute_edge_data: null or aliased argument");
    cudaStream_t st = as_stream(stream);
    const int64_t row = (int64_t)width * elem_bytes;
    const bool known = elem_bytes == 1 || elem_bytes == 2 || elem_bytes == 4 || elem_bytes == 8;
    // whole 16-byte chunks to a thread: 1.6 M rows of four floats 19 -> 12 us, of eight 46 -> 17 (an
    // element per thread, a division each)
    if (known && row % 16 == 0 && row <= 4096 && aligned16(in) && aligned16(out)) {
        launch_gather_rows(perm, E, in, (int)(row / 16), out, st);
        GNN_CHECK_LAUNCH("gnn_permute_edge_data");
        return GNN_OK;
    }
    switch (elem_bytes) {
        case 1: launch_permute<uint8_t>(E, width, perm, in, out, st); break;
        case 2: launch_permute<uint16_t>(E, width, perm, in, out, st); break;
        case 4: launch_permute<uint32_t>(E, width, perm, in, out, st); break;
        case 8: launch_permute<uint64_t>(E, width, perm, in, out, st); break;
        default: GNN_FAIL(GNN_ERR_UNSUPPORTED, "gnn_permute_edge_data: elem_bytes must be 1, 2, 4 or 8");
    }
    GNN_CHECK_LAUNCH("gnn_permute_edge_data");
    return GNN_OK;
}

}  // extern "C"
