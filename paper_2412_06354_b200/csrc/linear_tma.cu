// Pipelined tensor-core path of the dense node-wise transform for bf16: Y[N,Mo] = X[N,Kc] * B with
// B = W[Kc,Mo] as stored (b_transposed = 0: Y = X*W) or the transpose of W[Mo,Kc] (b_transposed = 1:
// dX = dY*W^T), and dW = X^T * dY.
//
// One persistent CTA per SM, three roles:
//   warp 0   loader: one thread issues bulk tensor copies (TMA).  The weight matrix is fetched once
//            per CTA; X arrives as slices of 128 rows x 64 contraction elements (128 bytes per row,
//            128-byte swizzle, 16 KB) into a ring of shared-memory slots, each copy signalling the
//            slot's "full" mbarrier with its byte count.
//   warp 1   MMA issuer: one thread waits for a slice, issues its four tcgen05.mma (128 x Mo x 16,
//            fp32 accumulator in tensor memory) and commits them to the slot's "empty" barrier, so the
//            loader can refill the slot as soon as the tensor core has read it.  Two accumulators
//            alternate between tiles.
//   warps 2..9  epilogue: wait for a tile's accumulator, read it back (tcgen05.ld), round to bf16,
//            write 32 rows x 64 columns at a time into a swizzled staging block that one bulk tensor
//            store sends to Y (rows past N are clipped by the copy engine), and hand the accumulator back.
// The contraction is short (Kc <= 512), so the kernel is bound by reading X and writing Y; the ring
// keeps 64-100 KB of loads in flight per SM.
//
// Every wait has an iteration limit: on expiry the role raises a status word and leaves its loop, the
// other roles run into their own limits, the loader waits (bounded) for copies still in flight, and
// the CTA frees its tensor memory and returns.
#include <cuda.h>  // CUtensorMap and its enums; the encoder itself is looked up through the runtime

#include <mutex>

#include "tc_common.cuh"

namespace gnn {

constexpr int TM_EPI_WARPS = 8;
constexpr int TM_THREADS = 32 * (2 + TM_EPI_WARPS);
constexpr int TM_KB = 64;                                    // contraction elements per slice = one 128-byte swizzle row
constexpr uint32_t TM_SLICE_BYTES = TC_ROWS * TM_KB * 2;     // 16 KB
constexpr uint32_t TM_STAGING_BYTES = 32 * 128;              // per epilogue warp: 32 rows x 64 bf16 columns of Y
constexpr int TM_MAX_STAGES = 8;
constexpr size_t TM_SMEM_MAX = 225 * 1024;                   // dynamic shared memory per CTA (227 KB less the static part)
constexpr uint32_t SW128 = 2;                                // descriptor layout code of the 128-byte swizzle

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "l"(policy)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar), "l"(policy)
        : "memory");
}

// the bias of the CTA's output columns in shared memory, zeros past the last, for the epilogue warps (256 threads from `first`)
__device__ __forceinline__ void stage_bias(float* to, const float* bias, int have, int first) {
    const int c = (int)threadIdx.x - first;
    to[c] = bias && c < have ? bias[c] : 0.f;
    asm volatile("bar.sync 1, 256;" ::: "memory");
}
// 16 columns of a row: + bias, max(., 0)
__device__ __forceinline__ void bias_relu16(float* f, const float* bias, bool add, bool relu) {
    if (add) {
#pragma unroll
        for (int q = 0; q < 16; q += 4) {
            const float4 b = *reinterpret_cast<const float4*>(bias + q);
            f[q] += b.x; f[q + 1] += b.y; f[q + 2] += b.z; f[q + 3] += b.w;
        }
    }
    if (relu) {
#pragma unroll
        for (int q = 0; q < 16; ++q) f[q] = fmaxf(f[q], 0.f);
    }
}

struct TmaParams {
    int64_t N;
    int Kc, Mo;        // contraction length, output columns
    int b_transposed;
    int w_box_rows;    // rows of one weight box (a box has at most 256 rows: taller blocks arrive as two boxes)
    int stages;        // ring slots
    int acc_stride;    // tensor-memory columns between the two accumulators
    int tmem_cols;
    int* status;
    int reset;          // first launch of a call: set the status word to 0
    const float* bias;  // [mo] added to every output row, or nullptr
    int relu;           // max(y, 0) after the bias
    int mo;             // output columns that exist (Kc and Mo are multiples of 16; what lies past the matrices arrives as zeros)
    __nv_bfloat16* Y;   // rows ldy apart, written directly where they do not start on 16 bytes; nullptr: bulk stores through mapY
    int64_t ldy;
};

__global__ void __launch_bounds__(TM_THREADS, 1)
linear_tma_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW,
                  const __grid_constant__ CUtensorMap mapY, const TmaParams P) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(16) float s_bias[256];
    __shared__ __align__(8) uint64_t bars[2 * TM_MAX_STAGES + 5];  // full[S], empty[S], wfull, acc_full[2], acc_empty[2]
    __shared__ uint32_t tmem_base_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Kc = P.Kc, Mo = P.Mo, S = P.stages;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // swizzle atoms are 1024-byte aligned
    const int kblocks = (Kc + TM_KB - 1) / TM_KB;
    // weight blocks: one per 64 elements of the stored matrix's contiguous dimension
    const int wblocks = P.b_transposed ? kblocks : (Mo + 63) / 64;
    const uint32_t wblock_bytes = (uint32_t)(P.b_transposed ? Mo : Kc) * 128u;
    const uint32_t w0 = base, stage0 = base + (uint32_t)wblocks * wblock_bytes;
    const uint32_t ring0 = stage0 + TM_EPI_WARPS * TM_STAGING_BYTES;
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(TM_MAX_STAGES + s); };
    const uint32_t wfull = bar0 + 8u * (2 * TM_MAX_STAGES);
    auto acc_full = [&](int a) { return bar0 + 8u * (uint32_t)(2 * TM_MAX_STAGES + 1 + a); };
    auto acc_empty = [&](int a) { return bar0 + 8u * (uint32_t)(2 * TM_MAX_STAGES + 3 + a); };

    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(wfull, 1);
        for (int a = 0; a < 2; ++a) { mbar_init(acc_full(a), 1); mbar_init(acc_empty(a), TM_EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapW)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapY)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)P.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_exclusive();
    if (P.reset && blockIdx.x == 0 && tid == 0) *P.status = 0;
    const uint32_t tmem_base = tmem_base_slot;
    const int64_t ntiles = (P.N + TC_ROWS - 1) / TC_ROWS;
    bool failed = false;

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t keep = policy_evict_last(), stream = policy_evict_first();
            mbar_arrive_expect_tx(wfull, (uint32_t)wblocks * wblock_bytes);
            const int w_rows = P.b_transposed ? Mo : Kc;
            for (int b = 0; b < wblocks; ++b)
                for (int r0 = 0; r0 < w_rows; r0 += P.w_box_rows)  // rows are 128 bytes apart: stacked boxes lie as one taller box would
                    tma_load_2d(w0 + (uint32_t)b * wblock_bytes + (uint32_t)r0 * 128u, &mapW, b * 64, r0, wfull, keep);
            uint32_t it = 0;
            for (int64_t t = blockIdx.x; t < ntiles && !failed; t += gridDim.x)
                for (int j = 0; j < kblocks; ++j, ++it) {
                    const int s = (int)(it % (uint32_t)S);
                    const uint32_t use = it / (uint32_t)S;
                    // the slot's previous contents have been consumed (first use: passes at once)
                    if (!mbar_wait_bounded(empty(s), (use & 1u) ^ 1u)) { failed = true; break; }
                    mbar_arrive_expect_tx(full(s), TM_SLICE_BYTES);
                    tma_load_2d(ring0 + (uint32_t)s * TM_SLICE_BYTES, &mapX, j * TM_KB, (int)(t * TC_ROWS), full(s), stream);
                }
            if (failed) {
                // do not leave while copies into this CTA's shared memory may still be in flight
                const uint32_t first = it > (uint32_t)S ? it - (uint32_t)S : 0u;
                for (uint32_t i = first; i < it; ++i) mbar_wait_bounded(full((int)(i % (uint32_t)S)), (i / (uint32_t)S) & 1u);
                mbar_wait_bounded(wfull, 0);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = make_idesc(Mo, P.b_transposed ? 0 : 1);
            failed = !mbar_wait_bounded(wfull, 0);
            uint32_t it = 0, lt = 0;
            for (int64_t t = blockIdx.x; t < ntiles && !failed; t += gridDim.x, ++lt) {
                const uint32_t a = lt & 1u;
                // the epilogue has drained this accumulator (first two tiles: passes at once)
                if (!mbar_wait_bounded(acc_empty((int)a), ((lt >> 1) & 1u) ^ 1u)) { failed = true; break; }
                tc_fence_after();
                const uint32_t dacc = tmem_base + a * (uint32_t)P.acc_stride;
                for (int j = 0; j < kblocks; ++j, ++it) {
                    const int s = (int)(it % (uint32_t)S);
                    if (!mbar_wait_bounded(full(s), (it / (uint32_t)S) & 1u)) { failed = true; break; }
                    tc_fence_after();
                    const uint32_t a_slice = ring0 + (uint32_t)s * TM_SLICE_BYTES;
                    const int ksteps = (Kc - j * TM_KB) >= TM_KB ? TM_KB / 16 : (Kc - j * TM_KB) / 16;
                    for (int kk = 0; kk < ksteps; ++kk) {
                        // A: rows 128 bytes apart, groups of 8 rows 1024 bytes apart; a k-step is 32 bytes along the row
                        const uint64_t adesc = make_smem_desc(a_slice + (uint32_t)kk * 32u, 16, 1024, SW128);
                        uint64_t bdesc;
                        if (P.b_transposed)  // K-major: block j holds Mo rows (output columns) of 64 contraction elements
                            bdesc = make_smem_desc(w0 + (uint32_t)j * wblock_bytes + (uint32_t)kk * 32u, 16, 1024, SW128);
                        else  // MN-major: block m holds Kc rows (contraction) of 64 output columns; blocks LBO apart
                            bdesc = make_smem_desc(w0 + (uint32_t)(j * TM_KB + kk * 16) * 128u, wblock_bytes, 1024, SW128);
                        mma_bf16_ss(dacc, adesc, bdesc, idesc, (j > 0 || kk > 0) ? 1u : 0u);
                    }
                    mma_commit(empty(s));  // slot reusable once these MMAs have read it
                }
                if (failed) break;
                mma_commit(acc_full((int)a));
            }
        }
    } else {
        const int ew = warp - 2, quarter = warp & 3, half = ew >> 2;  // tensor-memory lanes 32*(warp % 4)..: hardware rule
        const uint32_t stg = stage0 + (uint32_t)ew * TM_STAGING_BYTES;
        stage_bias(s_bias, P.bias, P.mo, 64);
        uint32_t lt = 0;
        for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++lt) {
            const uint32_t a = lt & 1u;
            if (!mbar_wait_bounded(acc_full((int)a), (lt >> 1) & 1u)) { failed = true; break; }
            tc_fence_after();
            const int64_t row0 = t * TC_ROWS + quarter * 32;  // first of this warp's 32 rows
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + a * (uint32_t)P.acc_stride;
            for (int cb = half; cb * 64 < Mo; cb += 2) {
                // the previous bulk store has finished reading the staging block
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
                const int groups = (Mo - cb * 64 >= 64 ? 64 : Mo - cb * 64) / 16;
                for (int g = 0; g < groups; ++g) {
                    uint32_t r[16];
                    tmem_ld16(taddr + (uint32_t)(cb * 64 + g * 16), r);
                    tmem_ld_wait();
                    float f[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) f[q] = __uint_as_float(r[q]);
                    if (P.bias || P.relu) bias_relu16(f, s_bias + cb * 64 + g * 16, P.bias != nullptr, P.relu != 0);
                    // row = lane, 128 bytes per row; 16-byte chunk c sits at position c ^ (row % 8)
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) {
                        const uint4 v = Chunk<__nv_bfloat16>::pack(f + 8 * h2);
                        const uint32_t dst = stg + (uint32_t)lane * 128u + ((uint32_t)((2 * g + h2) ^ (lane & 7)) << 4);
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
                    }
                }
                if (P.Y) {  // a row of up to 64 columns per step, two columns per lane
                    __syncwarp();
                    const int rows = (int)(P.N - row0 < 32 ? P.N - row0 : 32);
                    for (int r = 0; r < rows; ++r) {
                        __nv_bfloat16* yr = P.Y + (row0 + r) * P.ldy + cb * 64;
#pragma unroll
                        for (int h2 = 0; h2 < 2; ++h2) {
                            const int col = lane + 32 * h2;
                            if (cb * 64 + col < P.mo) {
                                uint16_t v;
                                asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(stg + (uint32_t)r * 128u + ((uint32_t)((col >> 3) ^ (r & 7)) << 4) + (uint32_t)(col & 7) * 2u) : "memory");
                                reinterpret_cast<uint16_t*>(yr)[col] = v;
                            }
                        }
                    }
                    __syncwarp();
                    continue;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0 && row0 < P.N) {  // rows past N are clipped by the copy engine
                    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                     reinterpret_cast<uint64_t>(&mapY)),
                                 "r"(cb * 64), "r"((int)row0), "r"(stg)
                                 : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty((int)a));
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // staging block is read, rows are written
    }
    if (failed) atomicExch(P.status, 7);  // GNN_ERR_TIMEOUT
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, (uint32_t)P.tmem_cols);
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encoder() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// row-major bf16 matrix [rows, cols]; box = 64 columns (128 bytes, swizzled) x box_rows rows; out-of-range reads give zeros
bool tensor_map_encoder_available() { return encoder() != nullptr; }

static bool make_map_ld(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int ld, int box_rows);
bool make_map(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int box_rows) { return make_map_ld(m, ptr, rows, cols, cols, box_rows); }
// a block of columns of a wider matrix: rows ld elements apart
static bool make_map_ld(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int ld, int box_rows) {
    EncodeTiledFn enc = encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int up16(int x) { return (x + 15) & ~15; }
static int up32(int x) { return (x + 31) & ~31; }
static size_t tma_w_bytes(int Kc, int Mo, int b_transposed) {
    return b_transposed ? (size_t)((Kc + 63) / 64) * Mo * 128 : (size_t)((Mo + 63) / 64) * Kc * 128;
}

// widest block of output columns whose weights fit shared memory beside the staging blocks and two slices; the MMA
// takes at most 256 columns and two accumulators of them fill tensor memory
static int tma_column_block(int Kc, int Mo, int b_transposed) {
    int mc = Mo < 256 ? Mo : 256;
    while (mc >= 16 && tma_w_bytes(Kc, mc, b_transposed) + TM_EPI_WARPS * TM_STAGING_BYTES + 2 * TM_SLICE_BYTES + 1024 > TM_SMEM_MAX) mc -= 16;
    return mc >= 16 ? mc : 0;
}

// Kc and Mo: any up to 512 and 1024 (inside, rounded up to 16 with zeros from the copy engine)
bool linear_tma_supported(int64_t N, int Kc, int Mo, int b_transposed, gnn_dtype dtype) {
    if (dtype != GNN_BF16 || N <= 0 || N >= ((int64_t)1 << 31) - TC_ROWS) return false;
    if (Kc < 1 || Kc > 512 || Mo < 1 || Mo > 1024) return false;
    if (tma_column_block(up16(Kc), up16(Mo), b_transposed) == 0) return false;
    return encoder() != nullptr;
}

// X: rows ldx elements apart, W: rows ldw apart, both on 16 bytes.  Y [N,Mo] is contiguous; rows that do not start on 16 bytes
// are written directly instead of by bulk stores.  More than 256 output columns, or weights too large for shared memory,
// run as one launch per block of output columns.
gnn_status linear_tma_forward(const void* X, int ldx, const void* W, int ldw, int64_t N, int Kc, int Mo, int b_transposed, void* Y, int* d_flag, int reset,
                              cudaStream_t st, const float* bias, int relu) {
    const char* who = "gnn_linear (pipelined tensor-core path)";
    const bool direct = (size_t)Mo * 2 % 16 != 0;
    GNN_REQUIRE(aligned16(X) && aligned16(W) && (direct || aligned16(Y)), GNN_ERR_INVALID_ARG, "%s: matrices must be 16-byte aligned", who);
    const int K16 = up16(Kc), block = tma_column_block(K16, up16(Mo), b_transposed);
    GNN_REQUIRE(block > 0, GNN_ERR_UNSUPPORTED, "%s: weights do not fit shared memory", who);
    CUtensorMap mapX;
    if (!make_map_ld(&mapX, X, N, Kc, ldx, TC_ROWS)) GNN_FAIL(GNN_ERR_CUDA, "%s: tensor map encoding failed", who);
    gnn_status rc = allow_big_smem(who, (const void*)linear_tma_kernel, 4, TM_SMEM_MAX);
    if (rc != GNN_OK) return rc;
    const int64_t ntiles = (N + TC_ROWS - 1) / TC_ROWS;
    const __nv_bfloat16* Wb = (const __nv_bfloat16*)W;
    for (int c0 = 0; c0 < Mo; c0 += block) {
        const int mc = Mo - c0 < block ? Mo - c0 : block, m16 = up16(mc);
        // stored [Kc,Mo]: a block of columns; stored [Mo,Kc]: a block of rows.  Boxes reach to the rounded sizes.
        const int w_rows = b_transposed ? mc : Kc, w_cols = b_transposed ? Kc : mc, box_span = b_transposed ? m16 : K16;
        const int box_rows = box_span > 256 ? box_span / 2 : box_span;
        CUtensorMap mapW, mapY;
        if (!make_map_ld(&mapW, b_transposed ? Wb + (size_t)c0 * ldw : Wb + c0, w_rows, w_cols, ldw, box_rows) ||
            (!direct && !make_map_ld(&mapY, (const __nv_bfloat16*)Y + c0, N, mc, Mo, 32)))
            GNN_FAIL(GNN_ERR_CUDA, "%s: tensor map encoding failed", who);
        if (direct) mapY = mapX;  // not used
        TmaParams P;
        P.N = N; P.Kc = K16; P.Mo = m16; P.mo = mc; P.b_transposed = b_transposed; P.w_box_rows = box_rows; P.status = d_flag;
        P.reset = reset && c0 == 0;
        P.bias = bias ? bias + c0 : nullptr; P.relu = relu;
        P.Y = direct ? (__nv_bfloat16*)Y + c0 : nullptr; P.ldy = Mo;
        const size_t wbytes = tma_w_bytes(K16, m16, b_transposed);
        const size_t fixed = 1024 + wbytes + (size_t)TM_EPI_WARPS * TM_STAGING_BYTES;
        int stages = (int)((TM_SMEM_MAX - fixed) / TM_SLICE_BYTES);
        P.stages = stages > TM_MAX_STAGES ? TM_MAX_STAGES : stages;
        P.acc_stride = (m16 + 31) & ~31;
        int cols = 32;
        while (cols < 2 * P.acc_stride) cols <<= 1;
        P.tmem_cols = cols;
        const size_t smem = fixed + (size_t)P.stages * TM_SLICE_BYTES;
        launch_overlapped(linear_tma_kernel, dim3((unsigned)(ntiles < 148 ? ntiles : 148)), dim3(TM_THREADS), smem, st, mapX, mapW, mapY, P);
        GNN_CHECK_LAUNCH(who);
    }
    return GNN_OK;
}

// ------------------------------------------------------------------ fp32: Y = X * B on the bf16 tensor cores
// Every fp32 value is split exactly into three bf16 terms (x = x1 + x2 + x3, 8 mantissa bits each) and the
// six products with i + j <= 4 are accumulated (the dropped ones are below 2^-23 of a product), which keeps
// the fp32 tolerance.  Roles of the persistent CTA:
//   warp 0      loader: X arrives as fp32 slices of 128 rows x 32 columns (128-byte rows, 128-byte swizzle)
//               in a ring of shared-memory slots;
//   converters  G groups of warps, slice i to group i mod G: read a slice, a row per lane, split it, and write the three
//               bf16 levels into one of G operand buffers in tensor memory (48 columns each), which the MMA reads as A;
//   warp 1      MMA issuer: 2 k-steps x 6 level pairs per slice into one of two accumulators;
//   epilogue    accumulator -> swizzled staging blocks of 32 rows x 32 columns -> bulk tensor stores to Y.
// The weight matrix is split once per CTA by all warps before the roles start.
// What bounds it: the chain of a slice (wait, read, split, write, fence, arrive), about 1 us however few its columns.  With
// all converter warps on one slice after the other that chain was the rate; now G slices are in it at a time.  Slots and
// operand buffers are multiples of G, so that each belongs to one group, which sees all its phases (a parity wait only
// tells the last two apart).  170k x 128 x 128: 46 us with one group, levels in shared memory and the tables below looked up
// per MMA; 36 us now; reading X and writing Y takes 27 us.  200k x 256 -> 256: 346 -> 233 us.
// G is 4 where tensor memory has room for four operand buffers beside two accumulators (up to 160 output columns) and shared
// memory for four slots, otherwise 2 (up to 192).  Wider outputs, and weights whose three levels do not fit shared memory,
// are divided among CTAs by blocks of columns (blockIdx.y): X then comes from L2 for all but one of them.
constexpr int TF_CONV_WARPS = 16, TF_EPI_WARPS = 8;
constexpr int TF_THREADS = 32 * (2 + TF_CONV_WARPS + TF_EPI_WARPS);
constexpr int TF_KB = 32;                                  // contraction elements per slice
constexpr uint32_t TF_SLICE_BYTES = TC_ROWS * TF_KB * 4;   // 16 KB of fp32
constexpr int TF_MAX_STAGES = 8;
constexpr int TF_MAX_OPS = 4;        // operand buffers, one per group
constexpr int TF_OP_COLS = 3 * TF_KB / 2;  // tensor memory columns of one: three levels of 32 bf16

// Levels of A and B of product q, small terms first: (2,0) (0,2) (1,1) (1,0) (0,1) (0,0).  Functions of an unrolled index, so
// that the issuing thread adds constants to a descriptor: with tables in constant memory and a descriptor built per MMA the
// issue alone took 150 cycles an MMA, five times what the tensor core takes for 128 x 128 x 16.
__device__ __forceinline__ constexpr uint32_t pair_a(int q) { return q == 0 ? 2u : q == 2 || q == 3 ? 1u : 0u; }
__device__ __forceinline__ constexpr uint32_t pair_b(int q) { return q == 1 ? 2u : q == 2 || q == 4 ? 1u : 0u; }

// 8 fp32 values -> three 16-byte chunks of bf16 (x = x1 + x2 + x3 exactly)
__device__ __forceinline__ void split8(const float* xin, uint4* lv) {
    float x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = xin[j];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            __nv_bfloat162 b = __floats2bfloat162_rn(x[j], x[j + 1]);
            w[j / 2] = *reinterpret_cast<uint32_t*>(&b);
            // remainders are exact in fp32: the rounded term shares the leading bits of x
            x[j] -= __uint_as_float(w[j / 2] << 16);
            x[j + 1] -= __uint_as_float(w[j / 2] & 0xFFFF0000u);
        }
        lv[l] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
__device__ __forceinline__ void st_shared16(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 ld_shared16(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

struct TmaF32Params {
    const float* W;  // [Kc,Mo] (b_transposed = 0) or [Mo,Kc] (b_transposed = 1), rows ldw elements apart
    int ldw;
    int64_t N;
    int Kc, Mo;         // multiples of 16: the contraction, the output columns of a block
    int b_transposed;
    int stages;         // a multiple of the groups
    int acc_bufs;       // 2: the next tile's products run beside this one's epilogue
    int acc_stride, tmem_cols;  // tensor memory columns of an accumulator buffer, and of all
    int split, half, corr;      // exact kernels: first k-step of the second main sum; columns of that sum and of the corrections in a buffer
    int* status;
    int reset;          // set the status word to 0
    const float* bias;  // [cols] added to every output row, or nullptr
    int relu;           // max(y, 0) after the bias
    int kc, cols;       // contraction and output columns that exist (the rest of the last block is zeros)
    int direct;         // rows of Y do not start on 16 bytes: written directly instead of by bulk stores through mapY
    float* Y;           // rows ldy apart
    int64_t ldy;
};

template <int G, bool EXACT>
__global__ void __launch_bounds__(TF_THREADS, 1)
linear_tma_f32_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapY, const TmaF32Params P) {
    extern __shared__ unsigned char smem_raw[];
    // f_full[S], f_empty[S], o_full[G], o_empty[G], acc_full[2], acc_empty[2]
    __shared__ __align__(8) uint64_t bars[2 * TF_MAX_STAGES + 2 * TF_MAX_OPS + 4];
    __shared__ __align__(16) float s_bias[256];
    __shared__ uint32_t tmem_base_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // this CTA's block of output columns: [c0, c0 + mo), as the MMA sees it Mo wide
    const int c0 = (int)blockIdx.y * P.Mo, mo = min(P.cols - c0, P.Mo);
    const int Kc = P.Kc, Mo = (mo + 15) & ~15, S = P.stages;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int kchunks = Kc / 8;                    // 16-byte chunks of bf16 along the whole contraction
    const uint32_t b_sbo = (uint32_t)kchunks * 128;  // weight levels: same layout as a whole-K operand
    const uint32_t b_level = (uint32_t)Mo * Kc * 2;
    const uint32_t w0 = base, ring0 = base + ((3 * b_level + 1023u) & ~1023u);
    const uint32_t stage0 = ring0 + (uint32_t)S * TF_SLICE_BYTES;  // per epilogue warp: 32 rows x 32 fp32 columns of Y
    const int nslices = (Kc + TF_KB - 1) / TF_KB;
    const uint32_t bar0 = smem_u32(bars);
    auto f_full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto f_empty = [&](int s) { return bar0 + 8u * (uint32_t)(TF_MAX_STAGES + s); };
    auto o_full = [&](int o) { return bar0 + 8u * (uint32_t)(2 * TF_MAX_STAGES + o); };
    auto o_empty = [&](int o) { return bar0 + 8u * (uint32_t)(2 * TF_MAX_STAGES + TF_MAX_OPS + o); };
    auto acc_full = [&](int a) { return bar0 + 8u * (uint32_t)(2 * TF_MAX_STAGES + 2 * TF_MAX_OPS + a); };
    auto acc_empty = [&](int a) { return bar0 + 8u * (uint32_t)(2 * TF_MAX_STAGES + 2 * TF_MAX_OPS + 2 + a); };
    constexpr int GW = TF_CONV_WARPS / G;  // warps per group

    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(f_full(s), 1); mbar_init(f_empty(s), GW); }
        for (int o = 0; o < G; ++o) { mbar_init(o_full(o), GW); mbar_init(o_empty(o), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(acc_full(a), 1); mbar_init(acc_empty(a), TF_EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapY)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)P.tmem_cols);
    pdl_wait_exclusive();
    if (P.reset && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *P.status = 0;
    const int64_t ntiles = (P.N + TC_ROWS - 1) / TC_ROWS;
    const uint64_t stream = policy_evict_first();
    auto load = [&](int64_t t, int j, uint32_t it) {
        const int s = (int)(it % (uint32_t)S);
        mbar_arrive_expect_tx(f_full(s), TF_SLICE_BYTES);
        tma_load_2d(ring0 + (uint32_t)s * TF_SLICE_BYTES, &mapX, j * TF_KB, (int)(t * TC_ROWS), f_full(s), stream);
    };
    uint32_t early = 0;  // slices of X that arrive while the weights are split: as many as there are slots, of the first tile
    if (tid == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (; early < (uint32_t)min(S, nslices); ++early) load(blockIdx.x, (int)early, early);
    }
    // weight levels.  16-byte chunk c of stored row r:
    //   stored [Kc,Mo] (MN-major B): r = k, c = 8 output columns: offset c*sbo + (k/8)*128 + (k%8)*16
    //   stored [Mo,Kc] (K-major  B): r = n, c = 8 k's:            offset (n/8)*sbo + c*128 + (n%8)*16
    // eight consecutive threads take the eight rows of one core matrix: contiguous 16-byte stores
    {
        const int rows = P.b_transposed ? Mo : Kc, chunks = (P.b_transposed ? Kc : Mo) / 8;
        const int have_rows = P.b_transposed ? mo : P.kc, have_cols = P.b_transposed ? P.kc : mo;
        const float* const Wc = P.W + (P.b_transposed ? (size_t)c0 * P.ldw : (size_t)c0);
        constexpr int U = 3;  // chunks per thread in flight
        for (int e0 = tid; e0 < rows * chunks; e0 += U * TF_THREADS) {
            float x[U][8];
            uint32_t off[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int e = e0 + u * TF_THREADS;
                const int q = e >> 3, rg = q / chunks, c = q - rg * chunks, r = rg * 8 + (e & 7);
                const float* srcf = Wc + (size_t)r * P.ldw + (size_t)c * 8;
                off[u] = P.b_transposed ? (uint32_t)(r >> 3) * b_sbo + (uint32_t)c * 128 + (uint32_t)(r & 7) * 16
                                        : (uint32_t)c * b_sbo + (uint32_t)(r >> 3) * 128 + (uint32_t)(r & 7) * 16;
                if (P.ldw % 4 == 0 && r < have_rows && c * 8 + 8 <= have_cols) {
                    const float4 lo = reinterpret_cast<const float4*>(srcf)[0], hi = reinterpret_cast<const float4*>(srcf)[1];
                    x[u][0] = lo.x; x[u][1] = lo.y; x[u][2] = lo.z; x[u][3] = lo.w; x[u][4] = hi.x; x[u][5] = hi.y; x[u][6] = hi.z; x[u][7] = hi.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) x[u][j] = (r < have_rows && c * 8 + j < have_cols) ? srcf[j] : 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (e0 + u * TF_THREADS >= rows * chunks) break;
                uint4 lv[3];
                split8(x[u], lv);
#pragma unroll
                for (int l = 0; l < 3; ++l) st_shared16(w0 + (uint32_t)l * b_level + off[u], lv[l]);
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot, nbuf = EXACT ? (uint32_t)P.acc_bufs : 2u;
    bool failed = false;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;
            for (int64_t t = blockIdx.x; t < ntiles && !failed; t += gridDim.x)
                for (int j = 0; j < nslices; ++j, ++it) {
                    if (it < early) continue;
                    if (!mbar_wait_bounded(f_empty((int)(it % (uint32_t)S)), ((it / (uint32_t)S) & 1u) ^ 1u)) { failed = true; break; }
                    load(t, j, it);
                }
            if (failed) {
                const uint32_t first = it > (uint32_t)S ? it - (uint32_t)S : 0u;
                for (uint32_t i = first; i < it; ++i) mbar_wait_bounded(f_full((int)(i % (uint32_t)S)), (i / (uint32_t)S) & 1u);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = make_idesc(Mo, P.b_transposed ? 0 : 1), b_level16 = b_level / 16;
            uint32_t it = 0, lt = 0;
            for (int64_t t = blockIdx.x; t < ntiles && !failed; t += gridDim.x, ++lt) {
                const uint32_t a = lt % nbuf;
                if (!mbar_wait_bounded(acc_empty((int)a), ((lt / nbuf) & 1u) ^ 1u)) { failed = true; break; }
                tc_fence_after();
                const uint32_t dacc = tmem_base + a * (uint32_t)P.acc_stride;
                for (int j = 0; j < nslices; ++j, ++it) {
                    const uint32_t o = it % G;
                    if (!mbar_wait_bounded(o_full((int)o), (it / G) & 1u)) { failed = true; break; }
                    tc_fence_after();
                    const uint32_t at = tmem_base + nbuf * (uint32_t)P.acc_stride + o * (uint32_t)TF_OP_COLS;
                    const uint64_t bdesc = make_smem_desc(w0 + (uint32_t)j * (TF_KB / 16) * 256u, 128, b_sbo);
                    const bool both = Kc - j * TF_KB >= TF_KB;  // else a last slice of 16
#pragma unroll
                    for (int kk = 0; kk < TF_KB / 16; ++kk) {
                        if (kk > 0 && !both) break;
#pragma unroll
                        for (int q = 0; q < 6; ++q) {  // offsets add to the descriptors' address field, in units of 16 bytes
                            const uint64_t bd = bdesc + (uint64_t)(pair_b(q) * b_level16 + (uint32_t)kk * 16u);
                            uint32_t to = dacc, more = (j > 0 || kk > 0 || q > 0) ? 1u : 0u;
                            if (EXACT) {
                                const int ks = j * (TF_KB / 16) + kk;
                                if (q < 5) to += (uint32_t)P.corr;
                                else {
                                    more = ks != 0 && ks != P.split;
                                    if (ks >= P.split) to += (uint32_t)P.half;
                                }
                            }
                            mma_bf16_ts(to, at + pair_a(q) * (TF_KB / 2) + (uint32_t)kk * 8u, bd, idesc, more);
                        }
                    }
                    mma_commit(o_empty((int)o));
                }
                if (failed) break;
                mma_commit(acc_full((int)a));
            }
        }
    } else if (warp < 2 + TF_CONV_WARPS) {
        const int grp = (warp - 2) / GW, wl = (warp - 2) % GW;
        uint32_t it = 0;
        for (int64_t t = blockIdx.x; t < ntiles && !failed; t += gridDim.x)
            for (int j = 0; j < nslices; ++j, ++it) {
                if (it % G != (uint32_t)grp) continue;
                const int s = (int)(it % (uint32_t)S);
                if (!mbar_wait_bounded(f_full(s), (it / (uint32_t)S) & 1u)) { failed = true; break; }
                if (!mbar_wait_bounded(o_empty(grp), ((it / G) & 1u) ^ 1u)) { failed = true; break; }
                tc_fence_after();
                const uint32_t src = ring0 + (uint32_t)s * TF_SLICE_BYTES;
                // a warp reaches the 32 lanes of tensor memory of its number modulo 4
                const int r = (warp & 3) * 32 + lane;
                const uint32_t to = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + nbuf * (uint32_t)P.acc_stride + (uint32_t)(grp * TF_OP_COLS);
#pragma unroll
                for (int rep = 0; rep < 16 / GW; ++rep) {
                    const int kc = (wl >> 2) + rep * (GW / 4);
                    // 8 values of row r: fp32 row of 128 bytes, 16-byte chunk c at position c ^ (r % 8)
                    const uint4 c0 = ld_shared16(src + (uint32_t)r * 128u + (uint32_t)(((2 * kc) ^ (r & 7)) << 4));
                    const uint4 c1 = ld_shared16(src + (uint32_t)r * 128u + (uint32_t)(((2 * kc + 1) ^ (r & 7)) << 4));
                    const float x[8] = {__uint_as_float(c0.x), __uint_as_float(c0.y), __uint_as_float(c0.z), __uint_as_float(c0.w),
                                        __uint_as_float(c1.x), __uint_as_float(c1.y), __uint_as_float(c1.z), __uint_as_float(c1.w)};
                    uint4 lv[3];
                    split8(x, lv);
#pragma unroll
                    for (int l = 0; l < 3; ++l) tmem_st4(to + (uint32_t)(l * (TF_KB / 2) + kc * 4), lv[l]);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { mbar_arrive(f_empty(s)); mbar_arrive(o_full(grp)); }
            }
    } else {
        const int ew = warp - (2 + TF_CONV_WARPS), quarter = warp & 3, half = ew >> 2;
        const uint32_t stg = stage0 + (uint32_t)ew * 4096u;
        stage_bias(s_bias, P.bias ? P.bias + c0 : nullptr, mo, 32 * (2 + TF_CONV_WARPS));
        uint32_t lt = 0;
        for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++lt) {
            const uint32_t a = lt % nbuf;
            if (!mbar_wait_bounded(acc_full((int)a), (lt / nbuf) & 1u)) { failed = true; break; }
            tc_fence_after();
            const int64_t row0 = t * TC_ROWS + quarter * 32;  // first of this warp's 32 rows
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + a * (uint32_t)P.acc_stride;
            for (int cb = half; cb * 32 < Mo; cb += 2) {  // blocks of 32 columns = 128-byte rows
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // staging block free again
                __syncwarp();
                const int groups = (Mo - cb * 32 >= 32 ? 32 : Mo - cb * 32) / 16;
                for (int g16 = 0; g16 < groups; ++g16) {
                    uint32_t r[16];
                    tmem_ld16(taddr + (uint32_t)(cb * 32 + g16 * 16), r);
                    tmem_ld_wait();
                    if (EXACT) {  // main + second main + corrections
                        for (int w = P.half > 0 ? 0 : 1; w < 2; ++w) {
                            uint32_t more[16];
                            tmem_ld16(taddr + (uint32_t)((w == 0 ? P.half : P.corr) + cb * 32 + g16 * 16), more);
                            tmem_ld_wait();
#pragma unroll
                            for (int q = 0; q < 16; ++q) r[q] = __float_as_uint(__uint_as_float(r[q]) + __uint_as_float(more[q]));
                        }
                    }
                    if (P.bias || P.relu) {
                        float f[16];
#pragma unroll
                        for (int q = 0; q < 16; ++q) f[q] = __uint_as_float(r[q]);
                        bias_relu16(f, s_bias + cb * 32 + g16 * 16, P.bias != nullptr, P.relu != 0);
#pragma unroll
                        for (int q = 0; q < 16; ++q) r[q] = __float_as_uint(f[q]);
                    }
                    // row = lane, 128 bytes per row; 16-byte chunk c sits at position c ^ (row % 8)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        st_shared16(stg + (uint32_t)lane * 128u + ((uint32_t)((4 * g16 + q) ^ (lane & 7)) << 4),
                                    make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]));
                }
                // a row of up to 32 columns per step, a column per lane; also where a box of 32 columns would reach into the next block
                if (P.direct || (cb * 32 + 32 > mo && c0 + mo < P.cols)) {
                    __syncwarp();
                    const int rows = (int)(P.N - row0 < 32 ? P.N - row0 : 32);
                    if (cb * 32 + lane < mo)
                        for (int r = 0; r < rows; ++r) {
                            float v;
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(stg + (uint32_t)r * 128u + ((uint32_t)((lane >> 2) ^ (r & 7)) << 4) + (uint32_t)(lane & 3) * 4u) : "memory");
                            P.Y[(row0 + r) * P.ldy + c0 + cb * 32 + lane] = v;
                        }
                    __syncwarp();
                    continue;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0 && row0 < P.N) {  // rows past N are clipped by the copy engine
                    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                     reinterpret_cast<uint64_t>(&mapY)),
                                 "r"(c0 + cb * 32), "r"((int)row0), "r"(stg)
                                 : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty((int)a));
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    if (failed) atomicExch(P.status, 7);  // GNN_ERR_TIMEOUT
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, (uint32_t)P.tmem_cols);
}

// ------------------------------------------------------------------ dW = X^T * dY
// Contraction over the N rows.  A = X^T (features x rows) and B = dY (rows x columns) are both
// MN-major as stored, so the same 64-column x 64-row swizzled boxes serve: a pipeline slot holds 64
// rows of X (K/64 boxes) and of dY (M/64 boxes).  The MMA warp issues, per slot, four k-steps of 16
// rows for each half of 128 features (MMA shape 128 x M x 16) into per-CTA accumulators that stay in
// tensor memory for the whole kernel; at the end the epilogue warps write one fp32 partial [K,M] per
// CTA, and the partials are summed in CTA order by the caller (fixed order: deterministic).
constexpr int DW_ROWS = 64;                         // rows of X / dY per slot
constexpr uint32_t DW_BOX_BYTES = DW_ROWS * 128;    // one 64 x 64 bf16 box

struct TmaDwParams {
    float* part;  // [gridDim.x][K][M]
    int64_t N;
    int K, M;
    int stages;
    int tmem_cols;
    int* status;
    int reset;  // first launch of a call: set the status word to 0
};

__global__ void __launch_bounds__(TM_THREADS, 1)
linear_tma_dw_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapD,
                     const __grid_constant__ CUtensorMap mapP, const TmaDwParams P) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * TM_MAX_STAGES + 1];  // full[S], empty[S], acc_full
    __shared__ uint32_t tmem_base_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = P.K, M = P.M, S = P.stages;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // whole blocks of the MMA's 128 feature rows: boxes that start past column K arrive as zeros
    const int halves = (K + 127) / 128, xboxes = 2 * halves, dboxes = (M + 63) / 64;
    const uint32_t slot_bytes = (uint32_t)(xboxes + dboxes) * DW_BOX_BYTES;
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(TM_MAX_STAGES + s); };
    const uint32_t acc_full = bar0 + 8u * (2 * TM_MAX_STAGES);

    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(acc_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapD)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapP)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)P.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_exclusive();
    if (P.reset && blockIdx.x == 0 && tid == 0) *P.status = 0;
    const uint32_t tmem_base = tmem_base_slot;
    const int64_t nchunks = (P.N + DW_ROWS - 1) / DW_ROWS;  // gridDim.x <= nchunks: every CTA has work
    bool failed = false;

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t stream = policy_evict_first();
            uint32_t it = 0;
            for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x, ++it) {
                const int s = (int)(it % (uint32_t)S);
                if (!mbar_wait_bounded(empty(s), ((it / (uint32_t)S) & 1u) ^ 1u)) { failed = true; break; }
                mbar_arrive_expect_tx(full(s), slot_bytes);
                const uint32_t slot = base + (uint32_t)s * slot_bytes;
                for (int b = 0; b < xboxes; ++b) tma_load_2d(slot + (uint32_t)b * DW_BOX_BYTES, &mapX, b * 64, (int)(c * DW_ROWS), full(s), stream);
                for (int b = 0; b < dboxes; ++b)
                    tma_load_2d(slot + (uint32_t)(xboxes + b) * DW_BOX_BYTES, &mapD, b * 64, (int)(c * DW_ROWS), full(s), stream);
            }
            if (failed) {
                const uint32_t first = it > (uint32_t)S ? it - (uint32_t)S : 0u;
                for (uint32_t i = first; i < it; ++i) mbar_wait_bounded(full((int)(i % (uint32_t)S)), (i / (uint32_t)S) & 1u);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = make_idesc(M, 1, 1);  // A and B both MN-major
            uint32_t it = 0;
            for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x, ++it) {
                const int s = (int)(it % (uint32_t)S);
                if (!mbar_wait_bounded(full(s), (it / (uint32_t)S) & 1u)) { failed = true; break; }
                tc_fence_after();
                const uint32_t sa = base + (uint32_t)s * slot_bytes, sb = sa + (uint32_t)xboxes * DW_BOX_BYTES;
                for (int h = 0; h < halves; ++h)
                    for (int kk = 0; kk < DW_ROWS / 16; ++kk) {
                        // rows (contraction) are 128 bytes apart, groups of 8 rows 1024 bytes, blocks of 64 features / columns one box
                        const uint64_t adesc = make_smem_desc(sa + (uint32_t)(2 * h) * DW_BOX_BYTES + (uint32_t)kk * 2048u, DW_BOX_BYTES, 1024, SW128);
                        const uint64_t bdesc = make_smem_desc(sb + (uint32_t)kk * 2048u, DW_BOX_BYTES, 1024, SW128);
                        mma_bf16_ss(tmem_base + (uint32_t)(h * M), adesc, bdesc, idesc, (it > 0 || kk > 0) ? 1u : 0u);
                    }
                mma_commit(empty(s));
            }
            if (!failed) mma_commit(acc_full);
        }
    } else {
        const int ew = warp - 2, quarter = warp & 3, half = ew >> 2;
        if (!mbar_wait_bounded(acc_full, 0)) {
            failed = true;
        } else {
            tc_fence_after();
            // the pipeline slots are idle now (every load was consumed before the last commit): each warp
            // stages 32 feature rows x 32 columns of fp32 there and sends them with a bulk tensor store
            const uint32_t stg = base + (uint32_t)ew * 4096u;
            for (int h = 0; h < halves; ++h) {
                if (h * 128 + quarter * 32 >= K) break;  // feature rows past K (K is a multiple of 32): the next CTA's rows of the partial matrix
                const int prow0 = (int)blockIdx.x * K + h * 128 + quarter * 32;  // row of the [parts*K, M] partial matrix
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(h * M);
                for (int cb = half; cb * 32 < M; cb += 2) {
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    __syncwarp();
                    const int groups = (M - cb * 32 >= 32 ? 32 : M - cb * 32) / 16;
                    for (int g16 = 0; g16 < groups; ++g16) {
                        uint32_t r[16];
                        tmem_ld16(taddr + (uint32_t)(cb * 32 + g16 * 16), r);
                        tmem_ld_wait();
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            st_shared16(stg + (uint32_t)lane * 128u + ((uint32_t)((4 * g16 + q) ^ (lane & 7)) << 4),
                                        make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]));
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                         reinterpret_cast<uint64_t>(&mapP)),
                                     "r"(cb * 32), "r"(prow0), "r"(stg)
                                     : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            }
            if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        }
    }
    if (failed) atomicExch(P.status, 7);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, (uint32_t)P.tmem_cols);
}

// K and M: any (inside, rounded up to 32 and 16 with zeros from the copy engine; that is the shape of the partials)
bool linear_tma_dw_supported(int64_t N, int K, int M, gnn_dtype dtype) {
    if (dtype != GNN_BF16 || N <= 0 || N >= ((int64_t)1 << 31) - TC_ROWS) return false;
    if (K < 1 || K > 512 || M < 1 || M > 256) return false;
    if (up16(M) * ((K + 127) / 128) > 512) return false;  // one accumulator [128, M] per block of 128 features: 512 columns of tensor memory
    return encoder() != nullptr;
}

int linear_tma_dw_partials(int64_t N) {
    const int64_t nchunks = (N + DW_ROWS - 1) / DW_ROWS;
    return (int)(nchunks < 148 ? (nchunks > 0 ? nchunks : 1) : 148);
}

bool make_map_f32(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int box_rows);

// writes linear_tma_dw_partials(N) fp32 partials [up32(K), up16(M)] to part; X and dY: rows ldx and ldd elements apart
gnn_status linear_tma_dw(const void* X, int ldx, const void* dY, int ldd, int64_t N, int K, int M, float* part, int* d_flag, int reset, cudaStream_t st) {
    const char* who = "gnn_linear_backward (pipelined tensor-core dW)";
    GNN_REQUIRE(aligned16(X) && aligned16(dY) && aligned16(part), GNN_ERR_INVALID_ARG, "%s: matrices must be 16-byte aligned", who);
    const int K32 = up32(K), M16 = up16(M);
    CUtensorMap mapX, mapD, mapP;
    if (!make_map_ld(&mapX, X, N, K, ldx, DW_ROWS) || !make_map_ld(&mapD, dY, N, M, ldd, DW_ROWS) ||
        !make_map_f32(&mapP, part, (int64_t)linear_tma_dw_partials(N) * K32, M16, 32))
        GNN_FAIL(GNN_ERR_CUDA, "%s: tensor map encoding failed", who);
    TmaDwParams P;
    P.part = part; P.N = N; P.K = K32; P.M = M16; P.status = d_flag; P.reset = reset;
    const size_t slot = (size_t)(2 * ((K32 + 127) / 128) + (M16 + 63) / 64) * DW_BOX_BYTES;
    int stages = (int)((TM_SMEM_MAX - 1024) / slot);
    P.stages = stages > TM_MAX_STAGES ? TM_MAX_STAGES : stages;
    int cols = 32;
    while (cols < M16 * ((K32 + 127) / 128)) cols <<= 1;
    P.tmem_cols = cols;
    gnn_status rc = allow_big_smem(who, (const void*)linear_tma_dw_kernel, 5, TM_SMEM_MAX);
    if (rc != GNN_OK) return rc;
    launch_overlapped(linear_tma_dw_kernel, dim3((unsigned)linear_tma_dw_partials(N)), dim3(TM_THREADS), 1024 + (size_t)P.stages * slot, st, mapX, mapD, mapP, P);
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

// row-major fp32 matrix [rows, cols]; box = 32 columns (128 bytes, swizzled) x box_rows rows
// the same for a block of columns of a wider matrix: rows ld elements apart
static bool make_map_f32_ld(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int ld, int box_rows);
bool make_map_f32(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int box_rows) {
    return make_map_f32_ld(m, ptr, rows, cols, cols, box_rows);
}
static bool make_map_f32_ld(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int ld, int box_rows) {
    EncodeTiledFn enc = encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
    const cuuint32_t box[2] = {32, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same with all columns in one box, stored as the boxes of 32 columns one after the other: dimensions (32 columns, rows,
// blocks of 32 columns).  Whole blocks only: the copy engine would read a partial one past the row.
static bool make_map_f32_blocks(CUtensorMap* m, const void* ptr, int64_t rows, int cols, int ld, int box_rows) {
    EncodeTiledFn enc = encoder();
    if (!enc) return false;
    const cuuint64_t dims[3] = {32, (cuuint64_t)rows, (cuuint64_t)(cols / 32)};
    const cuuint64_t strides[2] = {(cuuint64_t)ld * 4, 128};
    const cuuint32_t box[3] = {32, (cuuint32_t)box_rows, (cuuint32_t)(cols / 32)};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ------------------------------------------------------------------ fp32: dW = X^T * dY on the bf16 tensor cores, pipelined
// Contraction over the N rows, 32 rows per pipeline slot (16 where K or M is over 128, so that two operand buffers and a
// ring still fit shared memory).  Roles of the persistent CTA:
//   warp 0      loader: a slot is K/32 + M/32 boxes of 32 rows x 32 fp32 columns (128-byte rows, 128-byte swizzle)
//               of X and dY, in a ring of shared-memory slots;
//   warps 2..17 converters, P.groups groups of them, slot i to group i mod groups (see the kernel above): split every
//               value exactly into three bf16 terms and write the levels of both operands
//               into the group's operand buffer in the canonical no-swizzle layout, MN-major (16-byte chunk c = 8
//               features or columns of row n at c*512 + (n/8)*128 + (n%8)*16);
//   warp 1      MMA issuer: 2 k-steps of 16 rows x 6 level pairs per slot, all into one accumulator [128 features x M]
//               that stays in tensor memory for the whole kernel;
//   at the end the first eight converter warps write the accumulator as this CTA's fp32 partial [K,M]; the caller sums the
//   partials in CTA order (fixed order: deterministic).
// K a multiple of 32 up to 512 features (blocks of the MMA's 128 rows; those past K are zeros), M a multiple of 32 up to 256.
// Every wait is bounded.
// Two groups on slots of 32 rows, on slots of 16 four where four buffers and slots fit.  170k x 128 x 128: 50 us with 8 warps
// on one slot after the other, 47 us with 16, 58 us in four groups on slots of 16 rows, 42 us so; reading X and dY takes 27 us.
// Then the bound was shared memory's bandwidth (copies, conversion and both operands of every MMA: 80 % of a slot's time), so X's
// levels go to tensor memory (A_TMEM), transposed on the way: a feature per lane, which leaves room for four groups on slots of 32 rows.  On slots
// of 16 rows, which had four groups before, that gives little and often loses, by the features that do not fill their four warps and by narrow results:
// A in shared / in tensor memory, 120k rows, K x M of 96 x 64 1.02, 128 x 128 1.04, 160 x 160 1.04, 256 x 128 1.03, 128 x 256 1.04, but 64 x 256 0.95,
// 160 x 192 0.91, 256 x 64 0.97, exact ones 187 x 59 0.96, 91 x 219 0.98; 170k x 200 x 47 92 and 98 us, x 100 x 200 100 and 105 us.
// Exact form (K or M no multiple of 32): the accumulator truncates at every MMA, 1.8e-8 of the result each and one way, so that
// a CTA's hundreds of rows in one sum cost 7.8e-6 norm-wise at 170k rows and 2.3e-5 at 500k, where the FFMA kernel that these
// sizes took before has 1.1e-6.  There the five small products go to an accumulator of corrections, and after every FD_FLUSH
// rows (32 main MMAs) four warps of their own add the main accumulator to the partial in fp32 while the MMAs go on in a second
// one (where tensor memory has room: up to 160 accumulator columns): 4.7e-7 at either size.  170k x 100 x 47: 52 -> 60 us
// (FFMA 1149 us); 500k x 500 x 250, where half as many columns fit a launch: 0.90 -> 1.79 ms (FFMA 6.4 ms).
constexpr int FD_CONV_WARPS = 16, FD_FLUSH_WARPS = 4;
constexpr int FD_THREADS = 32 * (2 + FD_CONV_WARPS);
constexpr int FD_FLUSH = 512;
constexpr int FD_MAX_STAGES = 8;
constexpr int FD_MAX_GROUPS = 4;

struct TmaF32DwParams {
    float* part;  // [gridDim.x][K][M]
    int64_t N;
    int K, M;
    int x_whole, d_whole;  // the slot's boxes of X or dY arrive in one copy
    int groups;  // 4 or 2
    int stages;  // a multiple of groups
    int mains;   // exact: main accumulators, 2 or 1; the corrections' columns follow them
    int tmem_cols;
    int* status;
    int reset;  // first launch of a call: set the status word to 0
};

template <int FD_ROWS, bool EXACT, bool A_TMEM>
__global__ void __launch_bounds__(FD_THREADS + (EXACT ? 32 * FD_FLUSH_WARPS : 0), 1)
linear_tma_f32_dw_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapD, const TmaF32DwParams P) {
    extern __shared__ unsigned char smem_raw[];
    // f_full[S], f_empty[S], o_full[G], o_empty[G], acc_full[2], acc_empty[2]
    __shared__ __align__(8) uint64_t bars[2 * FD_MAX_STAGES + 2 * FD_MAX_GROUPS + 4];
    __shared__ uint32_t tmem_base_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = P.K, M = P.M, S = P.stages, halves = (K + 127) / 128;
    const uint32_t G = (uint32_t)P.groups;
    constexpr uint32_t FD_BOX_BYTES = (uint32_t)FD_ROWS * 128u;   // one box: FD_ROWS rows x 32 fp32 columns
    constexpr uint32_t FD_SBO = (uint32_t)(FD_ROWS / 8) * 128u;   // next chunk of 8 features / columns in an operand level
    const int xboxes = K / 32, dboxes = M / 32;
    const uint32_t slot_bytes = (uint32_t)(xboxes + dboxes) * FD_BOX_BYTES;
    // the A operand always has whole blocks of the MMA's 128 feature rows; with K < 128 the rows past K stay zero (in tensor memory:
    // whatever they are, they only reach accumulator rows that nobody reads)
    const uint32_t a_level = A_TMEM ? 0u : (uint32_t)halves * 128u * FD_ROWS * 2, b_level = (uint32_t)M * FD_ROWS * 2;
    constexpr uint32_t A_COLS = FD_ROWS / 2;  // tensor memory columns of one level of 128 features
    const uint32_t op_bytes = 3u * (a_level + b_level);
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t ring0 = base, op0 = ring0 + (uint32_t)S * slot_bytes;
    const uint32_t bar0 = smem_u32(bars);
    auto f_full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto f_empty = [&](int s) { return bar0 + 8u * (uint32_t)(FD_MAX_STAGES + s); };
    auto o_full = [&](int o) { return bar0 + 8u * (uint32_t)(2 * FD_MAX_STAGES + o); };
    auto o_empty = [&](int o) { return bar0 + 8u * (uint32_t)(2 * FD_MAX_STAGES + FD_MAX_GROUPS + o); };
    auto acc_full = [&](uint32_t b) { return bar0 + 8u * ((uint32_t)(2 * FD_MAX_STAGES + 2 * FD_MAX_GROUPS) + b); };
    auto acc_empty = [&](uint32_t b) { return bar0 + 8u * ((uint32_t)(2 * FD_MAX_STAGES + 2 * FD_MAX_GROUPS + 2) + b); };
    constexpr uint32_t FLUSH = FD_FLUSH / FD_ROWS;  // slots per main sum
    const uint32_t mains = EXACT ? (uint32_t)P.mains : 1u, acc_cols = (uint32_t)(halves * M);

    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(f_full(s), 1); mbar_init(f_empty(s), FD_CONV_WARPS / G); }
        for (int o = 0; o < (int)G; ++o) { mbar_init(o_full(o), FD_CONV_WARPS / G); mbar_init(o_empty(o), 1); }
        for (uint32_t b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), FD_FLUSH_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapD)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)P.tmem_cols);
    if (!A_TMEM && K % 128 != 0) {  // the converters never write the feature rows past K: zero the buffers' A levels once
        for (int o = 0; o < (int)G; ++o)
            for (uint32_t off = (uint32_t)tid * 16u; off < 3u * a_level; off += blockDim.x * 16u)
                st_shared16(op0 + (uint32_t)o * op_bytes + off, make_uint4(0u, 0u, 0u, 0u));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait_exclusive();
    if (P.reset && blockIdx.x == 0 && tid == 0) *P.status = 0;
    const uint32_t tmem_base = tmem_base_slot;
    const int64_t nslots = (P.N + FD_ROWS - 1) / FD_ROWS;
    const uint32_t a_tmem = tmem_base + (EXACT ? mains + 1u : 1u) * acc_cols;  // A_TMEM: operand buffers, [group][128 features][level]
    bool failed = false;

    if (warp == 0) {
        // ------------------------------------------------------------ loader
        if (lane == 0) {
            const uint64_t stream = policy_evict_first();
            uint32_t it = 0;
            for (int64_t t = blockIdx.x; t < nslots; t += gridDim.x, ++it) {
                const int s = (int)(it % (uint32_t)S);
                if (!mbar_wait_bounded(f_empty(s), ((it / (uint32_t)S) & 1u) ^ 1u)) { failed = true; break; }
                mbar_arrive_expect_tx(f_full(s), slot_bytes);  // rows past N arrive as zeros and count all the same
                const uint32_t dst = ring0 + (uint32_t)s * slot_bytes;
                const int row = (int)(t * FD_ROWS);
                if (P.x_whole) tma_load_3d(dst, &mapX, 0, row, 0, f_full(s), stream);
                else
                    for (int b = 0; b < xboxes; ++b) tma_load_2d(dst + (uint32_t)b * FD_BOX_BYTES, &mapX, b * 32, row, f_full(s), stream);
                if (P.d_whole) tma_load_3d(dst + (uint32_t)xboxes * FD_BOX_BYTES, &mapD, 0, row, 0, f_full(s), stream);
                else
                    for (int b = 0; b < dboxes; ++b) tma_load_2d(dst + (uint32_t)(xboxes + b) * FD_BOX_BYTES, &mapD, b * 32, row, f_full(s), stream);
            }
            if (failed) {  // let the copies in flight land before the CTA goes away
                const uint32_t first = it > (uint32_t)S ? it - (uint32_t)S : 0u;
                for (uint32_t i = first; i < it; ++i) mbar_wait_bounded(f_full((int)(i % (uint32_t)S)), (i / (uint32_t)S) & 1u);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = make_idesc(M, 1, A_TMEM ? 0 : 1);  // B MN-major, A too where it lies in shared memory
            uint32_t it = 0, acc = tmem_base, fresh = 1, v = 0;  // fresh: the main sum begins with this slot; v: how many began before
            for (int64_t t = blockIdx.x; t < nslots; t += gridDim.x, ++it) {
                const uint32_t o = it % G;
                if (EXACT && fresh) {
                    if (!mbar_wait_bounded(acc_empty(v % mains), ((v / mains) & 1u) ^ 1u)) { failed = true; break; }
                    acc = tmem_base + v % mains * acc_cols;
                }
                if (!mbar_wait_bounded(o_full((int)o), (it / G) & 1u)) { failed = true; break; }
                tc_fence_after();
                const uint32_t abuf = op0 + o * op_bytes, bbuf = abuf + 3u * a_level;
                const uint64_t adesc = make_smem_desc(abuf, 128, FD_SBO), bdesc = make_smem_desc(bbuf, 128, FD_SBO);
                const uint32_t at = a_tmem + o * (uint32_t)halves * 3u * A_COLS;
                for (int h = 0; h < halves; ++h) {  // features [128h, 128h + 128): chunks 16h.., accumulator columns h*M..
#pragma unroll
                    for (int kk = 0; kk < FD_ROWS / 16; ++kk)
#pragma unroll
                        for (int q = 0; q < 6; ++q) {  // offsets add to the descriptors' address field, in units of 16 bytes
                            uint32_t to = acc, more = (it > 0 || kk > 0 || q > 0) ? 1u : 0u;
                            if (EXACT) {
                                if (q < 5) to = tmem_base + mains * acc_cols;
                                else more = (!fresh || kk > 0) ? 1u : 0u;
                            }
                            const uint64_t bd = bdesc + (uint64_t)(pair_b(q) * (b_level / 16) + (uint32_t)kk * 16u);
                            if (A_TMEM) mma_bf16_ts(to + (uint32_t)h * (uint32_t)M, at + ((uint32_t)h * 3u + pair_a(q)) * A_COLS + (uint32_t)kk * 8u, bd, idesc, more);
                            else
                                mma_bf16_ss(to + (uint32_t)h * (uint32_t)M, adesc + (uint64_t)(pair_a(q) * (a_level / 16) + (uint32_t)h * FD_SBO + (uint32_t)kk * 16u), bd, idesc, more);
                        }
                }
                mma_commit(o_empty((int)o));
                fresh = 0;
                if (EXACT && (it % FLUSH == FLUSH - 1 || t + gridDim.x >= nslots)) {  // (commits cover everything issued so far)
                    mma_commit(acc_full(v % mains));
                    fresh = 1;
                    ++v;
                }
            }
            if (!EXACT && !failed) mma_commit(acc_full(0));
        }
    } else if (EXACT && warp >= 2 + FD_CONV_WARPS) {
        // ------------------------------------------------------------ flush: main sums, and at last the corrections, to this CTA's partial
        const int quarter = warp & 3;  // a warp reaches the 32 lanes of tensor memory of its number modulo 4
        const uint32_t slots = (uint32_t)((nslots - blockIdx.x + gridDim.x - 1) / gridDim.x), sums = (slots + FLUSH - 1) / FLUSH;
        for (uint32_t v = 0; v < sums; ++v) {
            if (!mbar_wait_bounded(acc_full(v % mains), (v / mains) & 1u)) { failed = true; break; }
            tc_fence_after();
            for (int h = 0; h < halves; ++h) {
                if (h * 128 + quarter * 32 >= K) break;  // feature rows past K
                float* prow = P.part + ((size_t)blockIdx.x * K + h * 128 + quarter * 32 + lane) * M;
                const uint32_t lanes = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)h * (uint32_t)M;
                for (int c0 = 0; c0 < M; c0 += 16) {
                    uint32_t r[16], c[16];
                    tmem_ld16(lanes + v % mains * acc_cols + (uint32_t)c0, r);
                    if (v + 1 == sums) tmem_ld16(lanes + mains * acc_cols + (uint32_t)c0, c);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float4* const to = reinterpret_cast<float4*>(prow + c0) + q;
                        float4 s = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]), __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
                        if (v > 0) {
                            const float4 b = *to;
                            s.x += b.x; s.y += b.y; s.z += b.z; s.w += b.w;
                        }
                        if (v + 1 == sums) {
                            s.x += __uint_as_float(c[4 * q]); s.y += __uint_as_float(c[4 * q + 1]);
                            s.z += __uint_as_float(c[4 * q + 2]); s.w += __uint_as_float(c[4 * q + 3]);
                        }
                        *to = s;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(v % mains));
        }
    } else {
        // ------------------------------------------------------------ converters
        // A unit of 32 lanes: 8 rows of a box x its 4 chunks of 8 columns, so that every address is a sum of the lane's part
        // and the unit's; eight lanes read eight rows (swizzled: no conflict) and write one core matrix.
        constexpr int BU = FD_ROWS / 8;  // units per box
        const int GW = FD_CONV_WARPS / (int)G;  // warps per group
        const uint32_t o = (uint32_t)((warp - 2) / GW);
        const int units = (xboxes + dboxes) * BU, r7 = lane & 7, kc = lane >> 3;
        const uint32_t from0 = (uint32_t)r7 * 128u + (uint32_t)(((2 * kc) ^ r7) << 4), from1 = (uint32_t)r7 * 128u + (uint32_t)(((2 * kc + 1) ^ r7) << 4);
        const uint32_t to_l = (uint32_t)kc * FD_SBO + (uint32_t)r7 * 16u;
        uint32_t it = 0;
        for (int64_t t = blockIdx.x; t < nslots && !failed; t += gridDim.x, ++it) {
            if (it % G != o) continue;
            const int s = (int)(it % (uint32_t)S);
            if (!mbar_wait_bounded(f_full(s), (it / (uint32_t)S) & 1u)) { failed = true; break; }
            if (!mbar_wait_bounded(o_empty((int)o), ((it / G) & 1u) ^ 1u)) { failed = true; break; }
            tc_fence_after();
            const uint32_t src0 = ring0 + (uint32_t)s * slot_bytes;
            const uint32_t abuf = op0 + o * op_bytes, bbuf = abuf + 3u * a_level;
            if (A_TMEM) {  // a feature per lane, eight rows at a time; a warp reaches the 32 lanes of tensor memory of its number modulo 4
                const int quarter = warp & 3;
                const uint32_t at = a_tmem + o * (uint32_t)halves * 3u * A_COLS + ((uint32_t)(quarter * 32) << 16);
                for (int h = 0; h < halves; ++h) {
                    const int box = 4 * h + quarter;
                    if (box >= xboxes) break;
                    const uint32_t src = src0 + (uint32_t)box * FD_BOX_BYTES + (uint32_t)(lane & 3) * 4u;
                    for (int rg = ((warp - 2) % GW) >> 2; rg < BU; rg += GW >> 2) {
                        float x[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x[j]) : "r"(src + (uint32_t)rg * 1024u + (uint32_t)j * 128u + (uint32_t)(((lane >> 2) ^ j) << 4)) : "memory");
                        uint4 lv[3];
                        split8(x, lv);
#pragma unroll
                        for (int l = 0; l < 3; ++l) tmem_st4(at + (uint32_t)(h * 3 + l) * A_COLS + (uint32_t)rg * 4u, lv[l]);
                    }
                }
                tmem_st_wait();
                tc_fence_before();
            }
#pragma unroll 2
            for (int u = (warp - 2) % GW + (A_TMEM ? xboxes * BU : 0); u < units; u += GW) {
                const int box = u / BU, rg = u % BU;
                const uint32_t rows8 = src0 + (uint32_t)box * FD_BOX_BYTES + (uint32_t)rg * 1024u;
                const uint4 c0 = ld_shared16(rows8 + from0), c1 = ld_shared16(rows8 + from1);
                const float x[8] = {__uint_as_float(c0.x), __uint_as_float(c0.y), __uint_as_float(c0.z), __uint_as_float(c0.w),
                                    __uint_as_float(c1.x), __uint_as_float(c1.y), __uint_as_float(c1.z), __uint_as_float(c1.w)};
                uint4 lv[3];
                split8(x, lv);
                const bool isx = box < xboxes;
                const uint32_t level = isx ? a_level : b_level;
                const uint32_t dst = (isx ? abuf + (uint32_t)box * 4u * FD_SBO : bbuf + (uint32_t)(box - xboxes) * 4u * FD_SBO) + (uint32_t)rg * 128u + to_l;
#pragma unroll
                for (int l = 0; l < 3; ++l) st_shared16(dst + (uint32_t)l * level, lv[l]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> visible to the tensor core
            __syncwarp();
            if (lane == 0) { mbar_arrive(f_empty(s)); mbar_arrive(o_full((int)o)); }
        }
        // accumulator -> this CTA's partial.  Lane = feature row; warps 2..5 take the lower half of the columns, 6..9 the upper
        if (!EXACT && !failed && !mbar_wait_bounded(acc_full(0), 0u)) failed = true;
        tc_fence_after();
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        for (int h = 0; h < halves && !failed && !EXACT && half < 2; ++h) {
            const int krow = h * 128 + quarter * 32 + lane;
            if (h * 128 + quarter * 32 >= K) break;  // tcgen05.ld is warp-wide: a warp whose 32 feature rows all lie past K skips it as one
            float* prow = P.part + ((size_t)blockIdx.x * K + krow) * M;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)h * (uint32_t)M;
            for (int c0 = half * (M / 2); c0 < (half + 1) * (M / 2); c0 += 16) {
                uint32_t r[16];
                tmem_ld16(taddr + (uint32_t)c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (krow < K)
                        *reinterpret_cast<float4*>(prow + c0 + 4 * q) = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                                                                                   __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
            }
        }
    }
    if (failed) atomicExch(P.status, 7);  // GNN_ERR_TIMEOUT
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, (uint32_t)P.tmem_cols);
}

// The exact form where the whole product (K features, Mo columns, of which a launch may take a block of M) is no multiple of 32
static bool fd_exact(int K, int Mo) { return K % 32 != 0 || Mo % 32 != 0; }

// K and M: any (inside, rounded up to 32 with zeros from the copy engine; that is the shape of the partials)
bool linear_tma_f32_dw_supported(int64_t N, int K, int M, int Mo, gnn_dtype dtype) {
    if (dtype != GNN_F32 || N <= 0 || N >= ((int64_t)1 << 31) - 32) return false;
    if (K < 1 || K > 512 || M < 1 || M > 256) return false;
    // accumulators [128, M] per block of 128 features, the exact form's main and corrections: 512 columns of tensor memory
    if (up32(M) * ((K + 127) / 128) * (fd_exact(K, Mo) ? 2 : 1) > 512) return false;
    return encoder() != nullptr;
}

// every CTA has at least one slot of 32 rows, so every partial is written
int linear_tma_f32_dw_partials(int64_t N) {
    const int64_t n = (N + 31) / 32;
    return (int)(n < 148 ? (n > 0 ? n : 1) : 148);
}

// writes linear_tma_f32_dw_partials(N) fp32 partials [up32(K), up32(M)] to part; X and dY: rows ldx and ldd elements apart
// (a block of Mr of the Mo columns of dY)
gnn_status linear_tma_f32_dw(const void* X, int ldx, const void* dY, int ldd, int64_t N, int Kr, int Mr, int Mo, float* part, int* d_flag, int reset, cudaStream_t st) {
    const char* who = "gnn_linear_backward (pipelined fp32 tensor-core dW)";
    GNN_REQUIRE(aligned16(X) && aligned16(dY) && aligned16(part), GNN_ERR_INVALID_ARG, "%s: matrices must be 16-byte aligned", who);
    const int K = up32(Kr), M = up32(Mr);
    CUtensorMap mapX, mapD;
    const int R = K > 128 || M > 128 ? 16 : 32, ka = (K + 127) / 128 * 128;
    TmaF32DwParams P;
    P.x_whole = Kr % 32 == 0; P.d_whole = Mr % 32 == 0;
    if (!(P.x_whole ? make_map_f32_blocks : make_map_f32_ld)(&mapX, X, N, Kr, ldx, R) || !(P.d_whole ? make_map_f32_blocks : make_map_f32_ld)(&mapD, dY, N, Mr, ldd, R))
        GNN_FAIL(GNN_ERR_CUDA, "%s: tensor map encoding failed", who);
    P.part = part; P.N = N; P.K = K; P.M = M; P.status = d_flag; P.reset = reset;
    const bool exact = fd_exact(Kr, Mo);
    const int acc_cols = M * (ka / 128);
    P.mains = exact && 3 * acc_cols <= 512 ? 2 : 1;
    const int acc_all = (exact ? P.mains + 1 : 1) * acc_cols;
    // X's levels in tensor memory (see above), where two buffers of them fit beside the accumulators (R = 32: always, 480 columns at most)
    const bool a_tmem = acc_all + 2 * (ka / 128) * 3 * (R / 2) <= 512 && (R == 32 || (!exact && (K > 128 ? M >= 128 && M <= 160 : K >= 96 && M == 256)));
    const size_t slot = (size_t)(K / 32 + M / 32) * R * 128, op = 3 * ((a_tmem ? 0 : (size_t)ka * R * 2) + (size_t)M * R * 2);
    auto columns = [&](int groups) { return acc_all + (a_tmem ? groups * (ka / 128) * 3 * (R / 2) : 0); };
    P.groups = (R == 16 || a_tmem) && 1024 + FD_MAX_GROUPS * (op + slot) <= TM_SMEM_MAX && columns(FD_MAX_GROUPS) <= 512 ? FD_MAX_GROUPS : 2;
    const size_t ops = (size_t)P.groups * op;
    int stages = (int)((TM_SMEM_MAX - 1024 - ops) / slot);
    if (stages > FD_MAX_STAGES) stages = FD_MAX_STAGES;
    P.stages = stages / P.groups * P.groups;
    int cols = 32;
    while (cols < columns(P.groups)) cols <<= 1;
    P.tmem_cols = cols;
    auto launch = [&](auto kernel, int which, int threads) {
        gnn_status rc = allow_big_smem(who, (const void*)kernel, which, TM_SMEM_MAX);
        if (rc != GNN_OK) return rc;
        launch_overlapped(kernel, dim3((unsigned)linear_tma_f32_dw_partials(N)), dim3((unsigned)threads), 1024 + ops + (size_t)P.stages * slot, st, mapX, mapD, P);
        GNN_CHECK_LAUNCH(who);
        return GNN_OK;
    };
    constexpr int more = FD_THREADS + 32 * FD_FLUSH_WARPS;
    if (R == 32) return exact ? launch(linear_tma_f32_dw_kernel<32, true, true>, 44, more) : launch(linear_tma_f32_dw_kernel<32, false, true>, 46, FD_THREADS);
    if (a_tmem) return launch(linear_tma_f32_dw_kernel<16, false, true>, 47, FD_THREADS);
    return exact ? launch(linear_tma_f32_dw_kernel<16, true, false>, 19, more) : launch(linear_tma_f32_dw_kernel<16, false, false>, 15, FD_THREADS);
}

static size_t tf_fixed_bytes(int Kc, int Mo) {
    return 1024 + (((size_t)3 * Mo * Kc * 2 + 1023) & ~(size_t)1023) + (size_t)TF_EPI_WARPS * 4096;
}

// Sizes that are no multiples of 16 take the exact form: their callers were given FFMA precision before they came to the
// tensor cores, whose accumulator truncates at every MMA (1.8e-8 of the result each, norm-wise, one way).  There the five
// small products of a k-step go to an accumulator of their own (2^-8 of the size, so are its truncations), and above ten
// k-steps the main products to two, added in fp32.  Distance to 64 bits, norm-wise, one sum -> separate sums (FFMA): contraction
// of 100 7.3e-7 -> 9.2e-8 (1.8e-7), of 512 3.4e-6 -> 2.1e-7 (4.1e-7), of 47 2.9e-7 -> 5.4e-8 (1.2e-7).  170k x 100 x 47 takes
// 32 us forward either way, 43 instead of 33 us for dX, which has one accumulator buffer only (FFMA 127 and 112 us).
static bool tf_exact(int Kc, int Mo) { return Kc % 16 != 0 || Mo % 16 != 0; }
static int tf_sums(int Kc, bool exact) { return !exact ? 1 : up16(Kc) / 16 > 10 ? 3 : 2; }

// do `bufs` buffers of `sums` accumulators and `groups` operand buffers fit the 512 columns of tensor memory?
static bool tf_tmem_fits(int width, int sums, int bufs, int groups) { return bufs * sums * up32(width) + groups * TF_OP_COLS <= 512; }

// widest block of output columns (a multiple of 16): two accumulator buffers (exact: at least one) and two operand buffers fit
// tensor memory, the three weight levels shared memory beside two slices
static int tf_column_block(int Kc, int Mo, bool exact) {
    int mc = Mo < 192 ? Mo : 192;
    while (mc >= 16 && (tf_fixed_bytes(Kc, mc) + 2 * TF_SLICE_BYTES > TM_SMEM_MAX || !tf_tmem_fits(mc, tf_sums(Kc, exact), exact ? 1 : 2, 2))) mc -= 16;
    return mc >= 16 ? mc : 0;
}

// Kc and Mo: any up to 512 and 1024 (inside, rounded up to 16 with zeros); a contraction of one is a single rounded product,
// which FFMA has exactly
bool linear_tma_f32_supported(int64_t N, int Kc, int Mo, gnn_dtype dtype) {
    if (dtype != GNN_F32 || N <= 0 || N >= ((int64_t)1 << 31) - TC_ROWS) return false;
    if (Kc < 2 || Kc > 512 || Mo < 1 || Mo > 1024) return false;
    if (tf_column_block(up16(Kc), up16(Mo), tf_exact(Kc, Mo)) == 0) return false;
    return encoder() != nullptr;
}

// X: rows ldx elements apart, on 16 bytes; Y [N,Mo] contiguous (rows that do not start on 16 bytes are written directly
// instead of by bulk stores).
// Blocks of output columns: as few as fit and equally wide (256 x 256 in three of 96, 96 and 64 at the side of one another;
// one launch after the other they took 233 us for 200k rows, 186 us now).  Few rows leave SMs idle: blocks of 32 columns
// for as long as there are SMs for them, which also divides the splitting of the weights (2000 x 128 x 128: 9.9 -> 7.8 us).
gnn_status linear_tma_f32_forward(const void* X, int ldx, const void* W, int64_t N, int Kc, int Mo, int b_transposed, void* Y, int* d_flag, int reset,
                                  cudaStream_t st, const float* bias, int relu) {
    const char* who = "gnn_linear (pipelined fp32 tensor-core path)";
    const bool direct = Mo % 4 != 0;
    GNN_REQUIRE(aligned16(X) && aligned16(W) && (direct || aligned16(Y)), GNN_ERR_INVALID_ARG, "%s: matrices must be 16-byte aligned", who);
    const bool exact = tf_exact(Kc, Mo);
    const int K16 = up16(Kc), sums = tf_sums(K16, exact), widest = tf_column_block(K16, up16(Mo), exact);
    GNN_REQUIRE(widest > 0, GNN_ERR_UNSUPPORTED, "%s: weights do not fit shared memory", who);
    CUtensorMap mapX, mapY;
    if (!make_map_f32_ld(&mapX, X, N, Kc, ldx, TC_ROWS) || (!direct && !make_map_f32_ld(&mapY, Y, N, Mo, Mo, 32)))
        GNN_FAIL(GNN_ERR_CUDA, "%s: tensor map encoding failed", who);
    if (direct) mapY = mapX;  // not used
    const int64_t ntiles = (N + TC_ROWS - 1) / TC_ROWS;
    int blocks = (int)ceil_div(Mo, widest), width = up16((int)ceil_div(Mo, blocks));
    if (ntiles * 2 * blocks <= 148 && width > 32) {
        const int more = (int)(148 / ntiles), w = up32((int)ceil_div(Mo, more));
        if (w < width) width = w;
    }
    blocks = (int)ceil_div(Mo, width);
    TmaF32Params P;
    P.W = (const float*)W; P.ldw = b_transposed ? Kc : Mo;
    P.N = N; P.Kc = K16; P.Mo = width; P.kc = Kc; P.cols = Mo; P.b_transposed = b_transposed; P.status = d_flag; P.reset = reset;
    P.bias = bias; P.relu = relu;
    P.direct = direct; P.Y = (float*)Y; P.ldy = Mo;
    const size_t fixed = tf_fixed_bytes(K16, width);
    int stages = (int)((TM_SMEM_MAX - fixed) / TF_SLICE_BYTES);  // at least two
    if (stages > TF_MAX_STAGES) stages = TF_MAX_STAGES;
    // four groups before a second accumulator buffer: only the exact form may be short of room for both
    const int most = stages >= 4 ? 4 : 2;
    P.acc_bufs = 2;
    int groups = most;
    if (!tf_tmem_fits(width, sums, 2, groups)) {
        if (tf_tmem_fits(width, sums, 1, groups) && exact) P.acc_bufs = 1;
        else {
            groups = 2;
            if (!tf_tmem_fits(width, sums, 2, 2)) P.acc_bufs = 1;
        }
    }
    P.acc_stride = sums * up32(width);
    P.half = sums == 3 ? up32(width) : 0; P.corr = (sums - 1) * up32(width);
    P.split = sums == 3 ? K16 / 32 : K16 / 16;
    P.stages = stages / groups * groups;
    int cols = 32;
    while (cols < P.acc_bufs * P.acc_stride + groups * TF_OP_COLS) cols <<= 1;
    P.tmem_cols = cols;
    auto launch = [&](auto kernel, int which) {
        gnn_status rc = allow_big_smem(who, (const void*)kernel, which, TM_SMEM_MAX);
        if (rc != GNN_OK) return rc;
        const int64_t per_block = blocks < 148 ? 148 / blocks : 1;
        launch_overlapped(kernel, dim3((unsigned)(ntiles < per_block ? ntiles : per_block), (unsigned)blocks), dim3(TF_THREADS),
                          fixed + (size_t)P.stages * TF_SLICE_BYTES, st, mapX, mapY, P);
        GNN_CHECK_LAUNCH(who);
        return GNN_OK;
    };
    if (exact) return groups == 4 ? launch(linear_tma_f32_kernel<4, true>, 16) : launch(linear_tma_f32_kernel<2, true>, 17);
    return groups == 4 ? launch(linear_tma_f32_kernel<4, false>, 6) : launch(linear_tma_f32_kernel<2, false>, 13);
}

}  // namespace gnn
