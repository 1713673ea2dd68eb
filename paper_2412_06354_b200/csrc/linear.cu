// Dense node-wise transform (the Dense layer / layer weight of the training example):
//   Y = X * W          X [N,K], W [K,M]
//   dX = dY * W^T      dY [N,M]
//   dW = X^T * dY      reduction over the N rows, split over row slabs and combined in slab order
//
// This file holds the entry points, their dispatch, and the fallback.  The products run on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory) through the pipelined kernels of linear_tma.cu for a contraction of up to
// 512 and up to 1024 output columns (dW: 512 x 256, or as much as fits tensor memory at a time), whatever the divisors of
// K and M: sizes are rounded up with zeros from the copy engine.  The copy engine wants rows that start on 16 bytes;
// matrices whose rows do not (K or M odd, say) are first copied to padded rows in the workspace, one pass at L2 or HBM
// speed.  Such shapes took the FFMA kernel before (170000 x 100 x 47 fp32, forward and backward: 1405 -> 121 us).
// Everything else, a driver without the tensor-map encoder and calls that lack the room or the alignment included, runs the
// shared-memory tiled FFMA kernel below with fp32 accumulation.  All sums have a fixed order.
#include "common.cuh"

namespace gnn {

// ------------------------------------------------------------------ FFMA path
// C[m,n] = sum_k A(m,k) * B(k,n) with arbitrary element strides, so transposed operands are
// stride swaps.  64x64 output tile per block, 16x16 threads, 4x4 outputs per thread, k in steps
// of 16.  k range [k0, k1) per blockIdx.z slab; slab results go to C + z*slab_stride.
constexpr int SG_TILE = 64, SG_K = 16;

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

template <typename TA, typename TB, typename TC>
__global__ void __launch_bounds__(256)
gemm_simt_kernel(const TA* __restrict__ A, int64_t sam, int64_t sak, const TB* __restrict__ B, int64_t sbk,
                 int64_t sbn, TC* __restrict__ C, int64_t Mr, int64_t Nc, int64_t Kd, int64_t k_per_slab,
                 int64_t slab_stride, const float* __restrict__ bias, int relu) {
    __shared__ float As[SG_K][SG_TILE + 1];
    __shared__ float Bs[SG_K][SG_TILE + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t m0 = (int64_t)blockIdx.y * SG_TILE, n0 = (int64_t)blockIdx.x * SG_TILE;
    const int64_t k0 = (int64_t)blockIdx.z * k_per_slab;
    const int64_t k1 = (k0 + k_per_slab < Kd) ? k0 + k_per_slab : Kd;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int64_t kb = k0; kb < k1; kb += SG_K) {
        for (int e = threadIdx.x; e < SG_K * SG_TILE; e += 256) {
            // A tile: consecutive threads walk the faster-varying of (m, k) in memory
            int kk, mm;
            if (sak <= sam) { kk = e % SG_K; mm = e / SG_K; } else { mm = e % SG_TILE; kk = e / SG_TILE; }
            const int64_t m = m0 + mm, k = kb + kk;
            As[kk][mm] = (m < Mr && k < k1) ? to_f32(A[m * sam + k * sak]) : 0.f;
            int kk2, nn;
            if (sbn <= sbk) { nn = e % SG_TILE; kk2 = e / SG_TILE; } else { kk2 = e % SG_K; nn = e / SG_K; }
            const int64_t n = n0 + nn, k2 = kb + kk2;
            Bs[kk2][nn] = (n < Nc && k2 < k1) ? to_f32(B[k2 * sbk + n * sbn]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < SG_K; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    TC* Cz = C + (size_t)blockIdx.z * slab_stride;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t m = m0 + ty * 4 + i;
        if (m >= Mr) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t n = n0 + tx * 4 + j;
            if (n < Nc) {
                float y = acc[i][j];
                if (bias) y += bias[n];  // the element-wise tail of a layer, before the single rounding
                if (relu) y = fmaxf(y, 0.f);
                Cz[m * Nc + n] = from_f32<TC>(y);
            }
        }
    }
}

// out[i] = sum over slabs of part[s][i] in a fixed order: eight contiguous groups of slabs, each summed in ascending order
// by one thread with eight loads in flight, then added in ascending group order.  64 elements x 8 groups per block, four
// elements to a load (V = 4); 32 x 8, one by one, where their number is no multiple of four.  Bound by instruction issue with
// single loads (61 % issued).
template <typename TC, int V>
__global__ void __launch_bounds__(V == 4 ? 128 : 256)
slab_sum_kernel(const float* part, int slabs, int64_t n, TC* __restrict__ out, int cols, int rows_out, int cols_out, int ld, int c0) {
    constexpr int L = V == 4 ? 16 : 32, E = L * V;
    __shared__ float gsum[8][E];
    pdl_wait();
    const int e = (threadIdx.x % L) * V, g = threadIdx.x / L;
    const int64_t i = blockIdx.x * (int64_t)E + e;
    const int per = (slabs + 7) / 8, z0 = g * per, z1 = min(slabs, z0 + per);
    float s[V];
#pragma unroll
    for (int j = 0; j < V; ++j) s[j] = 0.f;
    if (i < n) {
        for (int z = z0; z < z1; z += 8) {
            float v[8][V];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float* const p = part + (size_t)(z + u) * n + i;
                if constexpr (V == 4) {
                    const float4 q = z + u < z1 ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
                    v[u][0] = q.x; v[u][1] = q.y; v[u][2] = q.z; v[u][3] = q.w;
                } else {
                    v[u][0] = z + u < z1 ? *p : 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int j = 0; j < V; ++j) s[j] += v[u][j];
        }
    }
#pragma unroll
    for (int j = 0; j < V; ++j) gsum[g][e + j] = s[j];
    __syncthreads();
    // the partials are [rows, cols], of which [rows_out, cols_out] exist; the result may be a block of columns (c0 ..) of a
    // matrix with rows ld apart
    const int64_t k = blockIdx.x * (int64_t)E + threadIdx.x;
    if (threadIdx.x < E && k < n) {
        const int r = (int)(k / cols), c = (int)(k % cols);
        float t = gsum[0][threadIdx.x];
#pragma unroll
        for (int q = 1; q < 8; ++q) t += gsum[q][threadIdx.x];
        if (r < rows_out && c < cols_out) out[(int64_t)r * ld + c0 + c] = from_f32<TC>(t);
    }
}

// dst[r, 0..cols) = src[r, 0..cols), rows of dst `chunks` 16-byte chunks apart: a thread per chunk.  What follows the last
// column in a row of dst is zero and never read (the tensor maps know the real width).
template <typename TE, int PER>
__global__ void __launch_bounds__(256)
pad_rows_kernel(const TE* src, int64_t rows, int cols, TE* __restrict__ dst, int chunks) {
    pdl_wait();
    const int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x;
    if (i >= rows * chunks) return;
    const int64_t r = i / chunks;
    const int c = (int)(i - r * chunks) * PER;
    union { TE e[PER]; uint4 v; } u;
#pragma unroll
    for (int k = 0; k < PER; ++k) u.e[k] = c + k < cols ? src[r * cols + c + k] : TE(0);
    *reinterpret_cast<uint4*>(dst + (r * chunks) * PER + c) = u.v;
}

template <typename TA, typename TB, typename TC>
static void launch_simt(const TA* A, int64_t sam, int64_t sak, const TB* B, int64_t sbk, int64_t sbn, TC* C,
                        int64_t Mr, int64_t Nc, int64_t Kd, int64_t k_per_slab, int slabs, int64_t slab_stride,
                        cudaStream_t st, const float* bias = nullptr, int relu = 0) {
    dim3 grid((unsigned)ceil_div(Nc, SG_TILE), (unsigned)ceil_div(Mr, SG_TILE), (unsigned)slabs);
    gemm_simt_kernel<TA, TB, TC><<<grid, 256, 0, st>>>(A, sam, sak, B, sbk, sbn, C, Mr, Nc, Kd, k_per_slab, slab_stride, bias, relu);
}

// FFMA dW: rows of X / dY per partial.  128 rows while that gives at most 148 partials (small inputs
// still spread over many blocks), otherwise 4096.
static int dw_slab_rows(int64_t N) { return N <= 148 * 128 ? 128 : 4096; }
static int dw_slabs(int64_t N) { return (int)(N > 0 ? ceil_div(N, dw_slab_rows(N)) : 1); }

bool linear_tma_supported(int64_t N, int Kc, int Mo, int b_transposed, gnn_dtype dtype);
gnn_status linear_tma_forward(const void* X, int ldx, const void* W, int ldw, int64_t N, int Kc, int Mo, int b_transposed, void* Y, int* d_flag, int reset,
                              cudaStream_t st, const float* bias, int relu);
bool linear_tma_f32_supported(int64_t N, int Kc, int Mo, gnn_dtype dtype);
gnn_status linear_tma_f32_forward(const void* X, int ldx, const void* W, int64_t N, int Kc, int Mo, int b_transposed, void* Y, int* d_flag, int reset,
                                  cudaStream_t st, const float* bias, int relu);
bool linear_tma_dw_supported(int64_t N, int K, int M, gnn_dtype dtype);
int linear_tma_dw_partials(int64_t N);
gnn_status linear_tma_dw(const void* X, int ldx, const void* dY, int ldd, int64_t N, int K, int M, float* part, int* d_flag, int reset, cudaStream_t st);
bool linear_tma_f32_dw_supported(int64_t N, int K, int M, int Mo, gnn_dtype dtype);
int linear_tma_f32_dw_partials(int64_t N);
gnn_status linear_tma_f32_dw(const void* X, int ldx, const void* dY, int ldd, int64_t N, int K, int M, int Mo, float* part, int* d_flag, int reset, cudaStream_t st);

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

// elements between rows of a matrix of `cols` columns whose rows start on 16 bytes
static int padded(int cols, int s) { return round_up(cols, 16 / s); }

// Workspace layout: status word (256 bytes), dW partials, then the padded copies of X, dY and W.  The element type is not
// known where the size is asked for: rows that would be padded in either type count, in the larger one.
// least: what a backward call needs without the copies and the rounded partials (the FFMA kernel, and shapes without either).
// It grows with K and M, so that a workspace sized for the widest layer serves the others; `bytes` does not.
struct LinearWs {
    size_t part, x, dy, w, bytes, least;
    LinearWs(int64_t N, int K, int M) {
        const size_t parts = (size_t)(dw_slabs(N) > 148 ? dw_slabs(N) : 148);  // FFMA slabs or tensor-core CTA partials
        auto copy = [](int64_t rows, int cols) -> size_t {
            if (cols % 8 == 0) return 0;
            const size_t b2 = (size_t)rows * padded(cols, 2) * 2, b4 = cols % 4 == 0 ? 0 : (size_t)rows * padded(cols, 4) * 4;
            return up256(b2 > b4 ? b2 : b4);
        };
        part = 256;
        least = part + up256(parts * K * M * 4);
        x = part + up256(parts * round_up(K, 32) * round_up(M, 32) * 4);
        dy = x + copy(N, K);
        w = dy + copy(N, M);
        bytes = w + (M % 8 == 0 ? 0 : up256((size_t)K * padded(M, 2) * 2));
    }
};

// contraction and columns that the copy engine took before others were padded for it
static bool sixteens(int Kc, int Mo, int s) { return Kc % 16 == 0 && Mo % 16 == 0 && (Kc <= 256 || Kc % 32 == 0 || s == 4); }

// rows on 16 bytes: src itself, or its copy at dst
static const void* with_padded_rows(const void* src, int64_t rows, int cols, int s, void* dst, cudaStream_t st) {
    const int ld = padded(cols, s);
    if (ld == cols) return src;
    const int chunks = ld * s / 16;
    const dim3 grid((unsigned)ceil_div(rows * chunks, 256));
    if (s == 4) launch_overlapped(pad_rows_kernel<float, 4>, grid, dim3(256), 0, st, (const float*)src, rows, cols, (float*)dst, chunks);
    else launch_overlapped(pad_rows_kernel<uint16_t, 8>, grid, dim3(256), 0, st, (const uint16_t*)src, rows, cols, (uint16_t*)dst, chunks);
    return dst;
}

}  // namespace gnn

using namespace gnn;

extern "C" {

size_t gnn_linear_workspace(int32_t N, int K, int M) {
    if (N < 0 || K <= 0 || M <= 0) return 0;
    return LinearWs(N, K, M).bytes;
}

gnn_status gnn_linear(const void* X, const void* W, int32_t N, int K, int M, gnn_dtype dtype, void* Y,
                      void* ws, size_t ws_bytes, gnn_stream stream) {
    return gnn_linear_bias_act(X, W, N, K, M, dtype, nullptr, 0, Y, ws, ws_bytes, stream);
}

gnn_status gnn_linear_bias_act(const void* X, const void* W, int32_t N, int K, int M, gnn_dtype dtype,
                               const float* bias, int relu, void* Y, void* ws, size_t ws_bytes,
                               gnn_stream stream) {
    const char* who = "gnn_linear";
    GNN_REQUIRE(N >= 0 && K > 0 && M > 0, GNN_ERR_INVALID_ARG, "%s: bad shape", who);
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    if (N == 0) return GNN_OK;
    GNN_REQUIRE(X && W && Y, GNN_ERR_INVALID_ARG, "%s: null argument", who);
    const LinearWs lw(N, K, M);
    GNN_REQUIRE(ws && ws_bytes >= 256, GNN_ERR_WORKSPACE_TOO_SMALL, "%s: workspace of %zu bytes needed", who, lw.bytes);
    cudaStream_t st = as_stream(stream);
    const int s = elem_size(dtype);
    char* w8 = (char*)ws;
    // the status word alone is enough where no rows have to be padded; where they do, a caller with that little gets the
    // kernels that need no padding
    const bool pads = K * s % 16 != 0 || (s == 2 && M * s % 16 != 0);
    // Multiples of 16 have always asked for matrices on 16 bytes (the launches below refuse others); any other size takes
    // matrices on whole elements, and the FFMA kernel if one of them is off 16 bytes.
    const bool on16 = aligned16(X) && aligned16(W) && (aligned16(Y) || M * s % 16 != 0);
    if (sixteens(K, M, s) || ((!pads || (ws_bytes >= lw.bytes && aligned16(ws))) && on16)) {
        if (linear_tma_supported(N, K, M, 0, dtype)) {
            const void* Xp = with_padded_rows(X, N, K, s, w8 + lw.x, st);
            const void* Wp = with_padded_rows(W, K, M, s, w8 + lw.w, st);
            return linear_tma_forward(Xp, padded(K, s), Wp, padded(M, s), N, K, M, 0, Y, (int*)ws, 1, st, bias, relu);
        }
        if (linear_tma_f32_supported(N, K, M, dtype)) {
            const void* Xp = with_padded_rows(X, N, K, s, w8 + lw.x, st);
            return linear_tma_f32_forward(Xp, padded(K, s), W, N, K, M, 0, Y, (int*)ws, 1, st, bias, relu);
        }
    }
    if (cudaMemsetAsync(ws, 0, sizeof(int), st) != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: memset failed (is ws a device pointer?)", who);
    if (dtype == GNN_F32) {
        launch_simt<float, float, float>((const float*)X, K, 1, (const float*)W, M, 1, (float*)Y, N, M, K, K, 1, 0, st, bias, relu);
    } else {
        launch_simt<__nv_bfloat16, __nv_bfloat16, __nv_bfloat16>((const __nv_bfloat16*)X, K, 1, (const __nv_bfloat16*)W, M, 1,
                                                               (__nv_bfloat16*)Y, N, M, K, K, 1, 0, st, bias, relu);
    }
    GNN_CHECK_LAUNCH(who);
    return GNN_OK;
}

gnn_status gnn_linear_backward(const void* X, const void* W, const void* dY, int32_t N, int K, int M,
                               gnn_dtype dtype, void* dX, void* dW, void* ws, size_t ws_bytes,
                               gnn_stream stream) {
    const char* who = "gnn_linear_backward";
    GNN_REQUIRE(N >= 0 && K > 0 && M > 0, GNN_ERR_INVALID_ARG, "%s: bad shape", who);
    GNN_REQUIRE(dtype == GNN_F32 || dtype == GNN_BF16, GNN_ERR_INVALID_ARG, "%s: bad dtype", who);
    GNN_REQUIRE(dY || N == 0, GNN_ERR_INVALID_ARG, "%s: null dY", who);
    const LinearWs lw(N, K, M);
    GNN_REQUIRE(ws && ws_bytes >= lw.least, GNN_ERR_WORKSPACE_TOO_SMALL, "%s: workspace of %zu bytes needed", who, lw.bytes);
    GNN_REQUIRE(!dX || N == 0 || W, GNN_ERR_INVALID_ARG, "%s: dX needs W", who);
    GNN_REQUIRE(!dW || N == 0 || X, GNN_ERR_INVALID_ARG, "%s: dW needs X", who);
    cudaStream_t st = as_stream(stream);
    const int s = elem_size(dtype);
    char* w8 = (char*)ws;
    int* const status = (int*)ws;
    const bool room = ws_bytes >= lw.bytes && aligned16(ws);
    // dX[n,k] = sum_m dY[n,m] * W[k,m]
    const bool dx_on16 = aligned16(dY) && aligned16(W) && (aligned16(dX) || K * s % 16 != 0);
    const bool dx_tma = dX && N > 0 && (sixteens(M, K, s) || (dx_on16 && (room || M * s % 16 == 0))) && (dtype == GNN_F32 ? linear_tma_f32_supported(N, M, K, dtype) : linear_tma_supported(N, M, K, 1, dtype));
    // dW[k,m] = sum_n X[n,k] * dY[n,m]: one fp32 partial per CTA, then summed in CTA order.  More output columns than one
    // launch takes (256, or fewer where K fills tensor memory): one launch and one ordered sum per block of columns of dY.
    auto dw_supported = [&](int mc) { return dtype == GNN_F32 ? linear_tma_f32_dw_supported(N, K, mc, M, dtype) : linear_tma_dw_supported(N, K, mc, dtype); };
    int block = 0;
    if (dW && N > 0 && ((K % 32 == 0 && M % (dtype == GNN_F32 ? 32 : 16) == 0) || (room && aligned16(X) && aligned16(dY)))) {
        if (dw_supported(M)) block = M;
        else
            for (int mc = (M < 256 ? M : 256) / 32 * 32; mc >= 32 && !block; mc -= 32)
                if (dw_supported(mc)) block = mc;
    }
    int reset = 1;  // the first pipelined launch sets the status word
    if (!dx_tma && cudaMemsetAsync(ws, 0, sizeof(int), st) != cudaSuccess)
        GNN_FAIL(GNN_ERR_CUDA, "%s: memset failed (is ws a device pointer?)", who);
    if (!dx_tma) reset = 0;
    const void* dYp = dx_tma || block ? with_padded_rows(dY, N, M, s, w8 + lw.dy, st) : dY;
    const int ldd = padded(M, s);
    if (dX && N > 0) {
        if (dx_tma) {
            gnn_status rc;
            if (dtype == GNN_F32) {
                rc = linear_tma_f32_forward(dYp, ldd, W, N, M, K, 1, dX, status, reset, st, nullptr, 0);
            } else {
                const void* Wp = with_padded_rows(W, K, M, s, w8 + lw.w, st);
                rc = linear_tma_forward(dYp, ldd, Wp, ldd, N, M, K, 1, dX, status, reset, st, nullptr, 0);
            }
            if (rc != GNN_OK) return rc;
            reset = 0;
        } else if (dtype == GNN_F32) {
            launch_simt<float, float, float>((const float*)dY, M, 1, (const float*)W, 1, M, (float*)dX, N, K, M, M, 1, 0, st);
        } else {
            launch_simt<__nv_bfloat16, __nv_bfloat16, __nv_bfloat16>((const __nv_bfloat16*)dY, M, 1, (const __nv_bfloat16*)W, 1, M,
                                                                   (__nv_bfloat16*)dX, N, K, M, M, 1, 0, st);
        }
        GNN_CHECK_LAUNCH(who);
    }
    if (dW) {
        float* part = (float*)(w8 + lw.part);
        auto sum = [&](int slabs, int rows, int cols, int cols_out, int c0) {
            const int64_t n = (int64_t)rows * cols;
            auto run = [&](auto kernel, auto* to, int elements, int threads) {
                launch_overlapped(kernel, dim3((unsigned)ceil_div(n, (int64_t)elements)), dim3(threads), 0, st, part, slabs, n, to, cols, K, cols_out, M, c0);
            };
            // (148 partials of 16 Ki elements: 4.9 us one by one, 7.2 us by four, in too few blocks; of 64 Ki: 10.6 and 7.7 us.  With the product before
            // it, 170k rows bf16, one by one / by four: 16 Ki 22.6 / 24.7, 25 Ki 28.9 / 30.9, 36 Ki 34.5 / 35.1, 42 Ki 37.0 / 37.0, 49 Ki 39.3 / 38.9, 64 Ki 46.5 / 45.1)
            const bool four = n >= 48 * 1024 && n % 4 == 0 && aligned16(part);
            if (dtype == GNN_F32) four ? run(slab_sum_kernel<float, 4>, (float*)dW, 64, 128) : run(slab_sum_kernel<float, 1>, (float*)dW, 32, 256);
            else four ? run(slab_sum_kernel<__nv_bfloat16, 4>, (__nv_bfloat16*)dW, 64, 128) : run(slab_sum_kernel<__nv_bfloat16, 1>, (__nv_bfloat16*)dW, 32, 256);
        };
        if (block) {
            const void* Xp = with_padded_rows(X, N, K, s, w8 + lw.x, st);
            for (int c0 = 0; c0 < M; c0 += block) {
                const int mc = M - c0 < block ? M - c0 : block;
                const void* dYb = (const char*)dYp + (size_t)c0 * s;
                gnn_status rc = dtype == GNN_F32 ? linear_tma_f32_dw(Xp, padded(K, s), dYb, ldd, N, K, mc, M, part, status, reset, st)
                                                 : linear_tma_dw(Xp, padded(K, s), dYb, ldd, N, K, mc, part, status, reset, st);
                if (rc != GNN_OK) return rc;
                reset = 0;
                sum(dtype == GNN_F32 ? linear_tma_f32_dw_partials(N) : linear_tma_dw_partials(N), round_up(K, 32), round_up(mc, dtype == GNN_F32 ? 32 : 16), mc, c0);
                GNN_CHECK_LAUNCH(who);
            }
            return GNN_OK;
        }
        const int slabs = dw_slabs(N);
        const int64_t km = (int64_t)K * M;
        if (N == 0) {
            if (cudaMemsetAsync(part, 0, (size_t)km * 4, st) != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: memset failed", who);
        } else if (dtype == GNN_F32) {
            launch_simt<float, float, float>((const float*)X, 1, K, (const float*)dY, M, 1, part, K, M, N, dw_slab_rows(N), slabs, km, st);
        } else {
            launch_simt<__nv_bfloat16, __nv_bfloat16, float>((const __nv_bfloat16*)X, 1, K, (const __nv_bfloat16*)dY, M, 1, part, K, M, N,
                                                           dw_slab_rows(N), slabs, km, st);
        }
        sum(slabs, K, M, M, 0);
        GNN_CHECK_LAUNCH(who);
    }
    return GNN_OK;
}

}  // extern "C"
