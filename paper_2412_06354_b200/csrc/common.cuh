// Shared host/device helpers of libgnn_b200 (sm_100a only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "gnn.h"

#if defined(__CUDA_ARCH__) && (__CUDA_ARCH__ < 1000)
#error "libgnn_b200 is written for sm_100a"
#endif

namespace gnn {

void set_error(const char* fmt, ...);

#define GNN_FAIL(code, ...)            \
    do {                               \
        ::gnn::set_error(__VA_ARGS__); \
        return (code);                 \
    } while (0)

#define GNN_REQUIRE(cond, code, ...)              \
    do {                                          \
        if (!(cond)) GNN_FAIL(code, __VA_ARGS__); \
    } while (0)

// after a launch: report launch-configuration errors without synchronising
#define GNN_CHECK_LAUNCH(name)                                                                 \
    do {                                                                                       \
        cudaError_t e_ = cudaGetLastError();                                                   \
        if (e_ != cudaSuccess) GNN_FAIL(GNN_ERR_CUDA, "%s: %s", name, cudaGetErrorString(e_)); \
    } while (0)

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline cudaStream_t as_stream(gnn_stream s) { return reinterpret_cast<cudaStream_t>(s); }
static inline int elem_size(gnn_dtype d) { return d == GNN_F32 ? 4 : 2; }
static inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
static inline size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
// grid for a grid-stride loop over n items
static inline int grid_for(int64_t n, int threads) {
    int64_t b = ceil_div(n > 0 ? n : 1, threads);
    int64_t cap = 148 * 32;
    return (int)(b < cap ? b : cap);
}

#ifdef __CUDACC__
// ---------------------------------------------------------------- launches
// Launch whose blocks may be set up while the kernel before it in the stream drains (and, as every kernel lets its successor
// come up before it waits itself, while the one before that does).  The kernel's first statement is pdl_wait(): nothing of it
// touches global memory before all earlier work of the stream is complete and visible, so the order of the stream is kept;
// what overlaps is the launch latency (about 1 us of a 3-5 us kernel on a small graph).
// What griddepcontrol.wait makes visible are ordinary (coherent) loads.  Such a kernel is resident while what it reads is being
// written, so that the condition of the non-coherent path, data that is read-only as long as the kernel lives, does not hold:
// no ld.global.nc and no __ldg in it, and no __restrict__ on a pointer to const, from which the compiler would make them.
// (Outputs may be __restrict__: then loads can move ahead of stores.)  tests/test_overlapped_launches.py looks at the sources.
template <class... Params, class... Args>
static inline void launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);  // errors: GNN_CHECK_LAUNCH of the caller
}

// ---------------------------------------------------------------- device helpers
// every thread of a kernel started by launch_overlapped, before its first access to global memory
__device__ __forceinline__ void pdl_wait_exclusive() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// ... and in kernels that leave room on an SM (the persistent dense kernels take all of its shared memory): the next kernel
// of the stream may be set up from here on.
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    pdl_wait_exclusive();
}

// 16-byte global loads/stores with L2 cache policies (createpolicy + .L2::cache_hint).
//   feature rows that are gathered many times: keep in L2 (evict_last)
//   index / weight / output streams touched once: evict_first, no L1 allocation
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint4 ld_hint16(const void* p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
// VB 16-byte chunks, by one load: 16 or 32 bytes, aligned to their size
template <int VB> struct Vec16 { uint4 v[VB]; };
__device__ __forceinline__ void ld_hint(Vec16<1>& x, const void* p, uint64_t pol) { x.v[0] = ld_hint16(p, pol); }
__device__ __forceinline__ void ld_hint(Vec16<2>& x, const void* p, uint64_t pol) {
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
                 : "=r"(x.v[0].x), "=r"(x.v[0].y), "=r"(x.v[0].z), "=r"(x.v[0].w), "=r"(x.v[1].x), "=r"(x.v[1].y), "=r"(x.v[1].z), "=r"(x.v[1].w)
                 : "l"(p), "l"(pol));
}
__device__ __forceinline__ int ld_hint_i32(const int* p, uint64_t pol) {
    int v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ int ld_stream_i32(const int* p) {
    int v;
    asm volatile("ld.global.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_stream_f32(const float* p) {
    float v;
    asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
// coherent loads whose place among the other loads and stores in flight is kept
__device__ __forceinline__ uint4 ld_16(const void* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ int4 ld_int4(const int4* p) {
    const uint4 v = ld_16(p);
    return make_int4((int)v.x, (int)v.y, (int)v.z, (int)v.w);
}
__device__ __forceinline__ float ld_f32(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream16(void* p, uint4 v) {
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w)
                 : "memory");
}

// One 16-byte chunk of a feature row as fp32 lanes: 4 values for f32, 8 for bf16.
template <typename T>
struct Chunk;
template <>
struct Chunk<float> {
    static constexpr int N = 4;
    __device__ __forceinline__ static void unpack(uint4 u, float* f) {
        f[0] = __uint_as_float(u.x);
        f[1] = __uint_as_float(u.y);
        f[2] = __uint_as_float(u.z);
        f[3] = __uint_as_float(u.w);
    }
    __device__ __forceinline__ static uint4 pack(const float* f) {
        return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]),
                          __float_as_uint(f[3]));
    }
};
template <>
struct Chunk<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ __forceinline__ static void unpack(uint4 u, float* f) {
        // bf16 -> f32 is a 16-bit shift: exact
        f[0] = __uint_as_float(u.x << 16);
        f[1] = __uint_as_float(u.x & 0xFFFF0000u);
        f[2] = __uint_as_float(u.y << 16);
        f[3] = __uint_as_float(u.y & 0xFFFF0000u);
        f[4] = __uint_as_float(u.z << 16);
        f[5] = __uint_as_float(u.z & 0xFFFF0000u);
        f[6] = __uint_as_float(u.w << 16);
        f[7] = __uint_as_float(u.w & 0xFFFF0000u);
    }
    __device__ __forceinline__ static uint32_t pack2(float lo, float hi) {
        __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);  // round to nearest even
        return *reinterpret_cast<uint32_t*>(&b);
    }
    __device__ __forceinline__ static uint4 pack(const float* f) {
        return make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]),
                          pack2(f[6], f[7]));
    }
};

// first index r in [0, n] with a[r] >= v  (a non-decreasing, n entries)
__device__ __forceinline__ int lower_bound_i64(const int64_t* a, int n, int64_t v) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

#endif  // __CUDACC__
}  // namespace gnn
