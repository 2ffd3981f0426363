// Shared helpers of the CUDA path: error handling, complex arithmetic on
// float2/double2, launch geometry.  Part of the product library; independent
// of the CPU oracle.
#pragma once

#include <atomic>

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <stdexcept>
#include <string>

#include "mgmlmc.h"

namespace mg {

struct Error : std::runtime_error {
    int code;
    Error(int c, const std::string& m) : std::runtime_error(m), code(c) {}
};

#define MG_CUDA(call)                                                                  \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            throw ::mg::Error(MGMLMC_ECUDA, std::string(#call) + ": " +                 \
                                                cudaGetErrorString(e_));               \
    } while (0)

// Kernel launches issued by this library (process-wide), for launch accounting.
std::atomic<long long>& launch_counter();   // all contexts, thread-safe

#define MG_LAUNCHED()                                                                  \
    do {                                                                               \
        ++::mg::launch_counter();                                                      \
        cudaError_t e_ = cudaGetLastError();                                           \
        if (e_ != cudaSuccess)                                                         \
            throw ::mg::Error(MGMLMC_ECUDA, std::string("kernel launch in ") +         \
                                                __func__ + ": " + cudaGetErrorString(e_)); \
    } while (0)

#define MG_REQUIRE(cond, code, msg)                                                    \
    do {                                                                               \
        if (!(cond)) throw ::mg::Error((code), (msg));                                  \
    } while (0)

// ---- programmatic dependent launch
// Kernels of the solver's chain are launched so that a kernel is set up while the one before
// it in the stream still runs: without it each launch starts about 2 us after the end of its
// predecessor, as long as many of these kernels run.  Every kernel launched by MG_LAUNCH begins
// with `if (grid_dependency()) return;`: it waits until the kernels before it have completed
// and their writes are visible, so a chain orders as plain launches do.  No kernel lets its
// successor's CTAs in early (griddepcontrol.launch_dependents): they took the places of the
// CTAs that finished first, which left the grids sized to one even wave unevenly spread
// (512^2 step: 273 ms with it, 263 without dependent launches, 252 as it is; pilot draw at
// 64^2: 8.6, 12.0, 8.1).  The result is always false; the branch on it keeps the compiler from
// moving reads through const __restrict__ pointers, which it takes for invariant, above the
// wait.
__device__ __forceinline__ bool grid_dependency() {
    int z;
    asm volatile("griddepcontrol.wait;\n mov.u32 %0, 0;" : "=r"(z)::"memory");
    return z != 0;
}

template <typename... P, typename... A>
inline void launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    MG_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
}
// MG_LAUNCH(grid, block, smem, stream, (kernel<...>), args...)
#define MG_LAUNCH(g, b, sm, s, k, ...) ::mg::launch_dependent(k, g, b, sm, s, __VA_ARGS__)

// ---- complex type per real type --------------------------------------------------
template <typename R> struct Cx;
template <> struct Cx<double> { using T = double2; };
template <> struct Cx<float> { using T = float2; };
template <typename R> using cx_t = typename Cx<R>::T;
template <typename C> struct Re;
template <> struct Re<double2> { using T = double; };
template <> struct Re<float2> { using T = float; };
template <typename C> using re_t = typename Re<C>::T;

__host__ __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__host__ __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
template <typename C> __host__ __device__ __forceinline__ C czero();
template <> __host__ __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <> __host__ __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }

template <typename C> __host__ __device__ __forceinline__ C cadd(C a, C b) { return mk(a.x + b.x, a.y + b.y); }
template <typename C> __host__ __device__ __forceinline__ C csub(C a, C b) { return mk(a.x - b.x, a.y - b.y); }
// a * b
template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
    return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cmulc(C a, C b) {
    return mk(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
// acc += a * b
template <typename C> __host__ __device__ __forceinline__ void cfma(C& acc, C a, C b) {
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}
// acc += conj(a) * b
template <typename C> __host__ __device__ __forceinline__ void cfmac(C& acc, C a, C b) {
    acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(-a.y, b.x, acc.y));
}
template <typename C> __host__ __device__ __forceinline__ C cscale(C a, decltype(a.x) s) { return mk(a.x * s, a.y * s); }
// i * a
template <typename C> __host__ __device__ __forceinline__ C ctimesi(C a) { return mk(-a.y, a.x); }

__host__ __device__ __forceinline__ double2 to_d(float2 a) { return make_double2(a.x, a.y); }
__host__ __device__ __forceinline__ double2 to_d(double2 a) { return a; }

// ---- sums across threads: FP32 values as pairs, FP64 values plainly
struct PairF {
    float h = 0.f, l = 0.f;
    __host__ __device__ __forceinline__ void add(float v) {
        const float s = h + v, b = s - h;
        l += (h - (s - b)) + (v - b);
        h = s;
    }
    __host__ __device__ __forceinline__ void add(const PairF& o) {
        add(o.h);
        l += o.l;
    }
    __host__ __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};
struct SumD {
    double v = 0.0;
    __host__ __device__ __forceinline__ void add(double a) { v += a; }
    __host__ __device__ __forceinline__ void add(const SumD& o) { v += o.v; }
    __host__ __device__ __forceinline__ double value() const { return v; }
};
template <typename R> struct SumOf;
template <> struct SumOf<float> { using T = PairF; };
template <> struct SumOf<double> { using T = SumD; };
template <typename C> using sum_t = typename SumOf<re_t<C>>::T;

// Squares of V rhs over the rows of a thread.  FP32: plain accumulators, folded into the sums every
// kRowsPerSum rows, so that their error does not grow with the rows that a grid leaves a thread
// (a thread of a 2097152 x 128 block has 862).
constexpr int kRowsPerSum = 64;
template <typename R, int V> struct SquareSums {
    typename SumOf<R>::T total[V];
    R part[V] = {};
    int rows = 0;
    __host__ __device__ __forceinline__ void add(int q, R x, R y) { part[q] = fma(x, x, fma(y, y, part[q])); }
    __host__ __device__ __forceinline__ void end_row() {
        if (sizeof(R) == 4 && ++rows >= kRowsPerSum) fold();
    }
    __host__ __device__ __forceinline__ void fold() {
#pragma unroll
        for (int q = 0; q < V; ++q) {
            total[q].add(part[q]);
            part[q] = 0;
        }
        rows = 0;
    }
};
template <typename C> struct alignas(16) CSum { sum_t<C> re, im; };   // 16 B in both precisions
static_assert(sizeof(CSum<float2>) == 16 && sizeof(CSum<double2>) == 16, "partials are 16 bytes");

__device__ __forceinline__ void warp_sum(PairF& v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        PairF w;
        w.h = __shfl_down_sync(0xffffffffu, v.h, o);
        w.l = __shfl_down_sync(0xffffffffu, v.l, o);
        v.add(w);
    }
}
__device__ __forceinline__ void warp_sum(SumD& v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v.v += __shfl_down_sync(0xffffffffu, v.v, o);
}

// A thread's share of a stencil's dots as a partial of 16 bytes (FP32: CSum's layout), and
// their sums: FP64 adds and conversions run at 1/64 of the FP32 rate, and one CTA's epilogue
// of them took longer than its sites where the lattice is small.
__device__ __forceinline__ float4 dot_part(float2 v) { return make_float4(v.x, 0.f, v.y, 0.f); }
__device__ __forceinline__ double2 dot_part(double2 v) { return v; }
__device__ __forceinline__ float4 dot_part(float v) { return make_float4(v, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 dot_part(double v) { return make_double2(v, 0.0); }
__device__ __forceinline__ float4 dot_add(float4 a, float4 b) {
    PairF x{a.x, a.y}, y{a.z, a.w};
    x.add(PairF{b.x, b.y});
    y.add(PairF{b.z, b.w});
    return make_float4(x.h, x.l, y.h, y.l);
}
__device__ __forceinline__ double2 dot_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
template <typename C> using dot_t = decltype(dot_part(C()));
template <typename C> __device__ __forceinline__ dot_t<C>* dot_parts(double2* part) {
    return reinterpret_cast<dot_t<C>*>(part);
}
template <typename C> __host__ __device__ __forceinline__ C cvt(double2 a);
template <> __host__ __device__ __forceinline__ double2 cvt<double2>(double2 a) { return a; }
template <> __host__ __device__ __forceinline__ float2 cvt<float2>(double2 a) { return make_float2((float)a.x, (float)a.y); }
__host__ __device__ __forceinline__ float2 cvtc(float2 a, float2) { return a; }
__host__ __device__ __forceinline__ float2 cvtc(double2 a, float2) { return make_float2((float)a.x, (float)a.y); }
__host__ __device__ __forceinline__ double2 cvtc(float2 a, double2) { return make_double2(a.x, a.y); }
__host__ __device__ __forceinline__ double2 cvtc(double2 a, double2) { return a; }
template <typename C> __device__ __forceinline__ C from_d(double2 a);
template <> __device__ __forceinline__ double2 from_d<double2>(double2 a) { return a; }
template <> __device__ __forceinline__ float2 from_d<float2>(double2 a) { return make_float2((float)a.x, (float)a.y); }

// ---- launch geometry ---------------------------------------------------------------
constexpr int kNumSM = 152;          // GB300: 2 dies x 76 SMs
constexpr int kRhsTile = 32;         // right-hand sides per warp (threadIdx.x)
constexpr int kRowLanes = 8;         // rows per block (threadIdx.y)

inline int rhs_tiles(int N) { return (N + kRhsTile - 1) / kRhsTile; }
// Number of row groups for grid-stride kernels: about 4 resident blocks per SM.
inline int row_groups(long long rows, int N, int per_sm = 4) {
    long long want = (long long)kNumSM * per_sm / rhs_tiles(N);
    if (want < 1) want = 1;
    long long need = (rows + kRowLanes - 1) / kRowLanes;
    return (int)(need < want ? need : want);
}

}  // namespace mg
