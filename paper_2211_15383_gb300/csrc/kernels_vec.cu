// Multi-RHS vector kernels: Z2 noise, BLAS1 with per-rhs coefficients and
// deterministic per-rhs reductions.  Layout [row][rhs]; block (32 rhs, 8 rows);
// grid (rhs tiles, row groups) with a grid-stride loop over rows.  Arithmetic
// runs in the vector's own precision (FP32 vectors stay on the FP32 pipe);
// only the cross-block partial sums are FP64.
#include "kernels.cuh"

namespace mg {

__device__ __forceinline__ uint64_t sm64(uint64_t z) {
    // One splitmix64 step (Steele, Lea & Flood 2014): add the golden gamma, then mix.
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

template <typename C>
__global__ void k_noise(C* __restrict__ x, long long n, int N, uint64_t seed, uint64_t term, int64_t first) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    const uint64_t ks = sm64(sm64(seed ^ term) ^ (uint64_t)(first + j));
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n;
         i += (long long)gridDim.y * kRowLanes) {
        const uint64_t h = sm64(ks ^ (uint64_t)i);
        C v;
        v.x = (h & 1ull) ? -1 : 1;
        v.y = 0;
        x[i * N + j] = v;
    }
}

template <typename C>
__global__ void k_probes(C* __restrict__ x, const int8_t* __restrict__ p, long long n, int N) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n;
         i += (long long)gridDim.y * kRowLanes) {
        C v;
        v.x = p[(long long)j * n + i];
        v.y = 0;
        x[i * N + j] = v;
    }
}

template <typename Cout, typename Cin>
__global__ void k_convert(Cout* __restrict__ y, const Cin* __restrict__ x, long long count) {
    if (grid_dependency()) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x)
        y[i] = cvtc(x[i], Cout());
}

// Exponent e of a column's largest entry (in [2^(e-1), 2^e)); 0 for a zero or non-finite one.
__device__ __forceinline__ int unit_exponent(unsigned long long mx) {
    const int E = (int)(mx >> 52);
    return (mx == 0 || E == 0x7ff) ? 0 : E - 1022;
}
__global__ void k_to_unit(float2* __restrict__ y, const double2* __restrict__ x, const unsigned long long* __restrict__ mx,
                          long long n, int N) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    const int e = unit_exponent(mx[j]);
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n; i += (long long)gridDim.y * kRowLanes) {
        const double2 v = x[i * N + j];
        y[i * N + j] = make_float2((float)ldexp(v.x, -e), (float)ldexp(v.y, -e));
    }
}
__global__ void k_from_unit(double2* __restrict__ y, const float2* __restrict__ x,
                            const unsigned long long* __restrict__ mx, long long n, int N) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    const int e = unit_exponent(mx[j]);
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n; i += (long long)gridDim.y * kRowLanes) {
        const float2 v = x[i * N + j];
        y[i * N + j] = make_double2(ldexp((double)v.x, e), ldexp((double)v.y, e));
    }
}

template <typename C>
__global__ void k_zero(C* __restrict__ x, long long count) {
    if (grid_dependency()) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x)
        x[i] = czero<C>();
}

template <typename Cy, typename Cx_>
__global__ void k_scale_rhs(Cy* __restrict__ y, const Cx_* __restrict__ x, const double* __restrict__ scale,
                            bool invert, long long n, int N) {
    if (grid_dependency()) return;
    using R = re_t<Cy>;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    double sc = scale[j];
    if (invert) sc = (sc != 0.0) ? 1.0 / sc : 0.0;
    const R s = (R)sc;
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n;
         i += (long long)gridDim.y * kRowLanes) {
        Cy v = cvtc(x[i * N + j], Cy());
        y[i * N + j] = mk(v.x * s, v.y * s);
    }
}

template <typename Cy, typename Cx_>
__global__ void k_axpy_rhs(Cy* __restrict__ y, const double2* __restrict__ alpha, const double* __restrict__ beta,
                           double sign, const Cx_* __restrict__ x, long long n, int N) {
    if (grid_dependency()) return;
    using R = re_t<Cy>;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    double2 a = alpha ? alpha[j] : make_double2(1.0, 0.0);
    const double b = (beta ? beta[j] : 1.0) * sign;
    const Cy ar = mk((R)(a.x * b), (R)(a.y * b));
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n;
         i += (long long)gridDim.y * kRowLanes) {
        Cy acc = y[i * N + j];
        cfma(acc, ar, cvtc(x[i * N + j], Cy()));
        y[i * N + j] = acc;
    }
}

// ---------------------------------------------------------------- reductions
template <typename Cx_, typename Cy>
__global__ void k_dot(double2* __restrict__ part, const Cx_* __restrict__ x, const Cy* __restrict__ y,
                      long long n, int N) {
    if (grid_dependency()) return;
    using R = re_t<Cx_>;
    __shared__ double2 sh[kRowLanes][kRhsTile + 1];
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    using Ca = cx_t<R>;
    Ca acc = czero<Ca>();
    if (j < N)
        for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < n;
             i += (long long)gridDim.y * kRowLanes)
            cfmac(acc, x[i * N + j], cvtc(y[i * N + j], Ca()));
    sh[threadIdx.y][threadIdx.x] = to_d(acc);
    __syncthreads();
    if (threadIdx.y == 0 && j < N) {
        double2 s = sh[0][threadIdx.x];
        for (int r = 1; r < kRowLanes; ++r) s = cadd(s, sh[r][threadIdx.x]);
        part[(long long)blockIdx.y * N + j] = s;
    }
}

// Partials reduction: block (8 outputs, 32 group lanes); lane ty adds groups
// ty, ty+32, ... in order, then a fixed-order sum over the 32 lanes, so the result
// does not depend on timing (deterministic).  Few outputs per block: an SM does two FP64
// additions per clock, so a sum of many partials is spread over many SMs (32 outputs a
// block: 10 us for 608 groups).
__global__ void __launch_bounds__(256) k_finalize(double2* __restrict__ out, const double2* __restrict__ part,
                                                  int groups, int count) {
    if (grid_dependency()) return;
    __shared__ double2 sh[32][9];
    const int j = blockIdx.x * 8 + threadIdx.x;
    double2 acc = make_double2(0.0, 0.0);
    if (j < count) {
#pragma unroll 8
        for (int g = threadIdx.y; g < groups; g += 32) acc = cadd(acc, part[(long long)g * count + j]);
    }
    sh[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && j < count) {
        double2 s = sh[0][threadIdx.x];
        for (int r = 1; r < 32; ++r) s = cadd(s, sh[r][threadIdx.x]);
        out[j] = s;
    }
}

// ------------------------------------------------------------------ launchers
static inline dim3 blk() { return dim3(kRhsTile, kRowLanes); }

template <typename C>
void launch_noise(C* x, long long n, int N, uint64_t seed, uint64_t term, int64_t first, cudaStream_t s) {
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(n, N)), blk(), 0, s, (k_noise<C>), x, n, N, seed, term, first);
    MG_LAUNCHED();
}
template <typename C>
void launch_probes(C* x, const int8_t* p, long long n, int N, cudaStream_t s) {
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(n, N)), blk(), 0, s, (k_probes<C>), x, p, n, N);
    MG_LAUNCHED();
}
template <typename Cout, typename Cin>
void launch_convert(Cout* y, const Cin* x, long long count, cudaStream_t s) {
    if (count <= 0) return;
    long long b = (count + 255) / 256;
    if (b > kNumSM * 16) b = kNumSM * 16;
    MG_LAUNCH((int)b, 256, 0, s, (k_convert<Cout, Cin>), y, x, count);
    MG_LAUNCHED();
}
void launch_to_unit(float2* y, const double2* x, const unsigned long long* mx, long long n, int N, cudaStream_t s) {
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(n, N)), blk(), 0, s, k_to_unit, y, x, mx, n, N);
    MG_LAUNCHED();
}
void launch_from_unit(double2* y, const float2* x, const unsigned long long* mx, long long n, int N, cudaStream_t s) {
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(n, N)), blk(), 0, s, k_from_unit, y, x, mx, n, N);
    MG_LAUNCHED();
}
template <typename C>
void launch_zero(C* x, long long count, cudaStream_t s) {
    if (count <= 0) return;
    long long b = (count + 255) / 256;
    if (b > kNumSM * 16) b = kNumSM * 16;
    MG_LAUNCH((int)b, 256, 0, s, (k_zero<C>), x, count);
    MG_LAUNCHED();
}
template <typename Cy, typename Cx_>
void launch_scale_rhs(Cy* y, const Cx_* x, const double* scale, bool invert, long long n, int N, cudaStream_t s) {
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(n, N)), blk(), 0, s, (k_scale_rhs<Cy, Cx_>), y, x, scale, invert, n, N);
    MG_LAUNCHED();
}
template <typename Cy, typename Cx_>
void launch_axpy_rhs(Cy* y, const double2* alpha, const double* beta, double sign, const Cx_* x, long long n, int N,
                     cudaStream_t s) {
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(n, N)), blk(), 0, s, (k_axpy_rhs<Cy, Cx_>), y, alpha, beta, sign, x, n, N);
    MG_LAUNCHED();
}

int reduce_groups(long long n, int N) { return row_groups(n, N, 4); }
// The minimal-residual coefficient of every rhs from the row-major partials of its two
// dots (part[i * groups + g]): alpha_j = <y, x>_j / <y, y>_j (0 where <y, y> is 0).  One block
// per rhs, fixed order; FP32 dots are added as pairs, since FP64 adds run at 1/64 of the FP32
// rate (8 rhs of a 64^2 lattice: 4.0 -> 2.7 us; the stencil before it 4.4 -> 3.3).  The quotient
// is taken here, once per rhs: a division in the prologue of every thread of the update kernels
// was most of those kernels' time on small blocks (15 us for 4 MB, 8192 rows x 16 rhs).
template <typename C>
__global__ void __launch_bounds__(128) k_finalize_alpha(C* __restrict__ alpha, const double2* __restrict__ part,
                                                        int groups, int N) {
    if (grid_dependency()) return;
    using S = sum_t<C>;
    __shared__ double2 sh[3][4];                       // 16-byte slots, S in each
    const int j = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const CSum<C>* r0 = reinterpret_cast<const CSum<C>*>(part) + (long long)j * groups;
    const CSum<C>* r1 = reinterpret_cast<const CSum<C>*>(part) + (long long)(N + j) * groups;
    constexpr int U = sizeof(C) == 8 ? 4 : 1;
    S v[3];
#pragma unroll 4
    for (int g0 = threadIdx.x; g0 < groups; g0 += U * 128) {
        CSum<C> a[U];
        S b[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (g0 + 128 * u < groups) {
                a[u] = r0[g0 + 128 * u];
                b[u] = r1[g0 + 128 * u].re;
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (g0 + 128 * u < groups) {
                v[0].add(a[u].re);
                v[1].add(a[u].im);
                v[2].add(b[u]);
            }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        warp_sum(v[q]);
        if (lane == 0) *reinterpret_cast<S*>(&sh[q][wid]) = v[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            S s = *reinterpret_cast<const S*>(&sh[q][0]);
#pragma unroll
            for (int w = 1; w < 4; ++w) s.add(*reinterpret_cast<const S*>(&sh[q][w]));
            t[q] = s.value();
        }
        double ib = t[2] > 0.0 ? 1.0 / t[2] : 0.0;
        if (sizeof(C) == 16 && t[2] > 0.0 && t[2] < 0x1p-1022) {
            // FP64 vectors of norm 2^-511 and below: 1 / t overflows
            t[0] *= 0x1p100;
            t[1] *= 0x1p100;
            ib = 1.0 / (t[2] * 0x1p100);
        }
        alpha[j] = cvt<C>(make_double2(t[0] * ib, t[1] * ib));
    }
}

template <typename C>
void launch_finalize_alpha(C* alpha, const double2* part, int groups, int N, cudaStream_t s) {
    MG_LAUNCH(N, 128, 0, s, (k_finalize_alpha<C>), alpha, part, groups, N);
    MG_LAUNCHED();
}
template void launch_finalize_alpha<double2>(double2*, const double2*, int, int, cudaStream_t);
template void launch_finalize_alpha<float2>(float2*, const double2*, int, int, cudaStream_t);

void launch_finalize(double2* out, const double2* part, int groups, int count, cudaStream_t s) {
    MG_LAUNCH((count + 7) / 8, dim3(8, 32), 0, s, k_finalize, out, part, groups, count);
    MG_LAUNCHED();
}

template <typename Cx_, typename Cy>
void launch_dot(double2* out, const Cx_* x, const Cy* y, long long n, int N, double2* part, cudaStream_t s) {
    const int G = reduce_groups(n, N);
    MG_LAUNCH(dim3(rhs_tiles(N), G), blk(), 0, s, (k_dot<Cx_, Cy>), part, x, y, n, N);
    MG_LAUNCHED();
    launch_finalize(out, part, G, N, s);
}
#define INST_C(C)                                                                                   \
    template void launch_noise<C>(C*, long long, int, uint64_t, uint64_t, int64_t, cudaStream_t);    \
    template void launch_probes<C>(C*, const int8_t*, long long, int, cudaStream_t);                 \
    template void launch_zero<C>(C*, long long, cudaStream_t);
INST_C(double2)
INST_C(float2)
#define INST_CC(A, B)                                                                               \
    template void launch_convert<A, B>(A*, const B*, long long, cudaStream_t);                       \
    template void launch_scale_rhs<A, B>(A*, const B*, const double*, bool, long long, int,          \
                                         cudaStream_t);                                              \
    template void launch_axpy_rhs<A, B>(A*, const double2*, const double*, double, const B*,         \
                                        long long, int, cudaStream_t);
INST_CC(double2, double2)
INST_CC(float2, float2)
INST_CC(double2, float2)
INST_CC(float2, double2)
template void launch_dot<double2, double2>(double2*, const double2*, const double2*, long long, int, double2*,
                                           cudaStream_t);
template void launch_dot<float2, float2>(double2*, const float2*, const float2*, long long, int, double2*,
                                         cudaStream_t);

}  // namespace mg

namespace mg {
// out[c][r] = in[r][c] for a rows x cols complex matrix (32 x 32 tiles).
__global__ void k_transpose(double2* __restrict__ out, const double2* __restrict__ in, long long rows, int cols) {
    if (grid_dependency()) return;
    __shared__ double2 t[32][33];
    const int c0 = blockIdx.x * 32;
    const long long nrb = (rows + 31) / 32;
    for (long long rb = blockIdx.y; rb < nrb; rb += gridDim.y) {      // grid-stride over 32-row blocks
        const long long r0 = rb * 32;
        __syncthreads();
        for (int k = threadIdx.y; k < 32; k += blockDim.y) {
            const long long r = r0 + k;
            const int cc = c0 + threadIdx.x;
            if (r < rows && cc < cols) t[k][threadIdx.x] = in[r * cols + cc];
        }
        __syncthreads();
        for (int k = threadIdx.y; k < 32; k += blockDim.y) {
            const int cc = c0 + k;
            const long long r = r0 + threadIdx.x;
            if (r < rows && cc < cols) out[(long long)cc * rows + r] = t[threadIdx.x][k];
        }
    }
}
void launch_transpose(double2* out, const double2* in, long long rows, int cols, cudaStream_t s) {
    const long long nrb = (rows + 31) / 32;
    dim3 g((cols + 31) / 32, (unsigned)(nrb < 65535 ? nrb : 65535));
    MG_LAUNCH(g, dim3(32, 8), 0, s, k_transpose, out, in, rows, cols);
    MG_LAUNCHED();
}
}  // namespace mg
