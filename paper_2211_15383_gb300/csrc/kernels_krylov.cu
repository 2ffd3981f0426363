// Kernels of the multi-RHS flexible GMRES and of the refinement loop around it: block dot
// products, block updates, norms, their reductions, and the per-rhs bookkeeping (Givens
// rotations, triangular solve).  Layout [row][rhs].
//
// Two things bound these on small blocks, and shape them:
//  * FP64 arithmetic: an SM does 2 FP64 operations per clock, so summing partials, divisions
//    and square roots in every thread or on a single SM costs more than the memory traffic
//    (a sum of 608 x 32 FP64 partials on one SM takes 10 us).  FP32 accumulators are therefore
//    added across threads and blocks as unevaluated pairs of FP32 numbers (two-sum, about
//    2^-48, on the FP32 pipe); the FP64 result is formed once.  Reductions are spread over as
//    many SMs as they have outputs, and every coefficient is formed once, by the reduction
//    that has its sum, not in the prologue of the kernels that use it;
//  * launches: about 2 us each between dependent kernels.  Reductions write what the next
//    kernels read (scaled Hessenberg entries, update coefficients, range checks, the
//    convergence ratio), and the rotations of several columns are taken in one launch when
//    the residual estimate is looked at.
// All sums have a fixed order: results do not depend on timing.
#include <algorithm>

#include "kernels.cuh"

namespace mg {
namespace kr {

using u64 = unsigned long long;

template <typename C, int V> struct alignas(sizeof(C) * V) Vec { C v[V]; };

// A block is bx x by threads: bx (a power of two, at most 32) covers the N / V columns, by
// rows; narrow blocks keep every lane busy.
struct Shape2 {
    dim3 g, b;
};
static Shape2 shape(int N, int V, int groups) {
    const int cols = (N + V - 1) / V;
    int bx = 1;
    while (bx < cols && bx < 32) bx *= 2;
    return {dim3((cols + bx - 1) / bx, groups), dim3(bx, 256 / bx)};
}
static int groups_of(long long n, int N, int V, int per_sm) {
    const int cols = (N + V - 1) / V;
    int bx = 1;
    while (bx < cols && bx < 32) bx *= 2;
    const int by = 256 / bx, gx = (cols + bx - 1) / bx;
    const long long need = (n + by - 1) / by;
    return (int)std::max(1LL, std::min(need, (long long)per_sm * kNumSM / gx));
}
// FP32 blocks of even width: two rhs per thread (16-byte accesses).
template <typename C> static int width(int N) { return sizeof(C) == 8 && N % 2 == 0 ? 2 : 1; }

// Sums acc over the block's rows; the threads with threadIdx.y == 0 get the total.
template <typename S>
__device__ __forceinline__ S block_rows_sum(S acc, S* sh) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    sh[tid] = acc;
    __syncthreads();
    if (threadIdx.y == 0)
        for (int r = 1; r < (int)blockDim.y; ++r) acc.add(sh[r * blockDim.x + threadIdx.x]);
    __syncthreads();
    return acc;
}

// ---- <V_k, w> for k < m: partials [group][k][N] of mt vectors in all.  w is read once; the
// vectors of a row are loaded in chunks of 8 before their products.  HBM-bound on large blocks.
template <typename C, int M, int V, int R> struct DotRegs {
    static constexpr int words = 2 * (int)sizeof(C) / 8;
    static constexpr int need = (M + R * (M < 8 ? M : 8)) * V * words + 44;
    static constexpr int blocks = 256 / need < 1 ? 1 : (256 / need > 4 ? 4 : 256 / need);
};
template <typename C, int M, int V, int R>
__global__ void __launch_bounds__(256, (DotRegs<C, M, V, R>::blocks))
    k_multidot(CSum<C>* __restrict__ part, const C* __restrict__ Vb, int m, int mt, const C* __restrict__ w,
               long long n, int N) {
    if (grid_dependency()) return;
    constexpr int KC = 4;                        // vectors reduced at once
    constexpr int KL = M < 8 ? M : 8;            // vectors loaded at once
    __shared__ C sh[KC][256 * V];
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const long long stride = n * (long long)N;
    const long long S = (long long)gridDim.y * blockDim.y;
    C acc[M][V];
#pragma unroll
    for (int k = 0; k < M; ++k)
#pragma unroll
        for (int q = 0; q < V; ++q) acc[k][q] = czero<C>();
    if (j < N)
        for (long long i0 = (long long)blockIdx.y * blockDim.y + threadIdx.y; i0 < n; i0 += R * S) {
            Vec<C, V> wv[R];
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (i0 + r * S < n) wv[r] = *reinterpret_cast<const Vec<C, V>*>(w + (i0 + r * S) * N + j);
#pragma unroll
            for (int c0 = 0; c0 < M; c0 += KL) {
                if (c0 >= m) break;
                Vec<C, V> vv[R][KL];
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (i0 + r * S < n) {
#pragma unroll
                        for (int k = 0; k < KL; ++k)
                            if (c0 + k < m)
                                vv[r][k] = *reinterpret_cast<const Vec<C, V>*>(Vb + (c0 + k) * stride +
                                                                               (i0 + r * S) * N + j);
                    }
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (i0 + r * S < n) {
#pragma unroll
                        for (int k = 0; k < KL; ++k)
                            if (c0 + k < m)
#pragma unroll
                                for (int q = 0; q < V; ++q) cfmac(acc[c0 + k][q], vv[r][k].v[q], wv[r].v[q]);
                    }
            }
        }
    const int bxV = blockDim.x * V, tid = threadIdx.y * blockDim.x + threadIdx.x;
#pragma unroll
    for (int k0 = 0; k0 < M; k0 += KC) {
        if (k0 >= m) break;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KC; ++k)
            if (k0 + k < M)
#pragma unroll
                for (int q = 0; q < V; ++q) sh[k][threadIdx.y * bxV + threadIdx.x * V + q] = acc[k0 + k][q];
        __syncthreads();
        for (int o = tid; o < KC * bxV; o += 256) {
            const int k = o / bxV, col = o % bxV, jo = blockIdx.x * bxV + col;
            if (k0 + k >= m || jo >= N) continue;
            CSum<C> s;
            for (int r = 0; r < (int)blockDim.y; ++r) {
                const C v = sh[k][r * bxV + col];
                s.re.add(v.x);
                s.im.add(v.y);
            }
            part[((long long)blockIdx.y * mt + k0 + k) * N + jo] = s;
        }
    }
}

// h_k = sum of the partials of <w_k, u>; cf[k] = -h_k / eta_k^2 (the update u += cf w_k of an
// unnormalised basis), H[k] (+)= h_k / (eta_k eta_j), the Hessenberg entry.  Block (columns,
// groups); grid.y = k.
template <typename C>
__global__ void __launch_bounds__(256) k_finalize_dots(C* __restrict__ cf, double2* __restrict__ H,
                                                       const CSum<C>* __restrict__ part, int groups, int m, int N,
                                                       const double* __restrict__ ieta, bool add) {
    if (grid_dependency()) return;
    __shared__ CSum<C> sh[256];
    const int r = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    CSum<C> s;
    if (r < N) {
        const CSum<C>* p = part + (long long)k * N + r;
        const long long ld = (long long)m * N;
#pragma unroll 8
        for (int g = threadIdx.y; g < groups; g += blockDim.y) {
            const CSum<C> v = p[g * ld];
            s.re.add(v.re);
            s.im.add(v.im);
        }
    }
    sh[threadIdx.y * blockDim.x + threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && r < N) {
        for (int q = 1; q < (int)blockDim.y; ++q) {
            s.re.add(sh[q * blockDim.x + threadIdx.x].re);
            s.im.add(sh[q * blockDim.x + threadIdx.x].im);
        }
        const double re = s.re.value(), im = s.im.value();
        const double ik = ieta[(long long)k * N + r], f = -ik * ik, g = ik * ieta[(long long)(m - 1) * N + r];
        cf[(long long)k * N + r] = cvt<C>(make_double2(re * f, im * f));
        double2* h = H + (long long)k * N + r;
        *h = add ? make_double2(fma(re, g, h->x), fma(im, g, h->y)) : make_double2(re * g, im * g);
    }
}

// ---- w (=|+=) sum_{k < m} cf_k V_k, and (npart) the partials of |w * nscale|^2 of the result.
// Rows run from the last to the first: the dot products before read them in the other
// order, so what they left in L2 is met first.
template <typename C, int V>
__global__ void __launch_bounds__(256, 4) k_multiaxpy(C* __restrict__ w, const C* __restrict__ cf, int m,
                                                      const C* __restrict__ Vb, long long n, int N, bool accumulate,
                                                      sum_t<C>* __restrict__ npart,
                                                      const double* __restrict__ nscale) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    constexpr int KC = V * sizeof(C) == 8 ? 8 : 4;
    __shared__ Vec<C, V> cs[64 * 32];
    __shared__ sum_t<C> sh[256];
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const long long stride = n * (long long)N;
    for (int k = threadIdx.y; k < m; k += blockDim.y)
        if (j < N)
            cs[k * blockDim.x + threadIdx.x] = *reinterpret_cast<const Vec<C, V>*>(cf + (long long)k * N + j);
    __syncthreads();
    R ns[V];
    SquareSums<R, V> nrm;
#pragma unroll
    for (int q = 0; q < V; ++q) ns[q] = (nscale && j < N && nscale[j + q] != 0.0) ? (R)nscale[j + q] : (R)1;
    if (j < N)
        for (long long t = (long long)blockIdx.y * blockDim.y + threadIdx.y; t < n;
             t += (long long)gridDim.y * blockDim.y) {
            const long long i = n - 1 - t;
            Vec<C, V> acc;
            if (accumulate) acc = *reinterpret_cast<const Vec<C, V>*>(w + i * N + j);
            else
#pragma unroll
                for (int q = 0; q < V; ++q) acc.v[q] = czero<C>();
            for (int k0 = 0; k0 < m; k0 += KC) {
                Vec<C, V> vv[KC];
#pragma unroll
                for (int k = 0; k < KC; ++k)
                    if (k0 + k < m) vv[k] = *reinterpret_cast<const Vec<C, V>*>(Vb + (k0 + k) * stride + i * N + j);
#pragma unroll
                for (int k = 0; k < KC; ++k)
                    if (k0 + k < m) {
                        const Vec<C, V> a = cs[(k0 + k) * blockDim.x + threadIdx.x];
#pragma unroll
                        for (int q = 0; q < V; ++q) cfma(acc.v[q], a.v[q], vv[k].v[q]);
                    }
            }
            *reinterpret_cast<Vec<C, V>*>(w + i * N + j) = acc;
#pragma unroll
            for (int q = 0; q < V; ++q) nrm.add(q, acc.v[q].x * ns[q], acc.v[q].y * ns[q]);
            nrm.end_row();
        }
    if (npart) {
        nrm.fold();
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const sum_t<C> s = block_rows_sum(nrm.total[q], sh);
            if (threadIdx.y == 0 && j < N) npart[(long long)blockIdx.y * N + j + q] = s;
        }
    }
}

// ---- partials of |x|^2
template <typename C, int V>
__global__ void __launch_bounds__(256) k_norm2(sum_t<C>* __restrict__ npart, const C* __restrict__ x, long long n,
                                               int N) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    __shared__ sum_t<C> sh[256];
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    R nrm[V];
#pragma unroll
    for (int q = 0; q < V; ++q) nrm[q] = 0;
    if (j < N)
#pragma unroll 4
        for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n;
             i += (long long)gridDim.y * blockDim.y) {
            const Vec<C, V> v = *reinterpret_cast<const Vec<C, V>*>(x + i * N + j);
#pragma unroll
            for (int q = 0; q < V; ++q) nrm[q] = fma(v.v[q].x, v.v[q].x, fma(v.v[q].y, v.v[q].y, nrm[q]));
        }
#pragma unroll
    for (int q = 0; q < V; ++q) {
        sum_t<C> s;
        s.add(nrm[q]);
        s = block_rows_sum(s, sh);
        if (threadIdx.y == 0 && j < N) npart[(long long)blockIdx.y * N + j + q] = s;
    }
}

// ---- y = x scale (scale NULL: 1; inverse: 1 / scale, 0 where scale is 0) in another precision
// or the same, and the partials of |y|^2.
template <typename Cy, typename Cx_, int V>
__global__ void __launch_bounds__(256) k_scale_norm(Cy* __restrict__ y, const Cx_* __restrict__ x,
                                                    const double* __restrict__ scale, bool inverse, long long n, int N,
                                                    sum_t<Cy>* __restrict__ npart) {
    if (grid_dependency()) return;
    using R = re_t<Cy>;
    __shared__ sum_t<Cy> sh[256];
    __shared__ R sc[32 * V];
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    if (threadIdx.y == 0 && j < N)
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const double s = scale ? scale[j + q] : 1.0;
            sc[threadIdx.x * V + q] = (R)(inverse ? (s != 0.0 ? 1.0 / s : 0.0) : s);
        }
    __syncthreads();
    R nrm[V], s[V];
#pragma unroll
    for (int q = 0; q < V; ++q) {
        nrm[q] = 0;
        s[q] = j < N ? sc[threadIdx.x * V + q] : (R)0;
    }
    if (j < N)
#pragma unroll 4
        for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n;
             i += (long long)gridDim.y * blockDim.y) {
            Vec<Cy, V> o;
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const Cy v = cvtc(x[i * N + j + q], Cy());
                o.v[q] = mk(v.x * s[q], v.y * s[q]);
                nrm[q] = fma(o.v[q].x, o.v[q].x, fma(o.v[q].y, o.v[q].y, nrm[q]));
            }
            *reinterpret_cast<Vec<Cy, V>*>(y + i * N + j) = o;
        }
#pragma unroll
    for (int q = 0; q < V; ++q) {
        sum_t<Cy> t;
        t.add(nrm[q]);
        t = block_rows_sum(t, sh);
        if (threadIdx.y == 0 && j < N) npart[(long long)blockIdx.y * N + j + q] = t;
    }
}

// ---- refinement updates: y (=|+=) sign s_j x with FP32 x, FP64 y, and the partials of |x|^2
// (OF_X) or of the new |y|^2.
template <bool OF_X>
__global__ void __launch_bounds__(256) k_refine_axpy(double2* __restrict__ y, const double* __restrict__ s, double sign,
                                                     const float2* __restrict__ x, long long n, int N, bool accumulate,
                                                     void* __restrict__ npart) {
    if (grid_dependency()) return;
    __shared__ PairF shf[256];
    __shared__ SumD shd[256];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const double b = j < N ? s[j] * sign : 0.0;
    float nf = 0.f;
    double nd = 0.0;
    if (j < N)
#pragma unroll 4
        for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n;
             i += (long long)gridDim.y * blockDim.y) {
            const float2 v = x[i * N + j];
            double2 a = accumulate ? y[i * N + j] : make_double2(0.0, 0.0);
            a.x = fma(b, (double)v.x, a.x);
            a.y = fma(b, (double)v.y, a.y);
            y[i * N + j] = a;
            if (OF_X) nf = fmaf(v.x, v.x, fmaf(v.y, v.y, nf));
            else nd = fma(a.x, a.x, fma(a.y, a.y, nd));
        }
    if (!npart) return;
    if (OF_X) {
        PairF t;
        t.add(nf);
        t = block_rows_sum(t, shf);
        if (threadIdx.y == 0 && j < N) reinterpret_cast<PairF*>(npart)[(long long)blockIdx.y * N + j] = t;
    } else {
        SumD t;
        t.add(nd);
        t = block_rows_sum(t, shd);
        if (threadIdx.y == 0 && j < N) reinterpret_cast<SumD*>(npart)[(long long)blockIdx.y * N + j] = t;
    }
}

// Unnormalised basis vectors are kept while eta = |w| lies in [2^-32, 2^32]: their FP32
// entries, dot products and squared sums then stay far inside the normal range.
constexpr double kEtaLow = 0x1p-32, kEtaHigh = 0x1p32;

// Non-negative doubles order like their bit patterns, and NaN is above all of them.
__device__ __forceinline__ void atomic_max_double(u64* m, double v) {
    const u64 b = (u64)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
    if (b) atomicMax(m, b);
}

// norm_j = sqrt(sum of the partials), and with it what the caller's next kernels need (NormOut).
template <typename S>
__global__ void __launch_bounds__(256) k_finalize_norm(NormOut o, const S* __restrict__ part, int groups, int N) {
    if (grid_dependency()) return;
    __shared__ S sh[256];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    S s;
    if (r < N) {
#pragma unroll 8
        for (int g = threadIdx.y; g < groups; g += blockDim.y) s.add(part[(long long)g * N + r]);
    }
    s = block_rows_sum(s, sh);
    if (o.clear && blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) *o.clear = 0;
    if (threadIdx.y != 0 || r >= N) return;
    const double v = sqrt(s.value());
    if (o.norm) o.norm[r] = v;
    if (o.max) {
        const double d = o.den ? o.den[r] : v;
        // a zero right-hand side is solved; a NaN on either side is the maximum
        atomic_max_double(o.max, d == 0.0 ? 0.0 : (o.mul ? v * o.mul[r] : v) / d);
    }
    if (o.eta) {
        double en = v;
        if (o.hsub) {                            // v = |u / eta_j|, the Hessenberg subdiagonal
            const double ej = o.eta_prev[r];
            o.hsub[r] = ej != 0.0 ? v : 0.0;
            en = v * ej;
        }
        const bool out = en > 0.0 && (en < kEtaLow || en > kEtaHigh);
        const double ie = en != 0.0 ? 1.0 / en : 0.0;
        o.rsc[r] = out ? ie : 0.0;               // the vector is rescaled to unit norm where rsc != 0
        o.eta[r] = out ? 1.0 : en;
        o.ieta[r] = out ? 1.0 : ie;
        if (o.g0) o.g0[r] = make_double2(en, 0.0);
    }
}

// w[:, j] *= s[j] for the rhs with s[j] != 0; the others are left untouched (and their
// threads return after one load).
template <typename C>
__global__ void __launch_bounds__(256) k_scale_cols_if(C* __restrict__ w, const double* __restrict__ s, long long n,
                                                       int N) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const double sc = s[j];
    if (sc == 0.0) return;
    const R f = (R)sc;
    for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n;
         i += (long long)gridDim.y * blockDim.y) {
        const C v = w[i * N + j];
        w[i * N + j] = mk(v.x * f, v.y * f);
    }
}

// ---- Givens rotations of the Hessenberg columns j0 .. j1, one thread per rhs.  Column j:
// entries i <= j at H[(j (m + 1) + i) N + r] (overwritten by R), subdiagonal hsub[j N + r];
// rotation i: (a, b) <- (c a + s b, -conj(s) a + c b).  irr = 1 / R[j][j] (0 if it is 0).
// The square of the residual estimate after column j, divided by bnorm, goes to max[j] (the maximum
// over the rhs), or to host[j] where one warp holds all rhs: with the square root and the quotient
// of every column the first look of a cycle, at ten or more columns, took 10 us longer.
__global__ void __launch_bounds__(32) k_rotate(double2* __restrict__ H, const double* __restrict__ hsub,
                                               double* __restrict__ cs, double2* __restrict__ sn,
                                               double2* __restrict__ g, double2* __restrict__ irr,
                                               const double* __restrict__ bnorm, u64* max, double* host, int j0, int j1, int m,
                                               int N) {
    if (grid_dependency()) return;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = r < N;
    if (!in && !host) return;
    double2 gj = in ? g[(long long)j0 * N + r] : make_double2(0.0, 0.0);
    const double bn = in && bnorm ? bnorm[r] : 0.0;
    const double lift = bn < 0x1p-900 ? 0x1p200 : 1.0;         // 1 / |b| stays finite
    const double ib = bn == 0.0 ? 0.0 : 1.0 / (bn * lift);
    double resid = 0.0;
    auto column = [&](int j) {
        double2* col = H + (long long)j * (m + 1) * N + r;
        double2 a = col[0];
#pragma unroll 4
        for (int i = 0; i < j; ++i) {
            const double c = cs[(long long)i * N + r];
            const double2 s = sn[(long long)i * N + r], b = col[(long long)(i + 1) * N];
            col[(long long)i * N] = make_double2(fma(c, a.x, fma(s.x, b.x, -s.y * b.y)),
                                                 fma(c, a.y, fma(s.x, b.y, s.y * b.x)));
            a = make_double2(fma(c, b.x, -fma(s.x, a.x, s.y * a.y)), fma(c, b.y, -fma(s.x, a.y, -s.y * a.x)));
        }
        const double b = hsub[(long long)j * N + r];
        const double na2 = fma(a.x, a.x, a.y * a.y), t = fma(b, b, na2);
        double c = 1.0;
        double2 s = make_double2(0.0, 0.0), rr = s, ir = s;
        if (t > 0.0 && na2 > 0.0) {
            const double ia = rsqrt(na2), ir1 = rsqrt(t);
            const double2 ph = make_double2(a.x * ia, a.y * ia);
            c = na2 * ia * ir1;
            s = make_double2(ph.x * b * ir1, ph.y * b * ir1);      // (a / |a|) conj(b) / rho, b real
            rr = make_double2(ph.x * t * ir1, ph.y * t * ir1);
            ir = make_double2(ph.x * ir1, -ph.y * ir1);
        } else if (t > 0.0) {
            c = 0.0;
            s = make_double2(1.0, 0.0);
            rr = make_double2(b, 0.0);
            ir = make_double2(1.0 / b, 0.0);
        } else if (!(t == 0.0)) {
            rr = make_double2(t, 0.0);           // NaN stays visible
            c = t;
        }
        cs[(long long)j * N + r] = c;
        sn[(long long)j * N + r] = s;
        col[(long long)j * N] = rr;
        irr[(long long)j * N + r] = ir;
        g[(long long)j * N + r] = make_double2(c * gj.x, c * gj.y);
        const double2 sg = cmulc(s, gj);
        gj = make_double2(-sg.x, -sg.y);
        g[(long long)(j + 1) * N + r] = gj;
        if (!(t == t)) resid = t;
    };
    for (int j = j0; j <= j1; ++j) {
        if (in) column(j);
        if (!max && !host) continue;
        const double gx = gj.x * lift * ib, gy = gj.y * lift * ib;
        const double v = resid == resid ? fma(gx, gx, gy * gy) : resid;
        if (host) {
            u64 m8 = (u64)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const u64 w = __shfl_xor_sync(0xffffffffu, m8, o);
                m8 = w > m8 ? w : m8;
            }
            if (threadIdx.x == 0) host[j] = __longlong_as_double((long long)m8);
        } else {
            atomic_max_double(max + j, v);
        }
    }
}

// y = R^{-1} g (column-oriented back substitution) and the update coefficients
// cf[i] = y_i / eta_i: one warp per rhs, lane l holds rows l and l + 32.
template <typename C>
__global__ void __launch_bounds__(32) k_back_substitute(C* __restrict__ cf, const double2* __restrict__ H,
                                                        const double2* __restrict__ g, const double2* __restrict__ irr,
                                                        const double* __restrict__ ieta, int j, int m, int N) {
    if (grid_dependency()) return;
    const int r = blockIdx.x, l = threadIdx.x;
    double2 v[2], d[2], col[2], nxt[2];
    auto load = [&](int i, double2* c) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            c[q] = (l + 32 * q < i) ? H[((long long)i * (m + 1) + l + 32 * q) * N + r] : make_double2(0.0, 0.0);
    };
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = l + 32 * q;
        v[q] = i <= j ? g[(long long)i * N + r] : make_double2(0.0, 0.0);
        d[q] = i <= j ? irr[(long long)i * N + r] : make_double2(0.0, 0.0);
    }
    load(j, col);
    for (int i = j; i >= 0; --i) {
        load(i - 1, nxt);
        const int own = i & 31;
        const double2 y0 = i >= 32 ? cmul(v[1], d[1]) : cmul(v[0], d[0]);      // y_i in lane `own`
        const double2 y = make_double2(__shfl_sync(0xffffffffu, y0.x, own), __shfl_sync(0xffffffffu, y0.y, own));
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            if (l + 32 * p == i) v[p] = y;
            if (l + 32 * p < i) v[p] = csub(v[p], cmul(col[p], y));
            col[p] = nxt[p];
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = l + 32 * q;
        if (i <= j) {
            const double f = ieta[(long long)i * N + r];
            cf[(long long)i * N + r] = cvt<C>(make_double2(v[q].x * f, v[q].y * f));
        }
    }
}
}  // namespace kr

using namespace kr;

static int dot_groups(long long n, int N) { return groups_of(n, N, 1, 4); }
size_t dot_part_bytes(long long n, int N, int m) {
    return (size_t)std::max(groups_of(n, N, 1, 4), groups_of(n, N, 2, 4)) * m * N * 16;
}
// The updates of Gram-Schmidt stream m + 2 vectors with few loads per row: two waves of the four
// blocks that an SM holds.
static int axpy_groups(long long n, int N) { return groups_of(n, N, 1, 8); }
size_t norm_part_bytes(long long n, int N) { return (size_t)axpy_groups(n, N) * N * 8; }

template <typename C>
void launch_multidot(C* cf, double2* H, const C* V, int m, const C* w, long long n, int N, const double* ieta, bool add,
                     void* part, cudaStream_t s) {
    MG_REQUIRE(m >= 1 && m <= 64, MGMLMC_EINVAL, "multidot: 1 <= m <= 64");
    CSum<C>* p = reinterpret_cast<CSum<C>*>(part);
    const int W = width<C>(N);
    const int G = groups_of(n, N, W, 4);
    constexpr int W2 = sizeof(C) == 8 ? 2 : 1;   // FP64: one rhs per thread
    const Shape2 s2 = shape(N, W, G), s1 = shape(N, 1, G);
    // at most 32 vectors a launch (their sums are registers)
    for (int k0 = 0; k0 < m; k0 += 32) {
        const int mk_ = std::min(32, m - k0);
        const C* Vk = V + (size_t)k0 * n * N;
        CSum<C>* pk = p + (size_t)k0 * N;
        if (W == 2 && mk_ <= 16) {
            if (mk_ <= 4) MG_LAUNCH(s2.g, s2.b, 0, s, (k_multidot<C, 4, W2, 2>), pk, Vk, mk_, m, w, n, N);
            else if (mk_ <= 8) MG_LAUNCH(s2.g, s2.b, 0, s, (k_multidot<C, 8, W2, 1>), pk, Vk, mk_, m, w, n, N);
            else MG_LAUNCH(s2.g, s2.b, 0, s, (k_multidot<C, 16, W2, 1>), pk, Vk, mk_, m, w, n, N);
        } else {
            if (mk_ <= 4) MG_LAUNCH(s1.g, s1.b, 0, s, (k_multidot<C, 4, 1, 2>), pk, Vk, mk_, m, w, n, N);
            else if (mk_ <= 8) MG_LAUNCH(s1.g, s1.b, 0, s, (k_multidot<C, 8, 1, 1>), pk, Vk, mk_, m, w, n, N);
            else if (mk_ <= 16) MG_LAUNCH(s1.g, s1.b, 0, s, (k_multidot<C, 16, 1, 1>), pk, Vk, mk_, m, w, n, N);
            else MG_LAUNCH(s1.g, s1.b, 0, s, (k_multidot<C, 32, 1, 1>), pk, Vk, mk_, m, w, n, N);
        }
        MG_LAUNCHED();
    }
    int bx = 1;
    while (bx < N && bx < 16) bx *= 2;
    MG_LAUNCH(dim3((N + bx - 1) / bx, m), dim3(bx, 128 / bx), 0, s, (k_finalize_dots<C>), cf, H, p, G, m, N, ieta, add);
    MG_LAUNCHED();
}

template <typename C>
static void launch_finalize_norm(const NormOut& o, const void* part, int groups, int N, cudaStream_t s) {
    int bx = 1;
    while (bx < N && bx < 8) bx *= 2;
    MG_LAUNCH((N + bx - 1) / bx, dim3(bx, 256 / bx), 0, s, (k_finalize_norm<sum_t<C>>), o, reinterpret_cast<const sum_t<C>*>(part), groups, N);
    MG_LAUNCHED();
}

template <typename C>
void launch_multiaxpy(C* w, const C* cf, int m, const C* V, long long n, int N, bool accumulate, const NormOut* norm,
                      void* npart, const double* nscale, cudaStream_t s) {
    MG_REQUIRE(m >= 1 && m <= 64, MGMLMC_EINVAL, "multiaxpy: 1 <= m <= 64");
    sum_t<C>* np = norm ? reinterpret_cast<sum_t<C>*>(npart) : nullptr;
    constexpr int W2 = sizeof(C) == 8 ? 2 : 1;
    const int G = axpy_groups(n, N);
    if (width<C>(N) == 2) {
        const Shape2 sh = shape(N, W2, G);
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_multiaxpy<C, W2>), w, cf, m, V, n, N, accumulate, np, nscale);
    } else {
        const Shape2 sh = shape(N, 1, G);
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_multiaxpy<C, 1>), w, cf, m, V, n, N, accumulate, np, nscale);
    }
    MG_LAUNCHED();
    if (norm) launch_finalize_norm<C>(*norm, np, G, N, s);
}

template <typename C>
void launch_norm(const NormOut& o, const C* x, long long n, int N, void* part, cudaStream_t s) {
    sum_t<C>* np = reinterpret_cast<sum_t<C>*>(part);
    constexpr int W2 = sizeof(C) == 8 ? 2 : 1;
    const int G = dot_groups(n, N);
    if (width<C>(N) == 2) {
        const Shape2 sh = shape(N, W2, G);
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_norm2<C, W2>), np, x, n, N);
    } else {
        const Shape2 sh = shape(N, 1, G);
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_norm2<C, 1>), np, x, n, N);
    }
    MG_LAUNCHED();
    launch_finalize_norm<C>(o, np, G, N, s);
}

template <typename Cy, typename Cx_>
void launch_scale_norm(const NormOut& o, Cy* y, const Cx_* x, const double* scale, bool inverse, long long n, int N,
                       void* part, cudaStream_t s) {
    sum_t<Cy>* np = reinterpret_cast<sum_t<Cy>*>(part);
    constexpr int W2 = sizeof(Cy) == 8 ? 2 : 1;
    const int G = dot_groups(n, N);
    if (width<Cy>(N) == 2) {
        const Shape2 sh = shape(N, W2, G);
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_scale_norm<Cy, Cx_, W2>), y, x, scale, inverse, n, N, np);
    } else {
        const Shape2 sh = shape(N, 1, G);
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_scale_norm<Cy, Cx_, 1>), y, x, scale, inverse, n, N, np);
    }
    MG_LAUNCHED();
    launch_finalize_norm<Cy>(o, np, G, N, s);
}

void launch_refine_axpy(double2* y, const double* scale, double sign, const float2* x, long long n, int N,
                        bool accumulate, const NormOut* of_x, const NormOut* of_y, void* part, cudaStream_t s) {
    const int G = dot_groups(n, N);
    const Shape2 sh = shape(N, 1, G);
    if (of_y) {
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_refine_axpy<false>), y, scale, sign, x, n, N, accumulate, part);
        MG_LAUNCHED();
        launch_finalize_norm<double2>(*of_y, part, G, N, s);
    } else {
        MG_LAUNCH(sh.g, sh.b, 0, s, (k_refine_axpy<true>), y, scale, sign, x, n, N, accumulate, of_x ? part : nullptr);
        MG_LAUNCHED();
        if (of_x) launch_finalize_norm<float2>(*of_x, part, G, N, s);
    }
}

template <typename C>
void launch_scale_cols_if(C* w, const double* f, long long n, int N, cudaStream_t s) {
    const Shape2 sh = shape(N, 1, groups_of(n, N, 1, 4));
    MG_LAUNCH(sh.g, sh.b, 0, s, (k_scale_cols_if<C>), w, f, n, N);
    MG_LAUNCHED();
}

void launch_rotate(double2* H, const double* hsub, double* cs, double2* sn, double2* g, double2* irr,
                   const double* bnorm, unsigned long long* max, double* host, int j0, int j1, int m, int N,
                   cudaStream_t s) {
    MG_REQUIRE(!host || N <= kRotateWarp, MGMLMC_EINVAL, "rotations: one warp writes to the host");
    MG_LAUNCH((N + 31) / 32, 32, 0, s, k_rotate, H, hsub, cs, sn, g, irr, bnorm, max, host, j0, j1, m, N);
    MG_LAUNCHED();
}

template <typename C>
void launch_back_substitute(C* cf, const double2* H, const double2* g, const double2* irr, const double* ieta, int j,
                            int m, int N, cudaStream_t s) {
    MG_REQUIRE(j < 64, MGMLMC_EINVAL, "FGMRES restart length above 64");
    MG_LAUNCH(N, 32, 0, s, (k_back_substitute<C>), cf, H, g, irr, ieta, j, m, N);
    MG_LAUNCHED();
}

#define INST(C)                                                                                            \
    template void launch_multidot<C>(C*, double2*, const C*, int, const C*, long long, int, const double*, \
                                     bool, void*, cudaStream_t);                                            \
    template void launch_multiaxpy<C>(C*, const C*, int, const C*, long long, int, bool, const NormOut*,    \
                                      void*, const double*, cudaStream_t);                                  \
    template void launch_norm<C>(const NormOut&, const C*, long long, int, void*, cudaStream_t);            \
    template void launch_scale_cols_if<C>(C*, const double*, long long, int, cudaStream_t);                 \
    template void launch_scale_norm<C, C>(const NormOut&, C*, const C*, const double*, bool, long long, int, \
                                          void*, cudaStream_t);                                             \
    template void launch_back_substitute<C>(C*, const double2*, const double2*, const double2*,             \
                                            const double*, int, int, int, cudaStream_t);
INST(double2)
INST(float2)
template void launch_scale_norm<float2, double2>(const NormOut&, float2*, const double2*, const double*, bool, long long,
                                                 int, void*, cudaStream_t);

}  // namespace mg
