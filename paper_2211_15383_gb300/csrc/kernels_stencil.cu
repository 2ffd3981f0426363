// Stencil kernels: the fine Wilson-Schwinger operator D_1, the coarse 5-point
// block stencils D_l (l >= 2), restriction P^H, prolongation P, Gamma5 and the
// fused minimal-residual smoother update.
//
// The fine operator (the paper names the 2D Wilson-Schwinger discretisation,
// Sect. 1; its form is the standard Wilson one):
//   (D psi)(x) = (m0+2) psi(x) - 1/2 sum_mu [(1 - s_mu) U_mu(x) psi(x+mu)
//                                          + (1 + s_mu) U_mu(x-mu)^* psi(x-mu)]
// with s_0 = sigma_1, s_1 = sigma_2, antiperiodic in time.  Each hop needs a
// single complex multiply: (1 -+ s_mu) projects the 2-spinor onto one
// component (e.g. (1 - sigma_1) psi = (a, -a) with a = psi_0 - psi_1).
#include <algorithm>

#include "footprint.h"
#include "kernels.cuh"

namespace mg {

// BF16 pairs (one complex value per 32-bit word).
__device__ __forceinline__ float2 bf2_lo(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); }
__device__ __forceinline__ uint32_t f2_bf(float2 v) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t*>(&b);
}

// Threads of the one-rhs-per-thread CTAs: 128, or fewer for narrower blocks so that
// no lane idles (N = 64: two warps).
static int cta_threads(int N) { return std::min(128, (N + 31) / 32 * 32); }

template <typename C, int MODE>
__global__ void __launch_bounds__(256) k_wilson(C* __restrict__ y, const C* __restrict__ x, const C* __restrict__ b,
                                                const C* __restrict__ U, re_t<C> mass, int lx, int lt, int N,
                                                double2* __restrict__ part) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    const int V = lx * lt;
    const R half = (R)0.5;
    C dyx = czero<C>();
    R dyy = 0;
    if (j < N) {
        for (int site = blockIdx.y * kRowLanes + threadIdx.y; site < V; site += gridDim.y * kRowLanes) {
            const int xx = site % lx, t = site / lx;
            const int sxp = (xx + 1 == lx ? 0 : xx + 1) + lx * t;
            const int sxm = (xx == 0 ? lx - 1 : xx - 1) + lx * t;
            const int stp = xx + lx * (t + 1 == lt ? 0 : t + 1);
            const int stm = xx + lx * (t == 0 ? lt - 1 : t - 1);
            const R sgp = (t + 1 == lt) ? (R)-0.5 : half;   // antiperiodic time boundary, times 1/2
            const R sgm = (t == 0) ? (R)-0.5 : half;
            const C u0 = U[2 * site], u1 = U[2 * site + 1];
            const C u0m = U[2 * sxm], u1m = U[2 * stm + 1];
            const long long N2 = 2LL * N;
            const C p0 = x[site * N2 + j], p1 = x[site * N2 + N + j];
            C o0 = mk(mass * p0.x, mass * p0.y), o1 = mk(mass * p1.x, mass * p1.y);
            {   // +x: (1 - sigma_1) psi = (a, -a), a = psi0 - psi1
                const C q0 = x[sxp * N2 + j], q1 = x[sxp * N2 + N + j];
                const C u = cscale(cmul(u0, csub(q0, q1)), half);
                o0 = csub(o0, u);
                o1 = cadd(o1, u);
            }
            {   // -x: (1 + sigma_1) psi = (c, c), c = psi0 + psi1
                const C q0 = x[sxm * N2 + j], q1 = x[sxm * N2 + N + j];
                const C u = cscale(cmulc(u0m, cadd(q0, q1)), half);
                o0 = csub(o0, u);
                o1 = csub(o1, u);
            }
            {   // +t: (1 - sigma_2) psi = (a, -i a), a = psi0 + i psi1
                const C q0 = x[stp * N2 + j], q1 = x[stp * N2 + N + j];
                const C u = cscale(cmul(u1, cadd(q0, ctimesi(q1))), sgp);
                o0 = csub(o0, u);
                o1 = cadd(o1, ctimesi(u));
            }
            {   // -t: (1 + sigma_2) psi = (c, i c), c = psi0 - i psi1
                const C q0 = x[stm * N2 + j], q1 = x[stm * N2 + N + j];
                const C u = cscale(cmulc(u1m, csub(q0, ctimesi(q1))), sgm);
                o0 = csub(o0, u);
                o1 = csub(o1, ctimesi(u));
            }
            if (MODE == 1) {
                o0 = csub(b[site * N2 + j], o0);
                o1 = csub(b[site * N2 + N + j], o1);
            }
            if (MODE != 3) {
                y[site * N2 + j] = o0;
                y[site * N2 + N + j] = o1;
            }
            if (MODE >= 2) {
                cfmac(dyx, o0, p0);
                cfmac(dyx, o1, p1);
                dyy = fma(o0.x, o0.x, fma(o0.y, o0.y, fma(o1.x, o1.x, fma(o1.y, o1.y, dyy))));
            }
        }
    }
    if (MODE >= 2) {
        __shared__ dot_t<C> sh[2][kRowLanes][kRhsTile + 1];
        sh[0][threadIdx.y][threadIdx.x] = dot_part(dyx);
        sh[1][threadIdx.y][threadIdx.x] = dot_part(dyy);
        __syncthreads();
        if (threadIdx.y < 2 && j < N) {
            dot_t<C> s = sh[threadIdx.y][0][threadIdx.x];
            for (int r = 1; r < kRowLanes; ++r) s = dot_add(s, sh[threadIdx.y][r][threadIdx.x]);
            dot_parts<C>(part)[((long long)threadIdx.y * N + j) * gridDim.y + blockIdx.y] = s;
        }
    }
}


// One block per coarse site (grid-stride): A[site] (5 d^2 complex) staged in
// shared memory, each thread owns one rhs and RPT output rows.
template <typename C, int RPT, int MODE>
__global__ void __launch_bounds__(256) k_block_stencil(C* __restrict__ y, const C* __restrict__ x,
                                                       const C* __restrict__ b, const C* __restrict__ A, int lx,
                                                       int lt, int d, int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* As = reinterpret_cast<C*>(smem_raw);
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    const int V = lx * lt;
    const int nA = 5 * d * d;
    const int tid = threadIdx.y * kRhsTile + threadIdx.x;
    C dyx = czero<C>();
    R dyy = 0;
    for (int site = blockIdx.y; site < V; site += gridDim.y) {
        __syncthreads();
        for (int e = tid; e < nA; e += kRhsTile * kRowLanes) As[e] = A[(long long)site * nA + e];
        __syncthreads();
        if (j < N) {
            C acc[RPT];
#pragma unroll
            for (int r = 0; r < RPT; ++r) acc[r] = czero<C>();
            for (int dir = 0; dir < 5; ++dir) {
                const int nb = nbr_site(site, dir, lx, lt);
                const C* xn = x + (long long)nb * d * N + j;
                const C* Ad = As + dir * d * d;
                for (int bc = 0; bc < d; ++bc) {
                    const C xv = xn[(long long)bc * N];
#pragma unroll
                    for (int r = 0; r < RPT; ++r) {
                        const int c = threadIdx.y + kRowLanes * r;
                        if (c < d) cfma(acc[r], Ad[c * d + bc], xv);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int c = threadIdx.y + kRowLanes * r;
                if (c < d) {
                    const long long idx = ((long long)site * d + c) * N + j;
                    C o = acc[r];
                    if (MODE == 1) o = csub(b[idx], o);
                    if (MODE != 3) y[idx] = o;
                    if (MODE >= 2) {
                        cfmac(dyx, o, x[idx]);
                        dyy = fma(o.x, o.x, fma(o.y, o.y, dyy));
                    }
                }
            }
        }
    }
    if (MODE >= 2) {
        __syncthreads();
        dot_t<C>* sh = reinterpret_cast<dot_t<C>*>(smem_raw);   // reuse: [2][8][33]
        sh[(0 * kRowLanes + threadIdx.y) * (kRhsTile + 1) + threadIdx.x] = dot_part(dyx);
        sh[(1 * kRowLanes + threadIdx.y) * (kRhsTile + 1) + threadIdx.x] = dot_part(dyy);
        __syncthreads();
        if (threadIdx.y < 2 && j < N) {
            dot_t<C> s = sh[(threadIdx.y * kRowLanes) * (kRhsTile + 1) + threadIdx.x];
            for (int r = 1; r < kRowLanes; ++r)
                s = dot_add(s, sh[(threadIdx.y * kRowLanes + r) * (kRhsTile + 1) + threadIdx.x]);
            dot_parts<C>(part)[((long long)threadIdx.y * N + j) * gridDim.y + blockIdx.y] = s;
        }
    }
}

// Site-per-thread-row variant for compile-time d: block = 128 rhs, each thread
// computes all d outputs of one site for its rhs, so every input value loaded
// is used d times.  The blocks are staged transposed, At[dir][b][c], so the
// inner loop over output rows reads consecutive shared-memory words (broadcast
// to the whole warp).
template <typename C, int D, int MODE>
__global__ void __launch_bounds__(128) k_block_stencil_d(C* __restrict__ y, const C* __restrict__ x,
                                                         const C* __restrict__ b, const C* __restrict__ A, int lx,
                                                         int lt, int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    __shared__ C At[5 * D * D];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int V = lx * lt;
    C dyx = czero<C>();
    R dyy = 0;
    for (int site = blockIdx.y; site < V; site += gridDim.y) {
        __syncthreads();
        for (int e = threadIdx.x; e < 5 * D * D; e += blockDim.x) {
            const int dir = e / (D * D), r = e % (D * D), c = r / D, bb = r % D;
            At[(dir * D + bb) * D + c] = A[(long long)site * 5 * D * D + e];
        }
        __syncthreads();
        if (j < N) {
            C acc[D];
#pragma unroll
            for (int c = 0; c < D; ++c) acc[c] = czero<C>();
#pragma unroll 1
            for (int dir = 0; dir < 5; ++dir) {
                const int nb = nbr_site(site, dir, lx, lt);
                const C* xn = x + (long long)nb * D * N + j;
                const C* Ad = At + dir * D * D;
#pragma unroll 4
                for (int bc = 0; bc < D; ++bc) {
                    const C xv = xn[(long long)bc * N];
#pragma unroll
                    for (int c = 0; c < D; ++c) cfma(acc[c], Ad[bc * D + c], xv);
                }
            }
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const long long idx = ((long long)site * D + c) * N + j;
                C o = acc[c];
                if (MODE == 1) o = csub(b[idx], o);
                if (MODE != 3) y[idx] = o;
                if (MODE >= 2) {
                    cfmac(dyx, o, x[idx]);
                    dyy = fma(o.x, o.x, fma(o.y, o.y, dyy));
                }
            }
        }
    }
    if (MODE >= 2) {
        // per-rhs partials: one thread per rhs, no cross-thread reduction needed
        if (j < N) {
            dot_parts<C>(part)[((long long)0 * N + j) * gridDim.y + blockIdx.y] = dot_part(dyx);
            dot_parts<C>(part)[((long long)1 * N + j) * gridDim.y + blockIdx.y] = dot_part(dyy);
        }
    }
}

// FP32 variant with two adjacent right-hand sides per thread: one 16-byte load
// brings x for both, and every shared-memory read of the block serves two rhs.
// Block = 128 threads = 256 rhs.  N must be even.
template <int D, int MODE>
__global__ void __launch_bounds__(128) k_block_stencil_f2(float2* __restrict__ y, const float2* __restrict__ x,
                                                          const float2* __restrict__ b, const float2* __restrict__ A,
                                                          int lx, int lt, int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    __shared__ float2 At[5 * D * D];
    // blockDim.x threads (32..128) x 2 rhs each: blocks of 64 rhs use one-warp CTAs
    const int j = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int V = lx * lt;
    float2 dyx0 = make_float2(0.f, 0.f), dyx1 = make_float2(0.f, 0.f);
    float dyy0 = 0.f, dyy1 = 0.f;
    for (int site = blockIdx.y; site < V; site += gridDim.y) {
        __syncthreads();
        for (int e = threadIdx.x; e < 5 * D * D; e += blockDim.x) {
            const int dir = e / (D * D), r = e % (D * D), c = r / D, bb = r % D;
            At[(dir * D + bb) * D + c] = A[(long long)site * 5 * D * D + e];
        }
        __syncthreads();
        if (j < N) {
            float2 a0[D], a1[D];
#pragma unroll
            for (int c = 0; c < D; ++c) a0[c] = a1[c] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int dir = 0; dir < 5; ++dir) {
                const int nb = nbr_site(site, dir, lx, lt);
                const float2* xn = x + (long long)nb * D * N + j;
                const float2* Ad = At + dir * D * D;
                // the neighbour's rows in groups of 4, loads first (latency of L2 hits)
#pragma unroll 1
                for (int b0 = 0; b0 < D; b0 += 4) {
                    float4 xv[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) xv[q] = *reinterpret_cast<const float4*>(xn + (long long)(b0 + q) * N);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 x0 = make_float2(xv[q].x, xv[q].y), x1 = make_float2(xv[q].z, xv[q].w);
#pragma unroll
                        for (int c = 0; c < D; ++c) {
                            const float2 av = Ad[(b0 + q) * D + c];
                            cfma(a0[c], av, x0);
                            cfma(a1[c], av, x1);
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const long long idx = ((long long)site * D + c) * N + j;
                float2 o0 = a0[c], o1 = a1[c];
                if (MODE == 1) {
                    const float4 bv = *reinterpret_cast<const float4*>(b + idx);
                    o0 = make_float2(bv.x - o0.x, bv.y - o0.y);
                    o1 = make_float2(bv.z - o1.x, bv.w - o1.y);
                }
                if (MODE != 3) *reinterpret_cast<float4*>(y + idx) = make_float4(o0.x, o0.y, o1.x, o1.y);
                if (MODE >= 2) {
                    const float4 xv = *reinterpret_cast<const float4*>(x + idx);
                    cfmac(dyx0, o0, make_float2(xv.x, xv.y));
                    cfmac(dyx1, o1, make_float2(xv.z, xv.w));
                    dyy0 = fmaf(o0.x, o0.x, fmaf(o0.y, o0.y, dyy0));
                    dyy1 = fmaf(o1.x, o1.x, fmaf(o1.y, o1.y, dyy1));
                }
            }
        }
    }
    if (MODE >= 2 && j < N) {
        const long long G = gridDim.y;
        dot_parts<float2>(part)[((long long)0 * N + j) * G + blockIdx.y] = dot_part(dyx0);
        dot_parts<float2>(part)[((long long)0 * N + j + 1) * G + blockIdx.y] = dot_part(dyx1);
        dot_parts<float2>(part)[((long long)1 * N + j) * G + blockIdx.y] = dot_part(dyy0);
        dot_parts<float2>(part)[((long long)1 * N + j + 1) * G + blockIdx.y] = dot_part(dyy1);
    }
}

// FP32 variant for d = 16 with four adjacent right-hand sides per thread and the 16
// output rows of a site split over the two halves of the CTA (half h, uniform per warp,
// computes rows 8h .. 8h + 7).  Each shared-memory read of a block entry serves four
// rhs, 16 FMA per 8 bytes read, twice as many as with two rhs per thread, whose FMA pipe
// waits on the shared-memory reads.  Per output the sums run in the same order as in
// k_block_stencil_f2, so y is the same; the dots (MODE 2, 3) add the two halves last.
// Block = 2 T threads with T = blockDim.x / 2 a multiple of 32; N % 4 == 0.
template <int MODE>
__global__ void __launch_bounds__(128) k_block_stencil_f4(float2* __restrict__ y, const float2* __restrict__ x,
                                                          const float2* __restrict__ b, const float2* __restrict__ A,
                                                          int lx, int lt, int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    constexpr int D = 16, H = 8;
    __shared__ float2 At[5 * D * D];
    __shared__ float red[MODE >= 2 ? 64 * 12 : 1];     // half 1's dots, T <= 64
    const int T = blockDim.x >> 1;
    const int h = threadIdx.x >= T ? 1 : 0;
    const int tq = threadIdx.x - h * T;
    const int j = 4 * (blockIdx.x * T + tq);
    const int V = lx * lt;
    float2 dyx[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    float dyy[4] = {0.f, 0.f, 0.f, 0.f};
    for (int site = blockIdx.y; site < V; site += gridDim.y) {
        __syncthreads();
        for (int e = threadIdx.x; e < 5 * D * D; e += blockDim.x) {
            const int dir = e / (D * D), r = e % (D * D), c = r / D, bb = r % D;
            At[(dir * D + bb) * D + c] = A[(long long)site * 5 * D * D + e];
        }
        __syncthreads();
        if (j < N) {
            float2 a[H][4];
#pragma unroll
            for (int c = 0; c < H; ++c)
#pragma unroll
                for (int r = 0; r < 4; ++r) a[c][r] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int dir = 0; dir < 5; ++dir) {
                const int nb = nbr_site(site, dir, lx, lt);
                const float2* xn = x + (long long)nb * D * N + j;
                const float2* Ad = At + dir * D * D + h * H;
                // the neighbour's rows in groups of 4, loads first (latency of L2 hits)
#pragma unroll 1
                for (int b0 = 0; b0 < D; b0 += 4) {
                    float4 xv[4][2];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        xv[q][0] = *reinterpret_cast<const float4*>(xn + (long long)(b0 + q) * N);
                        xv[q][1] = *reinterpret_cast<const float4*>(xn + (long long)(b0 + q) * N + 2);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 x0 = make_float2(xv[q][0].x, xv[q][0].y), x1 = make_float2(xv[q][0].z, xv[q][0].w);
                        const float2 x2 = make_float2(xv[q][1].x, xv[q][1].y), x3 = make_float2(xv[q][1].z, xv[q][1].w);
#pragma unroll
                        for (int c = 0; c < H; ++c) {
                            const float2 av = Ad[(b0 + q) * D + c];
                            cfma(a[c][0], av, x0);
                            cfma(a[c][1], av, x1);
                            cfma(a[c][2], av, x2);
                            cfma(a[c][3], av, x3);
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < H; ++c) {
                const long long idx = ((long long)site * D + h * H + c) * N + j;
                float2 o[4] = {a[c][0], a[c][1], a[c][2], a[c][3]};
                if (MODE == 1) {
                    const float4 b0v = *reinterpret_cast<const float4*>(b + idx);
                    const float4 b1v = *reinterpret_cast<const float4*>(b + idx + 2);
                    o[0] = make_float2(b0v.x - o[0].x, b0v.y - o[0].y);
                    o[1] = make_float2(b0v.z - o[1].x, b0v.w - o[1].y);
                    o[2] = make_float2(b1v.x - o[2].x, b1v.y - o[2].y);
                    o[3] = make_float2(b1v.z - o[3].x, b1v.w - o[3].y);
                }
                if (MODE != 3) {
                    *reinterpret_cast<float4*>(y + idx) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                    *reinterpret_cast<float4*>(y + idx + 2) = make_float4(o[2].x, o[2].y, o[3].x, o[3].y);
                }
                if (MODE >= 2) {
                    const float4 x0v = *reinterpret_cast<const float4*>(x + idx);
                    const float4 x1v = *reinterpret_cast<const float4*>(x + idx + 2);
                    const float2 xs[4] = {make_float2(x0v.x, x0v.y), make_float2(x0v.z, x0v.w),
                                          make_float2(x1v.x, x1v.y), make_float2(x1v.z, x1v.w)};
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        cfmac(dyx[r], o[r], xs[r]);
                        dyy[r] = fmaf(o[r].x, o[r].x, fmaf(o[r].y, o[r].y, dyy[r]));
                    }
                }
            }
        }
    }
    if (MODE >= 2) {
        // half 1 hands its sums to half 0, which writes the per-rhs partials
        if (h == 1)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                red[tq * 12 + 3 * r] = dyx[r].x;
                red[tq * 12 + 3 * r + 1] = dyx[r].y;
                red[tq * 12 + 3 * r + 2] = dyy[r];
            }
        __syncthreads();
        if (h == 0 && j < N) {
            const long long G = gridDim.y;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float2 s = make_float2(dyx[r].x + red[tq * 12 + 3 * r], dyx[r].y + red[tq * 12 + 3 * r + 1]);
                dot_parts<float2>(part)[((long long)0 * N + j + r) * G + blockIdx.y] = dot_part(s);
                dot_parts<float2>(part)[((long long)1 * N + j + r) * G + blockIdx.y] =
                    dot_part(dyy[r] + red[tq * 12 + 3 * r + 2]);
            }
        }
    }
}

// Narrow-block variant (few rhs, as in the setup solves): thread (tx < 8 rhs,
// ty < D output row); the blocks of the site are staged in shared memory.
template <typename C, int D, int MODE>
__global__ void __launch_bounds__(8 * D) k_block_stencil_narrow(C* __restrict__ y, const C* __restrict__ x,
                                                                const C* __restrict__ b, const C* __restrict__ A,
                                                                int lx, int lt, int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    using R = re_t<C>;
    __shared__ C As[5 * D * (D + 1)];             // rows padded: the four rows of a warp in different banks
    __shared__ dot_t<C> red[2][D][8];
    const int tx = threadIdx.x, c = threadIdx.y, tid = c * 8 + tx;
    const int j = blockIdx.x * 8 + tx;
    const int V = lx * lt;
    C dyx = czero<C>();
    R dyy = 0;
    for (int site = blockIdx.y; site < V; site += gridDim.y) {
        // FP32: the five neighbours' rows all in flight while the blocks are staged (one after
        // another they were five round trips: 9 us a launch, 3 now)
        constexpr int PRE = sizeof(C) == 8 ? 5 : 1;
        C xv[PRE][D];
        if (PRE == 5 && j < N)
#pragma unroll
            for (int dir = 0; dir < PRE; ++dir) {
                const C* xn = x + (long long)nbr_site(site, dir, lx, lt) * D * N + j;
#pragma unroll
                for (int bc = 0; bc < D; ++bc) xv[dir][bc] = xn[(long long)bc * N];
            }
        __syncthreads();
        for (int e = tid; e < 5 * D * D; e += 8 * D) As[(e / D) * (D + 1) + e % D] = A[(long long)site * 5 * D * D + e];
        __syncthreads();
        if (j < N) {
            C acc = czero<C>();
#pragma unroll
            for (int dir = 0; dir < 5; ++dir) {
                const C* Ar = As + (dir * D + c) * (D + 1);
                if (PRE == 1) {
                    const C* xn = x + (long long)nbr_site(site, dir, lx, lt) * D * N + j;
#pragma unroll
                    for (int bc = 0; bc < D; ++bc) xv[0][bc] = xn[(long long)bc * N];
                }
#pragma unroll
                for (int bc = 0; bc < D; ++bc) cfma(acc, Ar[bc], xv[PRE == 5 ? dir : 0][bc]);
            }
            const long long idx = ((long long)site * D + c) * N + j;
            if (MODE == 1) acc = csub(b[idx], acc);
            if (MODE != 3) y[idx] = acc;
            if (MODE >= 2) {
                cfmac(dyx, acc, x[idx]);
                dyy = fma(acc.x, acc.x, fma(acc.y, acc.y, dyy));
            }
        }
    }
    if (MODE >= 2) {
        red[0][c][tx] = dot_part(dyx);
        red[1][c][tx] = dot_part(dyy);
        __syncthreads();
        if (c < 2 && j < N) {
            dot_t<C> s2 = red[c][0][tx];
            for (int r = 1; r < D; ++r) s2 = dot_add(s2, red[c][r][tx]);
            dot_parts<C>(part)[((long long)c * N + j) * gridDim.y + blockIdx.y] = s2;
        }
    }
}

// y[s] (+)= Minv[s] sum_q alpha_q x_q[s] over the K residuals x_q of a group of smoother
// steps (slots of the block x; K = 1 and no alpha: the plain product): block = 128 rhs,
// one site per iteration, Minv[s] in shared memory; generic d (<= 32).
template <typename C>
__device__ __forceinline__ C step_sum(const C* __restrict__ x, size_t slot, int K, const C* __restrict__ alpha,
                                      long long idx, int j, int N) {
    if (!alpha) return x[idx];
    C acc = czero<C>();
    for (int q = 0; q < K; ++q) cfma(acc, alpha[q * N + j], x[q * slot + idx]);
    return acc;
}

template <typename C>
__global__ void __launch_bounds__(128) k_block_diag_apply(C* __restrict__ y, const C* __restrict__ x, size_t slot,
                                                          int K, const C* __restrict__ alpha,
                                                          const C* __restrict__ Minv, int nsites, int d, int N,
                                                          bool accumulate) {
    if (grid_dependency()) return;
    __shared__ C Ms[32 * 32];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    for (int site = blockIdx.y; site < nsites; site += gridDim.y) {
        __syncthreads();
        for (int e = threadIdx.x; e < d * d; e += blockDim.x) Ms[e] = Minv[(long long)site * d * d + e];
        __syncthreads();
        if (j >= N) continue;
        C xv[32];
        for (int b = 0; b < d; ++b) xv[b] = step_sum(x, slot, K, alpha, ((long long)site * d + b) * N + j, j, N);
        for (int c = 0; c < d; ++c) {
            C acc = accumulate ? y[((long long)site * d + c) * N + j] : czero<C>();
            for (int b = 0; b < d; ++b) cfma(acc, Ms[c * d + b], xv[b]);
            y[((long long)site * d + c) * N + j] = acc;
        }
    }
}

// The same with the block size fixed at compile time: the input column stays in
// registers (a runtime d puts it in local memory), all loads issued before the FMAs.
template <typename C, int D>
__global__ void __launch_bounds__(128) k_block_diag_apply_d(C* __restrict__ y, const C* __restrict__ x, size_t slot,
                                                            int K, const C* __restrict__ alpha,
                                                            const C* __restrict__ Minv, int nsites, int N,
                                                            bool accumulate) {
    if (grid_dependency()) return;
    __shared__ C Ms[D * D];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    for (int site = blockIdx.y; site < nsites; site += gridDim.y) {
        __syncthreads();
        for (int e = threadIdx.x; e < D * D; e += blockDim.x) Ms[e] = Minv[(long long)site * D * D + e];
        __syncthreads();
        if (j >= N) continue;
        C xv[D], acc[D];
        const long long base = (long long)site * D * N + j;
        if (alpha) {
#pragma unroll
            for (int b = 0; b < D; ++b) xv[b] = czero<C>();
            for (int q = 0; q < K; ++q) {
                const C a = alpha[q * N + j];
#pragma unroll
                for (int b = 0; b < D; ++b) cfma(xv[b], a, x[q * slot + base + (long long)b * N]);
            }
        } else {
#pragma unroll
            for (int b = 0; b < D; ++b) xv[b] = x[base + (long long)b * N];
        }
#pragma unroll
        for (int b = 0; b < D; ++b) acc[b] = accumulate ? y[base + (long long)b * N] : czero<C>();
#pragma unroll
        for (int c = 0; c < D; ++c) {
#pragma unroll
            for (int b = 0; b < D; ++b) cfma(acc[c], Ms[c * D + b], xv[b]);
            y[base + (long long)c * N] = acc[c];
        }
    }
}

template <typename C>
void launch_block_diag_combine(C* y, const C* x, size_t slot, int K, const C* alpha, const C* Minv, int nsites, int d,
                               int N, bool accumulate, cudaStream_t s) {
    MG_REQUIRE(d <= 32, MGMLMC_EINVAL, "block-diagonal apply: d <= 32");
    const int th = cta_threads(N);
    const int tiles = (N + th - 1) / th;
    int G = 16 * kNumSM / tiles;
    if (G > nsites) G = nsites;
    if (G < 1) G = 1;
    const dim3 g(tiles, G);
    if (d == 16) MG_LAUNCH(g, th, 0, s, (k_block_diag_apply_d<C, 16>), y, x, slot, K, alpha, Minv, nsites, N, accumulate);
    else if (d == 8) MG_LAUNCH(g, th, 0, s, (k_block_diag_apply_d<C, 8>), y, x, slot, K, alpha, Minv, nsites, N, accumulate);
    else MG_LAUNCH(g, th, 0, s, (k_block_diag_apply<C>), y, x, slot, K, alpha, Minv, nsites, d, N, accumulate);
    MG_LAUNCHED();
}

template <typename C>
void launch_block_diag_apply(C* y, const C* x, const C* Minv, int nsites, int d, int N, bool accumulate,
                             cudaStream_t s) {
    launch_block_diag_combine<C>(y, x, 0, 1, nullptr, Minv, nsites, d, N, accumulate, s);
}

// xc[S][o] = sum_{site in S} sum_{a in spin block s(o)} conj(P[site][a][j(o)]) x[site][a]
template <typename C>
__global__ void k_restrict(C* __restrict__ xc, const C* __restrict__ x, const C* __restrict__ P, int lx, int lt,
                           int d, int ax, int at, int nvec, int N) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    const int cx = lx / ax, ct = lt / at, dc = 2 * nvec, hd = d / 2;
    for (int S = blockIdx.y; S < cx * ct; S += gridDim.y) {
        const int X = S % cx, T = S / cx;
        for (int o = threadIdx.y; o < dc; o += kRowLanes) {
            const int s = o / nvec, jv = o % nvec;
            C acc = czero<C>();
            for (int it = 0; it < at; ++it)
                for (int ix = 0; ix < ax; ++ix) {
                    const int site = (X * ax + ix) + lx * (T * at + it);
                    for (int a = s * hd; a < (s + 1) * hd; ++a)
                        cfmac(acc, P[((long long)site * d + a) * nvec + jv], x[((long long)site * d + a) * N + j]);
                }
            xc[((long long)S * dc + o) * N + j] = acc;
        }
    }
}

// x[site][a] (+)= sum_j P[site][a][j] xc[S(site)][s(a) nvec + j]
template <typename C>
__global__ void k_prolong(C* __restrict__ x, const C* __restrict__ xc, const C* __restrict__ P, int lx, int lt,
                          int d, int ax, int at, int nvec, int N, bool accumulate) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    const int cx = lx / ax, dc = 2 * nvec, hd = d / 2;
    const long long rows = (long long)lx * lt * d;
    for (long long row = (long long)blockIdx.y * kRowLanes + threadIdx.y; row < rows;
         row += (long long)gridDim.y * kRowLanes) {
        const int site = (int)(row / d), a = (int)(row % d);
        const int xx = site % lx, t = site / lx;
        const int S = xx / ax + cx * (t / at);
        const int s = a / hd;
        C acc = accumulate ? x[row * N + j] : czero<C>();
        const C* Pr = P + row * nvec;
        const C* xcs = xc + ((long long)S * dc + s * nvec) * N + j;
        for (int jv = 0; jv < nvec; ++jv) cfma(acc, Pr[jv], xcs[(long long)jv * N]);
        x[row * N + j] = acc;
    }
}

// Aggregate-per-block restriction / prolongation for compile-time nvec: block =
// 128 rhs, one coarse site S per block iteration; P restricted to S (ax*at*d*nvec
// values) staged in shared memory; each thread reads every fine value of its rhs
// once and keeps the 2 nvec coarse values in registers.
template <typename C, int NV>
__global__ void __launch_bounds__(128) k_restrict_nv(C* __restrict__ xc, const C* __restrict__ x,
                                                     const C* __restrict__ P, int lx, int lt, int d, int ax, int at,
                                                     int N) {
    if (grid_dependency()) return;
    extern __shared__ __align__(16) unsigned char smem_rp[];
    C* Ps = reinterpret_cast<C*>(smem_rp);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int cx = lx / ax, ct = lt / at, hd = d / 2, na = ax * at;
    const int nP = na * d * NV;
    for (int S = blockIdx.y; S < cx * ct; S += gridDim.y) {
        const int X = S % cx, T = S / cx;
        __syncthreads();
        for (int e = threadIdx.x; e < nP; e += blockDim.x) {
            const int q = e / (d * NV), r = e % (d * NV);
            const int site = (X * ax + q % ax) + lx * (T * at + q / ax);
            Ps[e] = P[(long long)site * d * NV + r];
        }
        __syncthreads();
        if (j >= N) continue;
        C acc[2 * NV];
#pragma unroll
        for (int o = 0; o < 2 * NV; ++o) acc[o] = czero<C>();
        for (int q = 0; q < na; ++q) {
            const int site = (X * ax + q % ax) + lx * (T * at + q / ax);
            const C* xs = x + (long long)site * d * N + j;
            const C* Pq = Ps + q * d * NV;
            for (int a = 0; a < d; ++a) {
                const C xv = xs[(long long)a * N];
                const C* Pa = Pq + a * NV;
                if (a < hd) {
#pragma unroll
                    for (int jv = 0; jv < NV; ++jv) cfmac(acc[jv], Pa[jv], xv);
                } else {
#pragma unroll
                    for (int jv = 0; jv < NV; ++jv) cfmac(acc[NV + jv], Pa[jv], xv);
                }
            }
        }
#pragma unroll
        for (int o = 0; o < 2 * NV; ++o) xc[((long long)S * 2 * NV + o) * N + j] = acc[o];
    }
}

template <typename C, int NV>
__global__ void __launch_bounds__(128) k_prolong_nv(C* __restrict__ x, const C* __restrict__ xc,
                                                    const C* __restrict__ P, int lx, int lt, int d, int ax, int at,
                                                    int N, bool accumulate) {
    if (grid_dependency()) return;
    extern __shared__ __align__(16) unsigned char smem_rp[];
    C* Ps = reinterpret_cast<C*>(smem_rp);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int cx = lx / ax, ct = lt / at, hd = d / 2, na = ax * at;
    const int nP = na * d * NV;
    for (int S = blockIdx.y; S < cx * ct; S += gridDim.y) {
        const int X = S % cx, T = S / cx;
        __syncthreads();
        for (int e = threadIdx.x; e < nP; e += blockDim.x) {
            const int q = e / (d * NV), r = e % (d * NV);
            const int site = (X * ax + q % ax) + lx * (T * at + q / ax);
            Ps[e] = P[(long long)site * d * NV + r];
        }
        __syncthreads();
        if (j >= N) continue;
        C cv[2 * NV];
#pragma unroll
        for (int o = 0; o < 2 * NV; ++o) cv[o] = xc[((long long)S * 2 * NV + o) * N + j];
        for (int q = 0; q < na; ++q) {
            const int site = (X * ax + q % ax) + lx * (T * at + q / ax);
            C* xs = x + (long long)site * d * N + j;
            const C* Pq = Ps + q * d * NV;
            for (int a = 0; a < d; ++a) {
                const C* Pa = Pq + a * NV;
                C acc = accumulate ? xs[(long long)a * N] : czero<C>();
                if (a < hd) {
#pragma unroll
                    for (int jv = 0; jv < NV; ++jv) cfma(acc, Pa[jv], cv[jv]);
                } else {
#pragma unroll
                    for (int jv = 0; jv < NV; ++jv) cfma(acc, Pa[jv], cv[NV + jv]);
                }
                xs[(long long)a * N] = acc;
            }
        }
    }
}

// Row j of a site's BF16 operand tile (128 rhs x 16 complex values, K-major core
// matrices of 8 rows x 16 bytes: the layout of the tensor-core stencil).
__device__ __forceinline__ void store_bf16_row(uint8_t* xt, int site, int j, int N, const float2* v) {
    const int T = (N + 127) / 128, r = j & 127;
    uint8_t* row = xt + ((size_t)site * T + (j >> 7)) * 8192 + (r >> 3) * 512 + (r & 7) * 16;
#pragma unroll
    for (int cg = 0; cg < 4; ++cg)
        *reinterpret_cast<uint4*>(row + cg * 128) =
            make_uint4(f2_bf(v[4 * cg]), f2_bf(v[4 * cg + 1]), f2_bf(v[4 * cg + 2]), f2_bf(v[4 * cg + 3]));
}

// The same two operators with the dofs per fine site (D) fixed at compile time: the
// loads of QB aggregate sites (QB * D values per rhs) are issued together before the FMAs,
// instead of one load per loop trip.  V adjacent rhs per thread (FP32: 2 where N is even, in
// 16-byte accesses): each value takes NV coefficients from shared memory, and with one rhs a
// read that pipe, not HBM, set the time (restriction of a d = 16 level of 128^2 sites x 128 rhs:
// 55 us of reads against 42 us of HBM).
template <typename C, int V> struct alignas(sizeof(C) * V) RhsOf { C v[V]; };

template <typename C, int NV, int D, int QB, int V>
__global__ void __launch_bounds__(128) k_restrict_nvd(C* __restrict__ xc, const C* __restrict__ x,
                                                      const C* __restrict__ P, int lx, int lt, int ax, int at, int N) {
    if (grid_dependency()) return;
    extern __shared__ __align__(16) unsigned char smem_rp[];
    C* Ps = reinterpret_cast<C*>(smem_rp);
    constexpr int HD = D / 2;
    using X = RhsOf<C, V>;
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const int cx = lx / ax, ct = lt / at, na = ax * at;
    const int nP = na * D * NV;
    for (int S = blockIdx.y; S < cx * ct; S += gridDim.y) {
        const int Xc = S % cx, T = S / cx;
        __syncthreads();
        for (int e = threadIdx.x; e < nP; e += blockDim.x) {
            const int q = e / (D * NV), r = e % (D * NV);
            const int site = (Xc * ax + q % ax) + lx * (T * at + q / ax);
            Ps[e] = P[(long long)site * D * NV + r];
        }
        __syncthreads();
        if (j >= N) continue;
        X acc[2 * NV];
#pragma unroll
        for (int o = 0; o < 2 * NV; ++o)
#pragma unroll
            for (int u = 0; u < V; ++u) acc[o].v[u] = czero<C>();
        for (int q0 = 0; q0 < na; q0 += QB) {
            X xv[QB][D];
#pragma unroll
            for (int qq = 0; qq < QB; ++qq) {
                const int q = q0 + qq;
                const int site = (Xc * ax + q % ax) + lx * (T * at + q / ax);
#pragma unroll
                for (int a = 0; a < D; ++a)
                    if (q < na) xv[qq][a] = *reinterpret_cast<const X*>(x + ((long long)site * D + a) * N + j);
            }
#pragma unroll
            for (int qq = 0; qq < QB; ++qq) {
                if (q0 + qq >= na) break;
                const C* Pq = Ps + (q0 + qq) * D * NV;
#pragma unroll
                for (int a = 0; a < D; ++a)
#pragma unroll
                    for (int jv = 0; jv < NV; ++jv) {
                        const C p = Pq[a * NV + jv];
#pragma unroll
                        for (int u = 0; u < V; ++u) cfmac(acc[(a < HD ? 0 : NV) + jv].v[u], p, xv[qq][a].v[u]);
                    }
            }
        }
#pragma unroll
        for (int o = 0; o < 2 * NV; ++o) *reinterpret_cast<X*>(xc + ((long long)S * 2 * NV + o) * N + j) = acc[o];
    }
}

// xt (FP32, D = 16; may be null): the BF16 operand tiles of the result as well (the
// tensor-core residual reads them), so that no pass over x packs them later.  SPLIT: the fine
// sites of an aggregate are shared out over threadIdx.y where the rhs leave room in a CTA of 128
// threads (8 rhs of a 64^2 lattice: d = 16 5.6 -> 3.6 us, fine level 5.9 -> 3.2).
template <typename C, int NV, int D, int QB, int V, bool SPLIT>
__global__ void __launch_bounds__(128) k_prolong_nvd(C* __restrict__ x, const C* __restrict__ xc,
                                                     const C* __restrict__ P, int lx, int lt, int ax, int at, int N,
                                                     bool accumulate, uint8_t* __restrict__ xt) {
    if (grid_dependency()) return;
    extern __shared__ __align__(16) unsigned char smem_rp[];
    C* Ps = reinterpret_cast<C*>(smem_rp);
    constexpr int HD = D / 2;
    using X = RhsOf<C, V>;
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const int cx = lx / ax, ct = lt / at, na = ax * at;
    const int nP = na * D * NV;
    const int y0 = SPLIT ? threadIdx.y : 0, ny = SPLIT ? blockDim.y : 1;
    for (int S = blockIdx.y; S < cx * ct; S += gridDim.y) {
        const int Xc = S % cx, T = S / cx;
        __syncthreads();
        for (int e = y0 * blockDim.x + threadIdx.x; e < nP; e += ny * blockDim.x) {
            const int q = e / (D * NV), r = e % (D * NV);
            const int site = (Xc * ax + q % ax) + lx * (T * at + q / ax);
            Ps[e] = P[(long long)site * D * NV + r];
        }
        __syncthreads();
        if (j >= N) continue;
        X cv[2 * NV];
#pragma unroll
        for (int o = 0; o < 2 * NV; ++o) cv[o] = *reinterpret_cast<const X*>(xc + ((long long)S * 2 * NV + o) * N + j);
        for (int q0 = QB * y0; q0 < na; q0 += QB * ny) {
            X ov[QB][D];
#pragma unroll
            for (int qq = 0; qq < QB; ++qq) {
                const int q = q0 + qq;
                const int site = (Xc * ax + q % ax) + lx * (T * at + q / ax);
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    if (accumulate && q < na)
                        ov[qq][a] = *reinterpret_cast<const X*>(x + ((long long)site * D + a) * N + j);
                    else
#pragma unroll
                        for (int u = 0; u < V; ++u) ov[qq][a].v[u] = czero<C>();
                }
            }
#pragma unroll
            for (int qq = 0; qq < QB; ++qq) {
                const int q = q0 + qq;
                if (q >= na) break;
                const int site = (Xc * ax + q % ax) + lx * (T * at + q / ax);
                const C* Pq = Ps + q * D * NV;
#pragma unroll
                for (int a = 0; a < D; ++a) {
#pragma unroll
                    for (int jv = 0; jv < NV; ++jv) {
                        const C p = Pq[a * NV + jv];
#pragma unroll
                        for (int u = 0; u < V; ++u) cfma(ov[qq][a].v[u], p, cv[(a < HD ? 0 : NV) + jv].v[u]);
                    }
                    *reinterpret_cast<X*>(x + ((long long)site * D + a) * N + j) = ov[qq][a];
                }
                if constexpr (sizeof(C) == 8 && D == 16) {
                    if (xt)
#pragma unroll
                        for (int u = 0; u < V; ++u) {
                            float2 row[D];
#pragma unroll
                            for (int a = 0; a < D; ++a) row[a] = ov[qq][a].v[u];
                            store_bf16_row(xt, site, j + u, N, row);
                        }
                }
            }
        }
    }
}

// The minimal-residual smoother keeps the residuals r_0 .. r_{K-1} of a group of steps
// (rs, one slot of n x N each) and adds sum_s alpha_s r_s to the correction once per
// group, instead of reading and writing the correction in every step: a step moves r and
// p in and the next r out (3 vectors instead of 5), and the last step of all forms no
// residual.  The sums run over the steps in order, as the step-by-step updates did.
// All are bound by HBM (or L2); V values of one row per thread in 16-byte accesses where
// N allows.  A block is bx x (256 / bx) threads with bx the power of two that covers the
// N / V columns (at most 32), so that narrow blocks keep every lane busy.
template <typename T, int V> struct alignas(sizeof(T) * V) VecOf { T v[V]; };

// rn = r - alpha p (rn may be r: every value is read before its place is written)
template <typename C, int V>
__global__ void __launch_bounds__(256) k_mr_update(C* rn, const C* r, const C* __restrict__ p,
                                                   const C* __restrict__ alpha, long long n, int N) {
    if (grid_dependency()) return;
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    if (j >= N) return;
    C a[V];
#pragma unroll
    for (int q = 0; q < V; ++q) a[q] = alpha[j + q];
    const long long S = (long long)gridDim.y * blockDim.y;
    for (long long i0 = (long long)blockIdx.y * blockDim.y + threadIdx.y; i0 < n; i0 += 2 * S) {
        VecOf<C, V> rv[2], pv[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const long long i = i0 + u * S;
            if (i < n) {
                rv[u] = *reinterpret_cast<const VecOf<C, V>*>(r + i * N + j);
                pv[u] = *reinterpret_cast<const VecOf<C, V>*>(p + i * N + j);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const long long i = i0 + u * S;
            if (i < n) {
#pragma unroll
                for (int q = 0; q < V; ++q) rv[u].v[q] = csub(rv[u].v[q], cmul(a[q], pv[u].v[q]));
                *reinterpret_cast<VecOf<C, V>*>(rn + i * N + j) = rv[u];
            }
        }
    }
}

// e (=|+=) sum_{s < K} alpha_s r_s
constexpr int kMrGroup = kSmootherGroup;
template <typename C, int V>
__global__ void __launch_bounds__(256) k_mr_combine(C* __restrict__ e, const C* __restrict__ rs, size_t slot, int K,
                                                    const C* __restrict__ alpha, long long n, int N, bool e_is_zero) {
    if (grid_dependency()) return;
    const int j = V * (blockIdx.x * blockDim.x + threadIdx.x);
    if (j >= N) return;
    for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n;
         i += (long long)gridDim.y * blockDim.y) {
        VecOf<C, V> rv[kMrGroup], ev;
#pragma unroll
        for (int s = 0; s < kMrGroup; ++s)
            if (s < K) rv[s] = *reinterpret_cast<const VecOf<C, V>*>(rs + s * slot + i * N + j);
        if (!e_is_zero) ev = *reinterpret_cast<const VecOf<C, V>*>(e + i * N + j);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            C acc = e_is_zero ? czero<C>() : ev.v[q];
#pragma unroll
            for (int s = 0; s < kMrGroup; ++s)
                if (s < K) cfma(acc, alpha[s * N + j + q], rv[s].v[q]);
            ev.v[q] = acc;
        }
        *reinterpret_cast<VecOf<C, V>*>(e + i * N + j) = ev;
    }
}

// The same two (the sum always adds to e) with the residuals and the image in BF16 (one bf16x2 word per complex
// value), four rhs per thread: 16-byte accesses.  N % 4 == 0.
__global__ void __launch_bounds__(256) k_mr_update_fine_bf16(uint32_t* rn, const uint32_t* r,
                                                             const uint32_t* __restrict__ p,
                                                             const float2* __restrict__ alpha, long long n, int N) {
    if (grid_dependency()) return;
    const int j = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (j >= N) return;
    float2 a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = alpha[j + q];
    const long long S = (long long)gridDim.y * blockDim.y;
    for (long long i0 = (long long)blockIdx.y * blockDim.y + threadIdx.y; i0 < n; i0 += 2 * S) {
        VecOf<uint32_t, 4> rv[2], pv[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const long long i = i0 + u * S;
            if (i < n) {
                rv[u] = *reinterpret_cast<const VecOf<uint32_t, 4>*>(r + i * N + j);
                pv[u] = *reinterpret_cast<const VecOf<uint32_t, 4>*>(p + i * N + j);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const long long i = i0 + u * S;
            if (i < n) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    rv[u].v[q] = f2_bf(csub(bf2_lo(rv[u].v[q]), cmul(a[q], bf2_lo(pv[u].v[q]))));
                *reinterpret_cast<VecOf<uint32_t, 4>*>(rn + i * N + j) = rv[u];
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_mr_combine_bf16(float2* __restrict__ e, const uint32_t* __restrict__ rs,
                                                         size_t slot, int K, const float2* __restrict__ alpha,
                                                         long long n, int N) {
    if (grid_dependency()) return;
    const int j = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (j >= N) return;
    for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n;
         i += (long long)gridDim.y * blockDim.y) {
        VecOf<uint32_t, 4> rv[kMrGroup];
        VecOf<float2, 2> ev[2];
        float2* er = e + i * N + j;
#pragma unroll
        for (int s = 0; s < kMrGroup; ++s)
            if (s < K) rv[s] = *reinterpret_cast<const VecOf<uint32_t, 4>*>(rs + s * slot + i * N + j);
        ev[0] = *reinterpret_cast<const VecOf<float2, 2>*>(er);
        ev[1] = *reinterpret_cast<const VecOf<float2, 2>*>(er + 2);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float2 acc = ev[q >> 1].v[q & 1];
#pragma unroll
            for (int s = 0; s < kMrGroup; ++s)
                if (s < K) cfma(acc, alpha[s * N + j + q], bf2_lo(rv[s].v[q]));
            ev[q >> 1].v[q & 1] = acc;
        }
        *reinterpret_cast<VecOf<float2, 2>*>(er) = ev[0];
        *reinterpret_cast<VecOf<float2, 2>*>(er + 2) = ev[1];
    }
}

template <typename C>
__global__ void k_gamma5(C* __restrict__ y, const C* __restrict__ x, long long rows, int d, int N) {
    if (grid_dependency()) return;
    const int j = blockIdx.x * kRhsTile + threadIdx.x;
    if (j >= N) return;
    for (long long i = (long long)blockIdx.y * kRowLanes + threadIdx.y; i < rows;
         i += (long long)gridDim.y * kRowLanes) {
        const C v = x[i * N + j];
        y[i * N + j] = ((int)(i % d) < d / 2) ? v : mk(-v.x, -v.y);
    }
}

// --------------------------------------------------------------------- launchers
static inline dim3 blk() { return dim3(kRhsTile, kRowLanes); }

int stencil_groups(int nsites, int N) { return row_groups(nsites, N, 8); }
// k_wilson_bf16 launches N / 128 (four rhs per thread) or N / 64 column blocks of 256
// threads, three resident per SM: row groups for one wave of three CTAs per SM.
int stencil_groups_bf16(int nsites, int N) {
    const int gx = (N % 128 == 0) ? N / 128 : (N / 2 + kRhsTile - 1) / kRhsTile;
    const long long need = (nsites + kRowLanes - 1) / kRowLanes;
    return (int)std::max(1LL, std::min(need, 3LL * kNumSM / gx));
}


// FP32 Wilson operator with two rhs per thread: 16-byte loads and stores (a warp
// moves 512 B per access), half the index arithmetic per rhs.  N even.
// MODE 4: the residual b - D x rounded to BF16 (one bf16x2 word per complex value).
template <int MODE>
__global__ void __launch_bounds__(256) k_wilson_f2(float2* __restrict__ y, const float2* __restrict__ x,
                                                   const float2* __restrict__ b, const float2* __restrict__ U,
                                                   float mass, int lx, int lt, int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    const int j = 2 * (blockIdx.x * kRhsTile + threadIdx.x);
    const int V = lx * lt;
    float2 dyx[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    float dyy[2] = {0.f, 0.f};
    auto ld2 = [&](const float2* base, long long idx, float2& a, float2& c) {
        const float4 v = *reinterpret_cast<const float4*>(base + idx);
        a = make_float2(v.x, v.y);
        c = make_float2(v.z, v.w);
    };
    if (j < N) {
        const long long N2 = 2LL * N;
        for (int site = blockIdx.y * kRowLanes + threadIdx.y; site < V; site += gridDim.y * kRowLanes) {
            const int xx = site % lx, t = site / lx;
            const int sxp = (xx + 1 == lx ? 0 : xx + 1) + lx * t;
            const int sxm = (xx == 0 ? lx - 1 : xx - 1) + lx * t;
            const int stp = xx + lx * (t + 1 == lt ? 0 : t + 1);
            const int stm = xx + lx * (t == 0 ? lt - 1 : t - 1);
            const float sgp = (t + 1 == lt) ? -0.5f : 0.5f;   // antiperiodic time boundary, times 1/2
            const float sgm = (t == 0) ? -0.5f : 0.5f;
            const float2 u0 = U[2 * site], u1 = U[2 * site + 1];
            const float2 u0m = U[2 * sxm], u1m = U[2 * stm + 1];
            float2 p0[2], p1[2], a0[2], a1[2], c0[2], c1[2], e0[2], e1[2], f0[2], f1[2];
            ld2(x, site * N2 + j, p0[0], p0[1]);
            ld2(x, site * N2 + N + j, p1[0], p1[1]);
            ld2(x, sxp * N2 + j, a0[0], a0[1]);
            ld2(x, sxp * N2 + N + j, a1[0], a1[1]);
            ld2(x, sxm * N2 + j, c0[0], c0[1]);
            ld2(x, sxm * N2 + N + j, c1[0], c1[1]);
            ld2(x, stp * N2 + j, e0[0], e0[1]);
            ld2(x, stp * N2 + N + j, e1[0], e1[1]);
            ld2(x, stm * N2 + j, f0[0], f0[1]);
            ld2(x, stm * N2 + N + j, f1[0], f1[1]);
            float2 o0[2], o1[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                o0[r] = mk(mass * p0[r].x, mass * p0[r].y);
                o1[r] = mk(mass * p1[r].x, mass * p1[r].y);
                {   // +x: (1 - sigma_1) psi = (a, -a), a = psi0 - psi1
                    const float2 u = cscale(cmul(u0, csub(a0[r], a1[r])), 0.5f);
                    o0[r] = csub(o0[r], u);
                    o1[r] = cadd(o1[r], u);
                }
                {   // -x: (1 + sigma_1) psi = (c, c), c = psi0 + psi1
                    const float2 u = cscale(cmulc(u0m, cadd(c0[r], c1[r])), 0.5f);
                    o0[r] = csub(o0[r], u);
                    o1[r] = csub(o1[r], u);
                }
                {   // +t: (1 - sigma_2) psi = (a, -i a), a = psi0 + i psi1
                    const float2 u = cscale(cmul(u1, cadd(e0[r], ctimesi(e1[r]))), sgp);
                    o0[r] = csub(o0[r], u);
                    o1[r] = cadd(o1[r], ctimesi(u));
                }
                {   // -t: (1 + sigma_2) psi = (c, i c), c = psi0 - i psi1
                    const float2 u = cscale(cmulc(u1m, csub(f0[r], ctimesi(f1[r]))), sgm);
                    o0[r] = csub(o0[r], u);
                    o1[r] = csub(o1[r], ctimesi(u));
                }
            }
            if (MODE == 1 || MODE == 4) {
                float2 b0[2], b1[2];
                ld2(b, site * N2 + j, b0[0], b0[1]);
                ld2(b, site * N2 + N + j, b1[0], b1[1]);
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    o0[r] = csub(b0[r], o0[r]);
                    o1[r] = csub(b1[r], o1[r]);
                }
            }
            if (MODE == 4) {
                uint32_t* yb = reinterpret_cast<uint32_t*>(y);
                *reinterpret_cast<uint2*>(yb + site * N2 + j) = make_uint2(f2_bf(o0[0]), f2_bf(o0[1]));
                *reinterpret_cast<uint2*>(yb + site * N2 + N + j) = make_uint2(f2_bf(o1[0]), f2_bf(o1[1]));
            } else if (MODE != 3) {
                *reinterpret_cast<float4*>(y + site * N2 + j) = make_float4(o0[0].x, o0[0].y, o0[1].x, o0[1].y);
                *reinterpret_cast<float4*>(y + site * N2 + N + j) = make_float4(o1[0].x, o1[0].y, o1[1].x, o1[1].y);
            }
            if (MODE == 2 || MODE == 3) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    cfmac(dyx[r], o0[r], p0[r]);
                    cfmac(dyx[r], o1[r], p1[r]);
                    dyy[r] = fmaf(o0[r].x, o0[r].x, fmaf(o0[r].y, o0[r].y,
                                  fmaf(o1[r].x, o1[r].x, fmaf(o1[r].y, o1[r].y, dyy[r]))));
                }
            }
        }
    }
    if (MODE == 2 || MODE == 3) {
        __shared__ float4 sh[2][kRowLanes][2 * kRhsTile + 1];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            sh[0][threadIdx.y][2 * threadIdx.x + r] = dot_part(dyx[r]);
            sh[1][threadIdx.y][2 * threadIdx.x + r] = dot_part(dyy[r]);
        }
        __syncthreads();
        // 64 rhs x 2 quantities: threads (x, y < 4) add the 8 row lanes of one each
        const int q = threadIdx.y >> 1, jj = 2 * threadIdx.x + (threadIdx.y & 1);
        const int jo = 2 * blockIdx.x * kRhsTile + jj;
        if (threadIdx.y < 4 && jo < N) {
            float4 acc = sh[q][0][jj];
            for (int r = 1; r < kRowLanes; ++r) acc = dot_add(acc, sh[q][r][jj]);
            dot_parts<float2>(part)[((long long)q * N + jo) * gridDim.y + blockIdx.y] = acc;
        }
    }
}

template <typename C>
static bool wilson_f2(C*, const C*, const C*, const C*, re_t<C>, int, int, int, int, double2*, int, cudaStream_t) {
    return false;
}
template <>
bool wilson_f2<float2>(float2* y, const float2* x, const float2* b, const float2* U, float mass, int lx, int lt, int N,
                       int mode, double2* part, int groups, cudaStream_t s) {
    if (N % 2) return false;
    dim3 g((N / 2 + kRhsTile - 1) / kRhsTile, groups);
    switch (mode) {
        case 0: MG_LAUNCH(g, blk(), 0, s, (k_wilson_f2<0>), y, x, b, U, mass, lx, lt, N, part); break;
        case 1: MG_LAUNCH(g, blk(), 0, s, (k_wilson_f2<1>), y, x, b, U, mass, lx, lt, N, part); break;
        case 2: MG_LAUNCH(g, blk(), 0, s, (k_wilson_f2<2>), y, x, b, U, mass, lx, lt, N, part); break;
        default: MG_LAUNCH(g, blk(), 0, s, (k_wilson_f2<3>), y, x, b, U, mass, lx, lt, N, part); break;
    }
    MG_LAUNCHED();
    return true;
}

// ---------------------------------------------------------------------------
// Fine-level smoother with the residual and its image held in BF16 ([row][rhs],
// one bf16x2 per complex value): the operator y = D x with the minimal-residual dots
// conj(y).x, |y|^2 (FP32 arithmetic, ten loads of a site in flight per thread; N % 4 == 0).
// The first residual comes from k_wilson_f2<4>, the updates are k_mr_update_fine_bf16 and
// k_mr_combine_bf16.
// RPT right-hand sides per thread (4: 16-byte accesses, a warp spans 128 rhs; 2: 8-byte
// accesses, 64 rhs, so that a block of 64 keeps every lane busy).
// STORE = false: the dots only (the last minimal-residual step needs no image).
template <int RPT, bool STORE>
__global__ void __launch_bounds__(256, 3) k_wilson_bf16(uint32_t* __restrict__ y, const uint32_t* __restrict__ x,
                                                        const float2* __restrict__ U, float mass, int lx, int lt,
                                                        int N, double2* __restrict__ part) {
    if (grid_dependency()) return;
    const int j = RPT * (blockIdx.x * kRhsTile + threadIdx.x);
    const int V = lx * lt;
    float2 dyx[RPT];
    float dyy[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        dyx[r] = make_float2(0.f, 0.f);
        dyy[r] = 0.f;
    }
    auto ld4 = [&](long long idx, float2* v) {
        if constexpr (RPT == 4) {
            const uint4 w = *reinterpret_cast<const uint4*>(x + idx);
            v[0] = bf2_lo(w.x);
            v[1] = bf2_lo(w.y);
            v[2] = bf2_lo(w.z);
            v[3] = bf2_lo(w.w);
        } else {
            const uint2 w = *reinterpret_cast<const uint2*>(x + idx);
            v[0] = bf2_lo(w.x);
            v[1] = bf2_lo(w.y);
        }
    };
    if (j < N) {
        const long long N2 = 2LL * N;
        for (int site = blockIdx.y * kRowLanes + threadIdx.y; site < V; site += gridDim.y * kRowLanes) {
            const int xx = site % lx, t = site / lx;
            const int sxp = (xx + 1 == lx ? 0 : xx + 1) + lx * t;
            const int sxm = (xx == 0 ? lx - 1 : xx - 1) + lx * t;
            const int stp = xx + lx * (t + 1 == lt ? 0 : t + 1);
            const int stm = xx + lx * (t == 0 ? lt - 1 : t - 1);
            const float sgp = (t + 1 == lt) ? -0.5f : 0.5f;   // antiperiodic time boundary, times 1/2
            const float sgm = (t == 0) ? -0.5f : 0.5f;
            const float2 u0 = U[2 * site], u1 = U[2 * site + 1];
            const float2 u0m = U[2 * sxm], u1m = U[2 * stm + 1];
            float2 p0[RPT], p1[RPT], a0[RPT], a1[RPT], c0[RPT], c1[RPT], e0[RPT], e1[RPT], f0[RPT], f1[RPT];
            ld4(site * N2 + j, p0);
            ld4(site * N2 + N + j, p1);
            ld4(sxp * N2 + j, a0);
            ld4(sxp * N2 + N + j, a1);
            ld4(sxm * N2 + j, c0);
            ld4(sxm * N2 + N + j, c1);
            ld4(stp * N2 + j, e0);
            ld4(stp * N2 + N + j, e1);
            ld4(stm * N2 + j, f0);
            ld4(stm * N2 + N + j, f1);
            uint32_t w0[RPT], w1[RPT];
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                float2 o0 = mk(mass * p0[r].x, mass * p0[r].y), o1 = mk(mass * p1[r].x, mass * p1[r].y);
                {   // +x: (1 - sigma_1) psi = (a, -a), a = psi0 - psi1
                    const float2 u = cscale(cmul(u0, csub(a0[r], a1[r])), 0.5f);
                    o0 = csub(o0, u);
                    o1 = cadd(o1, u);
                }
                {   // -x: (1 + sigma_1) psi = (c, c), c = psi0 + psi1
                    const float2 u = cscale(cmulc(u0m, cadd(c0[r], c1[r])), 0.5f);
                    o0 = csub(o0, u);
                    o1 = csub(o1, u);
                }
                {   // +t: (1 - sigma_2) psi = (a, -i a), a = psi0 + i psi1
                    const float2 u = cscale(cmul(u1, cadd(e0[r], ctimesi(e1[r]))), sgp);
                    o0 = csub(o0, u);
                    o1 = cadd(o1, ctimesi(u));
                }
                {   // -t: (1 + sigma_2) psi = (c, i c), c = psi0 - i psi1
                    const float2 u = cscale(cmulc(u1m, csub(f0[r], ctimesi(f1[r]))), sgm);
                    o0 = csub(o0, u);
                    o1 = csub(o1, ctimesi(u));
                }
                cfmac(dyx[r], o0, p0[r]);
                cfmac(dyx[r], o1, p1[r]);
                dyy[r] = fmaf(o0.x, o0.x, fmaf(o0.y, o0.y, fmaf(o1.x, o1.x, fmaf(o1.y, o1.y, dyy[r]))));
                w0[r] = f2_bf(o0);
                w1[r] = f2_bf(o1);
            }
            if constexpr (!STORE) {
            } else if constexpr (RPT == 4) {
                *reinterpret_cast<uint4*>(y + site * N2 + j) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
                *reinterpret_cast<uint4*>(y + site * N2 + N + j) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
            } else {
                *reinterpret_cast<uint2*>(y + site * N2 + j) = make_uint2(w0[0], w0[1]);
                *reinterpret_cast<uint2*>(y + site * N2 + N + j) = make_uint2(w1[0], w1[1]);
            }
        }
    }
    __shared__ float4 sh[2][kRowLanes][RPT * kRhsTile + 1];
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        sh[0][threadIdx.y][RPT * threadIdx.x + r] = dot_part(dyx[r]);
        sh[1][threadIdx.y][RPT * threadIdx.x + r] = dot_part(dyy[r]);
    }
    __syncthreads();
    // RPT * 32 rhs x 2 quantities: thread t < 2 * RPT * 32 adds the 8 row lanes of
    // quantity t / (RPT * 32), rhs t % (RPT * 32) of this block
    const int t = threadIdx.y * kRhsTile + threadIdx.x;
    if (t < 2 * RPT * kRhsTile) {
        const int q = t / (RPT * kRhsTile), jj = t % (RPT * kRhsTile);
        const int jo = RPT * blockIdx.x * kRhsTile + jj;
        if (jo < N) {
            float4 acc = sh[q][0][jj];
            for (int r = 1; r < kRowLanes; ++r) acc = dot_add(acc, sh[q][r][jj]);
            dot_parts<float2>(part)[((long long)q * N + jo) * gridDim.y + blockIdx.y] = acc;
        }
    }
}

void launch_wilson_bf16(uint32_t* y, const uint32_t* x, const float2* U, double m0, int lx, int lt, int N,
                        double2* part, int groups, cudaStream_t s) {
    MG_REQUIRE(N % 4 == 0, MGMLMC_EINVAL, "BF16 Wilson operator: N a multiple of 4");
    if (N % 128 == 0) {
        dim3 g(N / 128, groups);
        if (y) MG_LAUNCH(g, blk(), 0, s, (k_wilson_bf16<4, true>), y, x, U, (float)(m0 + 2.0), lx, lt, N, part);
        else MG_LAUNCH(g, blk(), 0, s, (k_wilson_bf16<4, false>), y, x, U, (float)(m0 + 2.0), lx, lt, N, part);
    } else {
        dim3 g((N / 2 + kRhsTile - 1) / kRhsTile, groups);
        if (y) MG_LAUNCH(g, blk(), 0, s, (k_wilson_bf16<2, true>), y, x, U, (float)(m0 + 2.0), lx, lt, N, part);
        else MG_LAUNCH(g, blk(), 0, s, (k_wilson_bf16<2, false>), y, x, U, (float)(m0 + 2.0), lx, lt, N, part);
    }
    MG_LAUNCHED();
}

void launch_wilson_residual_bf16(uint32_t* y, const float2* x, const float2* b, const float2* U, double m0, int lx,
                                 int lt, int N, int groups, cudaStream_t s) {
    MG_REQUIRE(N % 2 == 0, MGMLMC_EINVAL, "BF16 Wilson residual: N even");
    dim3 g((N / 2 + kRhsTile - 1) / kRhsTile, groups);
    MG_LAUNCH(g, blk(), 0, s, (k_wilson_f2<4>), reinterpret_cast<float2*>(y), x, b, U, (float)(m0 + 2.0), lx, lt, N, nullptr);
    MG_LAUNCHED();
}

template <typename C>
void launch_wilson(C* y, const C* x, const C* b, const C* U, double m0, int lx, int lt, int N, int mode,
                   double2* part, int groups, cudaStream_t s) {
    using R = re_t<C>;
    dim3 g(rhs_tiles(N), groups);
    const R mass = (R)(m0 + 2.0);
    if (wilson_f2<C>(y, x, b, U, mass, lx, lt, N, mode, part, groups, s)) return;
    switch (mode) {
        case 0: MG_LAUNCH(g, blk(), 0, s, (k_wilson<C, 0>), y, x, b, U, mass, lx, lt, N, part); break;
        case 1: MG_LAUNCH(g, blk(), 0, s, (k_wilson<C, 1>), y, x, b, U, mass, lx, lt, N, part); break;
        case 2: MG_LAUNCH(g, blk(), 0, s, (k_wilson<C, 2>), y, x, b, U, mass, lx, lt, N, part); break;
        default: MG_LAUNCH(g, blk(), 0, s, (k_wilson<C, 3>), y, x, b, U, mass, lx, lt, N, part); break;
    }
    MG_LAUNCHED();
}

template <typename C, int RPT>
static void bs_dispatch(C* y, const C* x, const C* b, const C* A, int lx, int lt, int d, int N, int mode,
                        double2* part, int groups, cudaStream_t s) {
    dim3 g(rhs_tiles(N), groups);
    size_t sm = (size_t)5 * d * d * sizeof(C);
    size_t smin = 2 * kRowLanes * (kRhsTile + 1) * sizeof(double2);
    if (sm < smin) sm = smin;
    if (sm > 48 * 1024) {
        MG_CUDA(cudaFuncSetAttribute(k_block_stencil<C, RPT, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        MG_CUDA(cudaFuncSetAttribute(k_block_stencil<C, RPT, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        MG_CUDA(cudaFuncSetAttribute(k_block_stencil<C, RPT, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        MG_CUDA(cudaFuncSetAttribute(k_block_stencil<C, RPT, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    }
    switch (mode) {
        case 0: MG_LAUNCH(g, blk(), sm, s, (k_block_stencil<C, RPT, 0>), y, x, b, A, lx, lt, d, N, part); break;
        case 1: MG_LAUNCH(g, blk(), sm, s, (k_block_stencil<C, RPT, 1>), y, x, b, A, lx, lt, d, N, part); break;
        case 2: MG_LAUNCH(g, blk(), sm, s, (k_block_stencil<C, RPT, 2>), y, x, b, A, lx, lt, d, N, part); break;
        default: MG_LAUNCH(g, blk(), sm, s, (k_block_stencil<C, RPT, 3>), y, x, b, A, lx, lt, d, N, part); break;
    }
    MG_LAUNCHED();
}

template <int D>
static bool bsd_f2(float2* y, const float2* x, const float2* b, const float2* A, int lx, int lt, int N, int mode,
                   double2* part, int groups, cudaStream_t s) {
    if (N % 2 != 0) return false;
    if (D == 16 && N % 4 == 0 && N >= 128) {
        // four rhs per thread; T threads per half of the output rows
        const int T = std::min(64, (N / 4 + 31) / 32 * 32);
        dim3 g((N / 4 + T - 1) / T, groups);
        switch (mode) {
            case 0: MG_LAUNCH(g, 2 * T, 0, s, (k_block_stencil_f4<0>), y, x, b, A, lx, lt, N, part); break;
            case 1: MG_LAUNCH(g, 2 * T, 0, s, (k_block_stencil_f4<1>), y, x, b, A, lx, lt, N, part); break;
            case 2: MG_LAUNCH(g, 2 * T, 0, s, (k_block_stencil_f4<2>), y, x, b, A, lx, lt, N, part); break;
            default: MG_LAUNCH(g, 2 * T, 0, s, (k_block_stencil_f4<3>), y, x, b, A, lx, lt, N, part); break;
        }
        MG_LAUNCHED();
        return true;
    }
    const int threads = std::min(128, (N / 2 + 31) / 32 * 32);
    dim3 g((N / 2 + threads - 1) / threads, groups);
    switch (mode) {
        case 0: MG_LAUNCH(g, threads, 0, s, (k_block_stencil_f2<D, 0>), y, x, b, A, lx, lt, N, part); break;
        case 1: MG_LAUNCH(g, threads, 0, s, (k_block_stencil_f2<D, 1>), y, x, b, A, lx, lt, N, part); break;
        case 2: MG_LAUNCH(g, threads, 0, s, (k_block_stencil_f2<D, 2>), y, x, b, A, lx, lt, N, part); break;
        default: MG_LAUNCH(g, threads, 0, s, (k_block_stencil_f2<D, 3>), y, x, b, A, lx, lt, N, part); break;
    }
    MG_LAUNCHED();
    return true;
}
template <int D>
static bool bsd_f2(double2*, const double2*, const double2*, const double2*, int, int, int, int, double2*, int,
                   cudaStream_t) {
    return false;
}

template <typename C, int D>
static void bsd_dispatch(C* y, const C* x, const C* b, const C* A, int lx, int lt, int N, int mode, double2* part,
                         int groups, cudaStream_t s) {
    if (bsd_f2<D>(y, x, b, A, lx, lt, N, mode, part, groups, s)) return;
    const int th = cta_threads(N);
    dim3 g((N + th - 1) / th, groups);
    switch (mode) {
        case 0: MG_LAUNCH(g, th, 0, s, (k_block_stencil_d<C, D, 0>), y, x, b, A, lx, lt, N, part); break;
        case 1: MG_LAUNCH(g, th, 0, s, (k_block_stencil_d<C, D, 1>), y, x, b, A, lx, lt, N, part); break;
        case 2: MG_LAUNCH(g, th, 0, s, (k_block_stencil_d<C, D, 2>), y, x, b, A, lx, lt, N, part); break;
        default: MG_LAUNCH(g, th, 0, s, (k_block_stencil_d<C, D, 3>), y, x, b, A, lx, lt, N, part); break;
    }
    MG_LAUNCHED();
}

template <typename C, int D>
static void bsn_dispatch(C* y, const C* x, const C* b, const C* A, int lx, int lt, int N, int mode, double2* part,
                         int groups, cudaStream_t s) {
    const dim3 g((N + 7) / 8, groups), th(8, D);
    switch (mode) {
        case 0: MG_LAUNCH(g, th, 0, s, (k_block_stencil_narrow<C, D, 0>), y, x, b, A, lx, lt, N, part); break;
        case 1: MG_LAUNCH(g, th, 0, s, (k_block_stencil_narrow<C, D, 1>), y, x, b, A, lx, lt, N, part); break;
        case 2: MG_LAUNCH(g, th, 0, s, (k_block_stencil_narrow<C, D, 2>), y, x, b, A, lx, lt, N, part); break;
        default: MG_LAUNCH(g, th, 0, s, (k_block_stencil_narrow<C, D, 3>), y, x, b, A, lx, lt, N, part); break;
    }
}

// The one-rhs-per-thread kernels need wide blocks; narrow blocks (the setup solves
// run 8 rhs) take the generic 32-rhs-tile kernel.
static bool use_site_kernel(int d, int N) { return (d == 8 || d == 16) && N >= 64; }
static bool use_narrow_kernel(int d, int N) { return (d == 8 || d == 16) && N <= 16; }

int block_stencil_groups(int nsites, int d, int N) {
    if (use_narrow_kernel(d, N)) return nsites < 32 * kNumSM ? nsites : 32 * kNumSM;   // grid-stride over sites
    if (use_site_kernel(d, N)) {
        // one site per CTA up to 16 CTAs per SM: staging and compute of different
        // sites overlap across CTAs
        const int tiles = (N + 127) / 128;
        int want = 16 * kNumSM / tiles;
        if (want < 1) want = 1;
        return nsites < want ? nsites : want;
    }
    int want = 8 * kNumSM / rhs_tiles(N);
    if (want < 1) want = 1;
    return nsites < want ? nsites : want;
}

template <typename C>
void launch_block_stencil(C* y, const C* x, const C* b, const C* A, int lx, int lt, int d, int N, int mode,
                          double2* part, int groups, cudaStream_t s) {
    MG_REQUIRE(d >= 2 && d <= 64, MGMLMC_EINVAL, "block stencil: 2 <= d <= 64");
    if (use_narrow_kernel(d, N)) {
        if (d == 16) bsn_dispatch<C, 16>(y, x, b, A, lx, lt, N, mode, part, groups, s);
        else bsn_dispatch<C, 8>(y, x, b, A, lx, lt, N, mode, part, groups, s);
        MG_LAUNCHED();
        return;
    }
    if (use_site_kernel(d, N) && d == 16) return bsd_dispatch<C, 16>(y, x, b, A, lx, lt, N, mode, part, groups, s);
    if (use_site_kernel(d, N) && d == 8) return bsd_dispatch<C, 8>(y, x, b, A, lx, lt, N, mode, part, groups, s);
    if (d <= 8) bs_dispatch<C, 1>(y, x, b, A, lx, lt, d, N, mode, part, groups, s);
    else if (d <= 16) bs_dispatch<C, 2>(y, x, b, A, lx, lt, d, N, mode, part, groups, s);
    else if (d <= 32) bs_dispatch<C, 4>(y, x, b, A, lx, lt, d, N, mode, part, groups, s);
    else bs_dispatch<C, 8>(y, x, b, A, lx, lt, d, N, mode, part, groups, s);
}

// Restriction of a d = 16 level for few rhs (N <= 32): thread = (rhs, coarse value), a CTA per
// coarse site and spin block.  With a thread per rhs a CTA is one half-empty warp whose 2 NV sums
// run one after another (10 us for 64 coarse sites x 16 rhs, this takes 5).
template <int NV>
__global__ void __launch_bounds__(32 * NV) k_restrict_few(float2* __restrict__ xc, const float2* __restrict__ x,
                                                          const float2* __restrict__ P, int lx, int lt, int ax, int at,
                                                          int N) {
    if (grid_dependency()) return;
    constexpr int D = 16, HD = 8;
    extern __shared__ __align__(16) unsigned char smem_rp[];
    float2* Ps = reinterpret_cast<float2*>(smem_rp);            // [aggregate site][a of the spin block][jv]
    const int j = threadIdx.x, jv = threadIdx.y, tid = jv * 32 + j;
    const int cx = lx / ax, na = ax * at;
    const int S = blockIdx.x >> 1, sp = blockIdx.x & 1;
    const int Xc = S % cx, T = S / cx;
    auto site_of = [&](int q) { return (Xc * ax + q % ax) + lx * (T * at + q / ax); };
    for (int e = tid; e < na * HD * NV; e += 32 * NV) {
        const int q = e / (HD * NV), r = e % (HD * NV);
        Ps[e] = P[((long long)site_of(q) * D + sp * HD) * NV + r];
    }
    __syncthreads();
    if (j >= N) return;
    float2 acc = make_float2(0.f, 0.f);
    constexpr int QB = 4;                                       // sites whose loads are issued together
    for (int q0 = 0; q0 < na; q0 += QB) {
        float2 xv[QB][HD];
#pragma unroll
        for (int u = 0; u < QB; ++u) {
            const float2* xs = x + ((long long)site_of(min(q0 + u, na - 1)) * D + sp * HD) * N + j;
#pragma unroll
            for (int a = 0; a < HD; ++a) xv[u][a] = xs[(long long)a * N];
        }
#pragma unroll
        for (int u = 0; u < QB; ++u) {
            if (q0 + u >= na) break;
#pragma unroll
            for (int a = 0; a < HD; ++a) cfmac(acc, Ps[((q0 + u) * HD + a) * NV + jv], xv[u][a]);
        }
    }
    xc[((long long)S * 2 * NV + sp * NV + jv) * N + j] = acc;
}

template <typename C, int NV>
static bool restrict_few(C* xc, const C* x, const C* P, int lx, int lt, int d, int ax, int at, int N, cudaStream_t s) {
    if constexpr (sizeof(C) == 8) {
        if (d != 16 || N > 32) return false;
        const size_t sm = (size_t)ax * at * 8 * NV * sizeof(C);
        MG_LAUNCH(dim3(2 * (lx / ax) * (lt / at)), dim3(32, NV), sm, s, k_restrict_few<NV>, xc, x, P, lx, lt, ax, at, N);
        MG_LAUNCHED();
        return true;
    }
    return false;
}

template <typename C, int NV, int D, int QB, int V>
static void rp_nvd(bool restrict_op, C* out, const C* in, const C* P, int lx, int lt, int ax, int at, int N,
                   bool accumulate, uint8_t* xt, cudaStream_t s) {
    const int ncs = (lx / ax) * (lt / at);
    const int cols = (N + V - 1) / V;
    const int th = std::min(128 / V, (cols + 31) / 32 * 32);
    const int tiles = (cols + th - 1) / th;
    const int G = std::max(1, std::min(ncs, 16 * kNumSM / tiles));
    const size_t sm = (size_t)ax * at * D * NV * sizeof(C);
    const int rows = std::min(128 / th, (ax * at + QB - 1) / QB);
    if (restrict_op)
        MG_LAUNCH(dim3(tiles, G), th, sm, s, (k_restrict_nvd<C, NV, D, QB, V>), out, in, P, lx, lt, ax, at, N);
    else if (rows > 1)
        MG_LAUNCH(dim3(tiles, G), dim3(th, rows), sm, s, (k_prolong_nvd<C, NV, D, QB, V, true>), out, in, P, lx, lt, ax,
                  at, N, accumulate, xt);
    else
        MG_LAUNCH(dim3(tiles, G), th, sm, s, (k_prolong_nvd<C, NV, D, QB, V, false>), out, in, P, lx, lt, ax, at, N,
                  accumulate, xt);
    MG_LAUNCHED();
}

template <typename C, int NV>
static void rp_launch(bool restrict_op, C* xc_or_x, const C* in, const C* P, int lx, int lt, int d, int ax, int at,
                      int N, bool accumulate, uint8_t* xt, cudaStream_t s) {
    constexpr int W = sizeof(C) == 8 ? 2 : 1;
    // two rhs per thread from 64 rhs on (below, they leave lanes idle), except in the d = 16
    // prolongation, which also writes the BF16 tiles (39 us with one, 47 with two)
    const bool two = W == 2 && N % 2 == 0 && N >= 64 && !(d == 16 && !restrict_op);
    if (restrict_op && restrict_few<C, NV>(xc_or_x, in, P, lx, lt, d, ax, at, N, s)) return;
    if (d == 2) {
        if (two) rp_nvd<C, NV, 2, 4, W>(restrict_op, xc_or_x, in, P, lx, lt, ax, at, N, accumulate, nullptr, s);
        else rp_nvd<C, NV, 2, 4, 1>(restrict_op, xc_or_x, in, P, lx, lt, ax, at, N, accumulate, nullptr, s);
        return;
    }
    if (d == 16) {
        if (two) rp_nvd<C, NV, 16, 1, W>(true, xc_or_x, in, P, lx, lt, ax, at, N, accumulate, xt, s);
        else rp_nvd<C, NV, 16, 1, 1>(restrict_op, xc_or_x, in, P, lx, lt, ax, at, N, accumulate, xt, s);
        return;
    }
    const int ncs = (lx / ax) * (lt / at);
    const int th = cta_threads(N);
    const int tiles = (N + th - 1) / th;
    const int G = std::max(1, std::min(ncs, 16 * kNumSM / tiles));
    const size_t sm = (size_t)ax * at * d * NV * sizeof(C);
    if (restrict_op)
        MG_LAUNCH(dim3(tiles, G), th, sm, s, (k_restrict_nv<C, NV>), xc_or_x, in, P, lx, lt, d, ax, at, N);
    else
        MG_LAUNCH(dim3(tiles, G), th, sm, s, (k_prolong_nv<C, NV>), xc_or_x, in, P, lx, lt, d, ax, at, N, accumulate);
    MG_LAUNCHED();
}

template <typename C>
static bool rp_fast(bool restrict_op, C* out, const C* in, const C* P, int lx, int lt, int d, int ax, int at,
                    int nvec, int N, bool accumulate, uint8_t* xt, cudaStream_t s) {
    if ((size_t)ax * at * d * nvec * sizeof(C) > 48 * 1024) return false;
    switch (nvec) {
        case 2: rp_launch<C, 2>(restrict_op, out, in, P, lx, lt, d, ax, at, N, accumulate, xt, s); return true;
        case 4: rp_launch<C, 4>(restrict_op, out, in, P, lx, lt, d, ax, at, N, accumulate, xt, s); return true;
        case 8: rp_launch<C, 8>(restrict_op, out, in, P, lx, lt, d, ax, at, N, accumulate, xt, s); return true;
        default: return false;
    }
}

template <typename C>
void launch_restrict(C* xc, const C* x, const C* P, int lx, int lt, int d, int ax, int at, int nvec, int N,
                     cudaStream_t s) {
    if (rp_fast<C>(true, xc, x, P, lx, lt, d, ax, at, nvec, N, false, nullptr, s)) return;
    const int ncs = (lx / ax) * (lt / at);
    int G = row_groups((long long)ncs * kRowLanes, N, 4);
    MG_LAUNCH(dim3(rhs_tiles(N), G), blk(), 0, s, (k_restrict<C>), xc, x, P, lx, lt, d, ax, at, nvec, N);
    MG_LAUNCHED();
}

template <typename C>
bool launch_prolong(C* x, const C* xc, const C* P, int lx, int lt, int d, int ax, int at, int nvec, int N,
                    bool accumulate, cudaStream_t s, void* xt) {
    uint8_t* tiles = (sizeof(C) == 8 && d == 16) ? reinterpret_cast<uint8_t*>(xt) : nullptr;
    if (rp_fast<C>(false, x, xc, P, lx, lt, d, ax, at, nvec, N, accumulate, tiles, s)) return tiles != nullptr;
    const long long rows = (long long)lx * lt * d;
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(rows, N)), blk(), 0, s, (k_prolong<C>), x, xc, P, lx, lt, d, ax, at, nvec, N,
                                                                             accumulate);
    MG_LAUNCHED();
    return false;
}

// Block shape and grid of the row kernels above: V values per thread along the rhs, at
// most `per_sm` CTAs of 256 threads per SM.
static void row_shape(long long n, int N, int V, int per_sm, dim3& g, dim3& b) {
    const int cols = (N + V - 1) / V;
    int bx = 1;
    while (bx < cols && bx < 32) bx *= 2;
    const int by = 256 / bx, gx = (cols + bx - 1) / bx;
    const long long need = (n + by - 1) / by;
    g = dim3(gx, (unsigned)std::max(1LL, std::min(need, (long long)per_sm * kNumSM / gx)));
    b = dim3(bx, by);
}

template <typename C>
void launch_mr_update(C* rn, const C* r, const C* p, const C* alpha, long long n, int N, cudaStream_t s) {
    dim3 g, b;
    if (sizeof(C) == 8 && N % 2 == 0) {
        row_shape(n, N, 2, 8, g, b);
        MG_LAUNCH(g, b, 0, s, (k_mr_update<C, sizeof(C) == 8 ? 2 : 1>), rn, r, p, alpha, n, N);
    } else {
        row_shape(n, N, 1, 8, g, b);
        MG_LAUNCH(g, b, 0, s, (k_mr_update<C, 1>), rn, r, p, alpha, n, N);
    }
    MG_LAUNCHED();
}

template <typename C>
void launch_mr_combine(C* e, const C* rs, size_t slot, int K, const C* alpha, long long n, int N, bool e_is_zero,
                       cudaStream_t s) {
    MG_REQUIRE(K >= 1 && K <= kMrGroup, MGMLMC_EINVAL, "smoother: group size");
    dim3 g, b;
    if (sizeof(C) == 8 && N % 2 == 0) {
        row_shape(n, N, 2, 8, g, b);
        MG_LAUNCH(g, b, 0, s, (k_mr_combine<C, sizeof(C) == 8 ? 2 : 1>), e, rs, slot, K, alpha, n, N, e_is_zero);
    } else {
        row_shape(n, N, 1, 8, g, b);
        MG_LAUNCH(g, b, 0, s, (k_mr_combine<C, 1>), e, rs, slot, K, alpha, n, N, e_is_zero);
    }
    MG_LAUNCHED();
}

void launch_mr_update_fine_bf16(uint32_t* rn, const uint32_t* r, const uint32_t* p, const float2* alpha, long long n,
                                int N, cudaStream_t s) {
    MG_REQUIRE(N % 4 == 0, MGMLMC_EINVAL, "BF16 MR update: N a multiple of 4");
    dim3 g, b;
    row_shape(n, N, 4, 8, g, b);
    MG_LAUNCH(g, b, 0, s, k_mr_update_fine_bf16, rn, r, p, alpha, n, N);
    MG_LAUNCHED();
}

void launch_mr_combine_bf16(float2* e, const uint32_t* rs, size_t slot, int K, const float2* alpha, long long n, int N,
                            cudaStream_t s) {
    MG_REQUIRE(N % 4 == 0 && K >= 1 && K <= kMrGroup, MGMLMC_EINVAL, "BF16 MR sum: N a multiple of 4, group size");
    dim3 g, b;
    row_shape(n, N, 4, 8, g, b);
    MG_LAUNCH(g, b, 0, s, k_mr_combine_bf16, e, rs, slot, K, alpha, n, N);
    MG_LAUNCHED();
}

template <typename C>
void launch_gamma5(C* y, const C* x, long long nsites, int d, int N, cudaStream_t s) {
    const long long rows = nsites * d;
    MG_LAUNCH(dim3(rhs_tiles(N), row_groups(rows, N)), blk(), 0, s, (k_gamma5<C>), y, x, rows, d, N);
    MG_LAUNCHED();
}

#define INST(C)                                                                                        \
    template void launch_wilson<C>(C*, const C*, const C*, const C*, double, int, int, int, int, double2*, \
                                   int, cudaStream_t);                                                 \
    template void launch_block_stencil<C>(C*, const C*, const C*, const C*, int, int, int, int, int,    \
                                          double2*, int, cudaStream_t);                                 \
    template void launch_restrict<C>(C*, const C*, const C*, int, int, int, int, int, int, int,         \
                                     cudaStream_t);                                                     \
    template bool launch_prolong<C>(C*, const C*, const C*, int, int, int, int, int, int, int, bool,    \
                                    cudaStream_t, void*);                                               \
    template void launch_mr_update<C>(C*, const C*, const C*, const C*, long long, int, cudaStream_t);  \
    template void launch_mr_combine<C>(C*, const C*, size_t, int, const C*, long long, int, bool,       \
                                       cudaStream_t);                                                   \
    template void launch_block_diag_combine<C>(C*, const C*, size_t, int, const C*, const C*, int, int, \
                                               int, bool, cudaStream_t);                                \
    template void launch_gamma5<C>(C*, const C*, long long, int, int, cudaStream_t);                  \
    template void launch_block_diag_apply<C>(C*, const C*, const C*, int, int, int, bool, cudaStream_t);
INST(double2)
INST(float2)

}  // namespace mg
