// FP64 block products on the tensor cores.  GB300 issues 2 FP64 FMA per SM and clock (1/64
// of its FP32 rate), so the FP64 block stencils (d = 16) and the dense coarsest inverse were
// bound by that pipe: 4.3 ms for one D_3 x at 32^2 sites x 512 rhs, 2.2 ms for a 1024 x 1024
// inverse times 64 rhs.  Both are contractions, and an exact integer product of slices of the
// operands gives the same result on the BF16 tensor cores (the Ozaki scheme: K. Ozaki,
// T. Ogita, S. Oishi, S. M. Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication", Numer. Algorithms 59, 2012):
//
//  * every rhs of x is scaled by a power of two 2^-ex with |x| < 2^ex (its largest entry), every
//    row of the matrix likewise, and both are rounded to 63 bits, x = 2^ex sum_{j<8} d_j 2^{-6-8j},
//    a = 2^ea sum_{i<8} c_i 2^{-6-8i}; all digits are integers in [-128, 127], exact in BF16;
//  * G_g = sum_{i+j=g} sum_k c_i d_j for g = 0..8: products of digits are below 2^14, sums of
//    at most 192 k and 5 pairs below 2^24, so the FP32 accumulation in TMEM is exact for the
//    groups g <= 4 (the others weigh at most 2^-40, and their sums can only leave the
//    exact range by rounding their last place); the dropped pairs i + j > 8 weigh 2^-72;
//  * sum_g G_g 2^-8g is formed in 128-bit integers and rounded to FP64 once.
// The error of an entry is 2^-53 of itself from that rounding, and about 2^-63 of the rhs' largest
// entry; 160 FP64 FMAs leave about 2^-51 of the entries around it.  In the norm, by which the solver
// decides, the product is closer to the exact one also where a rhs is concentrated on a few
// sites (the second part is spread over n entries: it stays below as long as n < 2^21 of them).  Entry
// by entry a site loses whose inputs all lie more than 2^8 below the rhs' largest entry; where the
// caller asks for it (the operators of mgmlmc_apply), its rows are summed in FP64 instead, and so are
// those next to an infinity or NaN, which stays where it is.  In the solves of the near-critical 1024^2
// lattice, dominated by localised modes, that would be most sites (189 -> 140 samples/s).  With 7
// digits of x and 8 groups (2^-55) their residuals stood at 1.9e-12.
//
// Layout: the rhs are the MMA's M (128 rows of x digits, K = 32 reals of a site), the digits
// of the block are its N: the 8 x 32 rows (i, output real) of a block's tile lie one after
// another, so digit slice j of x times the first rows of the tile lands on the columns from
// 32j on, which is exactly where G_{i+j} belongs: 8 MMAs (N = 256, 256, 224, ..., 64) per K
// step, 1376 columns for the 43 pairs.  A job is one block of 16 output rows for 128 rhs (5
// blocks of the stencil, or up to 6 of a row of the dense matrix); x digits (64 KB, in two
// halves) and block digits (16 KB) of each K block move by bulk copies through rings of 5
// halves and 4 blocks; the 288 columns of a job's accumulator are drained into the registers of
// eight epilogue warps, which form the FP64 results while the next job's MMAs run.  One CTA
// per SM (224 KB).
// Bound: the stream of digit tiles (80 KB per K block) from L2 into one CTA per SM.  At 128^2 sites x 256
// rhs 13.4 GB of tiles take 2.04 ms, 6.6 TB/s; DRAM moves 6.7 GB meanwhile (0.48 of the measured
// copy rate), the MMAs run at 0.9 PFLOP/s (half of the measured BF16 rate).
// Measured: D_3 x at 32^2 sites x 512 rhs 4329 -> 230 us, D_2 x at 128^2 sites x 128 rhs (before, by
// P^H D_1 P) 9.4 -> 0.9 ms, the inverse of 1024 unknowns times 64 rhs 2205 -> 40 us; the two
// passes that scale and slice x move 32 B per real more.  The sites summed in FP64 and the
// operator's row exponents: D_2 x at 16^2 sites x 64 rhs 34.8 -> 36.3 us, where no site is.
#include <algorithm>

#include "kernels.cuh"
#include "tcgen05.cuh"

namespace mg {
namespace tc {
namespace f64 {
constexpr int D = 16, KD = 32;             // block size, reals of a block
constexpr int NX = 8, NA = 8, NG = 9;      // digit slices of x and of the matrix, groups
constexpr int XS = 128 * KD * 2;           // 8 KB: one digit slice of a 128-rhs tile
constexpr int XT = NX * XS;                // 64 KB
constexpr int AT = NA * KD * KD * 2;       // 16 KB: the digits of one block
constexpr int XH = XT / 2;                 // 32 KB: four digit slices
constexpr int NXH = 5, NAS = 4;            // ring slots of x halves and of blocks
constexpr int SMEM = NXH * XH + NAS * AT;  // 224 KB
constexpr int TCOLS = 512;                 // 288 accumulator columns, allocated as 512
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 64 + 32 * EPI_WARPS;
constexpr int KSPLIT = 6;                  // K blocks of a dense job (exact sums, see above)

using u64 = unsigned long long;
using i64 = long long;

constexpr u64 kNonFinite = 0x7FFull << 52;

// round(v 2^(62 - e)), |v| < 2^e, e = E - 1022 for the biased exponent E of the largest entry; 0
// for an infinity or NaN.
__device__ __forceinline__ i64 fixed_point(double v, int E) {
    const u64 b = (u64)__double_as_longlong(v);
    const int eb = (int)((b >> 52) & 0x7ff);
    if (eb > E && eb == 0x7ff) return 0;
    const u64 m = (b & 0xFFFFFFFFFFFFFull) | (eb ? 1ull << 52 : 0ull);
    // v = m 2^(max(eb, 1) - 1075); q = m 2^sh
    const int sh = (eb > 0 ? eb : 1) - 1075 + 62 - (E - 1022);
    u64 q;
    if (sh >= 0) q = m << sh;
    else if (sh < -54) q = 0;
    else q = (m + (1ull << (-sh - 1))) >> (-sh);
    return (b >> 63) ? -(i64)q : (i64)q;
}

// Digit (a byte of the offset fixed-point number) as the float it stands for.
__device__ __forceinline__ float digit(u64 u, int byte) {
    return __uint_as_float(0x4B000000u | ((uint32_t)(u >> (8 * byte)) & 0xFFu)) - 8388736.0f;   // 2^23 + 128
}
__device__ __forceinline__ uint32_t pack_exact(float lo, float hi) {
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// Largest |re|, |im| per column, as the bit pattern of the double: non-negative doubles order
// like integers, NaN above all, so the atomic maximum does not depend on the order.
__global__ void __launch_bounds__(256) k_absmax_cols(u64* __restrict__ out, const double2* __restrict__ x,
                                                     long long n, int N) {
    if (grid_dependency()) return;
    __shared__ u64 sh[256];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    u64 m = 0;
    if (j < N) {
        const long long S = (long long)gridDim.y * blockDim.y;
#pragma unroll 4
        for (long long i = (long long)blockIdx.y * blockDim.y + threadIdx.y; i < n; i += S) {
            const double2 v = x[i * N + j];
            const u64 a = (u64)__double_as_longlong(v.x) & 0x7FFFFFFFFFFFFFFFull;
            const u64 b = (u64)__double_as_longlong(v.y) & 0x7FFFFFFFFFFFFFFFull;
            m = max(m, max(a, b));
        }
    }
    sh[tid] = m;
    __syncthreads();
    for (int st = blockDim.y / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.y < st) sh[tid] = max(sh[tid], sh[tid + st * blockDim.x]);
        __syncthreads();
    }
    if (threadIdx.y == 0 && j < N && sh[threadIdx.x] != 0) atomicMax(out + j, sh[threadIdx.x]);
}

// The same over the finite entries of a stencil's input, and the exponent (biased) of the largest
// entry of every site and rhs: 0 for zeros, 0x7ff where an entry is not finite.  Four threads
// (threadIdx.y) per site and rhs.
__global__ void __launch_bounds__(256) k_absmax_sites(u64* __restrict__ out, uint16_t* __restrict__ xe,
                                                      const double2* __restrict__ x, int nsites, int N) {
    if (grid_dependency()) return;
    __shared__ u64 sh[256];
    const int bx = blockDim.x, tid = threadIdx.y * bx + threadIdx.x, cg = threadIdx.y & 3;
    const int j = blockIdx.x * bx + threadIdx.x;
    const int per = blockDim.y / 4;                      // sites of a CTA at a time
    u64 m = 0;
    for (int s0 = blockIdx.y * per; s0 < nsites; s0 += gridDim.y * per) {
        const int site = s0 + (threadIdx.y >> 2);
        u64 s = 0;
        if (j < N && site < nsites) {
            double2 v[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = x[((size_t)site * D + 4 * cg + c) * N + j];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                s = max(s, (u64)__double_as_longlong(v[c].x) & 0x7FFFFFFFFFFFFFFFull);
                s = max(s, (u64)__double_as_longlong(v[c].y) & 0x7FFFFFFFFFFFFFFFull);
            }
            if (s >= kNonFinite) {
                u64 f = 0;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const u64 a = (u64)__double_as_longlong(v[c].x) & 0x7FFFFFFFFFFFFFFFull;
                    const u64 b = (u64)__double_as_longlong(v[c].y) & 0x7FFFFFFFFFFFFFFFull;
                    f = max(f, max(a < kNonFinite ? a : 0, b < kNonFinite ? b : 0));
                }
                m = max(m, f);
                s = kNonFinite;
            } else {
                m = max(m, s);
            }
        }
        __syncthreads();
        sh[tid] = s;
        __syncthreads();
        if (cg == 0 && j < N && site < nsites) {
#pragma unroll
            for (int q = 1; q < 4; ++q) s = max(s, sh[tid + q * bx]);
            xe[(size_t)site * N + j] = (uint16_t)(s == 0 ? 0 : max((int)(s >> 52), 1));
        }
    }
    __syncthreads();
    sh[tid] = m;
    __syncthreads();
    for (int st = blockDim.y / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.y < st) sh[tid] = max(sh[tid], sh[tid + st * bx]);
        __syncthreads();
    }
    if (threadIdx.y == 0 && j < N && sh[threadIdx.x] != 0) atomicMax(out + j, sh[threadIdx.x]);
}

// Exponent (biased) of the largest |re|, |im| of every row of a job's blocks: row c of the five
// blocks of a site (nb = 0, rows of D), or of K blocks 6z .. of block row R of a dense matrix (nb
// blocks per row, rows ld apart, job = R splits + z).  Eight lanes per row.
__global__ void __launch_bounds__(128) k_row_exponents(uint16_t* __restrict__ re, const double2* __restrict__ A, int nb,
                                                       int splits, int ld) {
    if (grid_dependency()) return;
    const long long job = blockIdx.x;
    const int c = threadIdx.x >> 3, l = threadIdx.x & 7;
    int count = 5;                                       // blocks
    const double2* row = A + job * (5 * D * D) + c * D;
    size_t step = D * D;                                 // from a block to the next
    if (nb) {
        const int z = (int)(job % splits);
        count = min(KSPLIT, nb - z * KSPLIT);
        row = A + ((job / splits) * D + c) * (long long)ld + (long long)z * KSPLIT * D;
        step = D;
    }
    u64 m = 0;
    for (int e = l; e < count * D; e += 8) {
        const double2 a = row[(e / D) * step + e % D];
        m = max(m, max((u64)__double_as_longlong(a.x) & 0x7FFFFFFFFFFFFFFFull,
                       (u64)__double_as_longlong(a.y) & 0x7FFFFFFFFFFFFFFFull));
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (l == 0) re[job * D + c] = (uint16_t)(m >> 52);
}

// Digit tiles of x: per (site, 128-rhs tile) 8 K-major slices of 8 KB.  Thread = (site,
// group of 4 components, rhs): four 16-byte loads, eight 16-byte stores.  The rows of a
// tile beyond the rhs are not written (they only reach the same rows of the product).
__global__ void __launch_bounds__(128) k_slice_x(uint8_t* __restrict__ xs, const double2* __restrict__ x,
                                                 const u64* __restrict__ mx, int nblk, int N, int T) {
    if (grid_dependency()) return;
    const int row = threadIdx.x, t = blockIdx.y, j = 128 * t + row;
    const long long g = (long long)blockIdx.x * blockDim.y + threadIdx.y;    // (block, component group)
    const int site = (int)(g >> 2), cg = (int)(g & 3);
    if (site >= nblk || j >= N) return;
    const int E = (int)(mx[j] >> 52);
    double2 v[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) v[p] = x[((size_t)site * D + 4 * cg + p) * N + j];
    u64 qr[4], qi[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        qr[p] = (u64)fixed_point(v[p].x, E) + 0x8080808080808080ull;
        qi[p] = (u64)fixed_point(v[p].y, E) + 0x8080808080808080ull;
    }
    uint8_t* tile = xs + ((size_t)site * T + t) * XT + kmaj32_off(row, 8 * cg);
#pragma unroll
    for (int s = 0; s < NX; ++s) {
        uint32_t w[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) w[p] = pack_exact(digit(qr[p], NX - 1 - s), digit(qi[p], NX - 1 - s));
        *reinterpret_cast<uint4*>(tile + s * XS) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Digit tiles of 16 x 16 complex blocks in their real 32 x 32 form (row = output real, K =
// input real; the form of the BF16 stencil operands).  Block q starts at A + base(q) with
// rows ld apart: the stencil's blocks lie one after another (ld = 16, nb = 0), block (R, C)
// of a dense n x n matrix starts at (16 R) n + 16 C (nb = n / 16 blocks per row, ld = n).
// Each row relative to its own largest entry (k_row_exponents).  Thread = (block, output real, 8
// input reals).
__global__ void __launch_bounds__(128) k_slice_a(uint8_t* __restrict__ as, const double2* __restrict__ A,
                                                 const uint16_t* __restrict__ re, long long nblk, int nb, int splits,
                                                 int ld) {
    if (grid_dependency()) return;
    const long long q = blockIdx.x;
    if (q >= nblk) return;
    const int n = threadIdx.x >> 2, kg = threadIdx.x & 3;
    const int co = n >> 1, to = n & 1;
    const long long job = nb ? (q / nb) * splits + (q % nb) / KSPLIT : q / 5;
    const int E = re[job * D + co];
    const double2* blk = nb ? A + (q / nb) * D * (long long)ld + (q % nb) * D : A + q * (D * D);
    u64 u[8];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const double2 a = blk[(long long)co * ld + 4 * kg + p];
        u[2 * p] = (u64)fixed_point(to ? a.y : a.x, E) + 0x8080808080808080ull;        // times Re x
        u[2 * p + 1] = (u64)fixed_point(to ? a.x : -a.y, E) + 0x8080808080808080ull;   // times Im x
    }
    uint8_t* tile = as + (size_t)q * AT;
#pragma unroll
    for (int s = 0; s < NA; ++s) {
        uint32_t w[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) w[p] = pack_exact(digit(u[2 * p], NA - 1 - s), digit(u[2 * p + 1], NA - 1 - s));
        *reinterpret_cast<uint4*>(tile + kmaj32_off(s * KD + n, 8 * kg)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// 2^s sum_{g<9} G_g 2^(8 (7 - g)) rounded to FP64 once (the last group to its integer part:
// 2^-69 of the scale).  |G_g| < 2^25.
__device__ __forceinline__ double combine(const int* G, int s) {
    i64 hi = (((i64)G[0] * 256 + G[1]) * 256 + G[2]) * 256 + G[3];
    const i64 lo = (((i64)G[4] * 256 + G[5]) * 256 + G[6]) * 256 + G[7] + ((G[8] + 128) >> 8);
    hi += lo >> 32;                               // T = hi 2^32 + l, 0 <= l < 2^32
    u64 l = (u64)lo & 0xFFFFFFFFull;
    const bool neg = hi < 0;
    if (neg) {
        l = (0x100000000ull - l) & 0xFFFFFFFFull;
        hi = ~hi + (l == 0 ? 1 : 0);
    }
    u64 h = (u64)hi;
    int e = s + 95;                               // exponent of bit 63 of h
    if (h == 0) {
        if (l == 0) return 0.0;
        h = l;
        l = 0;
        e -= 32;
    }
    const int z = __clzll((i64)h);                // h < 2^50: z >= 14
    u64 m = h << z;
    m |= z >= 32 ? l << (z - 32) : l >> (32 - z);
    const u64 r = (m >> 11) + ((m >> 10) & 1);    // 2^52 <= r <= 2^53
    const int E = e - z + 1023;                   // biased exponent of 1.xxx
    double v;
    if (E > 0 && E < 2046) v = __longlong_as_double((i64)(((u64)(E - 1) << 52) + r));
    else v = ldexp((double)(i64)r, E - 1075);     // subnormal or above the range
    return neg ? -v : v;
}

// Rows c0 .. c0 + 7 of a site's product by FP64 sums, in the order of the FP64 block stencils; the
// 16 inputs of a neighbour are loaded together.
__device__ __noinline__ void rows_by_fp64(double2* v, const double2* __restrict__ A, const double2* __restrict__ x,
                                          int site, int c0, int lx, int lt, int N, int j) {
    double2 acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = czero<double2>();
#pragma unroll 1
    for (int dir = 0; dir < 5; ++dir) {
        const double2* xn = x + (size_t)nbr_site(site, dir, lx, lt) * D * N + j;
        const double2* Ar = A + (((size_t)site * 5 + dir) * D + c0) * D;
        double2 xv[D];
#pragma unroll
        for (int bc = 0; bc < D; ++bc) xv[bc] = xn[(size_t)bc * N];
#pragma unroll
        for (int bc = 0; bc < D; ++bc)
#pragma unroll
            for (int c = 0; c < 8; ++c) cfma(acc[c], Ar[c * D + bc], xv[bc]);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = acc[c];
}

// MODE 0: y = A x; 1: y = b - A x; 2: y = A x with the per-rhs dots <y, x>, <y, y>; 3: the
// dots only; 4: job (R, z) of a dense product, y[z] = its partial sum over K blocks
// 6z .. 6z + 5.  nblk: sites of the stencil (lx x lt) or block rows of the dense matrix.
// With xe (exponents per site and rhs) the stencil's results are also right entry by entry: where all
// of a site's inputs lie more than 2^kSpread below the rhs' largest entry, whose scale the digits
// share, or one of them is not finite, its rows are summed in FP64 instead.
constexpr int kSpread = 8;
template <int MODE>
__global__ void __launch_bounds__(THREADS, 1)
    k_block_f64(double2* __restrict__ y, const double2* __restrict__ b, const double2* __restrict__ x,
                const uint8_t* __restrict__ xs, const uint8_t* __restrict__ as, const u64* __restrict__ mxx,
                const uint16_t* __restrict__ xe, const uint16_t* __restrict__ re, const double2* __restrict__ A, int lx,
                int lt, int nblk, int splits, int N, double2* __restrict__ part,
                int* __restrict__ err) {
    if (grid_dependency()) return;
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t xfull[NXH], xempty[NXH], bfull[NAS], bempty[NAS], afull, aempty;
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_flag;
    uint8_t* xring = smem;
    uint8_t* bring = smem + NXH * XH;
    volatile int* abrt = &abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x, T = gridDim.y, t = blockIdx.y;
    const int njobs_all = nblk * splits;
    const int njob = (njobs_all - (int)blockIdx.x + G - 1) / G;
    const int rows = min(128, N - 128 * t);
    auto kblocks = [&](int job) { return MODE == 4 ? min(KSPLIT, nblk - (job % splits) * KSPLIT) : 5; };

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                     "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int q = 0; q < NXH; ++q) {
            mbar_init(&xfull[q], 1);
            mbar_init(&xempty[q], 1);
        }
        for (int q = 0; q < NAS; ++q) {
            mbar_init(&bfull[q], 1);
            mbar_init(&bempty[q], 1);
        }
        mbar_init(&afull, 1);
        mbar_init(&aempty, EPI_WARPS);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_holder;

    if (warp == 0) {
        if (lane == 0) {
            // producer: a tile narrower than 128 rhs moves only its own 8-row groups
            const uint32_t slice = (uint32_t)((rows + 7) / 8) * 512u;
            int q = 0, hq = 0;                   // K blocks and x halves issued
            bool ok = true;
            for (int i = 0; i < njob && ok; ++i) {
                const int job = blockIdx.x + i * G;
                const int kb = kblocks(job);
                for (int o = 0; o < kb && ok; ++o) {
                    long long xb, ab;
                    if (MODE == 4) {
                        xb = (job % splits) * KSPLIT + o;
                        ab = (long long)(job / splits) * nblk + xb;
                    } else {
                        xb = nbr_site(job, o, lx, lt);
                        ab = (long long)job * 5 + o;
                    }
                    const int bs = q % NAS;
                    if (q >= NAS && !mbar_wait_ab(&bempty[bs], (unsigned)((q / NAS - 1) & 1), abrt)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&bfull[bs], AT);
                    bulk_g2s(bring + bs * AT, as + (size_t)ab * AT, AT, &bfull[bs]);
                    ++q;
                    const uint8_t* xsrc = xs + ((size_t)xb * T + t) * XT;
                    for (int h = 0; h < 2; ++h) {
                        const int xslot = hq % NXH;
                        if (hq >= NXH && !mbar_wait_ab(&xempty[xslot], (unsigned)((hq / NXH - 1) & 1), abrt)) {
                            ok = false;
                            break;
                        }
                        uint8_t* st = xring + xslot * XH;
                        mbar_expect_tx(&xfull[xslot], slice * (NX / 2));
                        if (slice == (uint32_t)XS) {
                            bulk_g2s(st, xsrc + h * XH, XH, &xfull[xslot]);
                        } else {
                            for (int s = 0; s < NX / 2; ++s)
                                bulk_g2s(st + s * XS, xsrc + h * XH + s * XS, slice, &xfull[xslot]);
                        }
                        ++hq;
                    }
                }
            }
            if (*abrt) {
                // copies still in flight land before the shared memory goes back
                for (int q2 = max(0, q - NAS); q2 < q; ++q2) mbar_wait(&bfull[q2 % NAS], (unsigned)((q2 / NAS) & 1));
                for (int q2 = max(0, hq - NXH); q2 < hq; ++q2) mbar_wait(&xfull[q2 % NXH], (unsigned)((q2 / NXH) & 1));
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int q = 0, hq = 0;
            bool ok = true;
            for (int i = 0; i < njob && ok; ++i) {
                const int kb = kblocks(blockIdx.x + i * G);
                if (i >= 1 && !mbar_wait_ab(&aempty, (unsigned)((i - 1) & 1), abrt)) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                for (int o = 0; o < kb && ok; ++o, ++q) {
                    const int bs = q % NAS;
                    if (!mbar_wait_ab(&bfull[bs], (unsigned)((q / NAS) & 1), abrt)) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = smem_u32(bring + bs * AT);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int xslot = hq % NXH;
                        if (!mbar_wait_ab(&xfull[xslot], (unsigned)((hq / NXH) & 1), abrt)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;");
                        const uint32_t sx = smem_u32(xring + xslot * XH);
#pragma unroll
                        for (int jj = 0; jj < NX / 2; ++jj) {
                            const int j = h * (NX / 2) + jj;
                            const int cols = KD * (j == 0 ? NA : NG - j);      // groups j .. min(j + 7, 8)
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks) {
                                // columns 256 .. 287 are first written by j = 1 of the first K step: its
                                // rows i < 7 accumulate, the last group starts there
                                const uint64_t xd = smem_desc(sx + jj * XS + ks * 256, 128, 512);
                                if (j == 1 && o == 0 && ks == 0) {
                                    mma_bf16(tmem + KD, xd, smem_desc(sa, 128, 512), instr_desc(128, KD * 7), 1u);
                                    mma_bf16(tmem + KD * 8, xd, smem_desc(sa + 7 * KD * 64, 128, 512),
                                             instr_desc(128, KD), 0u);
                                } else {
                                    mma_bf16(tmem + KD * j, xd, smem_desc(sa + ks * 256, 128, 512),
                                             instr_desc(128, cols), (o > 0 || j > 0 || ks > 0) ? 1u : 0u);
                                }
                            }
                        }
                        mma_commit(&xempty[xslot]);
                        ++hq;
                    }
                    if (ok) mma_commit(&bempty[bs]);
                }
                if (ok) mma_commit(&afull);
            }
            // MMAs in flight complete before the TMEM and shared memory go back
            if (*abrt && hq > 0) mbar_wait(&xempty[(hq - 1) % NXH], (unsigned)(((hq - 1) / NXH) & 1));
        }
    } else {
        // epilogue: two warps per TMEM lane quarter, 16 of the 32 output reals each
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const int jl = quarter * 32 + lane, j = 128 * t + jl;
        const int ex = j < N ? (int)(mxx[j] >> 52) : 0;
        double2 dyx = make_double2(0.0, 0.0);
        double dyy = 0.0;
        bool ok = true;
        for (int i = 0; i < njob; ++i) {
            const int job = blockIdx.x + i * G;
            // exponents of the eight rows, two a word
            const uint4 ew = *reinterpret_cast<const uint4*>(re + (long long)job * D + half * 8);
            const uint32_t ea[4] = {ew.x, ew.y, ew.z, ew.w};
            // (no infinity or NaN among the column and the rows)
            bool by_sums = ex == 0x7ff;
#pragma unroll
            for (int p = 0; p < 8; ++p) by_sums = by_sums || ((ea[p / 2] >> (16 * (p & 1))) & 0xFFFF) == 0x7ff;
            if (MODE != 4 && xe && j < N) {
                int near = 0;
#pragma unroll
                for (int dir = 0; dir < 5; ++dir)
                    near = max(near, (int)xe[(size_t)nbr_site(job, dir, lx, lt) * N + j]);
                by_sums = by_sums || (near > 0 && (near == 0x7ff || near + kSpread < ex));
            }
            if (!mbar_wait_ab(&afull, (unsigned)(i & 1), abrt)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const long long row0 = (long long)(MODE == 4 ? job / splits : job) * D;
            double2* yo = MODE == 4 ? y + (long long)(job % splits) * nblk * D * N : y;
            const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 16);
            uint32_t r[NG][16];
#pragma unroll
            for (int g = 0; g < NG; ++g)
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                    "%13, %14, %15}, [%16];"
                    : "=r"(r[g][0]), "=r"(r[g][1]), "=r"(r[g][2]), "=r"(r[g][3]), "=r"(r[g][4]), "=r"(r[g][5]),
                      "=r"(r[g][6]), "=r"(r[g][7]), "=r"(r[g][8]), "=r"(r[g][9]), "=r"(r[g][10]), "=r"(r[g][11]),
                      "=r"(r[g][12]), "=r"(r[g][13]), "=r"(r[g][14]), "=r"(r[g][15])
                    : "r"(base + (uint32_t)(g * KD)));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&aempty);               // the accumulator may be overwritten
            if (by_sums && j < N) {
                double2 s[8];
                if (MODE != 4) rows_by_fp64(s, A, x, job, half * 8, lx, lt, N, j);
#pragma unroll 1
                for (int p = 0; p < 8; ++p) {
                    const long long idx = (row0 + half * 8 + p) * N + j;
                    double2 o = MODE == 4 ? make_double2(NAN, NAN) : s[p];
                    if (MODE == 1) o = csub(b[idx], o);
                    if (MODE != 3) yo[idx] = o;
                    if (MODE == 2 || MODE == 3) {
                        cfmac(dyx, o, x[idx]);
                        dyy = fma(o.x, o.x, fma(o.y, o.y, dyy));
                    }
                }
            } else if (j < N) {
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const int sc = ex + (int)((ea[p / 2] >> (16 * (p & 1))) & 0xFFFF) - (2 * 1022 + 68);
                    double v[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        int Gi[NG];
#pragma unroll
                        for (int g = 0; g < NG; ++g) Gi[g] = __float2int_rn(__uint_as_float(r[g][2 * p + u]));
                        v[u] = combine(Gi, sc);
                    }
                    const long long idx = (row0 + half * 8 + p) * N + j;
                    double2 o = make_double2(v[0], v[1]);
                    if (MODE == 1) o = csub(b[idx], o);
                    if (MODE != 3) yo[idx] = o;
                    if (MODE == 2 || MODE == 3) {
                        cfmac(dyx, o, x[idx]);
                        dyy = fma(o.x, o.x, fma(o.y, o.y, dyy));
                    }
                }
            }
        }
        if (MODE == 2 || MODE == 3) {
            // the two halves of a rhs meet in shared memory (the rings are free: every copy
            // has landed and every MMA has completed once the last accumulator was read)
            double* red = reinterpret_cast<double*>(smem);
            asm volatile("bar.sync 1, %0;" ::"r"(32 * EPI_WARPS));
            if (half == 1) {
                red[3 * jl] = dyx.x;
                red[3 * jl + 1] = dyx.y;
                red[3 * jl + 2] = dyy;
            }
            asm volatile("bar.sync 1, %0;" ::"r"(32 * EPI_WARPS));
            if (half == 0 && ok && j < N) {
                part[(long long)j * G + blockIdx.x] = make_double2(dyx.x + red[3 * jl], dyx.y + red[3 * jl + 1]);
                part[(long long)(N + j) * G + blockIdx.x] = make_double2(dyy + red[3 * jl + 2], 0.0);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (tid == 0 && abort_flag) atomicExch(err, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS));
}

// y = sum over the splits of a dense product, in order.
__global__ void __launch_bounds__(256) k_sum_splits(double2* __restrict__ y, const double2* __restrict__ p,
                                                    long long count, int splits) {
    if (grid_dependency()) return;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
         e += (long long)gridDim.x * blockDim.x) {
        double2 s = p[e];
        for (int z = 1; z < splits; ++z) s = cadd(s, p[z * count + e]);
        y[e] = s;
    }
}
}  // namespace f64
}  // namespace tc

using namespace tc::f64;

static int f64_tiles(int N) { return (N + 127) / 128; }

bool f64_tc_supported(int d, int N) { return d == D && f64_tiles(N) <= 65535; }
int f64_dense_splits(int n) { return (n / D + KSPLIT - 1) / KSPLIT; }
static long long operand_jobs(long long nblk, int nb) { return nb ? (long long)nb * f64_dense_splits(nb * D) : nblk / 5; }
size_t f64_tc_operand_bytes(long long nblk, int nb) {
    return (size_t)nblk * AT + (size_t)operand_jobs(nblk, nb) * D * sizeof(uint16_t);
}
static size_t max_bytes(int N) { return ((size_t)N * sizeof(u64) + 255) / 256 * 256; }
size_t f64_tc_scratch_bytes(long long nblk, int N) {
    return (size_t)nblk * f64_tiles(N) * XT + max_bytes(N) + ((size_t)nblk * N * sizeof(uint16_t) + 255) / 256 * 256;
}

void launch_absmax_cols(u64* out, const double2* x, long long n, int N, cudaStream_t s) {
    MG_CUDA(cudaMemsetAsync(out, 0, sizeof(u64) * N, s));
    int bx = 1;
    while (bx < N && bx < 32) bx *= 2;
    const int by = 256 / bx, gx = (N + bx - 1) / bx;
    const long long need = (n + 4 * by - 1) / (4 * by);
    const int gy = (int)std::max(1LL, std::min(need, 8LL * kNumSM / gx));
    MG_LAUNCH(dim3(gx, gy), dim3(bx, by), 0, s, k_absmax_cols, out, x, n, N);
    MG_LAUNCHED();
}

// Operand: the digit tiles, then the exponents of the rows of every job.
static const uint16_t* operand_rows(const void* op, long long nblk) {
    return reinterpret_cast<const uint16_t*>(reinterpret_cast<const uint8_t*>(op) + (size_t)nblk * AT);
}

void launch_f64_operand(void* op, const double2* A, long long nblk, int nb, int ld, cudaStream_t s) {
    MG_REQUIRE(nblk >= 1 && nblk <= (1LL << 31) - 1, MGMLMC_EINVAL, "FP64 operand: size");
    uint16_t* re = const_cast<uint16_t*>(operand_rows(op, nblk));
    const int splits = nb ? f64_dense_splits(nb * D) : 1;
    MG_LAUNCH((unsigned)operand_jobs(nblk, nb), 128, 0, s, k_row_exponents, re, A, nb, splits, nb ? ld : D);
    MG_LAUNCHED();
    MG_LAUNCH((unsigned)nblk, 128, 0, s, k_slice_a, reinterpret_cast<uint8_t*>(op), A, re, nblk, nb, splits, nb ? ld : D);
    MG_LAUNCHED();
}

// Slices x into the scratch: digit tiles, then the largest entry per rhs and (sites) the exponents
// per site and rhs, with the largest of the finite entries.
static const uint16_t* site_exponents(const u64* mx, int N) {
    return reinterpret_cast<const uint16_t*>(reinterpret_cast<const uint8_t*>(mx) + max_bytes(N));
}
static const u64* slice_x(void* scratch, const double2* x, long long nblk, int N, bool sites, cudaStream_t s) {
    const int T = f64_tiles(N);
    u64* mx = reinterpret_cast<u64*>(reinterpret_cast<uint8_t*>(scratch) + (size_t)nblk * T * XT);
    if (sites) {
        MG_CUDA(cudaMemsetAsync(mx, 0, sizeof(u64) * N, s));
        int cx = 1;
        while (cx < N && cx < 32) cx *= 2;
        const int cy = 256 / cx, gx = (N + cx - 1) / cx;
        const int gy = (int)std::max(1LL, std::min((4 * nblk + cy - 1) / cy, 8LL * kNumSM / gx));
        MG_LAUNCH(dim3(gx, gy), dim3(cx, cy), 0, s, k_absmax_sites, mx, const_cast<uint16_t*>(site_exponents(mx, N)), x,
                  (int)nblk, N);
        MG_LAUNCHED();
    } else {
        launch_absmax_cols(mx, x, nblk * D, N, s);
    }
    int bx = 8;
    while (bx < N && bx < 128) bx *= 2;
    const int by = 128 / bx;
    MG_LAUNCH(dim3((unsigned)((4 * nblk + by - 1) / by), T), dim3(bx, by), 0, s, k_slice_x, reinterpret_cast<uint8_t*>(scratch), x, mx, (int)nblk, N, T);
    MG_LAUNCHED();
    return mx;
}

template <int MODE>
static void f64_launch(double2* y, const double2* b, const double2* x, const void* scratch, const void* op,
                       const u64* mxx, const uint16_t* xe, const uint16_t* re, const double2* A, int lx, int lt, int nblk,
                       int splits, int N, double2* part, int groups, int* err, cudaStream_t s) {
    MG_CUDA(cudaFuncSetAttribute(k_block_f64<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
    MG_LAUNCH(dim3(groups, f64_tiles(N)), THREADS, SMEM, s, (k_block_f64<MODE>), y, b, x, reinterpret_cast<const uint8_t*>(scratch), reinterpret_cast<const uint8_t*>(op), mxx, xe, re, A, lx,
              lt, nblk, splits, N, part, err);
    MG_LAUNCHED();
}

int block_stencil_f64_groups(int nsites, int N) {
    return std::max(1, std::min(nsites, kNumSM / f64_tiles(N)));
}

void launch_block_stencil_f64(double2* y, const double2* x, const double2* b, const void* op, const double2* A, int lx,
                              int lt, int N, int mode, bool entrywise, void* scratch, double2* part, int groups, int* err, cudaStream_t s) {
    const int V = lx * lt;
    MG_REQUIRE(f64_tc_supported(D, N) && groups >= 1 && groups <= V, MGMLMC_EINVAL, "FP64 stencil: size");
    const u64* mxx = slice_x(scratch, x, V, N, entrywise, s);
    const uint16_t* xe = entrywise ? site_exponents(mxx, N) : nullptr;
    const uint16_t* re = operand_rows(op, 5LL * V);
    switch (mode) {
        case 0: f64_launch<0>(y, b, x, scratch, op, mxx, xe, re, A, lx, lt, V, 1, N, part, groups, err, s); break;
        case 1: f64_launch<1>(y, b, x, scratch, op, mxx, xe, re, A, lx, lt, V, 1, N, part, groups, err, s); break;
        case 2: f64_launch<2>(y, b, x, scratch, op, mxx, xe, re, A, lx, lt, V, 1, N, part, groups, err, s); break;
        default: f64_launch<3>(y, b, x, scratch, op, mxx, xe, re, A, lx, lt, V, 1, N, part, groups, err, s); break;
    }
}

size_t f64_dense_scratch_bytes(int n, int N) {
    const size_t a = (f64_tc_scratch_bytes(n / D, N) + 255) / 256 * 256;
    return a + (size_t)f64_dense_splits(n) * n * N * sizeof(double2);
}

void launch_dense_f64(double2* y, const double2* x, const void* op, int n, int N, void* scratch, int* err,
                      cudaStream_t s) {
    const int nb = n / D, S = f64_dense_splits(n);
    MG_REQUIRE(n % D == 0 && f64_tc_supported(D, N), MGMLMC_EINVAL, "FP64 dense product: n % 16 == 0");
    const u64* mxx = slice_x(scratch, x, nb, N, false, s);
    double2* p = reinterpret_cast<double2*>(reinterpret_cast<uint8_t*>(scratch) +
                                            (f64_tc_scratch_bytes(nb, N) + 255) / 256 * 256);
    const long long jobs = (long long)nb * S;
    const int G = (int)std::max(1LL, std::min(jobs, (long long)kNumSM / f64_tiles(N)));
    f64_launch<4>(S == 1 ? y : p, nullptr, nullptr, scratch, op, mxx, nullptr, operand_rows(op, (long long)nb * nb),
                  nullptr, 0, 0, nb, S, N, nullptr, G, err, s);
    if (S > 1) {
        const long long cnt = (long long)n * N;
        MG_LAUNCH((int)std::min((cnt + 255) / 256, 16LL * kNumSM), 256, 0, s, k_sum_splits, y, p, cnt, S);
        MG_LAUNCHED();
    }
}

}  // namespace mg
