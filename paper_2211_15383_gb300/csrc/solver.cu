// Solver layer: operator application per level, the multigrid cycle used as a
// preconditioner (Sect. 3.1, Eq. two_level_mg_method applied recursively), the
// multi-RHS flexible GMRES, and the FP64 outer solve (plain FP64 FGMRES, or
// FP64 iterative refinement around an FP32 FGMRES for the mixed mode).
//
// The smoother S^(nu) is nu steps of minimal residual (GMRES(1)) per rhs: one
// of the Krylov smoothers Sect. 3.1 lists; FGMRES tolerates its
// non-linearity.  The coarsest level is solved by its stored dense inverse.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "context.h"

namespace mg {

template <typename C> static const C* links(Ctx& c);
template <> const double2* links<double2>(Ctx& c) { return c.U64; }
template <> const float2* links<float2>(Ctx& c) { return c.U32; }
template <typename C> static const C* blocks(const Level& L);
template <> const double2* blocks<double2>(const Level& L) { return L.A64; }
template <> const float2* blocks<float2>(const Level& L) { return L.A32; }
template <typename C> static const C* hat_blocks(const Level& L);
template <> const double2* hat_blocks<double2>(const Level& L) { return L.Ahat64; }
template <> const float2* hat_blocks<float2>(const Level& L) { return L.Ahat32; }
template <typename C> static const C* minv(const Level& L);
template <> const double2* minv<double2>(const Level& L) { return L.Minv64; }
template <> const float2* minv<float2>(const Level& L) { return L.Minv32; }
template <typename C> static const C* prol(const Level& L);
template <> const double2* prol<double2>(const Level& L) { return L.P64; }
template <> const float2* prol<float2>(const Level& L) { return L.P32; }

static std::string nm(const char* base, int l, size_t sz) {
    std::string s(base);
    s += '_';
    s += (char)('0' + l);
    s += '_';
    if (sz >= 10) s += '1';
    s += (char)('0' + sz % 10);
    return s;
}

static const char* prec_tag(size_t sz) { return sz == sizeof(double2) ? "f64" : "f32"; }

// On the first coarse level D_2 = P_1^H D_1 P_1 (the Galerkin product); in FP64,
// where the pipe issues 2 FMA per SM and clock, restrict(Wilson(prolong(x))) can be
// cheaper than the 5-point stencil with dense d x d blocks.
static bool galerkin_form_cheaper(const Ctx& c, int l) {
    if (l != 1) return false;
    const Level& F = c.lev[0];
    const Level& Cl = c.lev[1];
    const double galerkin = 16.0 * F.nvec * F.n + 60.0 * F.nsites;   // prolong + restrict + Wilson
    const double direct = 40.0 * Cl.d * Cl.d * Cl.nsites;            // 5 blocks of d x d per site
    return galerkin < direct;
}

// FP64 block stencils with d = 16 run on the tensor cores (exact integer digit products, in the
// norm as accurate as FP64 sums, entry by entry with c.entrywise) from kF64TcMinRhs right-hand sides on, where the level has its digits
// and their work space is granted.  op: the level's own pointer (an allocation may take the
// digits away).
template <typename C>
static bool f64_stencil(Ctx&, const Level&, C*, const C*, const C*, void* const&, const C*, int, int, double2*, int) {
    return false;
}
static bool f64_stencil_used(const Level& L, const void* op, int N) {
    return op && N >= kF64TcMinRhs && f64_tc_supported(L.d, N);
}
template <>
bool f64_stencil<double2>(Ctx& c, const Level& L, double2* y, const double2* x, const double2* b, void* const& op,
                          const double2* A, int N, int mode, double2* part, int groups) {
    int* err = device_error_flag(c);
    if (!f64_stencil_used(L, op, N)) return false;
    void* scr = c.try_scratch("f64_tc", f64_tc_scratch_bytes(L.nsites, N));
    if (!scr) return false;
    launch_block_stencil_f64(y, x, b, op, A, L.lx, L.lt, N, mode, c.entrywise, scr, part, groups, err, c.stream);
    return true;
}
template <typename C> static int bst_groups(const Level& L, const void* op, int N) {
    return sizeof(C) == 16 && f64_stencil_used(L, op, N) ? block_stencil_f64_groups(L.nsites, N)
                                                         : block_stencil_groups(L.nsites, L.d, N);
}

template <typename C> static bool galerkin_apply(Ctx&, C*, const C*, const C*, int, int) { return false; }
template <> bool galerkin_apply<double2>(Ctx& c, double2* y, const double2* x, const double2* b, int N, int mode) {
    if (mode >= 2 || f64_stencil_used(c.lev[1], c.lev[1].A64t, N) || !galerkin_form_cheaper(c, 1)) return false;
    const Level& F = c.lev[0];
    const Level& Cl = c.lev[1];
    double2* t = c.scratch<double2>("gal64_t", (size_t)F.n * N);
    double2* u = c.scratch<double2>("gal64_u", (size_t)F.n * N);
    apply_prolong<double2>(c, 0, t, x, N, false);
    apply_D<double2>(c, 0, u, t, nullptr, N, 0, nullptr);
    if (mode == 0) {
        apply_restrict<double2>(c, 0, y, u, N);
        return true;
    }
    double2* v = c.scratch<double2>("gal64_v", (size_t)Cl.n * N);
    apply_restrict<double2>(c, 0, v, u, N);
    MG_CUDA(cudaMemcpyAsync(y, b, sizeof(double2) * Cl.n * N, cudaMemcpyDeviceToDevice, c.stream));
    launch_axpy_rhs<double2, double2>(y, nullptr, nullptr, -1.0, v, Cl.n, N, c.stream);
    return true;
}

// The minimal-residual coefficients from a stencil's partial dots.
template <typename C>
static void mr_alpha(Ctx& c, C* alpha, const double2* part, int groups, int N) {
    ProfScope ps(c, "reduce", (double)groups * 2 * N * 16, (double)groups * 2 * N * 2);
    launch_finalize_alpha<C>(alpha, part, groups, N, c.stream);
}

template <typename C>
void apply_D(Ctx& c, int l, C* y, const C* x, const C* b, int N, int mode, C* alpha) {
    if (l == 1 && galerkin_apply<C>(c, y, x, b, N, mode)) return;
    const Level& L = c.lev[l];
    const int groups = (l == 0) ? stencil_groups(L.nsites, N) : bst_groups<C>(L, L.A64t, N);
    // algorithmic traffic: read x once, write y once (+ b for the residual form),
    // operator data once; flops: 60 per fine site and rhs, 8 d^2 * 5 per coarse site and rhs
    const double s = sizeof(C);
    const double vec = (double)L.n * N * s;
    const double bytes = vec * (mode == 1 ? 3 : mode == 3 ? 1 : 2) +
                         (l == 0 ? 2.0 * L.nsites * s : 5.0 * L.nsites * L.d * L.d * s);
    const double flops = (l == 0) ? 60.0 * L.nsites * N : 40.0 * L.d * L.d * (double)L.nsites * N;
    double2* part = nullptr;
    if (mode >= 2) part = c.scratch<double2>("part_st", (size_t)groups * 2 * N);
    {
        ProfScope ps(c, {"D", l + 1, ".", prec_tag(sizeof(C))}, bytes, flops);
        if (l == 0)
            launch_wilson<C>(y, x, b, links<C>(c), c.m0, L.lx, L.lt, N, mode, part, groups, c.stream);
        else if (!f64_stencil<C>(c, L, y, x, b, L.A64t, blocks<C>(L), N, mode, part, groups))
            launch_block_stencil<C>(y, x, b, blocks<C>(L), L.lx, L.lt, L.d, N, mode, part, groups, c.stream);
    }
    if (mode >= 2) mr_alpha<C>(c, alpha, part, groups, N);
}

int* device_error_flag(Ctx& c) {
    if (!c.dev_err) {
        c.dev_err = c.scratch<int>("dev_err", 1);
        MG_CUDA(cudaMemsetAsync(c.dev_err, 0, sizeof(int), c.stream));
    }
    return c.dev_err;
}

// The block stencil of D M^{-1} runs on the tensor cores (BF16 operands, FP32
// accumulation) when mg_precision is 16 and d = 16: the smoother only
// preconditions the FP32 FGMRES, whose own matrix-vector products stay FP32.
template <typename C> static bool tc_smoother(const Level&, int) { return false; }
template <> bool tc_smoother<float2>(const Level& L, int N) { return L.Ahat16 && tc_stencil_supported(L.d, N); }

// BF16 tiles of one level-l block vector.
static __nv_bfloat16* tc_tiles(Ctx& c, const char* name, int l, int N) {
    return reinterpret_cast<__nv_bfloat16*>(c.scratch_bytes(nm(name, l, 2), tc_tiles_bytes(c.lev[l].nsites, N)));
}

// A multigrid cycle (or a smoother operator) is running: its residuals are in use.
struct CycleScope {
    Ctx& c;
    explicit CycleScope(Ctx& ctx) : c(ctx) { ++c.cycles; }
    ~CycleScope() { --c.cycles; }
};

// y = (D_l M_l^{-1}) x on the tensor cores, x given as its BF16 tiles xt, y as FP32 rows
// (y) or BF16 tiles (yt), or only alpha (may be null) = <y, x> / <y, y> (against the BF16 x).
static void apply_Dhat_tc(Ctx& c, int l, float2* y, __nv_bfloat16* yt, const __nv_bfloat16* xt, int N,
                          float2* alpha) {
    const Level& L = c.lev[l];
    const int groups = block_stencil_tc_groups(L.nsites, N);
    double2* part = c.scratch<double2>("part_st", (size_t)groups * 2 * N);
    {
        // algorithmic traffic: BF16 x (4 B per complex) and y (FP32 8 B or BF16 4 B) once,
        // the BF16 operands once
        ProfScope ps(c, {"D", l + 1, ".bf16"},
                     (double)L.n * N * (4 + (yt ? 4 : y ? 8 : 0)) + 5.0 * L.nsites * 8.0 * L.d * L.d,
                     40.0 * L.d * L.d * (double)L.nsites * N);
        launch_block_stencil_tc(y, yt, nullptr, xt, L.Ahat16, L.lx, L.lt, N, part, groups, device_error_flag(c),
                                c.stream);
    }
    if (alpha) mr_alpha<float2>(c, alpha, part, groups, N);
}

static void pack_tiles(Ctx& c, int l, __nv_bfloat16* xt, const float2* x, int N) {
    const Level& L = c.lev[l];
    ProfScope ps(c, {"pack", l + 1, ".bf16"}, (double)L.n * N * (8 + 4), 0.0);
    launch_pack_tiles_bf16(xt, x, L.nsites, N, c.stream);
}

// y = (D_l M_l^{-1}) x with the precomputed block stencil (block-Jacobi smoother); mode 0, 2
// or 3 as apply_D.
template <typename C>
static void apply_Dhat(Ctx& c, int l, C* y, const C* x, int N, int mode, C* alpha) {
    const Level& L = c.lev[l];
    const int groups = bst_groups<C>(L, L.Ahat64t, N);
    const double s = sizeof(C);
    double2* part = mode >= 2 ? c.scratch<double2>("part_st", (size_t)groups * 2 * N) : nullptr;
    {
        ProfScope ps(c, {"D", l + 1, ".", prec_tag(sizeof(C))},
                     (double)L.n * N * s * (mode == 3 ? 1 : 2) + 5.0 * L.nsites * L.d * L.d * s,
                     40.0 * L.d * L.d * (double)L.nsites * N);
        if (!f64_stencil<C>(c, L, y, x, (const C*)nullptr, L.Ahat64t, hat_blocks<C>(L), N, mode, part, groups))
            launch_block_stencil<C>(y, x, nullptr, hat_blocks<C>(L), L.lx, L.lt, L.d, N, mode, part, groups, c.stream);
    }
    if (mode >= 2) mr_alpha<C>(c, alpha, part, groups, N);
}

template <typename C> static bool apply_smoother_tc(Ctx&, int, C*, const C*, int) { return false; }
template <> bool apply_smoother_tc<float2>(Ctx& c, int l, float2* y, const float2* x, int N) {
    if (!tc_smoother<float2>(c.lev[l], N)) return false;
    __nv_bfloat16* xt = tc_tiles(c, "mr_rt", l, N);
    pack_tiles(c, l, xt, x, N);
    apply_Dhat_tc(c, l, y, nullptr, xt, N, nullptr);
    return true;
}

template <typename C>
void apply_smoother_operator(Ctx& c, int l, C* y, const C* x, int N) {
    MG_REQUIRE(l >= 1 && l < c.L - 1 && hat_blocks<C>(c.lev[l]), MGMLMC_EINVAL,
               "smoother operator: only coarse levels above the coarsest");
    const CycleScope running(c);
    if (!apply_smoother_tc<C>(c, l, y, x, N)) apply_Dhat<C>(c, l, y, x, N, 0, nullptr);
}

template <typename C>
void apply_restrict(Ctx& c, int l, C* xc, const C* x, int N) {
    const Level& L = c.lev[l];
    const double s = sizeof(C);
    ProfScope ps(c, {"PH", l + 1, ".", prec_tag(sizeof(C))},
                 (double)L.n * N * s + (double)c.lev[l + 1].n * N * s + (double)L.n * L.nvec * s,
                 8.0 * L.nvec * (double)L.n * N);
    launch_restrict<C>(xc, x, prol<C>(L), L.lx, L.lt, L.d, L.ax, L.at, L.nvec, N, c.stream);
}

template <typename C>
bool apply_prolong(Ctx& c, int l, C* x, const C* xc, int N, bool accumulate, void* xt) {
    const Level& L = c.lev[l];
    const double s = sizeof(C);
    ProfScope ps(c, {"P", l + 1, ".", prec_tag(sizeof(C))},
                 (double)L.n * N * s * (accumulate ? 2 : 1) + (double)c.lev[l + 1].n * N * s + (double)L.n * L.nvec * s,
                 8.0 * L.nvec * (double)L.n * N);
    return launch_prolong<C>(x, xc, prol<C>(L), L.lx, L.lt, L.d, L.ax, L.at, L.nvec, N, accumulate, c.stream, xt);
}

// Few right-hand sides of a small level are solved by the FP32 inverse in one launch, whose time
// goes with n (its dependent loads) and with the power of two of columns that N fills (each
// matrix entry's arithmetic); the BF16 form on the tensor cores takes three launches, 15 us up
// to n = 1024 whatever N.  Measured, us (with the launch gaps), for 2, 4, 8, 16 and 32 columns:
//   n = 256: 8.0, 6.7, 6.5, 8.1, 10.5;  n = 512: 8.0, 7.5, 8.2, 10.2, 16.2;
//   n = 1024: 8.2, 9.6, 12.3, 18.3, 30.6;  n = 2048: 14, 21, 33, 57, 107 (BF16: 17).
// Solves on the levels above take the same iterations with either (16 to 19 at 64^2), those on the
// coarsest level itself fewer with the FP32 inverse (six inverse iterations of 16 rhs at n = 1024:
// 23 for 36 to 1e-12, 18 for 24 to 1e-7), so that 16 columns at n = 1024 pay there (deflation of
// 64^2 182 ms, 194 with BF16; the pilot draw 7.49 and 7.42) and 32 columns, at twice the other
// form's time, do not.  The line: columns times n.  A level without the BF16 inverse (n no multiple of 128) takes the one launch throughout (960 unknowns:
// 8.3 to 29 us, the tiled FP32 product 43 to 66).
constexpr long long kFewRhs = 32, kFewRhsWork = 16384, kFewRhsUnknowns = 1024;
static bool few_rhs(const Level& L, int N) {
    long long cols = 1;
    while (cols < N) cols *= 2;
    return N < kFewRhs && L.n <= kFewRhsUnknowns && (!L.Dinv16 || cols * L.n <= kFewRhsWork);
}
template <typename C> static void coarsest_apply(Ctx& c, C* e, const C* r, int N);
static double dinv_bytes(const Level& L, int N, double s) { return (double)L.n * L.n * s + 2.0 * L.n * N * s; }
static double dinv_flops(const Level& L, int N) { return 8.0 * (double)L.n * L.n * N; }
template <> void coarsest_apply<double2>(Ctx& c, double2* e, const double2* r, int N) {
    const Level& L = c.lev[c.L - 1];
    ProfScope ps(c, "Dinv.f64", dinv_bytes(L, N, 16), dinv_flops(L, N));
    int* err = device_error_flag(c);
    if (L.Dinv64t && N >= kF64TcMinRhs && f64_tc_supported(16, N)) {
        if (void* scr = c.try_scratch("f64_dense", f64_dense_scratch_bytes((int)L.n, N))) {
            launch_dense_f64(e, r, L.Dinv64t, (int)L.n, N, scr, err, c.stream);
            return;
        }
    }
    launch_gemm_nn<double2>(e, L.Dinv64, r, (int)L.n, (int)L.n, N, false, c.stream);
}
template <> void coarsest_apply<float2>(Ctx& c, float2* e, const float2* r, int N) {
    const Level& L = c.lev[c.L - 1];
    if (few_rhs(L, N)) {
        ProfScope ps(c, "Dinv.f32", dinv_bytes(L, N, 8), dinv_flops(L, N));
        launch_gemm_few(e, L.Dinv32, r, (int)L.n, N, c.stream);
        return;
    }
    if (L.Dinv16) {
        // BF16 inverse on the tensor cores; algorithmic bytes: the BF16 matrix once + FP32 in/out
        ProfScope ps(c, "Dinv.bf16", (double)L.n * 2 * L.n * 2 + 2.0 * L.n * N * 8, dinv_flops(L, N));
        void* scr = c.scratch_bytes("tc_scratch", coarse_inverse_bf16_scratch((int)L.n, N));
        launch_coarse_inverse_bf16(e, r, L.Dinv16, (int)L.n, N, scr, device_error_flag(c), c.stream);
        return;
    }
    ProfScope ps(c, "Dinv.f32", dinv_bytes(L, N, 8), dinv_flops(L, N));
    launch_gemm_nn<float2>(e, L.Dinv32, r, (int)L.n, (int)L.n, N, false, c.stream);
}

// Minimal-residual steps are taken in groups of at most kSmootherGroup: the residuals of a
// group stay in consecutive slots, and the correction takes sum_s alpha_s r_s once per
// group.  Slots for nu steps of `bytes` each, as many as the memory allows (one at least: it is
// updated in place); K: their number.
static void* mr_slots(Ctx& c, const std::string& name, size_t bytes, int nu, int& K) {
    for (K = std::min(smoother_slots(nu), c.smoother_group); K > 1; K = c.smoother_group = (K + 1) / 2)
        if (void* p = c.try_scratch(name, K * bytes)) {
            c.extra_residuals = true;
            return p;
        }
    return c.scratch_bytes(name, bytes);
}

// The group loop, for any form of the vectors: image(s, last) forms the image of slot s and
// its coefficient (the last step of all needs no image), flush(K, first) adds the K slots to
// the correction, update(s, t) forms the next residual from slot s in slot t.  Returns the
// slot of the final residual (with need_r), else -1.
template <typename Image, typename Flush, typename Update>
static int mr_steps(int nu, int K, bool need_r, Image image, Flush flush, Update update) {
    int slot = 0;
    for (int s = 0; s < nu; ++s) {
        const bool last = s + 1 == nu && !need_r;
        image(slot, last);
        if (slot + 1 == K || s + 1 == nu) flush(slot + 1, s < K);
        if (last) return -1;
        const int next = (slot + 1) % K;
        update(slot, next);
        slot = next;
    }
    return slot;
}

// Post-smoothing of the V-cycle on the tensor cores: the residual r - D_l e is formed
// from BF16 tiles of e (et) straight into the smoother's BF16 residual tiles (it only
// feeds the smoother, which needs a few digits), then nu block-Jacobi MR steps with r and p
// only as BF16 tiles; e += M^{-1} sum_s alpha_s r_s.
template <typename C> static bool post_smooth_tc(Ctx&, int, C*, const C*, int, bool) { return false; }
template <typename C> static bool post_smooths_tc(const Ctx&, int, int) { return false; }
template <> bool post_smooths_tc<float2>(const Ctx& c, int l, int N) {
    const Level& L = c.lev[l];
    return c.opt.nu_post > 0 && L.A16 && tc_smoother<float2>(L, N);
}

template <>
bool post_smooth_tc<float2>(Ctx& c, int l, float2* e, const float2* r, int N, bool have_et) {
    if (!post_smooths_tc<float2>(c, l, N)) return false;
    const Level& L = c.lev[l];
    const int nu = c.opt.nu_post;
    float2* alpha = c.scratch<float2>(nm("mr_al", l, sizeof(float2)), (size_t)kSmootherGroup * N);
    __nv_bfloat16* et = tc_tiles(c, "cyc_et", l, N);
    __nv_bfloat16* pt = tc_tiles(c, "mr_pt", l, N);
    int K = 1;
    __nv_bfloat16* rt = reinterpret_cast<__nv_bfloat16*>(mr_slots(c, nm("mr_rt", l, 2), tc_tiles_bytes(L.nsites, N), nu, K));
    const size_t slot = tc_tiles_bytes(L.nsites, N) / sizeof(__nv_bfloat16);
    if (!have_et) pack_tiles(c, l, et, e, N);
    {
        const int groups = block_stencil_tc_groups(L.nsites, N);
        // algorithmic traffic: e tiles (4 B per complex) and r (8 B) read, residual tiles written (4 B)
        ProfScope ps(c, {"D", l + 1, "res.bf16"},
                     (double)L.n * N * (4 + 8 + 4) + 5.0 * L.nsites * 8.0 * L.d * L.d,
                     40.0 * L.d * L.d * (double)L.nsites * N);
        launch_block_stencil_tc(nullptr, rt, r, et, L.A16, L.lx, L.lt, N, nullptr, groups, device_error_flag(c),
                                c.stream);
    }
    mr_steps(
        nu, K, false,
        [&](int s, bool last) { apply_Dhat_tc(c, l, nullptr, last ? nullptr : pt, rt + s * slot, N, alpha + (size_t)s * N); },
        [&](int k, bool) {
            // traffic: the K residuals (4 B per complex) read, e read and written
            ProfScope ps(c, {"bjac", l + 1, ".bf16"}, (double)L.n * N * (4 * k + 16),
                         8.0 * (L.d + k) * (double)L.n * N);
            launch_block_diag_tiles(e, rt, k, alpha, L.Minv32, L.nsites, N, c.stream);
        },
        [&](int s, int t) {
            // traffic: r and p tiles read, the next r tiles written (4 B per complex)
            ProfScope ps(c, {"mr", l + 1, ".bf16"}, (double)L.n * N * 12, 8.0 * L.n * N);
            launch_mr_update_tiles(rt + t * slot, rt + s * slot, pt, alpha + (size_t)s * N, L.nsites, N, c.stream);
        });
    return true;
}

// Pre-smoothing with the image on the tensor cores: the residual stays FP32 (the caller
// restricts it) and each update writes the next step's tiles.
template <typename C> static bool pre_smooth_tc(Ctx&, int, C*, C*, int, int) { return false; }
template <>
bool pre_smooth_tc<float2>(Ctx& c, int l, float2* e, float2* r, int N, int nu) {
    const Level& L = c.lev[l];
    if (!tc_smoother<float2>(L, N)) return false;
    float2* yh = c.scratch<float2>(nm("mr_y", l, sizeof(float2)), (size_t)L.n * N);
    float2* p = c.scratch<float2>(nm("mr_p", l, sizeof(float2)), (size_t)L.n * N);
    float2* alpha = c.scratch<float2>(nm("mr_al", l, sizeof(float2)), (size_t)kSmootherGroup * N);
    __nv_bfloat16* rt = tc_tiles(c, "mr_rt", l, N);
    pack_tiles(c, l, rt, r, N);
    for (int s = 0; s < nu; ++s) {
        apply_Dhat_tc(c, l, p, nullptr, rt, N, alpha);
        const bool more = s + 1 < nu;
        ProfScope ps(c, {"mr", l + 1, ".f32"}, (double)L.n * N * (5 * 8 + (more ? 4 : 0)),
                     16.0 * L.n * N);
        launch_mr_update_tc(yh, r, p, alpha, L.nsites, N, s == 0, more ? rt : nullptr, c.stream);
    }
    ProfScope ps(c, {"bjac", l + 1, ".f32"}, 3.0 * L.n * N * sizeof(float2),
                 8.0 * L.d * (double)L.n * N);
    launch_block_diag_apply<float2>(e, yh, L.Minv32, L.nsites, L.d, N, false, c.stream);
    return true;
}

// Post-smoothing of the fine level with r and p in BF16 (mg_precision 16): the same few
// digits as the coarse smoother, half the traffic of the FP32 vectors; the residual r - D e
// is formed in FP32 and rounded as it is written, the correction e stays FP32.
template <typename C> static bool post_smooth_fine_bf16(Ctx&, int, C*, const C*, int) { return false; }
template <>
bool post_smooth_fine_bf16<float2>(Ctx& c, int l, float2* e, const float2* r, int N) {
    const int nu = c.opt.nu_post;
    if (l != 0 || nu <= 0 || c.opt.mg_precision != 16 || N % 4) return false;
    const Level& L = c.lev[0];
    const size_t nN = (size_t)L.n * N;
    uint32_t* pb = c.scratch<uint32_t>("mrf_pb", nN);
    float2* alpha = c.scratch<float2>(nm("mr_al", 0, sizeof(float2)), (size_t)kSmootherGroup * N);
    const int groups = stencil_groups_bf16(L.nsites, N);
    double2* part = c.scratch<double2>("part_st", (size_t)groups * 2 * N);
    int K = 1;
    uint32_t* rb = reinterpret_cast<uint32_t*>(mr_slots(c, "mrf_rb", nN * sizeof(uint32_t), nu, K));
    {
        // algorithmic traffic: e and r read (8 B each), the BF16 residual written
        ProfScope ps(c, "D1res.bf16", (double)nN * 20 + 2.0 * L.nsites * 8, 60.0 * L.nsites * N);
        launch_wilson_residual_bf16(rb, e, r, c.U32, c.m0, L.lx, L.lt, N, stencil_groups(L.nsites, N), c.stream);
    }
    mr_steps(
        nu, K, false,
        [&](int s, bool last) {
            {
                // algorithmic traffic: BF16 x read, y written once (4 B per complex), links once
                ProfScope ps(c, "D1.bf16", (double)nN * (last ? 4 : 8) + 2.0 * L.nsites * 8, 60.0 * L.nsites * N);
                launch_wilson_bf16(last ? nullptr : pb, rb + s * nN, c.U32, c.m0, L.lx, L.lt, N, part, groups,
                                   c.stream);
            }
            mr_alpha<float2>(c, alpha + (size_t)s * N, part, groups, N);
        },
        [&](int k, bool) {
            ProfScope ps(c, "mr1sum.bf16", (double)nN * (4 * k + 16), 8.0 * k * nN);
            launch_mr_combine_bf16(e, rb, nN, k, alpha, L.n, N, c.stream);
        },
        [&](int s, int t) {
            // traffic: r and p read, the next r written (4 B each)
            ProfScope ps(c, "mr1.bf16", (double)nN * 12, 8.0 * nN);
            launch_mr_update_fine_bf16(rb + t * nN, rb + s * nN, pb, alpha + (size_t)s * N, L.n, N, c.stream);
        });
    return true;
}

// nu MR steps on D_l e = r0 starting from e (or 0); rs has K slots, the first
// holding the current residual.  Returns the slot with the final residual (need_r).  On
// coarse levels above the coarsest: block-Jacobi MR, minimal-residual steps on D M^{-1}
// whose preconditioned correction M^{-1} sum_s alpha_s r_s goes to e.
template <typename C>
static C* mr_smooth(Ctx& c, int l, C* e, C* rs, int K, int N, int nu, bool e_zero, bool need_r) {
    const Level& L = c.lev[l];
    const size_t nN = (size_t)L.n * N;
    C* p = c.scratch<C>(nm("mr_p", l, sizeof(C)), nN);
    C* alpha = c.scratch<C>(nm("mr_al", l, sizeof(C)), (size_t)kSmootherGroup * N);
    const bool jacobi = hat_blocks<C>(L) != nullptr;
    const int fin = mr_steps(
        nu, K, need_r,
        [&](int s, bool last) {
            const int mode = last ? 3 : 2;
            if (jacobi) apply_Dhat<C>(c, l, last ? nullptr : p, rs + s * nN, N, mode, alpha + (size_t)s * N);
            else apply_D<C>(c, l, last ? nullptr : p, rs + s * nN, nullptr, N, mode, alpha + (size_t)s * N);
        },
        [&](int k, bool first) {
            const bool zero = e_zero && first;
            if (jacobi) {
                ProfScope ps(c, {"bjac", l + 1, ".", prec_tag(sizeof(C))}, (k + (zero ? 1.0 : 2.0)) * nN * sizeof(C), 8.0 * (L.d + k) * (double)nN);
                launch_block_diag_combine<C>(e, rs, nN, k, alpha, minv<C>(L), L.nsites, L.d, N, !zero, c.stream);
            } else {
                ProfScope ps(c, {"mr", l + 1, "sum.", prec_tag(sizeof(C))},
                             (k + (zero ? 1.0 : 2.0)) * nN * sizeof(C), 8.0 * k * (double)nN);
                launch_mr_combine<C>(e, rs, nN, k, alpha, L.n, N, zero, c.stream);
            }
        },
        [&](int s, int t) {
            ProfScope ps(c, {"mr", l + 1, ".", prec_tag(sizeof(C))}, 3.0 * nN * sizeof(C), 8.0 * (double)nN);
            // with a single slot the update is in place
            launch_mr_update<C>(rs + t * nN, rs + s * nN, p, alpha + (size_t)s * N, L.n, N, c.stream);
        });
    return fin >= 0 ? rs + fin * nN : nullptr;
}

// A maximum that the next reduction writes (NormOut::max and ::clear, or launch_rotate's) and
// read_max returns.  Four in turn: at most two are taken between two reads.  Each is taken
// right before the launch that it is for (nothing in between may fail: that launch also
// clears the place of the turn after the next).
constexpr int kMaxSlots = 4;
constexpr int kMaxRestart = 64;   // columns of a cycle at most
struct MaxSlot {
    int i = 0;
    unsigned long long *at = nullptr, *clear = nullptr;
};
static MaxSlot take_max(Ctx& c) {
    if (!c.dev_max) {
        c.dev_max = c.scratch<unsigned long long>("dev_max", kMaxSlots);
        MG_CUDA(cudaMemsetAsync(c.dev_max, 0, kMaxSlots * sizeof(unsigned long long), c.stream));
        c.max_turn = 0;
    }
    MaxSlot m;
    m.i = c.max_turn;
    m.at = c.dev_max + m.i;
    m.clear = c.dev_max + (m.i + 2) % kMaxSlots;
    c.max_turn = (m.i + 1) % kMaxSlots;
    return m;
}
// Value of one slot (and of another read with it); waits for the stream.
static double read_max(Ctx& c, const MaxSlot& m, const MaxSlot* also = nullptr, double* also_v = nullptr) {
    MG_CUDA(cudaMemcpyAsync(c.hbuf, c.dev_max, kMaxSlots * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
    c.sync();
    if (also) *also_v = c.hbuf[also->i];
    return c.hbuf[m.i];
}

template <typename C>
static void norms(Ctx& c, const NormOut& o, const C* x, long long n, int N) {
    launch_norm<C>(o, x, n, N, c.scratch_bytes("part_nrm", norm_part_bytes(n, N)), c.stream);
}

// One Arnoldi basis of the multi-RHS flexible GMRES with its per-rhs bookkeeping.
//
// The basis is kept unnormalised, w_i = eta_i v_i with eta_i = |w_i| per rhs: the
// Gram-Schmidt coefficients are divided by eta_i^2, the Hessenberg column by eta_i eta_j, and
// the correction takes y_j / eta_j of z_j = M(w_j).  This is FGMRES on the normalised basis
// exactly (the preconditioner of each step is whatever maps v_j to z_j / eta_j: no property
// of M is assumed) and saves the pass that would scale each new vector.  A vector whose eta
// leaves [2^-32, 2^32] (an iteration run on past convergence shrinks it by the FP32
// rounding level each step) is rescaled to unit norm, only for that rhs.
template <typename C>
struct Basis {
    C *V, *Z, *cf;
    double2 *H, *g, *sn, *irr;
    double *hsub, *cs, *eta, *ieta, *rsc;
    void *part, *npart;
    long long n;
    int N, m;
    C* v(int j) const { return V + (size_t)j * n * N; }
    C* z(int j) const { return Z + (size_t)j * n * N; }
};

template <typename C>
static Basis<C> basis(Ctx& c, const char* name, int l, long long n, int m, int N) {
    const size_t sz = sizeof(C), nN = (size_t)n * N;
    const std::string p = name;
    Basis<C> B;
    B.n = n;
    B.N = N;
    B.m = m;
    B.V = c.scratch<C>(nm((p + "_V").c_str(), l, sz), (size_t)(m + 1) * nN);
    B.Z = c.scratch<C>(nm((p + "_Z").c_str(), l, sz), (size_t)m * nN);
    B.cf = c.scratch<C>(nm((p + "_cf").c_str(), l, sz), (size_t)(m + 1) * N);
    B.H = c.scratch<double2>(nm((p + "_H").c_str(), l, sz), (size_t)m * (m + 1) * N);
    B.g = c.scratch<double2>(nm((p + "_g").c_str(), l, sz), (size_t)(m + 1) * N);
    B.sn = c.scratch<double2>(nm((p + "_sn").c_str(), l, sz), (size_t)m * N);
    B.irr = c.scratch<double2>(nm((p + "_irr").c_str(), l, sz), (size_t)m * N);
    B.hsub = c.scratch<double>(nm((p + "_hs").c_str(), l, sz), (size_t)m * N);
    B.cs = c.scratch<double>(nm((p + "_cs").c_str(), l, sz), (size_t)m * N);
    B.eta = c.scratch<double>(nm((p + "_eta").c_str(), l, sz), (size_t)(m + 1) * N);
    B.ieta = c.scratch<double>(nm((p + "_ieta").c_str(), l, sz), (size_t)(m + 1) * N);
    B.rsc = c.scratch<double>(nm((p + "_rsc").c_str(), l, sz), N);
    // own partials: a K-cycle runs inside an outer step
    B.part = c.scratch_bytes(nm((p + "_part").c_str(), l, sz), dot_part_bytes(n, N, m));
    B.npart = c.scratch_bytes(nm((p + "_npart").c_str(), l, sz), norm_part_bytes(n, N));
    return B;
}

// The reduction of the first vector's norm: eta_0 and g_0 with it.
template <typename C>
static NormOut basis_start(const Basis<C>& B) {
    NormOut o;
    o.eta = B.eta;
    o.ieta = B.ieta;
    o.rsc = B.rsc;
    o.g0 = B.g;
    return o;
}

// Step j after u = D M(w_j) was formed in v(j + 1): classical Gram-Schmidt (passes times) and
// the Hessenberg column j.
template <typename C>
static void arnoldi_step(Ctx& c, const Basis<C>& B, int j, int passes) {
    const double nN = (double)B.n * B.N, sz = sizeof(C);
    // algorithmic bytes: the j+1 basis vectors read once per Gram-Schmidt pass; the
    // implementation reads them twice (dot products, then the update) and reads w twice and
    // writes it once per pass: (2j + 5) vectors
    ProfScope ps(c, {"orth.", -1, prec_tag(sizeof(C))}, passes * (j + 1) * nN * sz,
                 passes * 2.0 * 8.0 * (j + 1) * nN, passes * (2 * j + 5) * nN * sz);
    C* u = B.v(j + 1);
    double2* H = B.H + (size_t)j * (B.m + 1) * B.N;
    NormOut o;
    o.eta = B.eta + (size_t)(j + 1) * B.N;
    o.ieta = B.ieta + (size_t)(j + 1) * B.N;
    o.rsc = B.rsc;
    o.hsub = B.hsub + (size_t)j * B.N;
    o.eta_prev = B.eta + (size_t)j * B.N;
    for (int p = 0; p < passes; ++p) {
        launch_multidot<C>(B.cf, H, B.V, j + 1, u, B.n, B.N, B.ieta, p > 0, B.part, c.stream);
        // the norm is summed over u / eta_j (FP32 squares of a small vector would leave the
        // normal range)
        launch_multiaxpy<C>(u, B.cf, j + 1, B.V, B.n, B.N, true, p + 1 == passes ? &o : nullptr, B.npart,
                            B.ieta + (size_t)j * B.N, c.stream);
    }
    if (j + 1 < B.m) launch_scale_cols_if<C>(u, B.rsc, B.n, B.N, c.stream);
}

// x (=|+=) Z y after column j.
template <typename C>
static void basis_update(Ctx& c, const Basis<C>& B, int j, C* x, bool accumulate) {
    launch_back_substitute<C>(B.cf, B.H, B.g, B.irr, B.ieta, j, B.m, B.N, c.stream);
    launch_multiaxpy<C>(x, B.cf, j + 1, B.Z, B.n, B.N, accumulate, nullptr, nullptr, nullptr, c.stream);
}

// K-cycle coarse-grid correction: e ~ D_l^{-1} r by k steps of flexible GMRES from
// e = 0, preconditioned by the multigrid cycle of level l.  A fixed number of steps
// with no convergence test, so nothing is read back to the host; the Arnoldi
// bookkeeping (Givens rotations, least-squares solve) runs per rhs on the device.
template <typename C>
static void kcycle(Ctx& c, int l, C* e, const C* r, int N, int k) {
    const long long n = c.lev[l].n;
    const Basis<C> B = basis<C>(c, "kc", l, n, k, N);
    launch_scale_norm<C, C>(basis_start(B), B.V, r, nullptr, false, n, N, B.npart, c.stream);
    launch_scale_cols_if<C>(B.V, B.rsc, n, N, c.stream);
    for (int j = 0; j < k; ++j) {
        mg_cycle<C>(c, l, B.z(j), B.v(j), N);
        apply_D<C>(c, l, B.v(j + 1), B.z(j), nullptr, N, 0, nullptr);
        arnoldi_step<C>(c, B, j, 1);
    }
    launch_rotate(B.H, B.hsub, B.cs, B.sn, B.g, B.irr, nullptr, nullptr, nullptr, 0, k - 1, k, N, c.stream);
    basis_update<C>(c, B, k - 1, e, false);
}

template <typename C>
void mg_cycle(Ctx& c, int l, C* e, const C* r, int N) {
    if (l == c.L - 1) {
        coarsest_apply<C>(c, e, r, N);
        return;
    }
    const CycleScope running(c);
    const Level& L = c.lev[l];
    const Level& Lc = c.lev[l + 1];
    C* rc = c.scratch<C>(nm("cyc_rc", l + 1, sizeof(C)), (size_t)Lc.n * N);
    C* ec = c.scratch<C>(nm("cyc_ec", l + 1, sizeof(C)), (size_t)Lc.n * N);
    const size_t nN = (size_t)L.n * N;
    int K = 1;
    auto residual_slots = [&](int nu) { return reinterpret_cast<C*>(mr_slots(c, nm("cyc_res", l, sizeof(C)), sizeof(C) * nN, nu, K)); };
    bool e_zero = true;
    if (c.opt.nu_pre > 0) {
        // the pre-smoother on the tensor cores keeps one residual
        C* res = residual_slots(tc_smoother<C>(L, N) ? 1 : c.opt.nu_pre);
        MG_CUDA(cudaMemcpyAsync(res, r, sizeof(C) * nN, cudaMemcpyDeviceToDevice, c.stream));
        // leaves res = r - D e
        if (!pre_smooth_tc<C>(c, l, e, res, N, c.opt.nu_pre))
            res = mr_smooth<C>(c, l, e, res, K, N, c.opt.nu_pre, true, true);
        e_zero = false;
        apply_restrict<C>(c, l, rc, res, N);
    } else {
        apply_restrict<C>(c, l, rc, r, N);
    }
    if (c.opt.kcycle_iters > 0 && l + 2 < c.L)
        kcycle<C>(c, l + 1, ec, rc, N, c.opt.kcycle_iters);
    else
        mg_cycle<C>(c, l + 1, ec, rc, N);
    // the prolongation also writes the tensor-core smoother's tiles of e where it can
    void* et = post_smooths_tc<C>(c, l, N) ? tc_tiles(c, "cyc_et", l, N) : nullptr;
    const bool have_et = apply_prolong<C>(c, l, e, ec, N, !e_zero, et);
    if (c.opt.nu_post <= 0 || post_smooth_tc<C>(c, l, e, r, N, have_et) || post_smooth_fine_bf16<C>(c, l, e, r, N))
        return;
    C* res = residual_slots(c.opt.nu_post);
    apply_D<C>(c, l, res, e, r, N, 1, nullptr);
    mr_smooth<C>(c, l, e, res, K, N, c.opt.nu_post, false, false);
}

// One Arnoldi cycle from the started basis B (first vector, eta_0, g_0): at most B.m steps,
// ended once the residual estimate (relative to bnorm) reaches tol or it reaches maxit; then
// x (=|+=) the correction.
template <typename C>
static void fgmres_cycle(Ctx& c, int l, const Basis<C>& B, C* x, bool accumulate, const double* bnorm, double tol,
                         long long& it, long long maxit, bool inner) {
    const int N = B.N, m = B.m;
    // Inner cycles of the refinement loop converge in a repeatable number of steps per level
    // and tolerance: the host reads the residual estimates (a round trip that leaves the GPU
    // idle) only from two steps before the last such count on.  It reads those of every
    // column: a cycle ends with the first that meets tol, whatever steps were taken after it, so
    // that the counts of earlier calls change its time and nothing else.
    int* hint = nullptr;
    if (inner) {
        const int dec = std::min(15, std::max(0, (int)std::floor(-std::log10(tol))));
        hint = &c.cycle_hint[((long long)l * 16 + dec) * (1LL << 32) + N];
    }
    const int check_from = hint ? std::max(1, *hint - 2) : 1;
    // classical Gram-Schmidt: twice in FP64; once in the FP32 inner solve of the refinement
    // loop, whose FP64 residual absorbs the loss of orthogonality
    const int passes = sizeof(C) == sizeof(double2) ? 2 : 1;
    unsigned long long* dmax = nullptr;
    double* est = c.hbuf + kMaxSlots;            // squares of the estimates, per column
    if (N > kRotateWarp) {
        dmax = c.scratch<unsigned long long>("fg_est", kMaxRestart);
        MG_CUDA(cudaMemsetAsync(dmax, 0, m * sizeof(unsigned long long), c.stream));
    }
    int j = 0, rotated = 0;
    for (bool done = false; !done; ++j) {
        mg_cycle<C>(c, l, B.z(j), B.v(j), N);
        apply_D<C>(c, l, B.v(j + 1), B.z(j), nullptr, N, 0, nullptr);
        arnoldi_step<C>(c, B, j, passes);
        ++it;
        if (j + 1 < check_from && j + 1 < m && it < maxit) continue;
        // up to 32 rhs one warp writes the maxima to the host itself
        launch_rotate(B.H, B.hsub, B.cs, B.sn, B.g, B.irr, bnorm, dmax, dmax ? nullptr : est, rotated, j, m, N, c.stream);
        if (dmax)
            MG_CUDA(cudaMemcpyAsync(est + rotated, dmax + rotated, (j + 1 - rotated) * sizeof(double),
                                    cudaMemcpyDeviceToHost, c.stream));
        c.sync();
        for (; rotated <= j && !done; ++rotated) {
            if (est[rotated] != est[rotated]) throw Error(MGMLMC_ENAN, "FGMRES: NaN in Arnoldi");
            done = std::sqrt(est[rotated]) <= tol;
        }
        if (done) {
            it -= j + 1 - rotated;               // steps beyond it were not needed
            j = rotated - 1;
        }
        done |= it >= maxit || j + 1 >= m;
    }
    --j;                                         // the last column
    if (hint) *hint = j + 1;
    basis_update<C>(c, B, j, x, accumulate);
}

template <typename C>
long long fgmres(Ctx& c, int l, const C* b, C* x, int N, double tol, long long maxit, bool x_zero, int* ok,
                 int max_cycles) {
    const long long n = c.lev[l].n;
    const Basis<C> B = basis<C>(c, "fg", 0, n, c.opt.fgmres_restart, N);
    double* bnorm = c.scratch<double>(nm("fg_bn", 0, sizeof(C)), N);
    // x = 0 is not written: the first correction overwrites x (or x is zeroed on exit)
    bool x_unset = x_zero;
    long long it = 0;
    int cycles = 0;
    *ok = 0;
    if (!x_unset) {
        NormOut o;
        o.norm = bnorm;
        norms<C>(c, o, b, n, N);
    }
    for (;;) {
        if (!x_unset) apply_D<C>(c, l, B.V, x, b, N, 1, nullptr);
        const MaxSlot ms = take_max(c);
        NormOut o = basis_start(B);
        o.max = ms.at;
        o.clear = ms.clear;
        if (x_unset) {
            o.norm = bnorm;
            launch_scale_norm<C, C>(o, B.V, b, nullptr, false, n, N, B.npart, c.stream);
        } else {
            o.den = bnorm;
            launch_norm<C>(o, B.V, n, N, B.npart, c.stream);
        }
        const double ratio = read_max(c, ms);
        if (ratio != ratio) throw Error(MGMLMC_ENAN, "FGMRES: NaN residual");
        if (c.opt.verbose)
            fprintf(stderr, "[mgmlmc] fgmres level %d prec %zu it %lld true rel res %.3e\n", l + 1, sizeof(C) * 4, it,
                    ratio);
        if (ratio <= tol) {
            *ok = 1;
            break;
        }
        if (it >= maxit) break;
        launch_scale_cols_if<C>(B.V, B.rsc, n, N, c.stream);
        fgmres_cycle<C>(c, l, B, x, !x_unset, bnorm, tol, it, maxit, max_cycles == 1);
        x_unset = false;
        if (++cycles >= max_cycles) {
            *ok = 1;
            break;
        }
    }
    if (x_unset) launch_zero<C>(x, n * N, c.stream);
    return it;
}

static long long solve_block(Ctx& c, int l, const double2* b, double2* x, int N, double tol, int* ok);

// Blocks wider than opt.max_block_rhs (the eigensolvers' subspaces) are solved in
// column chunks of at most that width, so the Krylov work space stays bounded.
long long solve(Ctx& c, int l, const double2* b, double2* x, int N, double tol, int* ok) {
    const int blk = c.opt.max_block_rhs;
    if (N <= blk) return with_less_memory(c, [&] { return solve_block(c, l, b, x, N, tol, ok); });
    const long long n = c.lev[l].n;
    double2* bb = c.scratch<double2>("sv_chunk_b", (size_t)n * blk);
    double2* xb = c.scratch<double2>("sv_chunk_x", (size_t)n * blk);
    const size_t w = sizeof(double2);
    long long it = 0;
    int all = 1;
    for (int j0 = 0; j0 < N; j0 += blk) {
        const int nb = std::min(blk, N - j0);
        MG_CUDA(cudaMemcpy2DAsync(bb, nb * w, b + j0, (size_t)N * w, nb * w, (size_t)n, cudaMemcpyDeviceToDevice,
                                  c.stream));
        int okb = 0;
        it += with_less_memory(c, [&] { return solve_block(c, l, bb, xb, nb, tol, &okb); });
        all &= okb;
        MG_CUDA(cudaMemcpy2DAsync(x + j0, (size_t)N * w, xb, nb * w, nb * w, (size_t)n, cudaMemcpyDeviceToDevice,
                                  c.stream));
    }
    *ok = all;
    c.last_iters = it;
    return it;
}

static long long solve_block(Ctx& c, int l, const double2* b, double2* x, int N, double tol, int* ok) {
    const long long maxit = c.opt.max_iters;
    if (c.opt.mg_precision == 64) {
        const long long it = fgmres<double2>(c, l, b, x, N, tol, maxit, true, ok, 1 << 30);
        c.last_iters = it;
        check_device_error(c);
        return it;
    }
    // Mixed: FP64 iterative refinement, FP32 FGMRES + FP32 multigrid inside.
    const long long n = c.lev[l].n;
    const size_t nN = (size_t)n * N;
    double2* r = c.scratch<double2>("ir_r", nN);
    // the FP32 rhs of each inner cycle is built in the inner FGMRES's first basis vector
    const Basis<float2> B = basis<float2>(c, "fg", 0, n, c.opt.fgmres_restart, N);
    float2* e32 = c.scratch<float2>("ir_e32", nN);
    double* bnorm = c.scratch<double>("ir_bn", N);
    double* rnorm = c.scratch<double>("ir_rn", N);
    double* inorm = c.scratch<double>("ir_in", N);
    void* npart = c.scratch_bytes("part_nrm", norm_part_bytes(n, N));
    // In the estimator's solves (c.fp32_residual_updates) the next residual comes from an
    // FP32 product, r <- r - |r| D e, between FP64 ones.  Its error against
    // the FP64 residual b - D x is below kFp32Product ||D|| |e| |r| (rounding of the FP32
    // operator and of the product's sums), with ||D_l|| <= ||D_1|| <= |m0 + 2| + 4 (each
    // hopping term has norm 1, the prolongators have orthonormal columns).  On the 256^2
    // workload the errors measured at the FP64 recomputations were 11 to 14 times below
    // this bound on all levels (verbose mode prints both).  |e| carries the
    // cancellation: a correction much longer than its residual (a rhs near the
    // near-kernel, as in the setup's inverse iteration) makes the FP32 product inexact.
    // drift bounds the error accumulated since the last FP64 residual (relative to |b|,
    // max over the rhs); the FP64 residual is recomputed once drift exceeds 1 % of the
    // residual, and for the convergence decision unless drift is below tol / 20.  Cycles
    // that reduce the residual a little then share one FP64 residual, which on a coarse
    // level costs as much as tens of FP32 products (d = 16: 1/64 of the FP32 FMA rate).
    // Every other solve (the setup's inverse iteration and the eigensolvers, whose
    // right-hand sides lie near the near-kernel) takes the FP64 residual after every
    // cycle but the last: below 500 tol the FP32 product's error (under 1e-4 |r|) stays
    // below tol / 20 of |b|.
    constexpr double kFp32Product = 4.0 * 0x1p-24;
    constexpr double kRecursiveResidual = 500.0;
    const bool fp32_updates = c.fp32_residual_updates;
    const double dnorm = std::fabs(c.m0 + 2.0) + 4.0;
    double drift = 0.0;
    // r = b, its norm; a reduction that gives |r| also gives max |r| / |b|
    const double* rn = bnorm;
    auto residual_norm = [&](const MaxSlot& ms) {
        NormOut o;
        o.norm = rnorm;
        o.den = bnorm;
        o.max = ms.at;
        o.clear = ms.clear;
        rn = rnorm;
        return o;
    };
    double ratio;
    {
        const MaxSlot ms = take_max(c);
        NormOut o;
        o.norm = bnorm;
        o.max = ms.at;
        o.clear = ms.clear;
        launch_scale_norm<double2, double2>(o, r, b, nullptr, false, n, N, npart, c.stream);
        ratio = read_max(c, ms);
    }
    auto fp64_residual = [&] {
        apply_D<double2>(c, l, r, x, b, N, 1, nullptr);
        const MaxSlot ms = take_max(c);
        launch_norm<double2>(residual_norm(ms), r, n, N, npart, c.stream);
        ratio = read_max(c, ms);
    };
    long long it = 0;
    bool x_unset = true;                         // x = 0 is written by the first correction
    *ok = 0;
    // cycles until the FP64 residual meets tol or the iteration budget is spent
    for (int cycle = 0;; ++cycle) {
        if (ratio != ratio) throw Error(MGMLMC_ENAN, "refinement: NaN residual");
        if (drift > 0.0 && (drift > 1e-2 * ratio || (ratio <= tol && drift > tol / 20))) {
            double2* rrec = nullptr;
            if (c.opt.verbose) {
                rrec = c.scratch<double2>("ir_rrec", nN);
                MG_CUDA(cudaMemcpyAsync(rrec, r, sizeof(double2) * nN, cudaMemcpyDeviceToDevice, c.stream));
            }
            fp64_residual();
            if (rrec) {
                // the error the FP32 updates actually made, against the bound
                launch_axpy_rhs<double2, double2>(rrec, nullptr, nullptr, -1.0, r, n, N, c.stream);
                const MaxSlot ms = take_max(c);
                NormOut o;
                o.den = bnorm;
                o.max = ms.at;
                o.clear = ms.clear;
                launch_norm<double2>(o, rrec, n, N, npart, c.stream);
                fprintf(stderr, "[mgmlmc] refine level %d FP64 residual: FP32 drift %.3e (bound %.3e)\n", l + 1,
                        read_max(c, ms), drift);
            }
            drift = 0.0;
            continue;
        }
        if (c.opt.verbose)
            fprintf(stderr, "[mgmlmc] refine level %d cycle %d it %lld rel res %.3e\n", l + 1, cycle, it, ratio);
        if (ratio <= tol) {
            *ok = 1;
            break;
        }
        if (it >= maxit) break;
        // one FGMRES cycle in FP32 on r / |r|: its own FP32 residual cannot certify more than
        // ~1e-6 relative, so the FP64 residual of this loop decides on restarts
        const double inner_tol = std::max(c.inner.floor, c.inner.margin * tol / ratio);
        NormOut start = basis_start(B);
        start.norm = inorm;
        launch_scale_norm<float2, double2>(start, B.V, r, rn, true, n, N, npart, c.stream);
        fgmres_cycle<float2>(c, l, B, e32, false, inorm, inner_tol, it, maxit, true);
        if (!fp32_updates && ratio > kRecursiveResidual * tol) {
            launch_refine_axpy(x, rn, 1.0, e32, n, N, !x_unset, nullptr, nullptr, npart, c.stream);
            x_unset = false;
            fp64_residual();
            continue;
        }
        // x += |r| e and, for the bound of this update, max_j |e_j| |r_j| / |b_j|; then
        // r -= |r| D e (without fp32_updates the last cycle: accepted on this residual)
        const MaxSlot md = take_max(c);
        NormOut oe;
        oe.max = md.at;
        oe.clear = md.clear;
        oe.den = bnorm;
        oe.mul = rn;
        launch_refine_axpy(x, rn, 1.0, e32, n, N, !x_unset, &oe, nullptr, npart, c.stream);
        x_unset = false;
        float2* de = c.scratch<float2>("ir_de32", nN);
        apply_D<float2>(c, l, de, e32, nullptr, N, 0, nullptr);
        const MaxSlot ms = take_max(c);
        const double* scale = rn;
        const NormOut orr = residual_norm(ms);
        launch_refine_axpy(r, scale, -1.0, de, n, N, true, nullptr, &orr, npart, c.stream);
        double er = 0.0;
        ratio = read_max(c, ms, &md, &er);
        if (fp32_updates) drift += kFp32Product * dnorm * er;
    }
    if (x_unset) launch_zero<double2>(x, (long long)nN, c.stream);
    c.last_iters = it;
    check_device_error(c);
    return it;
}

void check_device_error(Ctx& c) {
    if (!c.dev_err) return;
    int h = 0;
    MG_CUDA(cudaMemcpyAsync(&h, c.dev_err, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    c.sync();
    if (h) {
        MG_CUDA(cudaMemsetAsync(c.dev_err, 0, sizeof(int), c.stream));
        throw Error(MGMLMC_ETIMEOUT, "a tensor-core kernel gave up waiting on an mbarrier (bounded wait)");
    }
}

#define INST(C)                                                                                           \
    template void apply_D<C>(Ctx&, int, C*, const C*, const C*, int, int, C*);                              \
    template void apply_restrict<C>(Ctx&, int, C*, const C*, int);                                          \
    template bool apply_prolong<C>(Ctx&, int, C*, const C*, int, bool, void*);                              \
    template void mg_cycle<C>(Ctx&, int, C*, const C*, int);                                                \
    template void apply_smoother_operator<C>(Ctx&, int, C*, const C*, int);                                 \
    template long long fgmres<C>(Ctx&, int, const C*, C*, int, double, long long, bool, int*, int);
INST(double2)
INST(float2)

}  // namespace mg

namespace mg {
void column_norms(Ctx& c, double* out, const double2* x, long long n, int N) {
    NormOut o;
    o.norm = out;
    norms<double2>(c, o, x, n, N);
}

void approx_inverse(Ctx& c, int l, const double2* b, double2* x, int N) {
    int ok = 0;
    if (c.opt.mg_precision == 64) {
        with_less_memory(c, [&] { return fgmres<double2>(c, l, b, x, N, 1e-14, c.opt.fgmres_restart, true, &ok, 1); });
        return;
    }
    const size_t nN = (size_t)c.lev[l].n * N;
    float2* b32 = c.scratch<float2>("ai_b32", nN);
    float2* x32 = c.scratch<float2>("ai_x32", nN);
    unsigned long long* mx = c.scratch<unsigned long long>("unit_mx", N);
    const long long n = c.lev[l].n;
    launch_absmax_cols(mx, b, n, N, c.stream);
    launch_to_unit(b32, b, mx, n, N, c.stream);
    with_less_memory(c, [&] { return fgmres<float2>(c, l, b32, x32, N, 1e-6, c.opt.fgmres_restart, true, &ok, 1); });
    launch_from_unit(x, x32, mx, n, N, c.stream);
}
}  // namespace mg
