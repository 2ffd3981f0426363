"""The calls that a user of this library makes, as measurable cases.

A user sets up a trace problem (gauge field, mass, multigrid hierarchy, deflation)
once and then draws Hutchinson samples of the terms of the telescoping sum, in blocks
of right-hand sides, until the statistical error is small enough.  The kinds of case:

* ``samples``  one step of the estimator: ``estimate_level`` on every term (or one
  term) of the sum, one block of device-drawn Z2 vectors each;
* ``probes``   the same for one term with the caller's own Z2 vectors (host int8);
* ``solve``    ``D_l x = b`` for a handful of host right-hand sides;
* ``setup``    gauge upload, inverse iteration and the Galerkin hierarchy;
* ``deflate``  the k smallest singular triplets of the coarsest operator;
* ``trace``    the whole multilevel Monte Carlo loop to a relative error.

Lattices, couplings, masses, aggregates and blocks are those of the workloads in
``inputs``, of the benchmark's serving mix and of the GPU tests.  Gauge fields are
drawn here (von Mises plaquettes in a random gauge: the 2D U(1) Wilson action's local
distribution), so that a lattice of any size takes milliseconds; test vectors are
relaxed random vectors handed over with ``setup_iters = 0``, so that the hierarchy is
a function of the inputs alone.
"""
import math

import numpy as np
import torch

import paper_2211_15383_gb300 as pkg

DEV = "cuda" if torch.cuda.is_available() else "cpu"
C128 = torch.complex128


def _case(name, kind, lx, lt, beta, m0, agg, nvec, prec, n, **kw):
    c = dict(name=name, kind=kind, lx=lx, lt=lt, beta=beta, m0=m0, agg=agg, nvec=nvec, prec=prec, n=n,
             k=0, terms=len(agg.split(",")) + 1, term=-1, restart=24, nu=4, kcycle=0, level=1, tol=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest estimate: the 16x16 workload with the library's default options
        # (FP64 throughout), every term, one block of 64 samples.  Latency and launches.
        _case("step-16x16-f64", "samples", 16, 16, 3.0, -0.10, "4x4", "4", 64, 64, k=16),
        # The pilot draw that starts every multilevel loop: 16 samples per term on the
        # smallest lattice that the serving mix holds.
        _case("pilot-64x64", "samples", 64, 64, 3.0, -0.09, "4x4,2x2", "8,8", 16, 16, k=32),
        # A block of the 128x128 workload: 256 samples on each of three terms in the
        # benchmark's precision, the last term deflated.
        _case("step-128x128", "samples", 128, 128, 3.0, -0.10, "4x4,2x2", "8,8", 16, 256, k=64),
        # A ragged problem: oblong lattice, levels of d = 8 and 16, an odd number of
        # samples, the FP32 multigrid.
        _case("ragged-160x96-f32", "samples", 160, 96, 5.0, -0.03, "4x4,2x2", "4,8", 32, 75),
        # The FP64 multigrid (the default precision) on a middle-sized lattice.
        _case("step-64x64-f64", "samples", 64, 64, 5.0, -0.03, "4x4,2x2", "8,8", 64, 64),
        # The last, deflated term of the 256x256 workload (level 3, k = 128, a
        # solver-only level below it) with the caller's own noise vectors, 512 at a time.
        _case("probes-256x256-last", "probes", 256, 256, 5.0, -0.05, "4x4,2x2,2x2", "8,8,8", 16, 512, k=128,
              terms=3, term=2),
        # The largest lattice of the serving mix: a block of 128 samples on each of the
        # three terms (levels of 524288 / 262144 / 65536 unknowns, 4096 below).
        _case("step-512x512", "samples", 512, 512, 5.0, -0.03, "4x4,2x2,4x4", "8,8,8", 16, 128, terms=3, restart=8),
        # A few right-hand sides solved through the host interface, as a caller with its
        # own sources does (and as the setup's inverse iteration does inside).
        _case("solve-128x128-8rhs", "solve", 128, 128, 3.0, -0.09, "4x4,2x2", "8,8", 16, 8),
        # The setup of a served 64x64 request: four rounds of inverse iteration.
        _case("setup-64x64", "setup", 64, 64, 5.0, 0.02, "4x4,2x2", "8,8", 16, 1),
        # The deflation of a served 64x64 request's coarsest operator (1024 unknowns).
        _case("deflate-64x64", "deflate", 64, 64, 3.0, -0.04, "4x4,2x2", "8,8", 32, 1, k=32),
        # A whole multilevel Monte Carlo estimate to relative error 2e-3: many small
        # blocks of whatever width the allocation asks for.
        _case("trace-32x32", "trace", 32, 32, 3.0, -0.09, "4x4,2x2", "8,8", 16, 1, k=16, tol=2e-3),
    ]


def draw(rng):
    """One more case: a kind by its share of use, sizes over the ranges above."""
    def even(lo, hi, step):   # log-uniform multiple of step
        return max(lo, min(hi, step * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)))

    kind = rng.choice(("samples", "samples", "samples", "samples", "samples", "probes", "solve", "setup", "deflate",
                       "trace"))
    beta = rng.choice((3.0, 5.0))
    m0 = round(rng.uniform(-0.09, 0.0) if beta == 3.0 else rng.uniform(-0.04, 0.05), 4)
    prec = rng.choice((16, 16, 16, 32, 64))
    if kind in ("setup", "deflate", "trace"):
        lx, lt = even(32, 64, 8), even(32, 64, 8)
        if kind == "deflate":
            prec = rng.choice((32, 16))
        return {k: v for k, v in _case("", kind, lx, lt, beta, max(m0, -0.05), "4x4,2x2", "8,8", 16 if kind == "setup"
                                       else prec if prec != 64 else 32, 1, k=rng.choice((8, 16, 24)) if
                                       kind != "setup" else 0, tol=3e-3 if kind == "trace" else 0.0).items()
                if k != "name"}
    hi = 64 if prec == 64 else 320
    lx, lt = even(16, hi, 16), even(16, hi, 16)
    # the stored inverse holds at most 4096 unknowns here: a third coarsening where the
    # first two leave more
    nv = rng.choice(("8,8", "8,8", "8,8", "4,8", "4,4"))
    agg, nvec, terms = "4x4,2x2", nv, 3
    if (lx // 8) * (lt // 8) * 2 * int(nv[-1]) > 4096 or (lx * lt >= 128 * 128 and rng.random() < 0.3):
        lx, lt = max(32, lx // 32 * 32), max(32, lt // 32 * 32)
        agg, nvec = "4x4,2x2,4x4", nv + "," + nv[-1]
    budget = 512 * 512 * 128 if prec != 64 else 64 * 64 * 64
    if kind == "solve":
        n = rng.randint(1, 24)
    else:
        n = max(1, min(512, int(budget / (lx * lt)), int(math.exp(rng.uniform(math.log(8), math.log(512))))))
        if rng.random() < 0.5:   # the even blocks that callers choose
            n = max(8, n // 8 * 8)
    c = _case("", kind, lx, lt, beta, m0, agg, nvec, prec, n, terms=terms,
              term=rng.randrange(terms) if kind == "probes" else -1, restart=rng.choice((8, 16, 24)),
              nu=rng.choice((2, 4, 4, 6)), kcycle=rng.choice((0, 0, 0, 2)) if agg.count(",") == 2 else 0,
              level=rng.choice((1, 2)) if kind == "solve" else 1)
    del c["name"]
    return c


# --------------------------------------------------------------------- inputs
def _shape(c):
    agg = [tuple(int(v) for v in a.split("x")) for a in c["agg"].split(",")]
    return agg, [int(v) for v in c["nvec"].split(",")]


def _dims(c):
    agg, nvec = _shape(c)
    dims = [(c["lx"], c["lt"], 2)]
    for (ax, at), nv in zip(agg, nvec):
        dims.append((dims[-1][0] // ax, dims[-1][1] // at, 2 * nv))
    return dims


def _gauge(c, seed):
    """Link angles [t][x][mu]: von Mises plaquettes (zero sum along every time line, as a
    periodic lattice needs) in a random gauge, with random holonomies."""
    rng = np.random.default_rng([seed, 1])
    lt, lx = c["lt"], c["lx"]
    plaq = rng.vonmises(0.0, c["beta"], (lt, lx))
    plaq -= plaq.mean(axis=0, keepdims=True)
    th = np.zeros((lt, lx, 2))
    th[1:, :, 0] = -np.cumsum(plaq, axis=0)[:-1]
    th += rng.uniform(-math.pi, math.pi, 2) / np.array([lx, lt])
    g = rng.uniform(-math.pi, math.pi, (lt, lx))
    th[..., 0] += g - np.roll(g, -1, axis=1)
    th[..., 1] += g - np.roll(g, -1, axis=0)
    return np.remainder(th + math.pi, 2 * math.pi) - math.pi


def _random(shape, seed, stream):
    gen = torch.Generator(device=DEV).manual_seed(seed * 64 + stream)
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, dtype=torch.float64, device=DEV)) / math.sqrt(2.0)


class _Op:
    """A level operator as 5-point block stencil A[t][x][dir][d][d], dir = self, +x, -x, +t, -t."""

    def __init__(self, A):
        self.A = A
        self.lt, self.lx, _, self.d, _ = A.shape

    def __call__(self, v):   # v: [lt][lx][d][N]
        y = torch.matmul(self.A[:, :, 0], v)
        for k, (s, dim) in enumerate(((-1, 1), (1, 1), (-1, 0), (1, 0)), start=1):
            y += torch.matmul(self.A[:, :, k], torch.roll(v, s, dim))
        return y


def _wilson(theta, m0):
    """D_1 = (m0 + 2) - 1/2 sum_mu [(1 - s_mu) U_mu T_+mu + (1 + s_mu) U_mu^* T_-mu],
    antiperiodic in time, s_0 = sigma_1, s_1 = sigma_2."""
    lt, lx, _ = theta.shape
    u = torch.exp(1j * torch.tensor(theta, device=DEV, dtype=torch.float64))
    eye = torch.eye(2, dtype=C128, device=DEV)
    s = [torch.tensor([[0, 1], [1, 0]], dtype=C128, device=DEV), torch.tensor([[0, -1j], [1j, 0]], dtype=C128, device=DEV)]
    u0, u1 = u[..., 0], u[..., 1].clone()
    u1[-1] *= -1.0
    A = torch.zeros(lt, lx, 5, 2, 2, dtype=C128, device=DEV)
    A[:, :, 0] = (m0 + 2.0) * eye
    A[:, :, 1] = -0.5 * u0[..., None, None] * (eye - s[0])
    A[:, :, 2] = -0.5 * torch.roll(u0, 1, 1).conj()[..., None, None] * (eye + s[0])
    A[:, :, 3] = -0.5 * u1[..., None, None] * (eye - s[1])
    A[:, :, 4] = -0.5 * torch.roll(u1, 1, 0).conj()[..., None, None] * (eye + s[1])
    return _Op(A)


def _to_agg(v, ax, at):
    """[lt][lx][d][n] -> [ct][cx][2][at ax d/2][n]: the rows of each (aggregate, spin block)."""
    lt, lx, d, n = v.shape
    v = v.reshape(lt // at, at, lx // ax, ax, 2, d // 2, n).permute(0, 2, 4, 1, 3, 5, 6)
    return v.reshape(lt // at, lx // ax, 2, at * ax * (d // 2), n)


def _from_agg(w, ax, at, d):
    ct, cx, _, _, n = w.shape
    w = w.reshape(ct, cx, 2, at, ax, d // 2, n).permute(0, 3, 1, 4, 2, 5, 6)
    return w.reshape(ct * at, cx * ax, d, n)


class _Prolong:
    """P from test vectors [lt][lx][d][nvec]: per (aggregate, spin block) Gram-Schmidt in vector order."""

    def __init__(self, v, ax, at):
        self.ax, self.at, self.d = ax, at, v.shape[2]
        q = _to_agg(v, ax, at).clone()
        for j in range(q.shape[-1]):
            for i in range(j):
                q[..., j] -= (q[..., i].conj() * q[..., j]).sum(-1, keepdim=True) * q[..., i]
            q[..., j] /= torch.linalg.vector_norm(q[..., j], dim=-1, keepdim=True)
        self.q = q                       # [ct][cx][2][rows][nvec]

    def restrict(self, v):
        y = torch.matmul(self.q.transpose(-1, -2).conj(), _to_agg(v, self.ax, self.at))
        return y.reshape(*y.shape[:2], -1, y.shape[-1])

    def prolong(self, x):
        ct, cx, _, n = x.shape
        return _from_agg(torch.matmul(self.q, x.reshape(ct, cx, 2, -1, n)), self.ax, self.at, self.d)

    def galerkin(self, op):
        """P^H D P: each hop goes to the coarse direction of the aggregate face that it crosses."""
        nv = self.q.shape[-1]
        full = torch.zeros(*self.q.shape[:4], 2 * nv, dtype=C128, device=DEV)
        full[:, :, 0, :, :nv] = self.q[:, :, 0]
        full[:, :, 1, :, nv:] = self.q[:, :, 1]
        p = _from_agg(full, self.ax, self.at, self.d)            # [lt][lx][d][2 nvec]
        ct, cx = op.lt // self.at, op.lx // self.ax
        out = torch.zeros(ct, cx, 5, 2 * nv, 2 * nv, dtype=C128, device=DEV)
        x = torch.arange(op.lx, device=DEV) % self.ax
        t = torch.arange(op.lt, device=DEV) % self.at
        for k in range(5):
            s, dim = ((0, 0), (-1, 1), (1, 1), (-1, 0), (1, 0))[k]
            m = torch.matmul(p.transpose(-1, -2).conj(), torch.matmul(op.A[:, :, k], torch.roll(p, s, dim)))
            edge = (None, x == self.ax - 1, x == 0, t == self.at - 1, t == 0)[k]
            if k == 0:
                cross = torch.zeros(op.lt, op.lx, dtype=torch.bool, device=DEV)
            else:
                cross = edge[None, :].expand(op.lt, -1) if k < 3 else edge[:, None].expand(-1, op.lx)
            for mask, to in ((cross, k), (~cross, 0)):
                g = m * mask[..., None, None]
                out[:, :, to] += g.reshape(ct, self.at, cx, self.ax, 2 * nv, 2 * nv).sum(dim=(1, 3))
        return _Op(out)


def _relax(op, v, steps):
    for _ in range(steps):
        v = v - 0.4 * op(v)
    return v / torch.linalg.vector_norm(v.reshape(-1, v.shape[-1]), dim=0)


def _hierarchy(c, seed, vectors=None):
    """(theta, operators, prolongators, start vectors per level as (nvec, n) arrays).  The
    start vectors are relaxed random vectors (restricted to the coarser levels), or given."""
    theta = _gauge(c, seed)
    agg, nvec = _shape(c)
    ops, pros, starts = [_wilson(theta, c["m0"])], [], []
    v = None
    for l, ((ax, at), nv) in enumerate(zip(agg, nvec)):
        op = ops[-1]
        if vectors is not None:
            v = vectors(l, op)
        elif l == 0:
            v = _relax(op, _random((op.lt, op.lx, op.d, max(nvec)), seed, 2), 80)
        else:
            v = _relax(op, pros[-1].restrict(v), 4)
        w = v[..., :nv].contiguous()
        pros.append(_Prolong(w, ax, at))
        starts.append(w.reshape(-1, nv).T.contiguous())
        ops.append(pros[-1].galerkin(op))
    return theta, ops, pros, starts


def _raw_vectors(c, seed):
    """The Gaussian start vectors that the setup case iterates on."""
    _, nvec = _shape(c)
    dims = _dims(c)
    return [_random((dims[l][1], dims[l][0], dims[l][2], nv), seed, 20 + l) for l, nv in enumerate(nvec)]


def _deflation_vectors(c, seed, op):
    """k orthonormal relaxed vectors of the last term's level, (k, n)."""
    v = _relax(op, _random((op.lt, op.lx, op.d, c["k"]), seed, 40), 12)
    q, _ = torch.linalg.qr(v.reshape(-1, c["k"]))
    return q.T.contiguous()


def _skip(c):
    return list(range(c["terms"] + 1, len(_shape(c)[0]) + 2))


def _noise_seed(seed):
    return 1000003 * (seed + 1)


def _probes(c, seed, n):
    return (2 * np.random.default_rng([seed, 3]).integers(0, 2, (c["n"], n), dtype=np.int8) - 1).astype(np.int8)


def _costs(c):
    n = [x * t * d for x, t, d in _dims(c)][: c["terms"]]
    return [(a + b) / n[0] for a, b in zip(n, n[1:] + [0])]


def prepare(case, seed):
    c = case
    agg, nvec = _shape(c)
    ctx = pkg.Context(mg_precision=c["prec"], max_block_rhs=min(512, max(16, c["n"])), fgmres_restart=c["restart"],
                      nu_post=c["nu"], kcycle_iters=c["kcycle"])
    s = {"case": c, "seed": seed, "ctx": ctx}
    if c["kind"] == "setup":
        s["theta"] = _gauge(c, seed)
        s["start"] = [v.reshape(-1, v.shape[-1]).T.contiguous().cpu().numpy() for v in _raw_vectors(c, seed)]
        return s
    theta, ops, pros, starts = _hierarchy(c, seed)
    ctx.set_gauge(theta)
    ctx.set_mass(c["m0"])
    ctx.set_hierarchy(agg, nvec, [v.cpu().numpy() for v in starts], setup_iters=0)
    ctx.set_terms(_skip(c))
    last = c["terms"] - 1
    if c["k"] and c["kind"] not in ("deflate",):
        ctx.set_term_deflation_vectors(last, _deflation_vectors(c, seed, ops[last]).cpu().numpy())
    if c["kind"] == "probes":
        s["probes"] = _probes(c, seed, ctx.level_info(c["term"] + 1)[3])
    if c["kind"] == "solve":
        n = ctx.level_info(c["level"])[3]
        s["b"] = _random((c["n"], n), seed, 50).cpu().numpy()
    return s


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "samples":
        return [ctx.estimate_level(t, 0, c["n"], _noise_seed(state["seed"]))[0] for t in range(c["terms"])]
    if kind == "probes":
        return [ctx.estimate_level_probes(c["term"], state["probes"])[0]]
    if kind == "solve":
        return [ctx.solve(c["level"], state["b"])[0]]
    if kind == "setup":
        agg, nvec = _shape(c)
        ctx.set_gauge(state["theta"])
        ctx.set_mass(c["m0"])
        ctx.set_hierarchy(agg, nvec, state["start"], setup_iters=4, setup_tol=1e-13)
        return [ctx.get_test_vectors(l + 1, nv) for l, nv in enumerate(nvec)]
    if kind == "deflate":
        ctx.compute_deflation(c["k"], 1e-10, 600)
        lam, sigma, _, _, tau = ctx.get_deflation(c["k"], c["terms"])
        return {"lambda": np.sort(lam), "sigma": sigma, "tau": np.array([tau])}
    r = ctx.estimate_trace(c["tol"], 1 << 20, _noise_seed(state["seed"]), _costs(c))
    return {"trace": np.array([r["trace"]]), "rel_err": r["rel_err"],
            "n": np.array([t["nsamples"] for t in r["terms"]], np.int64),
            "mean": np.array([complex(t["mean_re"], t["mean_im"]) for t in r["terms"]]),
            "variance": np.array([t["variance"] for t in r["terms"]])}


# ----------------------------------------------------------------------- work
def work(case):
    """A lower bound that no method that solves with these operators can go below: the
    operators and prolongators once (FP64), every solve's block read and its solution
    written once, and one application of its operator.  Iterations are not counted."""
    c = case
    dims = _dims(c)
    _, nvec = _shape(c)
    n = [x * t * d for x, t, d in dims]
    op_bytes = [2.0 * c["lx"] * c["lt"] * 16] + [5.0 * x * t * d * d * 16 for x, t, d in dims[1:]]
    op_flops = [60.0 * c["lx"] * c["lt"]] + [40.0 * x * t * d * d for x, t, d in dims[1:]]
    solves = []                                             # (level, right-hand sides)
    if c["kind"] in ("samples", "trace"):
        nb = c["n"] if c["kind"] == "samples" else 16       # every loop draws at least its pilot
        for t in range(c["terms"]):
            solves += [(t, nb)] + ([(t + 1, nb)] if t + 1 < c["terms"] else [])
    elif c["kind"] == "probes":
        solves = [(c["term"], c["n"])] + ([(c["term"] + 1, c["n"])] if c["term"] + 1 < c["terms"] else [])
    elif c["kind"] == "solve":
        solves = [(c["level"] - 1, c["n"])]
    elif c["kind"] == "setup":
        solves = [(l, 4 * nv) for l, nv in enumerate(nvec)]
    else:
        solves = [(c["terms"] - 1, c["k"])]
    bytes_ = sum(op_bytes) + sum(16.0 * n[l] * nv for l, nv in enumerate(nvec))
    return {"bytes": bytes_ + sum(32.0 * n[l] * m for l, m in solves),
            "flops": sum(op_flops[l] * m for l, m in solves)}


# ---------------------------------------------------------------------- exact
class _Direct:
    """D x = b by block elimination over the time slices (cyclic block tridiagonal),
    the last slice as the separator, with one step of iterative refinement."""

    def __init__(self, op):
        self.op, lt, lx, d = op, op.lt, op.lx, op.d
        m = lx * d
        A = op.A
        i = torch.arange(lx, device=DEV)

        def diag(k, t):                                     # the slice's hop k as an m x m matrix
            M = torch.zeros(lx, d, lx, d, dtype=C128, device=DEV)
            for kk, j in ((0, i), (1, (i + 1) % lx), (2, (i - 1) % lx)) if k == 0 else ((k, i),):
                M.index_put_((i[:, None, None], torch.arange(d, device=DEV)[None, :, None], j[:, None, None],
                              torch.arange(d, device=DEV)[None, None, :]), A[t, :, kk], accumulate=True)
            return M.reshape(m, m)

        self.m, self.small = m, lt <= 2
        if self.small:
            M = torch.zeros(lt, m, lt, m, dtype=C128, device=DEV)
            for t in range(lt):
                M[t, :, t] += diag(0, t)
                M[t, :, (t + 1) % lt] += diag(3, t)
                M[t, :, (t - 1) % lt] += diag(4, t)
            self.lu = torch.linalg.lu_factor(M.reshape(lt * m, lt * m))
            return
        # S_t = B_t - A_t S_{t-1}^{-1} C_{t-1}; W_t = S_t^{-1} [C_t | border column]
        self.S, self.C, self.W = [], [], []
        border = -diag(4, 0)                                # slice 0 couples to the last slice
        prev = None
        for t in range(lt - 1):
            S = diag(0, t)
            if prev is not None:
                S = S - self._hop(4, t, prev[:, :m])
                border = -self._hop(4, t, prev[:, m:])
            C = diag(3, t)
            if t == lt - 2:
                border = border - C
                C = torch.zeros_like(C)
            f = torch.linalg.lu_factor(S)
            prev = torch.linalg.lu_solve(*f, torch.cat((C, border), 1))
            self.S.append(f)
            self.W.append(prev)
        Z = [None] * (lt - 1)                               # x_t = y_t + Z_t x_last
        Z[-1] = self.W[-1][:, m:]
        for t in range(lt - 3, -1, -1):
            Z[t] = self.W[t][:, m:] - self.W[t][:, :m] @ Z[t + 1]
        self.Z = Z
        self.last = torch.linalg.lu_factor(diag(0, lt - 1) + self._hop(3, lt - 1, Z[0]) + self._hop(4, lt - 1, Z[-1]))

    def _hop(self, k, t, M):                                # the block-diagonal hop k of slice t times M
        op = self.op
        return torch.matmul(op.A[t, :, k], M.reshape(op.lx, op.d, -1)).reshape(self.m, -1)

    def _solve(self, b):
        op, m = self.op, self.m
        lt = op.lt
        r = b.reshape(lt, m, -1)
        if self.small:
            return torch.linalg.lu_solve(*self.lu, r.reshape(lt * m, -1)).reshape(b.shape)
        y = []
        for t in range(lt - 1):
            y.append(torch.linalg.lu_solve(*self.S[t], r[t] - self._hop(4, t, y[-1]) if t else r[t]))
        for t in range(lt - 3, -1, -1):
            y[t] = y[t] - self.W[t][:, :m] @ y[t + 1]
        x = torch.linalg.lu_solve(*self.last, r[-1] - self._hop(3, lt - 1, y[0]) - self._hop(4, lt - 1, y[-1]))
        return torch.stack([v + z @ x for v, z in zip(y, self.Z)] + [x]).reshape(b.shape)

    def __call__(self, b):
        x = self._solve(b)
        return x + self._solve(b - self.op(x))


def _sm(z):
    """One splitmix64 step on int64 tensors (arithmetic modulo 2^64, logical shifts)."""
    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)

    z = z + (0x9E3779B97F4A7C15 - (1 << 64))
    z = (z ^ shr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ shr(z, 31)


def _z2(seed, level, first, count, n):
    """The estimator's Z2 vectors as [n][count]: the low bit of sm(sm(sm(seed ^ level) ^ j) ^ i)."""
    k = _sm(torch.tensor([seed ^ level], device=DEV, dtype=torch.int64))
    ks = _sm(k ^ torch.arange(first, first + count, device=DEV, dtype=torch.int64))
    h = _sm(ks[None, :] ^ torch.arange(n, device=DEV, dtype=torch.int64)[:, None])
    return (1 - 2 * (h & 1)).to(torch.float64).to(C128)


def _block(x, op):
    return x.reshape(op.lt, op.lx, op.d, -1)


def _dot(a, b):
    return (a.conj() * b).reshape(-1, a.shape[-1]).sum(0)


class _Terms:
    """Samples of the terms of the telescoping sum from direct solves."""

    def __init__(self, c, ops, pros, vectors):
        self.c, self.ops, self.pros, self.solver = c, ops, pros, {}
        self.V = vectors                                    # (k, n) of the last term, or None
        self.tau = 0.0
        if vectors is not None:
            op = ops[c["terms"] - 1]
            self.AV = self.solve(c["terms"] - 1, _block(vectors.T, op)).reshape(-1, c["k"])
            self.tau = complex((vectors.conj().T * self.AV).sum())

    def solve(self, l, b):
        if l not in self.solver:
            self.solver[l] = _Direct(self.ops[l])
        return self.solver[l](b)

    def samples(self, t, x):
        """x: [n][count] on the level of term t."""
        b = _block(x, self.ops[t])
        s = _dot(b, self.solve(t, b))
        if t + 1 < self.c["terms"]:
            bc = self.pros[t].restrict(b)
            s = s - _dot(bc, self.solve(t + 1, bc))
        elif self.V is not None:
            s = s - _dot(self.AV.conj().T @ x, self.V.conj() @ x)
        return s.cpu().numpy()


def _exact_trace(c, seed, terms):
    """The multilevel loop: pilot of 16, then N_l towards eps^-2 sqrt(V_l / C_l) sum_m sqrt(V_m C_m), at most doubled."""
    T, cost = c["terms"], np.array(_costs(c))
    have = [np.zeros(0, complex) for _ in range(T)]
    want = [16] * T
    while True:
        for t in range(T):
            if want[t] > len(have[t]):
                op = terms.ops[t]
                x = _z2(_noise_seed(seed), t + 1, len(have[t]), want[t] - len(have[t]), op.lt * op.lx * op.d)
                have[t] = np.concatenate([have[t], terms.samples(t, x)])
        N = np.array([len(h) for h in have])
        mean = np.array([h.mean() for h in have])
        V = np.array([(np.abs(h - h.mean()) ** 2).sum() / (len(h) - 1) for h in have])
        est = mean.sum() + terms.tau
        rel = math.sqrt((V / N).sum()) / abs(est)
        if rel <= c["tol"]:
            return {"trace": np.array([est]), "rel_err": rel, "n": N.astype(np.int64), "mean": mean, "variance": V}
        eps = c["tol"] * abs(est)
        goal = np.ceil(np.sqrt(V / cost) * np.sqrt(V * cost).sum() / eps ** 2)
        want = [int(min(max(g, n), 2 * n)) for g, n in zip(goal, N)]
        if all(w == n for w, n in zip(want, N)):
            worst = int(np.argmax(V / N))
            want[worst] = 2 * int(N[worst])


def exact(case, seed):
    """What run() returns, from block-direct FP64 solves; None where those take too long (above 320 x 320)."""
    c = case
    if c["lx"] * c["lt"] > 320 * 320:
        return None
    if c["kind"] == "setup":
        raw, found = _raw_vectors(c, seed), []

        def iterate(l, op):
            v, solve = raw[l], _Direct(op)
            for _ in range(4):
                v = solve(v)
                v = v / torch.linalg.vector_norm(v.reshape(-1, v.shape[-1]), dim=0)
            found.append(v.reshape(-1, v.shape[-1]).T.contiguous().cpu().numpy())
            return v

        _hierarchy(c, seed, iterate)
        return found
    _, ops, pros, _ = _hierarchy(c, seed)
    if c["kind"] == "deflate":
        op = ops[-1]
        n = op.lt * op.lx * op.d
        D = op(_block(torch.eye(n, dtype=C128, device=DEV), op))
        g5 = torch.ones(op.d, device=DEV, dtype=torch.float64)
        g5[op.d // 2:] = -1.0
        Q = (g5[:, None] * D).reshape(n, n)
        lam, X = torch.linalg.eigh((Q + Q.conj().T) / 2)
        at = torch.argsort(lam.abs())[: c["k"]]
        lam, X = lam[at], X[:, at]
        g = g5.repeat(n // op.d)[:, None]
        tau = ((X.conj() * (g * X)).sum(0) / lam).sum()
        return {"lambda": np.sort(lam.cpu().numpy()), "sigma": lam.abs().cpu().numpy(),
                "tau": np.array([complex(tau)])}
    last = c["terms"] - 1
    terms = _Terms(c, ops, pros, _deflation_vectors(c, seed, ops[last]) if c["k"] else None)
    if c["kind"] == "solve":
        op = ops[c["level"] - 1]
        b = _random((c["n"], op.lt * op.lx * op.d), seed, 50)
        return [terms.solve(c["level"] - 1, _block(b.T, op)).reshape(-1, c["n"]).T.contiguous().cpu().numpy()]
    if c["kind"] == "trace":
        return _exact_trace(c, seed, terms)
    if c["kind"] == "probes":
        t = c["term"]
        x = torch.tensor(_probes(c, seed, ops[t].lt * ops[t].lx * ops[t].d).T.astype(np.float64), device=DEV).to(C128)
        return [terms.samples(t, x)]
    return [terms.samples(t, _z2(_noise_seed(seed), t + 1, 0, c["n"], ops[t].lt * ops[t].lx * ops[t].d))
            for t in range(c["terms"])]
