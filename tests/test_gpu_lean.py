"""The memory that a context can do without (digits of the FP64 operators, the residuals of a
smoother's group): not held where blocks are too narrow to use it, given back when an allocation is
refused, left out of a served request or a tuned context that only fits without it."""
import numpy as np
import pytest

from gpu_common import make_ctx, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0, N = ((4, 4), (2, 2)), (8, 8), 0.1, 256
SITES = (256, 64)                                    # of the levels with d = 16
UNKNOWNS = (8192, 4096)                              # of the smoothed levels
DIGITS = 5 * 16384                                   # bytes a site
SEED = 11


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.fixture(scope="module")
def problem():
    return small_problem(64, 64, 3.0, M0, AGG, NVEC)


def optional_bytes(prec, nu, n):
    tiles = -(-n // 128)
    slots = nu - 1
    if prec == 64:
        dense = 1024 ** 2 * 64 + 64 * tiles * 65536 + 11 * 1024 * n * 16
        return (2 * SITES[0] + SITES[1]) * DIGITS + SITES[0] * tiles * 65536 + dense + slots * sum(UNKNOWNS) * n * 16
    return sum(SITES) * DIGITS + SITES[0] * tiles * 65536 + slots * (UNKNOWNS[0] * n * 4 + SITES[0] * tiles * 8192)


def estimate(ctx, n):
    return np.array([ctx.estimate_level(t, 0, n, SEED)[0] for t in range(3)])


@pytest.mark.parametrize("nu", [4, 8])
@pytest.mark.parametrize("prec", [64, 16])
def test_refused_memory(pkg, problem, monkeypatch, prec, nu):
    import torch
    theta, sv = problem
    opts = dict(mg_precision=prec, nu_post=nu, max_block_rhs=N, fgmres_restart=8)
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, **opts) as ctx:
        ref = estimate(ctx, N)
        peak = ctx.memory()[1]
    # most of the optional memory beyond what the context is granted (and without digits the
    # products of level 2 go through three blocks of the Galerkin form)
    limit = peak - int(0.9 * optional_bytes(prec, nu, N)) + (2 * UNKNOWNS[0] + UNKNOWNS[1]) * N * 16
    assert limit < peak
    empty, held = torch.empty, []

    def limited(nbytes, **kw):
        ctx = held[0]
        if sum(t.numel() for t in ctx._mem.values()) + nbytes > limit:
            raise RuntimeError("refused")
        return empty(nbytes, **kw)

    with pkg.Context(**opts) as ctx:
        held.append(ctx)
        monkeypatch.setattr(torch, "empty", limited)
        ctx.set_gauge(theta)
        ctx.set_mass(M0)
        ctx.set_hierarchy(AGG, NVEC, sv, setup_iters=0, setup_tol=1e-13)
        for _ in range(2):
            got = estimate(ctx, N)
            assert np.abs(got - ref).max() < 1e-9 * np.abs(ref).max()
        assert ctx.memory()[1] <= limit
        monkeypatch.setattr(torch, "empty", empty)
        # a new hierarchy asks for it again
        ctx.set_hierarchy(AGG, NVEC, sv, setup_iters=0, setup_tol=1e-13)
        assert np.abs(estimate(ctx, N) - ref).max() < 1e-9 * np.abs(ref).max()
        assert ctx.memory()[1] > limit


@pytest.mark.parametrize("prec", [64, 16])
def test_narrow_blocks_hold_no_digits(pkg, problem, prec):
    theta, sv = problem
    digits = (2 * SITES[0] + SITES[1] if prec == 64 else sum(SITES)) * DIGITS
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, max_block_rhs=16) as ctx:
        wide = ctx.memory()[0]
        ref = estimate(ctx, 32)
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, max_block_rhs=15) as ctx:
        assert ctx.memory()[0] <= wide - digits
        assert np.abs(estimate(ctx, 32) - ref).max() < 1e-9 * np.abs(ref).max()
        before = ctx.memory()[0]
        ctx.set_options(max_block_rhs=16)
        assert ctx.memory()[0] >= before + digits
        assert np.abs(estimate(ctx, 32) - ref).max() < 1e-9 * np.abs(ref).max()


@pytest.mark.parametrize("prec,fraction", [(64, 0.7), (16, 0.88)])
def test_server_and_autotuner(pkg, problem, prec, fraction):
    theta, sv = problem
    opts = dict(mg_precision=prec, nu_post=8, max_block_rhs=N, fgmres_restart=4)
    req = pkg.make_request(theta, M0, AGG, NVEC, sv, 1e-3, SEED, setup_iters=0, costs=[1.0, 0.3, 0.1], **opts)
    full = pkg.request_footprint(req)
    res = []
    for budget in (2 * full, int(fraction * full), int(fraction * full)):
        with pkg.Server(hbm_budget=budget, max_active=1) as srv:
            res.append([srv.wait(srv.submit(req), 600.0) for _ in range(2)])
    for first, second in res:
        assert first["status"] == 0 and first["peak_bytes"] <= first["reserved_bytes"]
        assert second["status"] == 0 and second["peak_bytes"] <= second["reserved_bytes"]
    a, b = res[0][0]["result"]["trace"], res[1][0]["result"]["trace"]
    assert abs(a - b) < 1e-8 * abs(a)
    assert res[1][0]["peak_bytes"] < res[0][0]["peak_bytes"] - optional_bytes(prec, 8, N) // 4
    # less than the autotuner's narrowest candidate (32) takes with that memory
    narrow = pkg.make_request(theta, M0, AGG, NVEC, sv, 1e-3, SEED, setup_iters=0,
                              **{**opts, "max_block_rhs": 32})
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, **opts) as ctx:
        t = ctx.autotune(hbm_budget=int(0.9 * pkg.request_footprint(narrow)), max_trials=1)
        assert t["block_rhs"] >= 32 and t["footprint"] <= t["budget"]
