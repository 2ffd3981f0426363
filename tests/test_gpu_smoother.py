"""The multigrid cycle against a plain numpy restatement on the oracle's hierarchy: the
smoother's groups of steps (up to, at and past a group of 8, before and after the
coarse correction), narrow and ragged blocks, every precision."""
import numpy as np
import pytest

from oracle import hierarchy as ohier

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0 = ((4, 4), (2, 1)), (8, 8), 0.1


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.fixture(scope="module")
def problem():
    theta, sv = small_problem(16, 16, 3.0, M0, AGG, NVEC)
    return theta, sv, ohier.build_hierarchy(theta, M0, AGG, NVEC, sv, 0)


def minimal_residual(A, r, nu):
    y = np.zeros_like(r)
    for _ in range(nu):
        p = A @ r
        a = (p.conj() * r).sum(0) / (np.abs(p) ** 2).sum(0)
        y += a * r
        r = r - a * p
    return y, r


def cycle(H, l, r, nu_pre, nu_post):
    D = H.D[l].toarray()
    if l == H.nlevels - 1:
        return np.linalg.solve(D, r)
    P = H.P[l].toarray()
    M = np.eye(D.shape[0])
    if l > 0:                                # block Jacobi on the coarse levels
        d = H.dims[l][2]
        M = np.zeros_like(D)
        for s in range(0, D.shape[0], d):
            M[s:s + d, s:s + d] = np.linalg.inv(D[s:s + d, s:s + d])
    e, res = np.zeros_like(r), r
    if nu_pre:
        y, res = minimal_residual(D @ M, r, nu_pre)
        e = M @ y
    e = e + P @ cycle(H, l + 1, P.conj().T @ res, nu_pre, nu_post)
    y, _ = minimal_residual(D @ M, r - D @ e, nu_post)
    return e + M @ y


@pytest.mark.parametrize("nu_pre,nu_post", [(0, 1), (0, 8), (0, 9), (1, 2), (9, 17)])
@pytest.mark.parametrize("nrhs", [1, 3, 12, 130])
# FP64: rounding through the MR quotients of up to 17 steps; FP32 and BF16: the coarsest
# solve and the smoother's vectors are BF16 (2^-9 a rounding, a few dozen of them)
@pytest.mark.parametrize("prec,tol", [(64, 1e-10), (32, 5e-2), (16, 1e-1)])
def test_cycle(pkg, problem, prec, tol, nrhs, nu_pre, nu_post):
    theta, sv, H = problem
    x = rand_complex(np.random.default_rng(nrhs), (nrhs, H.D[0].shape[0]))
    ref = cycle(H, 0, x.T, nu_pre, nu_post).T
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, nu_pre=nu_pre, nu_post=nu_post) as ctx:
        got = ctx.apply(pkg.OP_PREC, 1, x, x.shape[1])
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() < tol, err.max()
