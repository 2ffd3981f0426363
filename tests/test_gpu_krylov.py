"""The block FGMRES with a weak preconditioner (one smoothing step, one rough test vector: one
cycle runs to the restart length): restart lengths below, at and above 32 vectors,
narrow and ragged blocks, zero right-hand sides among the others."""
import numpy as np
import pytest

from oracle import hierarchy as ohier

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0 = ((2, 2),), (1,), 0.4


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.mark.parametrize("restart", [5, 32, 33, 63])
@pytest.mark.parametrize("nrhs", [1, 2, 7, 33, 66])
@pytest.mark.parametrize("prec", [64, 32])
def test_solve(pkg, prec, nrhs, restart):
    theta, sv = small_problem(16, 12, 3.0, M0, AGG, NVEC)
    D = ohier.build_hierarchy(theta, M0, AGG, NVEC, sv, 0).D[0]
    b = rand_complex(np.random.default_rng(nrhs), (nrhs, D.shape[0]))
    b *= np.exp2(np.arange(nrhs) % 5 * 20.0 - 40.0)[:, None]
    if nrhs > 2:
        b[1] = 0
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, fgmres_restart=restart, nu_post=1,
                  max_iters=20000) as ctx:
        x, iters = ctx.solve(1, b)
        zero, none = ctx.solve(1, np.zeros_like(b))
    assert iters > 40 and none == 0 and not zero.any()
    norm = np.linalg.norm(b, axis=1)
    # solve_tol 1e-12 of each rhs; D x formed here in FP64 adds a few rounding errors of |x|
    res = np.linalg.norm((D @ x.T).T - b, axis=1)
    assert np.all(res <= 1e-12 * norm + 32 * 2.0 ** -53 * np.linalg.norm(x, axis=1))
    if nrhs > 2:
        assert not x[1].any()
