"""A solve gives the same bits and iteration counts whatever the context has solved before: what
it remembers of earlier cycles only decides when the host looks at the residual estimates."""
import numpy as np
import pytest

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, HARD, EASY = ((2, 2),), (1,), 0.4, 1.5


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


# up to 32 rhs the estimates come from one warp, above from device maxima; a restart inside and none
@pytest.mark.parametrize("restart", [7, 40])
@pytest.mark.parametrize("nrhs", [2, 32, 70])
@pytest.mark.parametrize("prec", [64, 32, 16])
def test_after_other_solves(pkg, prec, nrhs, restart):
    theta, sv = small_problem(16, 12, 3.0, EASY, AGG, NVEC)
    opts = dict(mg_precision=prec, fgmres_restart=restart, nu_post=1)
    b = rand_complex(np.random.default_rng(nrhs), (nrhs, 384))
    with make_ctx(pkg, theta, EASY, AGG, NVEC, sv, 0, **opts) as ctx:
        ref, iters = ctx.solve(1, b)
        again = ctx.solve(1, b)
    with make_ctx(pkg, theta, HARD, AGG, NVEC, sv, 0, **opts) as ctx:
        _, hard = ctx.solve(1, b)
        ctx.set_mass(EASY)
        ctx.set_hierarchy(AGG, NVEC, sv, setup_iters=0, setup_tol=1e-13)
        after = ctx.solve(1, b)
    assert hard > iters + 6
    for x, n in (again, after):
        assert n == iters and np.array_equal(x, ref)
