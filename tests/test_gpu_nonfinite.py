"""A right-hand side that is not finite is an error, alone and among good ones; it is not
taken for a solved one."""
import numpy as np
import pytest

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0 = ((2, 2), (2, 2)), (2, 2), 0.2
ENAN = -7


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


# up to 32 rhs the residual estimate goes to the host from one warp, above through a device maximum
@pytest.mark.parametrize("nrhs", [1, 5, 32, 33, 70])
@pytest.mark.parametrize("prec", [64, 32, 16])
def test_solve_reports_it(pkg, prec, nrhs):
    theta, sv = small_problem(8, 8, 3.0, M0, AGG, NVEC)
    b = rand_complex(np.random.default_rng(nrhs), (nrhs, 128))
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec) as ctx:
        good, _ = ctx.solve(1, b)
        for bad in (np.nan, np.inf, 1j * np.nan):
            for j in {0, nrhs // 2, nrhs - 1}:
                c = b.copy()
                c[j, 17] = bad
                with pytest.raises(pkg.MgmlmcError) as err:
                    ctx.solve(1, c)
                assert err.value.code == ENAN
        # the context is as good as before, and a zero right-hand side is still a solved one
        again, _ = ctx.solve(1, b)
        assert np.abs(again - good).max() < 1e-10 * np.abs(good).max()
        zero, iters = ctx.solve(1, np.zeros_like(b))
        assert iters == 0 and not zero.any()
