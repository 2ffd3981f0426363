"""The device-memory model bounds what an estimate holds, pre-smoothing included."""
import pytest

from gpu_common import require_gpu, small_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


# three levels of d = 16 with as many unknowns as the finest has, and a short restart: the
# smoother's blocks are most of what is held
AGG, NVEC, M0, N0 = ((4, 2), (1, 1), (1, 1), (8, 8)), (8, 8, 8, 4), 0.3, 2 * 64 * 64


def peak_and_model(pkg, prec, nu_pre, nu_post):
    theta, sv = small_problem(64, 64, 3.0, M0, AGG, NVEC)
    opts = dict(mg_precision=prec, nu_pre=nu_pre, nu_post=nu_post, max_block_rhs=512, fgmres_restart=2)
    req = pkg.make_request(theta, M0, AGG, NVEC, sv, 1e-2, 1, setup_iters=0, **opts)
    with pkg.Context(**opts) as ctx:
        ctx.set_gauge(theta)
        ctx.set_mass(M0)
        ctx.set_hierarchy(AGG, NVEC, sv, setup_iters=0, setup_tol=1e-12)
        for t in range(len(AGG) + 1):
            ctx.estimate_level(t, 0, 512, 7)
        return ctx.memory()[1], pkg.request_footprint(req)


@pytest.mark.parametrize("nu_pre,nu_post", [(4, 4), (8, 8), (8, 0), (0, 8)])
@pytest.mark.parametrize("prec", [16, 32, 64])
def test_bound(pkg, prec, nu_pre, nu_post):
    peak, model = peak_and_model(pkg, prec, nu_pre, nu_post)
    assert peak <= model


def test_tensor_core_pre_smoother_keeps_one_residual(pkg):
    one, eight = [peak_and_model(pkg, 16, nu, 8)[0] for nu in (1, 8)]
    # seven more residuals of the finest level, which smooths in FP32, and of no other
    assert eight - one <= 7 * N0 * 512 * 8 * 1.01
