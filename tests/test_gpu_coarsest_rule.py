"""Which form solves the coarsest level of the mixed modes: the FP32 inverse in one launch where that
is the faster one (columns, rounded up to a power of two, times unknowns up to 16384, or no BF16
inverse), the BF16 inverse on the tensor cores elsewhere; on both sides of every line."""
import numpy as np
import pytest

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.mark.parametrize("lattice,nrhs,form", [
    ((32, 32), 31, "f32"), ((32, 32), 32, "bf16"),                              # 256 unknowns
    ((64, 32), 31, "f32"), ((64, 32), 32, "bf16"),                              # 512
    ((64, 64), 16, "f32"), ((64, 64), 17, "bf16"), ((64, 64), 31, "bf16"),      # 1024
    ((128, 64), 1, "bf16"),                                                     # 2048
    ((40, 24), 31, "f32"),                                                      # 240: no BF16 inverse
])
def test_form(pkg, lattice, nrhs, form):
    agg, nvec = ((4, 4), (2, 2)), (8, 8)
    theta, sv = small_problem(*lattice, 3.0, 0.3, agg, nvec, sweeps=3)
    with make_ctx(pkg, theta, 0.3, agg, nvec, sv, 0, mg_precision=16) as ctx:
        n = ctx.level_info(3)[3]
        y = rand_complex(np.random.default_rng(nrhs), (nrhs, n))
        x = ctx.apply(pkg.OP_D, 3, y, n)
        ctx.profile(True, True)
        got = ctx.apply(pkg.OP_DINV_C, 3, x, n)
        assert [k for k in ctx.profile_report() if k.startswith("Dinv")] == ["Dinv." + form]
    # the inverse in FP32 (its condition is below 1e3), or rounded to BF16 (2^-9 an entry)
    assert np.linalg.norm(got - y) < (1e-4 if form == "f32" else 3e-2) * np.linalg.norm(y)
