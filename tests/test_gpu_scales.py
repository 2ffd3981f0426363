"""Vectors of any scale: the multigrid cycle is homogeneous and every step of it commutes with
powers of two, so a scaled input gives the scaled result to the last bit, although the FP32
cycle's sums of squares have only FP32's range."""
import numpy as np
import pytest

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0 = ((4, 4), (2, 1)), (8, 8), 0.1


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.mark.parametrize("nrhs", [1, 6, 40])
@pytest.mark.parametrize("prec,kcycle", [(32, 0), (16, 0), (16, 2)])
def test_cycle(pkg, prec, kcycle, nrhs):
    theta, sv = small_problem(16, 16, 3.0, M0, AGG, NVEC)
    x = rand_complex(np.random.default_rng(nrhs), (nrhs, 512))
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, nu_pre=1, kcycle_iters=kcycle) as ctx:
        ref = ctx.apply(pkg.OP_PREC, 1, x, 512)
        assert np.isfinite(ref).all()
        for e in (59, 62, 90, 600, -60, -100, -600):
            got = ctx.apply(pkg.OP_PREC, 1, np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e), 512)
            assert np.array_equal(got, np.ldexp(ref.real, e) + 1j * np.ldexp(ref.imag, e)), e
        x[0] = 0
        assert not ctx.apply(pkg.OP_PREC, 1, x, 512)[0].any()


@pytest.mark.parametrize("prec", [32, 16])
def test_start_vectors(pkg, prec):
    theta, sv = small_problem(16, 16, 3.0, M0, AGG, NVEC)
    out = []
    for e in (0, 62):
        with make_ctx(pkg, theta, M0, AGG, NVEC, [v * 2.0 ** e for v in sv], 2, mg_precision=prec) as ctx:
            out.append([ctx.get_test_vectors(l + 1, nv) for l, nv in enumerate(NVEC)])
    # each solve of the inverse iteration to 1e-13, its start only scaled
    for a, b in zip(*out):
        assert np.abs(a - b).max() < 1e-11 * np.abs(a).max()
