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


# |D r|^2 of a few hundred entries of 2^e: its reciprocal overflows, its own digits are few
@pytest.mark.parametrize("e", [-508, -516, -520, -524])
def test_fp64_cycle_of_tiny_vectors(pkg, e):
    theta, sv = small_problem(16, 16, 3.0, M0, AGG, NVEC)
    x = rand_complex(np.random.default_rng(3), (3, 512))
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=64) as ctx:
        ref = ctx.apply(pkg.OP_PREC, 1, x, 512)
        got = ctx.apply(pkg.OP_PREC, 1, np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e), 512)
    got = np.ldexp(got.real, -e) + 1j * np.ldexp(got.imag, -e)
    # squares of 2^(2e) on a grid of 2^-1074, a step down in scale per smoothing step
    tol = max(1e-12, 64 * 2.0 ** (-1074 - 2 * e + 4))
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
