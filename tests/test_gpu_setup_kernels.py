"""Setup kernels where their work splits: the panel cluster of the coarsest inverse (fewer rows
than CTAs, a partial last panel, above its largest size), and aggregates with more rows
than a warp has lanes or than fit in shared memory."""
import numpy as np
import pytest

from oracle import hierarchy as ohier

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


# coarsest unknowns: 2 x 1 x 2 = 4, 12, 90, 1000, 2000 (two rows of a CTA apart from even shares)
@pytest.mark.parametrize("lattice,agg,nv", [((4, 2), (2, 2), 1), ((12, 4), (4, 2), 1), ((30, 6), (2, 2), 1),
                                            ((50, 40), (2, 2), 1), ((20, 50), (1, 1), 1)])
@pytest.mark.parametrize("prec,tol", [(64, 1e-10), (32, 3e-2)])
def test_inverse(pkg, lattice, agg, nv, prec, tol):
    theta, sv = small_problem(*lattice, 3.0, 0.2, (agg,), (nv,))
    D = ohier.build_hierarchy(theta, 0.2, (agg,), (nv,), sv, 0).D[-1].toarray()
    x = rand_complex(np.random.default_rng(1), (3, D.shape[0]))
    ref = np.linalg.solve(D, x.T).T
    with make_ctx(pkg, theta, 0.2, (agg,), (nv,), sv, 0, mg_precision=prec) as ctx:
        got = ctx.apply(pkg.OP_DINV_C, 2, x, D.shape[0])
    # FP64: cond eps with some room; FP32: the inverse itself to FP32, applied in FP32 or BF16
    assert np.linalg.norm(got - ref) < tol * np.linalg.norm(ref)


def test_inverse_above_the_panel_cluster(pkg):
    lattice, agg, nv = (112, 56), (1, 1), 1          # 12544 unknowns: 1568 rows a CTA
    theta, sv = small_problem(*lattice, 3.0, 0.2, (agg,), (nv,), sweeps=5)
    D = ohier.build_hierarchy(theta, 0.2, (agg,), (nv,), sv, 0).D[-1]
    y = rand_complex(np.random.default_rng(1), (2, D.shape[0]))
    with make_ctx(pkg, theta, 0.2, (agg,), (nv,), sv, 0, mg_precision=32) as ctx:
        got = ctx.apply(pkg.OP_DINV_C, 2, (D @ y.T).T, D.shape[0])
    assert np.linalg.norm(got - y) < 3e-2 * np.linalg.norm(y)


@pytest.mark.parametrize("agg,nvec", [(((2, 2), (2, 2)), (2, 3)), (((8, 8), (2, 2)), (6, 12)), (((8, 16), (1, 1)), (20, 20))])
def test_prolongator_and_smoother(pkg, agg, nvec):
    theta, sv = small_problem(16, 32, 3.0, 0.2, agg, nvec)
    H = ohier.build_hierarchy(theta, 0.2, agg, nvec, sv, 0)
    rng = np.random.default_rng(2)
    with make_ctx(pkg, theta, 0.2, agg, nvec, sv, 0) as ctx:
        for lev in (1, 2):
            x = rand_complex(rng, (3, H.P[lev - 1].shape[1]))
            got = ctx.apply(pkg.OP_P, lev, x, H.P[lev - 1].shape[0])
            ref = (H.P[lev - 1] @ x.T).T
            # Gram-Schmidt of random vectors: condition of the blocks times eps
            assert np.abs(got - ref).max() < 1e-10 * np.abs(ref).max()
        D, d = H.D[1].toarray(), H.dims[1][2]
        M = np.zeros_like(D)
        for s in range(0, D.shape[0], d):
            M[s:s + d, s:s + d] = np.linalg.inv(D[s:s + d, s:s + d])
        x = rand_complex(rng, (2, D.shape[0]))
        got = ctx.apply(pkg.OP_SMOOTH, 2, x, D.shape[0])
        ref = (D @ (M @ x.T)).T
        assert np.abs(got - ref).max() < 1e-10 * np.abs(ref).max()
