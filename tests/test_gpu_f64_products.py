"""The FP64 block products on the tensor cores (digit slices, exact sums) against extended
precision and against the FP64 pipe, which blocks of fewer than 16 rhs take."""
import numpy as np
import pytest

from oracle import hierarchy as ohier

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
M0, NARROW = 0.1, 15


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


def by_pipe(ctx, op, level, x):
    return np.concatenate([ctx.apply(op, level, x[i:i + NARROW], x.shape[1]) for i in range(0, len(x), NARROW)])


def extended(D, x):
    """D x for a sparse D with the sums in extended precision: [nrhs][n] real and imaginary parts."""
    D = D.tocoo()
    out = [np.zeros(x.shape, np.longdouble) for _ in range(2)]
    ar, ai = D.data.real.astype(np.longdouble), D.data.imag.astype(np.longdouble)
    for j in range(len(x)):
        xr, xi = x[j, D.col].real.astype(np.longdouble), x[j, D.col].imag.astype(np.longdouble)
        np.add.at(out[0][j], D.row, ar * xr - ai * xi)
        np.add.at(out[1][j], D.row, ar * xi + ai * xr)
    return out


# level 2 with 4 x 2 sites (neighbours that coincide in one direction), level 3 below it
@pytest.mark.parametrize("nrhs", [16, 17, 127, 128, 130])
@pytest.mark.parametrize("prec", [64, 16])
def test_stencil(pkg, prec, nrhs):
    agg, nvec = ((4, 4), (2, 1)), (8, 8)
    theta, sv = small_problem(16, 8, 3.0, M0, agg, nvec)
    H = ohier.build_hierarchy(theta, M0, agg, nvec, sv, 0)
    rng = np.random.default_rng(nrhs)
    with make_ctx(pkg, theta, M0, agg, nvec, sv, 0, mg_precision=prec) as ctx:
        for level in (2, 3):
            D = H.D[level - 1]
            x = rand_complex(rng, (nrhs, D.shape[0]))
            x *= np.exp2(rng.integers(-600, 600, nrhs))[:, None]     # every rhs has its own scale
            x[1] = 0
            x[2, rng.random(D.shape[0]) < 0.9] *= 2.0 ** -40          # mostly far below the largest entry
            got, pipe = ctx.apply(pkg.OP_D, level, x, D.shape[0]), by_pipe(ctx, pkg.OP_D, level, x)
            ref = extended(D, x)
            big = np.maximum(np.abs(x.real).max(1), np.abs(x.imag).max(1))
            # the oracle's blocks agree with the library's to a few rounding errors: the
            # digits add 2^-63 of the rhs' largest entry per term, one rounding at the end
            rows = np.abs(D).sum(1).A1 if hasattr(np.abs(D).sum(1), "A1") else np.asarray(np.abs(D).sum(1)).ravel()
            bound = (64 * 2.0 ** -53) * rows.max() * big
            for y, r in ((got.real, ref[0]), (got.imag, ref[1])):
                assert np.all(np.abs(y - r).max(1) <= bound)
            assert np.all(np.abs(got - pipe).max(1) <= bound)
            assert not got[1].any()
            x[3, 5] = np.nan
            x[4, 7] = np.inf
            bad = ctx.apply(pkg.OP_D, level, x, D.shape[0])
            assert np.isnan(bad[3]).any() and not np.isfinite(bad[4]).all()
            keep = [j for j in range(nrhs) if j not in (3, 4)]
            assert np.array_equal(bad[keep], got[keep])


@pytest.mark.parametrize("nrhs", [16, 65, 128, 200])
@pytest.mark.parametrize("lattice,agg,nvec", [((8, 8), ((4, 4),), (4,)),            # 32 unknowns: one split
                                              ((16, 24), ((4, 4), (2, 1)), (8, 8))])   # 192: two splits
def test_dense_inverse(pkg, lattice, agg, nvec, nrhs):
    theta, sv = small_problem(*lattice, 3.0, M0, agg, nvec)
    H = ohier.build_hierarchy(theta, M0, agg, nvec, sv, 0)
    D = H.D[-1].toarray()
    x = rand_complex(np.random.default_rng(nrhs), (nrhs, D.shape[0]))
    with make_ctx(pkg, theta, M0, agg, nvec, sv, 0, mg_precision=64) as ctx:
        got = ctx.apply(pkg.OP_DINV_C, len(agg) + 1, x, D.shape[0])
        pipe = by_pipe(ctx, pkg.OP_DINV_C, len(agg) + 1, x)
    ref = np.linalg.solve(D, x.T).T
    assert np.abs(got - pipe).max() < 1e-13 * np.abs(ref).max()      # one inverse, two products
    assert np.abs(got - ref).max() < 1e-10 * np.abs(ref).max()


# spread over the lattice, and concentrated on ever fewer of its 256 unknowns
@pytest.mark.parametrize("decay", [0.0, 0.02, 0.2, 2.0])
def test_closer_than_fp64_sums(pkg, decay):
    """On one operator (taken from the context itself, so that its blocks are exact) the digit
    product is nearer to extended precision than the FP64 sums are, rhs by rhs."""
    agg, nvec = ((4, 4), (2, 2)), (8, 8)
    theta, sv = small_problem(16, 16, 3.0, M0, agg, nvec)
    with make_ctx(pkg, theta, M0, agg, nvec, sv, 0, mg_precision=64) as ctx:
        n = ctx.level_info(2)[3]
        D = ctx.apply(pkg.OP_D, 2, np.eye(n, dtype=np.complex128), n).T      # columns: exact products with 1
        x = rand_complex(np.random.default_rng(9), (32, n)) * np.exp(-decay * np.arange(n))
        got, pipe = ctx.apply(pkg.OP_D, 2, x, n), by_pipe(ctx, pkg.OP_D, 2, x)
    Dr, Di = D.real.astype(np.longdouble), D.imag.astype(np.longdouble)
    xr, xi = x.real.T.astype(np.longdouble), x.imag.T.astype(np.longdouble)
    re, im = (Dr @ xr - Di @ xi).T, (Dr @ xi + Di @ xr).T

    def err(y):
        return np.sqrt(((y.real - re) ** 2).sum(1) + ((y.imag - im) ** 2).sum(1))

    assert np.all(err(got) <= err(pipe))
