"""FP64 block products of 16 and more right-hand sides, entry by entry: as accurate as FP64 sums
also far below a right-hand side's largest entry and beside operator rows of very different size,
and what is not finite stays next to where it is."""
import numpy as np
import pytest

from oracle import hierarchy as ohier

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, NARROW = ((4, 4), (2, 2)), (8, 8), 15
U = 2.0 ** -53


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


def by_sums(ctx, op, level, x):
    return np.concatenate([ctx.apply(op, level, x[i:i + NARROW], x.shape[1]) for i in range(0, len(x), NARROW)])


def check(ctx, op, level, x):
    n = x.shape[1]
    A = np.abs(by_sums(ctx, op, level, np.eye(n, dtype=np.complex128)))        # |A|^T
    size = np.abs(x) @ A                                                        # sum |a| |x| per entry
    got, ref = ctx.apply(op, level, x, n), by_sums(ctx, op, level, x)
    # 80 complex products each in FP64 sums (two FMAs per part), and the same again for the digits
    assert np.all(np.abs(got - ref) <= 2 * 4 * 80 * U * size)
    return got


def scaled(rng, nrhs, n, d=16):
    """Sites from 1 down to 2^-300 of the largest, in no order; decaying ones; single sites."""
    x = rand_complex(rng, (nrhs, n))
    sites = n // d
    e = -rng.integers(0, 300, (nrhs, sites))
    e[1::3] = -np.arange(sites) * 7
    x = x * np.exp2(np.repeat(e, d, axis=1).astype(float))
    x[2::3] *= np.repeat(np.arange(sites) == 3, d)
    return x


@pytest.mark.parametrize("nrhs", [16, 40, 130])
@pytest.mark.parametrize("prec", [64, 16])
def test_sites_of_every_scale(pkg, prec, nrhs):
    theta, sv = small_problem(32, 16, 3.0, 0.1, AGG, NVEC)
    rng = np.random.default_rng(nrhs)
    with make_ctx(pkg, theta, 0.1, AGG, NVEC, sv, 0, mg_precision=prec) as ctx:
        for level in (2, 3):
            n = ctx.level_info(level)[3]
            x = scaled(rng, nrhs, n)
            got = check(ctx, pkg.OP_D, level, x)
            x[3, 5], x[4, n - 1], x[7] = np.nan, np.inf, np.nan
            bad, ref = ctx.apply(pkg.OP_D, level, x, n), by_sums(ctx, pkg.OP_D, level, x)
            assert np.array_equal(np.isfinite(bad), np.isfinite(ref))
            assert np.isfinite(bad[3]).any() and not np.isfinite(bad[7]).any()
            keep = [j for j in range(nrhs) if j not in (3, 4, 7)]
            assert np.array_equal(bad[keep], got[keep])


def test_rows_of_every_scale(pkg):
    """The smoother's operator D M^-1 with one nearly singular diagonal block."""
    theta, sv = small_problem(32, 16, 3.0, 0.0, AGG, NVEC)
    D = ohier.build_hierarchy(theta, 0.0, AGG, NVEC, sv, 0).D[1].toarray()
    real = []
    for s in range(0, D.shape[0], 16):
        lam = np.linalg.eigvals(D[s:s + 16, s:s + 16])
        real += [v.real for v in lam if abs(v.imag) < 1e-9]
    m0 = -min(real) + 1e-7                        # the blocks of D_2 shift by the mass
    x = rand_complex(np.random.default_rng(5), (32, D.shape[0]))
    with make_ctx(pkg, theta, m0, AGG, NVEC, sv, 0, mg_precision=64) as ctx:
        n = D.shape[0]
        A = np.abs(by_sums(ctx, pkg.OP_SMOOTH, 2, np.eye(n, dtype=np.complex128)))
        rows = A.max(axis=0)
        assert rows.max() > 2.0 ** 18 * np.median(rows)
        check(ctx, pkg.OP_SMOOTH, 2, x)


def gemm_check(ctx, op, level, x):
    """As check for a dense operator of n unknowns: n complex products an entry."""
    n = x.shape[1]
    A = np.abs(by_sums(ctx, op, level, np.eye(n, dtype=np.complex128)))
    got, ref = ctx.apply(op, level, x, n), by_sums(ctx, op, level, x)
    assert np.all(np.abs(got - ref) <= 2 * 4 * n * U * (np.abs(x) @ A))


def test_inverse(pkg):
    """A heavy mass: the inverse decays with the distance, and so do its rows' products with a
    right-hand side of one large entry."""
    agg, nvec = ((2, 2),), (4,)
    theta, sv = small_problem(32, 32, 3.0, 6.0, agg, nvec)
    with make_ctx(pkg, theta, 6.0, agg, nvec, sv, 0, mg_precision=64) as ctx:
        n = ctx.level_info(2)[3]
        rng = np.random.default_rng(7)
        x = scaled(rng, 18, n, d=8)
        x[:, 100] = 1.0                            # far above the rest
        gemm_check(ctx, pkg.OP_DINV_C, 2, x)
