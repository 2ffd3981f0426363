"""The smoother's groups of steps, close enough to see one step: the FP32 cycle at FP32 accuracy
(the coarsest level of few right-hand sides is solved in FP32), and the BF16 cycle against a
restatement that rounds where the kernels do (operators, residuals and images of the smoother),
which it has to be five times closer to than one step less or more would leave it."""
import numpy as np
import pytest

from oracle import hierarchy as ohier

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0 = ((4, 4), (2, 1)), (8, 8), 0.1
STEPS = [(0, 1), (0, 2), (0, 7), (0, 8), (0, 9), (0, 16), (0, 17)]


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.fixture(scope="module")
def problem():
    theta, sv = small_problem(16, 16, 3.0, M0, AGG, NVEC)
    H = ohier.build_hierarchy(theta, M0, AGG, NVEC, sv, 0)
    D = [d.toarray() for d in H.D]
    M = [np.eye(len(D[0]))]
    M.append(np.zeros_like(D[1]))
    for s in range(0, len(D[1]), 16):
        M[1][s:s + 16, s:s + 16] = np.linalg.inv(D[1][s:s + 16, s:s + 16])
    return theta, sv, D, M, [p.toarray() for p in H.P]


def bf16(z):
    """Real and imaginary parts rounded to BF16, to nearest even."""
    def one(x):
        u = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
        return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32)
    return one(z.real) + 1j * one(z.imag).astype(np.float64)


def exact(z):
    return z


def cycle(problem, l, r, nu, prec):
    _, _, D, M, P = problem
    if l == 2:
        return np.linalg.solve(D[2], r)
    e = P[l] @ cycle(problem, l + 1, P[l].conj().T @ r, nu, prec)
    rnd = bf16 if prec == 16 else exact
    # level 1 in BF16: operators rounded as well, and e where the residual is formed
    A, hat, et = (rnd(D[1]), rnd(D[1] @ M[1]), rnd(e)) if l == 1 else (D[0], D[0], e)
    res = rnd(r - A @ et)
    y = np.zeros_like(r)
    for _ in range(nu):
        p = hat @ res
        a = (p.conj() * res).sum(0) / (np.abs(p) ** 2).sum(0)
        y = y + a * res
        res = rnd(res - a * rnd(p))
    return e + M[l] @ y


def distance(a, b):
    return (np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)).max()


# FP32: a few rounding errors a step.  BF16: a value that falls to the other side of a rounding
# moves by 2^-8 and takes all later residuals with it, so the step itself is the measure
@pytest.mark.parametrize("nu_pre,nu", STEPS)
@pytest.mark.parametrize("prec,nrhs", [(32, 3), (32, 12), (16, 12), (16, 28)])
def test_steps(pkg, problem, prec, nrhs, nu_pre, nu):
    theta, sv = problem[:2]
    x = rand_complex(np.random.default_rng(nrhs), (nrhs, 512))
    ref = cycle(problem, 0, x.T, nu, prec)
    step = distance(cycle(problem, 0, x.T, nu + 1, prec), ref)     # the steps get smaller
    tol = 1e-4 if prec == 32 else step / 5
    assert tol <= step / 5
    with make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, nu_pre=nu_pre, nu_post=nu) as ctx:
        got = ctx.apply(pkg.OP_PREC, 1, x, 512)
    assert distance(got.T, ref) < tol
