"""The FP32 coarsest inverse (one panel: up to 32 unknowns) bit for bit against Gauss-Jordan in
numpy: pivots by |a|^2 in FP64, their reciprocals formed in FP64 and rounded once, everything
else in FP32 (of each pair of products the compiler fuses one, either one, in the scaling of
the pivot row and in the elimination)."""
import itertools

import numpy as np
import pytest

from gpu_common import make_ctx, require_gpu, small_problem

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


def pair(a, b, c, d, sign, first):
    """a b + sign c d in FP32 with the first or the second product fused."""
    if first:
        return (a.astype(float) * b + sign * (c * d).astype(float)).astype(F)
    return (sign * c.astype(float) * d + (a * b).astype(float)).astype(F)


def inverse(D, fuse):
    re, im = D.real.astype(F), D.imag.astype(F)
    n = len(re)

    def mul(ar, ai, br, bi, fuse):
        ar, ai, br, bi = np.broadcast_arrays(ar, ai, br, bi)
        return pair(ar, br, ai, bi, -1.0, fuse[0]), pair(ar, bi, ai, br, 1.0, fuse[1])

    perm = []
    for k in range(n):
        size = re[k:, k].astype(float) ** 2 + im[k:, k].astype(float) ** 2
        p = k + int(np.argmax(size))
        perm.append(p)
        for m in (re, im):
            m[[k, p]] = m[[p, k]]
        x, y = float(re[k, k]), float(im[k, k])
        den = x * x + y * y
        re[k, k], im[k, k] = 1, 0
        re[k], im[k] = mul(re[k], im[k], F(x / den), F(-y / den), fuse[:2])
        fr, fi = re[:, k].copy(), im[:, k].copy()
        for i in range(n):
            if i != k:
                re[i, k] = im[i, k] = 0
                pr, pi = mul(fr[i], fi[i], re[k], im[k], fuse[2:])
                re[i], im[i] = re[i] - pr, im[i] - pi
    for k in reversed(range(n)):
        for m in (re, im):
            m[:, [k, perm[k]]] = m[:, [perm[k], k]]
    return re, im


@pytest.mark.parametrize("lattice,agg,nv", [((4, 4), (4, 4), 4), ((12, 4), (4, 2), 1), ((12, 10), (2, 5), 1),
                                            ((8, 8), (4, 4), 3)])
def test_bits(pkg, lattice, agg, nv):
    theta, sv = small_problem(*lattice, 3.0, 0.2, (agg,), (nv,))
    with make_ctx(pkg, theta, 0.2, (agg,), (nv,), sv, 0, mg_precision=32) as ctx:
        n = ctx.level_info(2)[3]
        eye = np.eye(n, dtype=np.complex128)
        D, got = [np.concatenate([ctx.apply(op, 2, eye[i:i + 8], n) for i in range(0, n, 8)]).T
                  for op in (pkg.OP_D, pkg.OP_DINV_C)]
    same = []
    for fuse in itertools.product((True, False), repeat=4):
        re, im = inverse(D, fuse)
        same.append(np.mean((got.real == re) & (got.imag == im)))
    # a fused product formed in FP64 is rounded twice once in 2^29 times
    assert max(same) > 0.99, same
