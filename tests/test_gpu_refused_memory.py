"""A device allocation that is refused leaves a context as good as before: the same call, with
the memory granted, gives what it gives on a fresh context, in as many iterations (to rounding:
the context has given up the memory that it can do without)."""
import numpy as np
import pytest

from gpu_common import make_ctx, rand_complex, require_gpu, small_problem

pytestmark = pytest.mark.gpu
AGG, NVEC, M0 = ((4, 4), (2, 2)), (8, 8), 0.1
ENOMEM, ENOTCONVERGED = -2, -3


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


class Allocations:
    """Counts a context's device allocations and refuses the given one."""

    def __init__(self, monkeypatch):
        import torch
        self.count, self.refuse = 0, -1
        empty = torch.empty

        def counted(*a, **kw):
            i = self.count
            self.count += 1
            if i == self.refuse:
                raise RuntimeError("refused")
            return empty(*a, **kw)

        monkeypatch.setattr(torch, "empty", counted)

    def start(self, refuse=-1):
        self.count, self.refuse = 0, refuse


def prepared(pkg, prec, n):
    """A context whose last solve (one rhs fewer) stopped far from its tolerance."""
    theta, sv = small_problem(32, 16, 3.0, M0, AGG, NVEC)
    ctx = make_ctx(pkg, theta, M0, AGG, NVEC, sv, 0, mg_precision=prec, nu_pre=2, nu_post=0, fgmres_restart=50,
                   max_iters=2)
    b = rand_complex(np.random.default_rng(1), (n - 1, 1024))
    with pytest.raises(pkg.MgmlmcError) as err:
        ctx.solve(1, b)
    assert err.value.code == ENOTCONVERGED
    ctx.set_options(max_iters=2000)
    return ctx


@pytest.mark.parametrize("prec,n", [(64, 3), (64, 40), (32, 3), (16, 40)])
def test_solve(pkg, monkeypatch, prec, n):
    b = rand_complex(np.random.default_rng(2), (n, 512))
    alloc = Allocations(monkeypatch)
    with prepared(pkg, prec, n) as ctx:
        alloc.start()
        ref, iters = ctx.solve(2, b)
        count = alloc.count
    assert count > 0
    for i in range(count):
        with prepared(pkg, prec, n) as ctx:
            alloc.start(refuse=i)
            try:
                ctx.solve(2, b)
            except pkg.MgmlmcError as e:
                assert e.code == ENOMEM
            alloc.start()
            x, it = ctx.solve(2, b)
            assert it == iters and np.abs(x - ref).max() < 1e-10 * np.abs(ref).max(), i
