"""The deflation eigensolver's dense pieces at the block sizes where their work splits:
rotations formed by every CTA (blocks of up to 128) or once for all, odd blocks, blocks of
fewer items than SMs, the Cholesky factor in a cluster (up to 144) or over the grid."""
import numpy as np
import pytest

from oracle import deflation as odefl
from oracle import hierarchy as ohier

from gpu_common import make_ctx, require_gpu, small_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


# the block holds max(2k, k + 16) vectors (at most n): 17, 24, 66, 128, 130, 144, 146, 180
@pytest.mark.parametrize("k", [1, 8, 33, 64, 65, 72, 73, 90])
def test_triplets(pkg, k):
    agg, nvec, m0 = ((2, 2), (2, 2)), (2, 4), 0.05
    theta, sv = small_problem(32, 24, 3.0, m0, agg, nvec)
    H = ohier.build_hierarchy(theta, m0, agg, nvec, sv, 0)
    defl = odefl.coarsest_deflation(H.D[-1], H.g5[-1], k)
    with make_ctx(pkg, theta, m0, agg, nvec, sv, 0, mg_precision=64) as ctx:
        ctx.compute_deflation(k, 1e-9, 2000)
        lam, sig, U, V, tau = ctx.get_deflation(k, 3)
    # residuals of 1e-9 |lambda| leave the eigenvalues of a Hermitian matrix within 1e-9 |lambda|
    assert np.abs(np.sort(sig) - np.sort(1.0 / defl.a)).max() < 1e-8 * sig.max()
    assert np.abs(V.conj() @ V.T - np.eye(k)).max() < 1e-10
    D = H.D[-1].toarray()
    assert np.abs((D @ V.T) - (U.T * sig)).max() < 1e-8 * sig.max()
