"""Gradients with respect to the state on grids of one level are repeatable to the last bit: the halo
targets of same-level faces are gathered by the block that holds the points, in a fixed order."""
import numpy as np
import pytest

from tests.gpu_util import smooth_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_05371_gb300 import acm
    acm.lib()
    return acm


@pytest.mark.parametrize("prec,Bs,J", [(32, 9, 2), (32, 17, 2), (32, 33, 1), (64, 9, 2), (64, 17, 2)])
def test_state_gradients_on_one_level_are_bitwise_repeatable(A, prec, Bs, J):
    M, n = Bs - 1, 2 ** J
    N = n * M
    f = A.Forest(dict(nroot=(1, 1, 1), root_len=1.0, Bs=Bs, g=4, Jmin=J, Jmax=J, precision=prec, max_blocks=n ** 3,
                      fd_scheme=1, wavelet=40),
                 dict(nu=1e-2, c0=3.0, C_eta=1e-2, C_gamma=0.5, cfl=0.5, eps=1e-3))
    f.init_uniform(J)
    f.set_mask(A.ACM_MASK_SPHERE, (0.45, 0.5, 0.55, 0.2, 0.04))
    x = np.arange(N) / N
    Z, Y, X = np.meshgrid(x, x, x, indexing="ij")
    t = f.topology()
    at = [np.ix_(range(4), *((g * M + np.arange(Bs)) % N for g in (gz, gy, gx)))
          for gx, gy, gz in zip(t["gx"].tolist(), t["gy"].tolist(), t["gz"].tolist())]
    u, w = (smooth_field(X, Y, Z, (1.0, 1.0, 1.0), s) for s in (3, 4))
    f.write_fields(np.stack([u[i] for i in at]))
    lam = np.stack([w[i] for i in at])
    first, _ = f.adjoint_vjp(3, 1e-3, lam)
    first = np.array(first, copy=True)
    assert np.isfinite(first).all() and np.abs(first).max() > 0
    for _ in range(6):
        again, _ = f.adjoint_vjp(3, 1e-3, lam)
        assert np.array_equal(np.asarray(again), first)
