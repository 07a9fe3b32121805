"""The max norms of the state on grids on both sides of the reduction's split over CTAs (acm_diagnostics):
exact, and a NaN anywhere in the state is reported."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_05371_gb300 import acm
    acm.lib()
    return acm


@pytest.mark.parametrize("nroot", [(1, 1, 1), (5, 5, 5), (6, 6, 6)], ids=["1", "125", "216"])
@pytest.mark.parametrize("prec,Bs", [(32, 9), (64, 9), (32, 17), (64, 17), (32, 33)])
def test_max_norms_are_exact(A, prec, Bs, nroot):
    import torch
    n = nroot[0] * nroot[1] * nroot[2]
    f = A.Forest(dict(nroot=nroot, root_len=1.0, Bs=Bs, g=4, Jmin=0, Jmax=0, precision=prec, max_blocks=n, fd_scheme=1),
                 dict(nu=1e-2, c0=3.0, cfl=0.5))
    f.init_uniform(0)
    g = torch.Generator(device="cuda").manual_seed(n + Bs)
    U = torch.randn((n, 4, Bs, Bs, Bs), generator=g, device="cuda", dtype=torch.float64 if prec == 64 else torch.float32)
    f.write_fields(U)
    d = f.diagnostics()
    want = U.abs().amax(dim=(0, 2, 3, 4)).double().cpu().numpy()
    assert np.array_equal(np.asarray(d["norms"]), want)
    # the speed is rounded three times before its root and once after it
    speed = float((U[:, :3].double() ** 2).sum(1).amax().sqrt())
    assert abs(d["u_max"] - speed) <= 4 * np.finfo(f.dtype).eps * speed
    for block, point in ((0, 0), (n - 1, Bs ** 3 - 1), (n // 2, Bs ** 3 // 2)):
        V = U.clone()
        V.view(n, 4, -1)[block, 2, point] = float("nan")
        f.write_fields(V)
        with pytest.raises(A.AcmError):
            f.diagnostics()
