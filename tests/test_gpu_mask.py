"""The mask kernel's whole-block and per-point shortcuts: blocks and points that lie beyond the
distance at which chi rounds to 0 or 1 take that value without the distance and tanh.  Against the
FP64 formula on every block of a graded grid, for thin and thick surfaces and bodies near the
periodic seam."""
import math

import numpy as np
import pytest

from oracle import acm as oacm
from oracle.plate import Plate
from tests.gpu_util import oracle_forest

pytestmark = pytest.mark.gpu

LEAVES = [(1, x, y, z) for x in range(4) for y in range(2) for z in range(2) if (x, y, z) != (2, 0, 0)]
LEAVES += [(2, 4 + (c & 1), (c >> 1) & 1, (c >> 2) & 1) for c in range(8)]


@pytest.fixture(scope="module")
def A():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_05371_gb300 import acm
    acm.lib()
    return acm


@pytest.mark.parametrize("body", ["sphere", "seam", "plate"])
@pytest.mark.parametrize("delta", [0.01, 0.004, 0.05])
@pytest.mark.parametrize("prec,Bs", [(64, 9), (64, 17), (32, 9), (32, 17), (32, 33)])
def test_mask_matches_the_formula(A, prec, Bs, delta, body):
    grid = dict(nroot=(2, 1, 1), root_len=1.0, Bs=Bs, g=4, Jmin=1, Jmax=2, precision=prec, max_blocks=64, fd_scheme=1)
    f = A.Forest(grid, dict(nu=1e-2, c0=3.0, C_eta=1e-2, C_gamma=0.5, cfl=0.5))
    f.set_leaves(LEAVES)
    if body == "plate":
        P = dict(chord=0.3, span=0.4, thickness=0.1, phi_m=math.radians(60.0), alpha_m=math.radians(45.0), freq=1.0,
                 root=(1.2, 0.4, 0.5), delta=delta)
        f.set_time(0.07)
        f.set_mask(A.ACM_MASK_PLATE, [P["chord"], P["span"], P["thickness"], P["phi_m"], P["alpha_m"], P["freq"],
                                      *P["root"], delta], t=0.07)
        plate = Plate(**P)
        chi_of = lambda X, Y, Z: plate.fields(X, Y, Z, 0.07)[0]
    else:
        p = (1.3, 0.4, 0.5, 0.35, delta) if body == "sphere" else (1.95, 0.97, 0.03, 0.2, delta)
        f.set_mask(A.ACM_MASK_SPHERE, p)
        chi_of = lambda X, Y, Z: oacm.sphere_mask(X, Y, Z, p[:3], p[3], delta)
    fo = oracle_forest(grid, leaves=LEAVES, max_blocks=64)
    ref = np.stack([chi_of(*oacm.block_coords(fo, l)) for l in fo.sorted_leaves()])
    got = f.read_mask().astype(np.float64).reshape(ref.shape)
    # eight roundings of the distance (coordinates up to 3), carried through tanh(d / delta) (slope 1/2)
    tol = 8 * (2.0 ** -53 if prec == 64 else 2.0 ** -24) * 3 / delta / 2
    assert np.abs(got - ref).max() <= tol
    # where the formula's tanh is exactly +-1 chi is 0 or 1 to its last bit
    assert np.abs(got - ref)[(ref == 0.0) | (ref == 1.0)].max(initial=0.0) <= 2.0 ** -53
