"""The fused stage kernel on the smallest and on graded grids: whole RK4 steps (stage states
point-major inside a step, no accumulator away from finer boundaries) against the FP64 oracle."""
import numpy as np
import pytest

from tests.gpu_util import (block_order_fields, fill_from_function, oracle_forest, oracle_solver, rel_linf,
                            smooth_field, sphere_fn, sponge_fn)

pytestmark = pytest.mark.gpu

# the step parity tolerances of the repository: FP64 rounding of a few steps, FP32 fields
TOL = {64: 1e-12, 32: 2e-5}
ONE = [(0, 0, 0, 0)]                                    # one block, its own neighbour on every side
PAIR = [(0, 0, 0, 0), (0, 1, 0, 0)]                     # a second root: same-level faces only
GRADED = [(0, 0, 0, 0)] + [(1, 2 + (c & 1), (c >> 1) & 1, (c >> 2) & 1) for c in range(8)]


@pytest.fixture(scope="module")
def A():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_05371_gb300 import acm
    acm.lib()
    return acm


def _grid(leaves, Bs, prec):
    return dict(nroot=(1, 1, 1) if leaves == ONE else (2, 1, 1), root_len=1.0, Bs=Bs, g=4, Jmin=0, Jmax=1,
                precision=prec, max_blocks=96, fd_scheme=1, wavelet=40)


def _phys(extras):
    p = dict(nu=1e-2, c0=3.0, C_eta=1e-2, C_gamma=0.5, cfl=0.5, eps=1e-3, dealias=0, mask_range_thr=1e-5)
    if extras:
        p.update(sponge=1, C_sp=0.05, u_inf=(0.4, -0.1, 0.2), p_inf=0.1, sponge_L=(2.0, 1.0, 1.0), sponge_width=0.2,
                 sponge_delta=0.05)
    return p


@pytest.mark.parametrize("extras", [False, True])
@pytest.mark.parametrize("leaves", [ONE, PAIR, GRADED], ids=["one", "pair", "graded"])
@pytest.mark.parametrize("prec,Bs", [(64, 9), (64, 17), (32, 9), (32, 17), (32, 33)])
def test_steps_match_oracle(A, prec, Bs, leaves, extras):
    if Bs == 33 and leaves == GRADED and not extras:
        pytest.skip("the 33^3 tests hold this layout")
    grid, phys = _grid(leaves, Bs, prec), _phys(extras)
    mask = (0.8, 0.5, 0.5, 0.2, 0.04) if extras else None
    f = A.Forest(grid, phys)
    f.set_leaves(leaves)
    S = oracle_solver(oracle_forest(grid, leaves=leaves, max_blocks=96), phys, mask=sphere_fn(mask) if mask else None,
                      sponge=sponge_fn(phys) if extras else None)
    L = tuple(float(n) for n in grid["nroot"])
    fill_from_function(S, lambda X, Y, Z: smooth_field(X, Y, Z, L, 5))
    S.eval_mask()
    if mask:
        f.set_mask(A.ACM_MASK_SPHERE, mask)
    f.write_fields(block_order_fields(S))
    for _ in range(2):
        f.rk4_step(1e-3)
        S.rk4(1e-3)
    err = rel_linf(f.read_fields().astype(np.float64), block_order_fields(S))
    assert max(err) < TOL[prec], err


@pytest.mark.parametrize("leaves", [ONE, PAIR, GRADED], ids=["one", "pair", "graded"])
@pytest.mark.parametrize("Bs", [9, 17])
def test_vjp_is_the_transpose_of_the_steps(A, Bs, leaves):
    """<w, dF v> = <dF^T w, v> for two FP64 steps F with mask and sponge: dF v by central differences
    of the steps, dF^T w by the vector-Jacobian product (kept stage states point-major; same-level,
    finer and coarser faces).  The perturbation 1e-4 leaves a difference error of 1e-8 of the second
    and third derivatives (order 1 here) and a rounding error of 1e-16 / 1e-4: 1e-6 of the norms
    bounds both."""
    f = A.Forest(_grid(leaves, Bs, 64), _phys(True))
    f.set_leaves(leaves)
    f.set_mask(A.ACM_MASK_SPHERE, (0.8, 0.5, 0.5, 0.2, 0.04))
    fo = oracle_forest(_grid(leaves, Bs, 64), leaves=leaves, max_blocks=96)
    S = oracle_solver(fo, _phys(True))
    L = (1.0, 1.0, 1.0) if leaves == ONE else (2.0, 1.0, 1.0)

    def field(seed):
        fill_from_function(S, lambda X, Y, Z: smooth_field(X, Y, Z, L, seed))
        return block_order_fields(S).copy()

    U, v, w, e = field(5), field(6), field(7), 1e-4
    out = []
    for s in (1.0, -1.0):
        f.write_fields(U + s * e * v)
        for _ in range(2):
            f.rk4_step(1e-3)
        out.append(f.read_fields().copy())
    f.write_fields(U)
    g, _ = f.adjoint_vjp(2, 1e-3, w)
    a, b = float((w * (out[0] - out[1])).sum() / (2 * e)), float((g * v).sum())
    assert abs(a - b) <= 1e-6 * np.linalg.norm(w) * np.linalg.norm(v), (a, b)
