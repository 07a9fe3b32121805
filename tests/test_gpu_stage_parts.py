"""The fused stage kernel with a block's planes split over several CTAs along z, on grids of the sizes at
which a part starts three planes below the top of its block (its upper halo planes are wanted in its
second iteration): whole RK4 steps against the FP64 oracle, alone and in a batch."""
import numpy as np
import pytest

from tests.gpu_util import (block_order_fields, fill_from_function, oracle_forest, oracle_solver, rel_linf,
                            smooth_field, sphere_fn)

pytestmark = pytest.mark.gpu

# the step parity tolerances of the repository: FP64 rounding of a few steps, FP32 fields
TOL = {64: 1e-12, 32: 2e-5}
PHYS = dict(nu=1e-2, c0=3.0, C_eta=1e-2, C_gamma=0.5, cfl=0.5, eps=1e-3, dealias=0, mask_range_thr=1e-5)
SPHERE = (0.45, 0.5, 0.55, 0.2, 0.04)


@pytest.fixture(scope="module")
def A():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_05371_gb300 import acm
    acm.lib()
    return acm


def refined(k):
    """One root refined and k of its children refined again: 8 + 7 k leaves, with same-level, finer and
    coarser faces in every direction for 0 < k < 8."""
    kids = [(1, c & 1, (c >> 1) & 1, (c >> 2) & 1) for c in range(8)]
    fine = [(2, 2 * x + (c & 1), 2 * y + ((c >> 1) & 1), 2 * z + ((c >> 2) & 1))
            for _, x, y, z in kids[:k] for c in range(8)]
    return fine + kids[k:]


def roots(nx, ny, nz):
    return [(0, x, y, z) for z in range(nz) for y in range(ny) for x in range(nx)]


def pair(A, leaves, Bs, prec, nroot=(1, 1, 1), stream=None, seed=5):
    """A forest on the leaves with a body and smooth fields, and the oracle's solver in the same state."""
    grid = dict(nroot=nroot, root_len=1.0, Bs=Bs, g=4, Jmin=0, Jmax=2, precision=prec, max_blocks=96, fd_scheme=1,
                wavelet=40)
    f = A.Forest(grid, PHYS, **({"stream": stream} if stream is not None else {}))
    f.set_leaves(leaves)
    S = oracle_solver(oracle_forest(grid, leaves=leaves, max_blocks=96), PHYS, mask=sphere_fn(SPHERE))
    fill_from_function(S, lambda X, Y, Z: smooth_field(X, Y, Z, tuple(map(float, nroot)), seed))
    S.eval_mask()
    f.set_mask(A.ACM_MASK_SPHERE, SPHERE)
    f.write_fields(block_order_fields(S))
    return f, S


@pytest.mark.parametrize("prec,Bs,leaves,nroot", [
    (32, 17, refined(7), (1, 1, 1)), (64, 17, refined(3), (1, 1, 1)), (32, 33, roots(3, 2, 1), (3, 2, 1)),
    (32, 9, refined(7), (1, 1, 1)), (64, 9, refined(3), (1, 1, 1))],
    ids=["f32-17-57", "f64-17-29", "f32-33-6", "f32-9-57", "f64-9-29"])
def test_steps_match_oracle(A, prec, Bs, leaves, nroot):
    f, S = pair(A, leaves, Bs, prec, nroot)
    for _ in range(2):
        f.rk4_step(1e-3)
        S.rk4(1e-3)
    err = rel_linf(f.read_fields().astype(np.float64), block_order_fields(S))
    assert max(err) < TOL[prec], err


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_batch_of_52_blocks_matches_oracle(A, mode):
    """Instances of 29, 22 and 1 blocks of 17^3: their number of parts follows the sum, 52 (launched one by
    one, or as one graph; the persistent form keeps whole blocks)."""
    import torch
    layouts = [refined(3), refined(2), roots(1, 1, 1)]
    assert sum(len(l) for l in layouts) == 52
    made = [pair(A, l, 17, 32, stream=torch.cuda.Stream(), seed=7 + i) for i, l in enumerate(layouts)]
    A.rk4_steps_batch([f for f, _ in made], 2, 1e-3, graph=mode)
    for f, S in made:
        for _ in range(2):
            S.rk4(1e-3)
        err = rel_linf(f.read_fields().astype(np.float64), block_order_fields(S))
        assert max(err) < TOL[32], err


# plate: chord, span, thickness, stroke and pitch amplitudes, frequency, pivot, delta
PLATE = (0.3, 0.4, 0.15, 0.5, 0.6, 1.0, 0.45, 0.3, 0.55, 0.04)
SPONGE = dict(sponge=1, C_sp=0.05, u_inf=(0.4, -0.1, 0.2), p_inf=0.1, sponge_L=(1.0, 1.0, 1.0), sponge_width=0.2,
              sponge_delta=0.05)


def set_parts(f, parts):
    """The parts of a block along z in this forest's stage launches (an internal entry of the library)."""
    import ctypes as C
    fn = f.L.acm_internal_stage_parts
    fn.argtypes, fn.restype = [C.c_void_p, C.c_int], C.c_int
    return fn(f.h, parts)


@pytest.mark.parametrize("prec,Bs,body", [(32, 9, "sphere"), (32, 17, "sphere"), (32, 33, "sphere"),
                                          (64, 9, "sphere"), (64, 17, "sphere"), (32, 17, "plate"),
                                          (32, 33, "plate"), (64, 17, "plate")])
def test_every_part_count_is_bitwise_the_whole_block(A, prec, Bs, body):
    """Every number of parts the rule may choose, 2 .. Bs / 2, gives bitwise the steps of whole blocks, on a
    grid with same-level, finer and coarser faces in z, with a body and a sponge."""
    grid = dict(nroot=(1, 1, 1), root_len=1.0, Bs=Bs, g=4, Jmin=0, Jmax=2, precision=prec, max_blocks=96, fd_scheme=1,
                wavelet=40)
    leaves, phys = refined(3), dict(PHYS, **SPONGE)
    f = A.Forest(grid, phys)
    f.set_leaves(leaves)
    S = oracle_solver(oracle_forest(grid, leaves=leaves, max_blocks=96), phys)
    fill_from_function(S, lambda X, Y, Z: smooth_field(X, Y, Z, (1.0, 1.0, 1.0), 11))
    U = block_order_fields(S)
    f.set_mask(A.ACM_MASK_SPHERE if body == "sphere" else A.ACM_MASK_PLATE, SPHERE if body == "sphere" else PLATE)

    def steps(parts):
        assert set_parts(f, parts) == 0
        f.write_fields(U)
        f.set_time(0.1)
        for _ in range(2):
            f.rk4_step(1e-3)
        return f.read_fields().copy()

    whole = steps(1)
    assert np.isfinite(whole).all() and np.abs(whole - U).max() > 1e-4
    for parts in range(2, Bs // 2 + 1):
        assert np.array_equal(steps(parts), whole), parts
    assert set_parts(f, Bs // 2 + 1) == 1 and set_parts(f, -1) == 1      # refused: ACM_EINVAL
    assert np.array_equal(steps(0), whole)


@pytest.mark.parametrize("prec,Bs,body", [(32, 9, "plate"), (32, 17, "sphere"), (32, 17, "plate"), (32, 33, "plate"),
                                          (64, 17, "sphere"), (64, 17, "plate")])
@pytest.mark.parametrize("parts", [1, 4])
def test_copies_of_a_point_stay_bitwise_equal(A, prec, Bs, body, parts):
    """Points stored by several blocks of one level (fine wins relies on their copies being equal): on 2^3
    blocks of a periodic box all copies of a point hold the same bits after three steps, the pencils that
    the loading warp computes included."""
    M, N = Bs - 1, 2 * (Bs - 1)
    grid = dict(nroot=(2, 2, 2), root_len=0.5, Bs=Bs, g=4, Jmin=0, Jmax=1, precision=prec, max_blocks=16, fd_scheme=1,
                wavelet=40)
    f = A.Forest(grid, dict(PHYS, **SPONGE))
    f.set_leaves(roots(2, 2, 2))
    f.set_mask(A.ACM_MASK_SPHERE if body == "sphere" else A.ACM_MASK_PLATE, SPHERE if body == "sphere" else PLATE)
    f.set_time(0.1)
    x = np.arange(N) / N
    Z, Y, X = np.meshgrid(x, x, x, indexing="ij")
    lat = smooth_field(X, Y, Z, (1.0, 1.0, 1.0), 13)
    t = f.topology()
    corner = list(zip(t["gx"].tolist(), t["gy"].tolist(), t["gz"].tolist()))
    at = [np.ix_(range(4), *((g * M + np.arange(Bs)) % N for g in (gz, gy, gx))) for gx, gy, gz in corner]
    f.write_fields(np.stack([lat[i] for i in at]))
    assert set_parts(f, parts) == 0
    for _ in range(3):
        f.rk4_step(1e-3)
    U = f.read_fields()
    full = np.full(lat.shape, np.nan, U.dtype)
    for i, b in zip(at, U):
        full[i] = b
    assert np.isfinite(full).all()
    for i, b in zip(at, U):
        assert np.array_equal(full[i], b)
