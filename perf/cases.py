"""The work whose speed this repository is measured by, through its public Python entry points.

What a user's program does with this framework: it makes a block grid, hands a state over, takes
time steps on it (one call per step, many steps per call, or whole refine - evolve - coarsen
cycles), reads the state back, and for an inverse problem takes the gradient of a loss of the
final state.  Every case below is one such call sequence; a case is a dict of plain values:

``kind``
    ``step``   one ``rk4_step`` per pass on a fixed grid (the call per step of a coupled program);
    ``steps``  ``rk4_steps`` on a fixed grid, several steps per call;
    ``batch``  ``rk4_steps_batch`` over several independent instances of uneven size;
    ``cycle``  the paper's whole time step, ``step``: refine every block, one RK4 step, coarsen;
    ``vjp``    ``adjoint_vjp``: the gradient of a loss of the final state with respect to the
               initial state and the body's parameters, by the discrete adjoint.
``grid``
    ``uniform`` (level ``J0``), ``random`` (a random 2:1-graded layout of about ``target`` blocks,
    levels ``J0..Jmax``, drawn from ``layout``), ``sphere`` or ``plate`` (the initial grid of that
    body: blocks that the body's smoothed surface crosses are refined up to level ``Jmax - 1``).

Physics, geometries and sizes are those of ``paper_1912_05371_gb300/workloads.py`` and of
``bench.py``'s workloads: the periodic unit cube of Taylor-Green type, the penalised sphere in its
4 x 2 x 2 box with the sponge, the flapping plate in its 8^3 box, random graded grids, and the
batched instances with a pressure pulse and a vortex ring.  A pass begins from the caller's own
state (``write_fields`` from device memory) and ends with the state in the caller's hands
(``read_fields`` into device memory).  Gradients are returned in the forest's precision, as an
optimiser that holds its parameters in that precision keeps them.

:func:`exact` computes the same outputs in 64 bits with plain torch on dense lattices, one per
level, instead of blocks: it shares nothing with the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1912_05371_gb300 import acm as A

# ---- the cases -----------------------------------------------------------------------------------


def listed():
    return [
        # The smallest call: one RK4 step of the paper's non-adaptive case (64 blocks of 17^3, FP64)
        # per call with the CFL time step, as a program that couples to another code every step.
        dict(name="tg64-step-f64", kind="step", grid="uniform", Bs=17, precision=64, J0=2, Jmax=2, target=64,
             layout=0, nsteps=1),
        # The same small grid in FP32, 20 steps per call (graph replay): launches and latency.
        dict(name="tg64-steps20-f32", kind="steps", grid="uniform", Bs=17, precision=32, J0=2, Jmax=2, target=64,
             layout=0, nsteps=20),
        # A small adaptive run with the smallest blocks (9^3): host, launches and small kernels.
        dict(name="random71-cycle-bs9-f32", kind="cycle", grid="random", Bs=9, precision=32, J0=1, Jmax=3, target=71,
             layout=7, nsteps=1, wavelet=40),
        # Independent instances of uneven size (8 to 512 blocks) in one call, 10 steps from each
        # instance's own initial field: an ensemble.
        dict(name="batch12-steps10-f32", kind="batch", grid="random", Bs=17, precision=32, J0=1, Jmax=5, target=512,
             layout=3, instances=12, nsteps=10),
        # The largest grid: uniform level 5, 32,768 blocks of 17^3 (161 M points), FP32.
        dict(name="uniform32768-steps4-f32", kind="steps", grid="uniform", Bs=17, precision=32, J0=5, Jmax=5,
             target=32768, layout=0, nsteps=4),
        # The flagship: the penalised sphere at levels 2..5 with its sponge, one whole adaptive time
        # step (576 stored blocks, 4608 evolved), thresholds active, FP32.
        dict(name="sphere5-cycle-f32", kind="cycle", grid="sphere", Bs=17, precision=32, J0=2, Jmax=5, target=576,
             layout=0, nsteps=1, wavelet=40),
        # The same with the lifted wavelet the paper uses for its later results.
        dict(name="sphere5-cycle44-f32", kind="cycle", grid="sphere", Bs=17, precision=32, J0=2, Jmax=5, target=576,
             layout=0, nsteps=1, wavelet=44),
        # The sphere in FP64 (levels 2..4: 184 stored blocks, 1472 evolved), for verification runs.
        dict(name="sphere4-cycle-f64", kind="cycle", grid="sphere", Bs=17, precision=64, J0=2, Jmax=4, target=184,
             layout=0, nsteps=1, wavelet=40),
        # The paper's performance study: a random graded grid of about 1000 blocks, refined to about
        # 8000, evolved and coarsened back everywhere, FP32.
        dict(name="random1000-cycle-f32", kind="cycle", grid="random", Bs=17, precision=32, J0=3, Jmax=4, target=1009,
             layout=5, nsteps=1, wavelet=40),
        # The flapping plate with the 33^3 blocks of the full-scale case, at levels 2..5: the mask and
        # the solid velocity move at every stage.
        dict(name="plate5-cycle-bs33-f32", kind="cycle", grid="plate", Bs=33, precision=32, J0=2, Jmax=5, target=0,
             layout=0, nsteps=1, wavelet=40),
        # The gradient through 10 steps of the sphere on its frozen grid (levels 2..5, 576 blocks),
        # checkpoints every 5, FP32.
        dict(name="sphere5-vjp10-f32", kind="vjp", grid="sphere", Bs=17, precision=32, J0=2, Jmax=5, target=576,
             layout=0, nsteps=10, ckpt=5, snapshots=0),
        # The gradient of the moving plate (levels 2..5, 33^3 blocks), 4 steps, checkpoints every 2, FP32.
        dict(name="plate5-vjp4-bs33-f32", kind="vjp", grid="plate", Bs=33, precision=32, J0=2, Jmax=5, target=0,
             layout=0, nsteps=4, ckpt=2, snapshots=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any kind, block size, precision and layout that the listed
    ones stand for, sizes spread over their logarithm and capped below the largest listed case."""
    kind = rng.choice(["step", "steps", "steps", "batch", "cycle", "cycle", "cycle", "vjp"])
    c = dict(kind=kind, grid="random", precision=rng.choice([32, 32, 32, 64]), layout=rng.randrange(1 << 20))
    c["Bs"] = rng.choice([9, 17, 17, 33] if c["precision"] == 32 and kind != "batch" else [9, 17, 17])
    # about the points a pass may evolve: FP64 costs an order of magnitude more than FP32, a cycle
    # evolves 8 times its stored blocks, a gradient step costs several steps
    pts = 3.0e8 / (16 if c["precision"] == 64 else 1)
    if kind == "step":
        c["nsteps"] = 1
    elif kind == "steps":
        c["nsteps"] = _log_int(rng, 2, 30)
    elif kind == "batch":
        c["nsteps"], c["instances"] = rng.randint(2, 12), rng.randint(2, 20)
        pts /= 2 * c["instances"]
    elif kind == "cycle":
        c["nsteps"] = 1
        pts /= 16
    else:
        c["nsteps"] = rng.randint(1, 12)
        pts /= 32
    most = int(min(pts / c["nsteps"], 8.0e7) / c["Bs"] ** 3)
    if kind == "batch":
        c.update(J0=1, Jmax=5, target=max(16, min(512, most)))
        return c
    if kind in ("cycle", "vjp") and rng.random() < 0.5:
        # a body: the sphere (any precision) or the plate
        if c["Bs"] == 33 or rng.random() < 0.3:
            c.update(grid="plate", J0=2, Jmax=rng.choice([4, 5]) if c["Bs"] == 33 else rng.choice([4, 5, 6]), target=0)
        else:
            c.update(grid="sphere", J0=2, Jmax=rng.choice([3, 4]) if c["precision"] == 64 else rng.choice([3, 4, 5]),
                     target=0)
            if kind == "cycle":
                c["Bs"] = 17     # 9^3 blocks resolve this case too coarsely: its grid grows with every step
    else:
        lo = 8 if kind != "vjp" else 16
        target = _log_int(rng, lo, max(lo + 1, min(most, 12000)))
        J0 = 1 if target < 100 else (2 if target < 1500 else 3)
        if kind == "steps" and rng.random() < 0.25:
            J = 1 if target < 64 else (2 if target < 512 else 3)
            c.update(grid="uniform", J0=J, Jmax=J, target=8 ** J)
        else:
            c.update(J0=J0, Jmax=J0 + (2 if kind != "cycle" else 1), target=target)
    if kind == "cycle":
        c["wavelet"] = 44 if c["Bs"] != 33 and rng.random() < 0.2 else 40
    if kind == "vjp":
        c["ckpt"] = rng.randint(1, max(1, min(5, c["nsteps"])))
        c["snapshots"] = rng.randint(2, 4) if c["nsteps"] > 3 and rng.random() < 0.3 else 0
    return c


# ---- grids ---------------------------------------------------------------------------------------


def _grade(refined):
    """26-neighbour 2:1 grading: a refined box's neighbours exist, so their parents are refined."""
    for J in range(len(refined) - 1, 0, -1):
        r = refined[J]
        for ax in range(3):
            r = r | np.roll(r, 1, ax) | np.roll(r, -1, ax)
        nz, ny, nx = (s // 2 for s in r.shape)
        refined[J - 1] |= r.reshape(nz, 2, ny, 2, nx, 2).any(axis=(1, 3, 5))


def _leaf_masks(refined):
    out, exist = [], np.ones_like(refined[0])
    for J, r in enumerate(refined):
        out.append(exist & ~r)
        if J + 1 < len(refined):
            exist = (exist & r).repeat(2, 0).repeat(2, 1).repeat(2, 2)
    return out


def _block_order(leaves, nroot):
    """Leaves (J, x, y, z) sorted as the library lists them: root, then octal digits x + 2y + 4z
    from the coarsest level down (18 levels), then level."""
    a = np.asarray(leaves, dtype=np.int64).reshape(-1, 4)
    J, x, y, z = a.T
    code = ((x >> J) + nroot[0] * ((y >> J) + nroot[1] * (z >> J))) << 56
    for lev in range(1, int(J.max()) + 1):
        sh = np.maximum(J - lev, 0)
        d = ((x >> sh) & 1) | (((y >> sh) & 1) << 1) | (((z >> sh) & 1) << 2)
        code |= np.where(J >= lev, d, 0) << (3 * (18 - lev))
    return a[np.lexsort((J, code))].astype(np.int32)


def _random_layout(nroot, J0, Jmax, target, seed):
    rng = np.random.default_rng(seed)
    refined = [np.full((nroot[2] << J, nroot[1] << J, nroot[0] << J), J < J0) for J in range(Jmax + 1)]
    while True:
        leaf = _leaf_masks(refined)
        idx = [np.argwhere(m) for m in leaf]
        n, can = sum(len(i) for i in idx), sum(len(i) for i in idx[:Jmax])
        if n >= target or can == 0:
            break
        for p in np.sort(rng.choice(can, size=min(can, max(1, (target - n) // 60)), replace=False)):
            for J in range(Jmax):
                if p < len(idx[J]):
                    refined[J][tuple(idx[J][p])] = True
                    break
                p -= len(idx[J])
        _grade(refined)
    return _block_order([(J, x, y, z) for J in range(Jmax + 1) for z, y, x in idx[J].tolist()], nroot)


def _body_layout(cs, chi_of, level_h):
    """The initial grid of a body: a box at level J <= Jmax - 1 is kept if chi varies over it (by more
    than the mask-range threshold), together with its seven sisters; boxes at Jmax always merge."""
    nroot, M, J0, Jmax = cs["nroot"], cs["Bs"] - 1, cs["J0"], cs["Jmax"]
    refined = [np.full((nroot[2] << J, nroot[1] << J, nroot[0] << J), J < J0) for J in range(Jmax)]
    off = np.arange(M + 1)
    for J in range(J0 + 1, Jmax):
        # boxes whose parent is kept (or at the coarsest level) and may be crossed by the surface
        par = np.argwhere(_kept(refined, J - 1))
        kids = (2 * par[:, None, :] + np.array([[c >> 2, (c >> 1) & 1, c & 1] for c in range(8)])).reshape(-1, 3)
        h = level_h(J)
        for i0 in range(0, len(kids), 64):
            k = kids[i0:i0 + 64]
            N = [(nroot[a] << J) * M for a in range(3)]
            z, y, x = (((k[:, a][:, None] * M + off) % N[2 - a]) * h for a in range(3))
            chi = chi_of(torch.from_numpy(x)[:, None, None, :], torch.from_numpy(y)[:, None, :, None],
                         torch.from_numpy(z)[:, :, None, None]).reshape(len(k), -1)
            hit = ((chi.amax(1) - chi.amin(1)) > cs["phys"]["mask_range_thr"]).numpy()
            for z_, y_, x_ in k[hit] // 2:
                refined[J - 1][z_, y_, x_] = True
        _grade(refined)
    leaf = _leaf_masks(refined)
    return _block_order([(J, x, y, z) for J in range(Jmax) for z, y, x in np.argwhere(leaf[J]).tolist()], nroot)


def _kept(refined, J):
    """Boxes of level J that exist."""
    exist = np.ones_like(refined[0])
    for K in range(J):
        exist = (exist & refined[K]).repeat(2, 0).repeat(2, 1).repeat(2, 2)
    return exist


_SETUPS = {}


def _setup(case):
    """Grid and physics parameters, body and leaves of a case (kept per case: they are the problem's
    definition, drawn from the case alone)."""
    key = repr(sorted((k, v) for k, v in case.items() if k not in ("name", "nsteps", "ckpt", "snapshots")))
    if key not in _SETUPS:
        _SETUPS[key] = _make_setup(case)
    return _SETUPS[key]


def _make_setup(case):
    kind, body, Bs, J0, Jmax = case["kind"], case["grid"], case["Bs"], case["J0"], case["Jmax"]
    cs = dict(Bs=Bs, J0=J0, Jmax=Jmax, mask=None, ic="modes", amp=0.3, base=(0.0, 0.0, 0.0))
    phys = dict(nu=1e-2, c0=10.0, C_eta=1e-3, C_gamma=1.0, cfl=0.5, cfl_eta=1.0, cfl_nu=0.25, eps=1e-3, dealias=0,
                mask_range_thr=1e-5)
    if body == "sphere":
        cs.update(nroot=(2, 1, 1), root_len=2.0, base=(1.0, 0.0, 0.0), amp=0.02)
        delta = 1.5 * 2.0 / ((1 << Jmax) * (Bs - 1))
        cs["mask"] = (A.ACM_MASK_SPHERE, (1.0, 1.0, 1.0, 0.25, delta))
        phys.update(nu=1e-3, c0=20.0, C_gamma=0.0, C_sp=0.25 / (20.0 * 20.0), u_inf=(1.0, 0.0, 0.0), dealias=1,
                    sponge=1, sponge_L=(4.0, 2.0, 2.0), sponge_width=0.25, sponge_delta=delta)
    elif body == "plate":
        cs.update(nroot=(1, 1, 1), root_len=8.0, amp=0.02)
        delta = 1.5 * 8.0 / ((1 << Jmax) * (Bs - 1))
        cs["mask"] = (A.ACM_MASK_PLATE, (1.0, 3.0, 0.05, math.radians(60.0), math.radians(45.0), 1.0, 4.0, 4.0, 4.0,
                                         delta))
        phys.update(nu=1.0 / 2000.0, c0=30.0, C_eta=1e-4, C_gamma=0.0, dealias=1)
    else:
        cs.update(nroot=(1, 1, 1), root_len=1.0)
        if body == "uniform":
            cs["ic"] = "taylor_green"
        if kind == "batch":
            cs["ic"] = "pulse_ring"
            phys.update(nu=1e-3, C_gamma=0.0)
        if kind == "cycle":
            phys["coarsen_everywhere"] = 1       # the performance study's cycle: the grid comes back
    cs["phys"] = phys
    h = lambda J: cs["root_len"] / ((1 << J) * (Bs - 1))  # noqa: E731
    cs["h"] = h
    if body == "uniform":
        n = 1 << J0
        cs["leaves"] = _block_order([(J0, x, y, z) for z in range(n) for y in range(n) for x in range(n)], (1, 1, 1))
    elif body == "random" and kind == "batch":
        rng = np.random.default_rng(case["layout"])
        lo = math.log(min(16, case["target"]))
        sizes = [int(round(math.exp(rng.uniform(lo, math.log(case["target"]))))) for _ in range(case["instances"])]
        sizes[0] = case["target"]
        cs["instances"] = [_random_layout((1, 1, 1), 1 if s < 64 else 2, Jmax, s, int(rng.integers(1 << 30)))
                           for s in sizes]
        cs["leaves"] = np.concatenate(cs["instances"])
    elif body == "random":
        cs["leaves"] = _random_layout((1, 1, 1), J0, Jmax, case["target"], case["layout"])
    else:
        cs["leaves"] = _body_layout(cs, lambda x, y, z: _chi(cs, x, y, z, 0.0), h)
    return cs


# ---- inputs --------------------------------------------------------------------------------------


def _coords(cs, leaves, dev):
    """Coordinates (n, 1, 1, Bs) x, (n, 1, Bs, 1) y, (n, Bs, 1, 1) z of the leaves' points, FP64."""
    a = torch.as_tensor(np.asarray(leaves), device=dev, dtype=torch.int64)
    i, M = torch.arange(cs["Bs"], device=dev), cs["Bs"] - 1
    h = cs["root_len"] / (torch.pow(2.0, a[:, 0].double()) * M)
    x, y, z = ((((a[:, 1 + d][:, None] * M + i) % ((cs["nroot"][d] * M) << a[:, 0])[:, None]).double() * h[:, None])
               for d in range(3))
    return x[:, None, None, :], y[:, None, :, None], z[:, :, None, None]


def _field(cs, leaves, seed, dev, dtype):
    """The initial state (n, 4, Bs, Bs, Bs) in block order, a function of position: smooth periodic
    modes on top of the case's flow (Taylor-Green, uniform inflow, rest), or a pressure pulse and a
    vortex ring."""
    rng = np.random.default_rng([seed, 17])
    L = [n * cs["root_len"] for n in cs["nroot"]]
    kmax = 2
    out = torch.empty((len(leaves), 4) + (cs["Bs"],) * 3, dtype=dtype, device=dev)
    amps, ks, phs = rng.uniform(0.2, 1.0, (4, 3)), rng.integers(-kmax, kmax + 1, (4, 3, 3)), rng.uniform(0, 2 * math.pi,
                                                                                                         (4, 3))
    pulse, ring = rng.uniform(0.0, 1.0, 3), rng.uniform(0.0, 1.0, 3)
    width, pamp, R, gam = rng.uniform(0.05, 0.2), rng.uniform(0.01, 1.0), rng.uniform(0.1, 0.3), rng.uniform(0.5, 2.0)
    axis = rng.normal(size=3)
    axis /= np.linalg.norm(axis)
    for i0 in range(0, len(leaves), 2048):
        sl = slice(i0, i0 + 2048)
        x, y, z = _coords(cs, leaves[sl], dev)
        if cs["ic"] == "pulse_ring":
            near = lambda c, c0: (c - c0) - torch.round(c - c0)  # noqa: E731
            r2 = near(x, pulse[0]) ** 2 + near(y, pulse[1]) ** 2 + near(z, pulse[2]) ** 2
            d = [near(c, ring[a]) for a, c in enumerate((x, y, z))]
            zeta = d[0] * axis[0] + d[1] * axis[1] + d[2] * axis[2]
            rp = [d[a] - zeta * axis[a] for a in range(3)]
            rho = torch.sqrt(rp[0] ** 2 + rp[1] ** 2 + rp[2] ** 2)
            s2 = (0.25 * R) ** 2
            K = gam * torch.exp(-((rho - R) ** 2 + zeta ** 2) / s2) / (2 * math.pi * R)
            for a in range(3):
                out[sl, a] = K * (2 * zeta / s2 * rp[a] + (2 - 2 * rho * (rho - R) / s2) * axis[a])
            out[sl, 3] = pamp * torch.exp(-r2 / width ** 2)
            continue
        v = [torch.full_like(x + y + z, b) for b in (*cs["base"], 0.0)]
        amp = cs["amp"]
        if cs["phys"].get("sponge"):
            # the sponge holds the inflow: the disturbances fade out before they reach it
            for c, Lc in zip((x, y, z), L):
                s = ((torch.minimum(c, Lc - c) - 0.3) / 0.5).clamp(0.0, 1.0)
                amp = amp * s ** 3 * (10.0 - 15.0 * s + 6.0 * s * s)
        if cs["ic"] == "taylor_green":
            k = 2 * math.pi
            v[0] = v[0] + torch.sin(k * x) * torch.cos(k * y) * torch.cos(k * z)
            v[1] = v[1] - torch.cos(k * x) * torch.sin(k * y) * torch.cos(k * z)
        for f in range(4):
            for m in range(3):
                kx, ky, kz = (2 * math.pi * float(ks[f, m, a]) / L[a] for a in range(3))
                v[f] = v[f] + amp * amps[f, m] * torch.sin(kx * x + ky * y + kz * z + phs[f, m])
            out[sl, f] = v[f]
    return out


def _cotangent(cs, leaves, seed, dev):
    """dL/dU_N of a tracking loss (FP64): smooth, weighted by each block's cell volume."""
    lam = _field(dict(cs, ic="modes", base=(0.0, 0.0, 0.0), amp=1.0), leaves, seed + 1000003, dev, torch.float64)
    h = torch.tensor([cs["h"](int(J)) for J in leaves[:, 0]], dtype=torch.float64, device=dev)
    return lam * (h ** 3 / cs["h"](int(leaves[:, 0].max())) ** 3)[:, None, None, None, None]


def _fixed_dt(cs):
    h, p = cs["h"](int(cs["leaves"][:, 0].max())), cs["phys"]
    return min(0.25 * h / p["c0"], 0.1 * h * h / p["nu"], p["C_eta"] / 2 if cs["mask"] else 1.0)


def _point_keys(cs, leaves, dev):
    """One whole number per stored point, the same for every copy of a physical point."""
    a, top = torch.as_tensor(leaves, device=dev, dtype=torch.int64), int(leaves[:, 0].max())
    i, M = torch.arange(cs["Bs"], device=dev), cs["Bs"] - 1
    N = [(cs["nroot"][d] * M) << top for d in range(3)]
    x, y, z = (((a[:, 1 + d][:, None] * M + i) << (top - a[:, 0])[:, None]) % N[d] for d in range(3))
    return (((z[:, :, None, None] * N[1] + y[:, None, :, None]) * N[0]) + x[:, None, None, :]).reshape(-1)


# ---- the passes ----------------------------------------------------------------------------------


def _forest(cs, case, leaves, stream):
    room = len(leaves) * 8 if case["kind"] == "cycle" else len(leaves)
    g = dict(nroot=cs["nroot"], root_len=cs["root_len"], Bs=cs["Bs"], g=4, Jmin=min(cs["J0"], int(leaves[:, 0].min())),
             Jmax=cs["Jmax"] + (1 if case["kind"] == "cycle" and cs["mask"] is None else 0),
             precision=case["precision"], max_blocks=room + 64, fd_scheme=1, wavelet=case.get("wavelet", 40))
    f = A.Forest(g, cs["phys"], stream=stream)
    f.set_leaves(leaves)
    if cs["mask"]:
        f.set_mask(cs["mask"][0], cs["mask"][1])
    return f


def prepare(case, seed):
    dev = torch.device("cuda")
    cs, kind = _setup(case), case["kind"]
    dtype = torch.float64 if case["precision"] == 64 else torch.float32
    parts = cs["instances"] if kind == "batch" else [cs["leaves"]]
    st = dict(kind=kind, case=case, forests=[], U0=[], out=[])
    for i, leaves in enumerate(parts):
        stream = torch.cuda.Stream()
        u0 = _field(cs, leaves, seed * 64 + i, dev, dtype)
        torch.cuda.current_stream().synchronize()
        with torch.cuda.stream(stream):
            f = _forest(cs, case, leaves, stream)
            f.write_fields(u0)
        st["forests"].append(f)
        st["U0"].append(u0)
        st["out"].append(torch.empty_like(u0))
    if kind == "vjp":
        st["lam"] = _cotangent(cs, cs["leaves"], seed, dev)
        st["dt"] = _fixed_dt(cs)
        keys, st["point"] = torch.unique(_point_keys(cs, cs["leaves"], dev), return_inverse=True)
        st["n_points"] = len(keys)
    if kind == "cycle" and cs["mask"] and case["grid"] == "plate":
        st["moving"] = True
    if kind == "cycle":
        # the cycle has to bring the grid back, or the next pass could not begin from U0
        f = st["forests"][0]
        f.step(0.0)
        t = f.topology()
        back = np.stack([t["level"], t["gx"], t["gy"], t["gz"]], axis=1)
        if back.shape != cs["leaves"].shape or not np.array_equal(back, cs["leaves"]):
            raise RuntimeError("the cycle left another grid: %d blocks for %d" % (len(back), len(cs["leaves"])))
    torch.cuda.synchronize()
    return st


def run(state):
    case, kind, fs = state["case"], state["kind"], state["forests"]
    if kind == "vjp":
        f = fs[0]
        kw = dict(snapshots=case["snapshots"]) if case["snapshots"] else dict(ckpt_every=case["ckpt"])
        g, th = f.adjoint_vjp(case["nsteps"], state["dt"], state["lam"], **kw)
        # the gradients as an optimiser of the flow field keeps them: one value per physical point
        # (the blocks' copies of a point are one unknown), in its parameters' precision
        dtype = state["U0"][0].dtype
        out = torch.zeros((4, state["n_points"]), dtype=torch.float64, device=g.device)
        for c in range(4):
            out[c].index_add_(0, state["point"], g[:, c].reshape(-1))
        return [out.to(dtype), torch.as_tensor(th, dtype=dtype)]
    for f, u in zip(fs, state["U0"]):
        f.write_fields(u)
    if kind == "step":
        fs[0].rk4_step(0.0)
    elif kind == "steps":
        fs[0].rk4_steps(case["nsteps"], 0.0)
    elif kind == "batch":
        A.rk4_steps_batch(fs, case["nsteps"], 0.0)
    else:
        if state.get("moving"):
            fs[0].set_time(0.0)
        fs[0].step(0.0)
    return [f.read_fields(o) for f, o in zip(fs, state["out"])]


def work(case):
    """One pass: the caller's state in and out, and per RK4 stage the stage's state read once and the
    next one written once (a stage needs its neighbours' values of the stage before, over the whole
    grid), with chi where there is a body; operations of the four right-hand sides.  A gradient
    needs the forward steps and their adjoints: three times a step."""
    cs = _setup(case)
    es = case["precision"] // 8
    pts = len(cs["leaves"]) * cs["Bs"] ** 3
    evolved = pts * (8 if case["kind"] == "cycle" else 1)
    words = 32 + (4 if cs["mask"] else 0)
    mult = 3 if case["kind"] == "vjp" else 1
    return {"bytes": 8.0 * pts * es + mult * case["nsteps"] * evolved * words * es,
            "flops": mult * case["nsteps"] * evolved * 4 * 224.0}


# ---- the same in 64 bits on dense lattices ---------------------------------------------------------

_A3 = 0.0265199520614978
_D1 = (2.0 / 3.0 + 5.0 * _A3, -1.0 / 12.0 - 4.0 * _A3, _A3)


def _pose(q, t, alpha_m=None):
    """(R, omega) of the flapping plate at time t."""
    w = 2.0 * math.pi * q[5]
    am = torch.tensor(q[4], dtype=torch.float64) if alpha_m is None else alpha_m
    phi, dphi = q[3] * math.sin(w * t), q[3] * w * math.cos(w * t)
    al, dal = am * math.cos(w * t), -am * w * math.sin(w * t)
    cp, sp, ca, sa = math.cos(phi), math.sin(phi), torch.cos(al), torch.sin(al)
    R = [[cp * ca, -sp, cp * sa], [sp * ca, cp, sp * sa], [-sa, 0.0, ca]]
    return R, [-dal * sp, dal * cp, dphi]


def _root(v):
    """Square root with derivative 0 at 0."""
    return torch.where(v > 0, torch.sqrt(torch.where(v > 0, v, torch.ones_like(v))), torch.zeros_like(v))


def _chi(cs, x, y, z, t, theta=None):
    kind, q = cs["mask"]
    if kind == A.ACM_MASK_SPHERE:
        c = q[:4] if theta is None else theta
        d = _root((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) - c[3]
        return 0.5 * (1.0 - torch.tanh(d / q[4]))
    R, _ = _pose(q, t, theta)
    r = [x - q[6], y - q[7], z - q[8]]
    xb = [R[0][k] * r[0] + R[1][k] * r[1] + R[2][k] * r[2] for k in range(3)]
    xb[1] = xb[1] - 0.5 * q[1]
    s = [xb[k].abs() - 0.5 * w for k, w in enumerate((q[0], q[1], q[2]))]
    out2 = s[0].clamp(min=0) ** 2 + s[1].clamp(min=0) ** 2 + s[2].clamp(min=0) ** 2
    d = _root(out2) + torch.maximum(torch.maximum(s[0], s[1]), s[2]).clamp(max=0)
    return 0.5 * (1.0 - torch.tanh(d / q[9]))


def _us(cs, x, y, z, t, theta=None):
    q = cs["mask"][1]
    w = _pose(q, t, theta)[1]
    r = (x - q[6], y - q[7], z - q[8])
    return [w[1] * r[2] - w[2] * r[1], w[2] * r[0] - w[0] * r[2], w[0] * r[1] - w[1] * r[0]]


class _Dense:
    """The grid as one periodic lattice per level.  A state is {J: (4, Nz, Ny, Nx)} with the leaves' own
    values at the points of level-J leaves."""

    def __init__(self, cs, leaves, dev):
        self.cs, self.dev, self.M = cs, dev, cs["Bs"] - 1
        self.levels = sorted(set(int(J) for J in leaves[:, 0]))
        self.N = {J: tuple((cs["nroot"][a] << J) * self.M for a in (2, 1, 0)) for J in range(self.levels[0], self.levels[-1] + 1)}
        self.idx, self.rank, self.own = {}, {}, {}
        i = torch.arange(cs["Bs"], device=dev)
        for J in self.N:
            sel = np.nonzero(leaves[:, 0] == J)[0]
            b = torch.as_tensor(leaves[sel], device=dev, dtype=torch.int64)
            z, y, x = ((b[:, 3 - a][:, None] * self.M + i) % self.N[J][a] for a in range(3))
            lin = (z[:, :, None, None] * self.N[J][1] + y[:, None, :, None]) * self.N[J][2] + x[:, None, None, :]
            self.idx[J], self.rank[J] = lin.reshape(-1), torch.as_tensor(sel, device=dev)
            m = torch.zeros(math.prod(self.N[J]), dtype=torch.bool, device=dev)
            m[self.idx[J]] = True
            self.own[J] = m.reshape(self.N[J])
        # held[J]: points of the level-J lattice that some leaf of level >= J holds
        self.held = {}
        for J in reversed(list(self.N)):
            self.held[J] = self.own[J].clone()
            if J + 1 in self.N:
                self.held[J] |= self.held[J + 1][::2, ::2, ::2]

    def coords(self, J):
        h = self.cs["h"](J)
        z, y, x = (torch.arange(n, device=self.dev).double() * h for n in self.N[J])
        return x[None, None, :], y[None, :, None], z[:, None, None]

    def put(self, blocks):
        B3 = self.cs["Bs"] ** 3
        out = {}
        for J in self.N:
            o = torch.zeros((4, math.prod(self.N[J])), dtype=torch.float64, device=self.dev)
            v = blocks[self.rank[J]].double().permute(1, 0, 2, 3, 4).reshape(4, -1)
            o = o.index_copy(1, self.idx[J], v) if len(self.rank[J]) * B3 else o
            out[J] = o.reshape((4,) + self.N[J])
        return out

    def get(self, state, n):
        out = torch.empty((n, 4) + (self.cs["Bs"],) * 3, dtype=torch.float64, device=self.dev)
        for J in self.N:
            if len(self.rank[J]):
                v = state[J].reshape(4, -1)[:, self.idx[J]].reshape((4, -1) + (self.cs["Bs"],) * 3)
                out[self.rank[J]] = v.permute(1, 0, 2, 3, 4)
        return out

    def direct(self, own):
        """Values of the finest leaf holding each point (where held)."""
        out = {}
        for J in reversed(list(self.N)):
            d = own[J]
            if J + 1 in self.N:
                d = torch.where(self.held[J + 1][::2, ::2, ::2], out[J + 1][:, ::2, ::2, ::2], d)
            out[J] = d
        return out

    @staticmethod
    def predict(c):
        """The tensor DD-4 prediction of the next finer lattice."""
        for dim in (3, 2, 1):
            odd = (-torch.roll(c, 1, dim) + 9.0 * c + 9.0 * torch.roll(c, -1, dim) - torch.roll(c, -2, dim)) / 16.0
            c = torch.stack((c, odd), dim + 1).flatten(dim, dim + 1)
        return c

    def fill(self, own):
        """Every lattice point's value: the finest leaf holding it, else predicted from below."""
        d, out = self.direct(own), {}
        for J in self.N:
            out[J] = d[J] if J - 1 not in self.N else torch.where(self.held[J], d[J], self.predict(out[J - 1]))
        return out

    def sync(self, own):
        """Leaves' own values with finer leaves' values on shared points."""
        return self.direct(own)

    def rhs(self, F, J, t, theta=None):
        p, h, u = self.cs["phys"], self.cs["h"](J), F

        def d1(a, dim):
            return sum(c * (torch.roll(a, -k - 1, dim) - torch.roll(a, k + 1, dim)) for k, c in enumerate(_D1)) / h

        def d2(a, dim):
            return (16.0 * (torch.roll(a, 1, dim) + torch.roll(a, -1, dim)) - torch.roll(a, 2, dim) - torch.roll(a, -2, dim)
                    - 30.0 * a) / (12.0 * h * h)

        x, y, z = self.coords(J)
        chi = _chi(self.cs, x, y, z, t, theta) if self.cs["mask"] else None
        us = _us(self.cs, x, y, z, t, theta) if self.cs["mask"] and self.cs["mask"][0] == A.ACM_MASK_PLATE else (0, 0, 0)
        sp = None
        if p.get("sponge"):
            prof = [0.5 * (1.0 - torch.tanh((torch.minimum(c, L - c) - p["sponge_width"]) / p["sponge_delta"]))
                    for c, L in zip((x, y, z), p["sponge_L"])]
            sp = torch.maximum(torch.maximum(prof[0], prof[1]), prof[2])
        out = []
        div = 0
        for i in range(3):
            g = d1(u[i], 2)
            r = -u[0] * g
            div = div + (g if i == 0 else 0)
            g = d1(u[i], 1)
            r = r - u[1] * g
            div = div + (g if i == 1 else 0)
            g = d1(u[i], 0)
            r = r - u[2] * g
            div = div + (g if i == 2 else 0)
            r = r - d1(u[3], 2 - i) + p["nu"] * (d2(u[i], 0) + d2(u[i], 1) + d2(u[i], 2))
            if chi is not None:
                r = r - chi / p["C_eta"] * (u[i] - us[i])
            if sp is not None:
                r = r - sp / p["C_sp"] * (u[i] - p["u_inf"][i])
            out.append(r)
        r = -p["c0"] ** 2 * div - p["C_gamma"] * u[3]
        out.append(r if sp is None else r - sp / p["C_sp"] * u[3])
        return torch.stack(out)

    def dt(self, own):
        """The CFL time step of a state."""
        p = self.cs["phys"]
        um = max(float(torch.sqrt((own[J][:3] ** 2).sum(0))[self.own[J]].max()) for J in self.levels)
        h = self.cs["h"](self.levels[-1])
        dt = p["cfl"] * h / (um + math.sqrt(um * um + p["c0"] ** 2))
        if self.cs["mask"]:
            dt = min(dt, p["cfl_eta"] * p["C_eta"])
        return min(dt, p["cfl_nu"] * h * h / p["nu"])

    def K(self, own, t, theta=None):
        F = self.fill(own)
        return {J: self.rhs(F[J], J, t, theta) if J in self.levels else torch.zeros_like(F[J]) for J in self.N}

    def rk4(self, own, dt, t, theta=None):
        U = self.sync(own)
        acc, y = U, U
        for s, (ca, co, ts) in enumerate(((1, 0.5, 0.0), (2, 0.5, 0.5), (2, 1.0, 0.5), (1, 0.0, 1.0))):
            if theta is None:
                k = self.K(y, t + ts * dt)
            else:                            # differentiated: keep the stage's state only
                k = checkpoint(self.K, y, t + ts * dt, theta, use_reentrant=False)
            acc = {J: acc[J] + ca * dt / 6.0 * k[J] for J in self.N}
            if s < 3:
                y = {J: U[J] + co * dt * k[J] for J in self.N}
        return acc


def _lowpass44(c, dim):
    """The CDF 4/4 analysis low-pass at the even points along one axis."""
    w = (348.0, 144.0, -63.0, -16.0, 18.0, 0.0, -1.0)
    v = w[0] * c
    for k in range(1, 7):
        v = v + w[k] * (torch.roll(c, k, dim) + torch.roll(c, -k, dim))
    return v / 512.0


def exact(case, seed):
    cs, kind = _setup(case), case["kind"]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    dtype = torch.float64 if case["precision"] == 64 else torch.float32
    top = max(int(cs["leaves"][:, 0].max()), 0) + (1 if kind == "cycle" else 0)
    finest = math.prod((n << top) * (cs["Bs"] - 1) for n in cs["nroot"])
    grad = kind == "vjp"
    if finest * case["nsteps"] > (1.6e9 if not grad else 6.0e8) or finest > 3.0e8:
        return None
    uniform = len(set(cs["leaves"][:, 0].tolist())) == 1
    if case.get("wavelet") == 44 and not uniform:
        return None          # merged in several passes, each changing what its neighbours' parents read
    outs = []
    for i, leaves in enumerate(cs["instances"] if kind == "batch" else [cs["leaves"]]):
        u0 = _field(cs, leaves, seed * 64 + i, dev, dtype)
        D = _Dense(cs, leaves, dev)
        own = D.put(u0)
        if kind == "vjp":
            return _exact_gradients(cs, case, D, own, seed, dev)
        if kind == "cycle":
            outs.append(_exact_cycle(cs, case, D, own, leaves, dev))
            continue
        for _ in range(case["nsteps"]):
            own = D.rk4(own, D.dt(own), 0.0)
        outs.append(D.get(own, len(leaves)))
    return outs


def _exact_cycle(cs, case, D, own, leaves, dev):
    """Refine every block, one RK4 step, merge everything back."""
    kids = np.concatenate([np.stack([leaves[:, 0] + 1, 2 * leaves[:, 1] + (c & 1), 2 * leaves[:, 2] + ((c >> 1) & 1),
                                     2 * leaves[:, 3] + (c >> 2)], axis=1) for c in range(8)])
    E = _Dense(cs, kids, dev)
    F = D.fill(own)
    fine = {J: D.predict(F[J - 1]) for J in E.N}
    del F, own
    fine = E.rk4(fine, E.dt(fine), 0.0)
    if case.get("wavelet") == 44:
        J = E.levels[-1]
        V = E.fill(fine)[J]
        low = V
        for dim in (3, 2, 1):
            low = _lowpass44(low, dim)
        out = D.get({J - 1: V[:, ::2, ::2, ::2]}, len(leaves))
        inner = D.get({J - 1: low[:, ::2, ::2, ::2]}, len(leaves))
        out[:, :, 1:-1, 1:-1, 1:-1] = inner[:, :, 1:-1, 1:-1, 1:-1]
        return out
    d = E.sync(fine)
    return D.get({J: d[J + 1][:, ::2, ::2, ::2] for J in D.N}, len(leaves))


def _exact_gradients(cs, case, D, own, seed, dev):
    """dL/dU_0 per physical point and dL/d(centre, radius) of the sphere or dL/d(pitch amplitude) of the
    plate, by reverse-mode differentiation of the lattice steps."""
    dt, n, keys = _fixed_dt(cs), len(cs["leaves"]), list(D.N)
    sphere = cs["mask"] and cs["mask"][0] == A.ACM_MASK_SPHERE
    q = (cs["mask"][1][:4] if sphere else cs["mask"][1][4]) if cs["mask"] else 0.0
    theta = torch.tensor(q, dtype=torch.float64, device=dev, requires_grad=True)
    lam = _cotangent(cs, cs["leaves"], seed, dev)
    start = [own[J].requires_grad_() for J in keys]

    def one(t, th, *arrays):
        r = D.rk4(dict(zip(keys, arrays)), dt, t, th)
        return tuple(r[J] for J in keys)

    y = tuple(start)
    for k in range(case["nsteps"]):
        y = checkpoint(one, k * dt, theta, *y, use_reentrant=False)
    L = (D.get(dict(zip(keys, y)), n) * lam).sum()
    g = torch.autograd.grad(L, [theta, *start], allow_unused=True)
    out = torch.zeros(4, dtype=torch.float64, device=dev)
    if cs["mask"]:
        out[:4 if sphere else 1] = g[0]
    # every level's lattice points under the points' common numbers
    points = torch.unique(_point_keys(cs, cs["leaves"], dev))
    G = torch.zeros((4, len(points)), dtype=torch.float64, device=dev)
    top = keys[-1]
    for J, gj in zip(keys, g[1:]):
        if gj is None:
            continue
        z, y_, x = torch.nonzero(D.own[J], as_tuple=True)
        lin = ((z << (top - J)) * D.N[top][1] + (y_ << (top - J))) * D.N[top][2] + (x << (top - J))
        G.index_add_(1, torch.searchsorted(points, lin), gj[:, D.own[J]])
    return [G, out]
